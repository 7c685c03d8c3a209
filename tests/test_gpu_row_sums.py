"""The gradient's per-lane row sums against exact ones.

Each of the 15 sums is of products of two floats (one of three: rounded once),
which FP64 holds exactly, so n additions are off by at most n 2^-53 of the sum
of the terms' moduli (2 n 2^-53 for the one of three).
"""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.test_gpu_parity import G  # noqa: F401

pytestmark = pytest.mark.gpu

SOURCE = """
#include "icrs_rays_der.cuh"
__global__ void rows(const float* v, const float* r, const int* row, int n, double* out) {
  __shared__ double sums[icrs::DSUM * 32];
  for (int k = 0; k < icrs::DSUM; ++k) sums[k * 32 + threadIdx.x] = 0.0;
  for (int i = 0; i < n; ++i) {
    const size_t o = (size_t)i * 32 + threadIdx.x;
    icrs::RowTerms x;
    for (int k = 0; k < 12; ++k) x.v[k] = v[o * 12 + k];
    icrs::row_add(sums, threadIdx.x, row[o], r[o], x);
  }
  for (int k = 0; k < icrs::DSUM; ++k) out[k * 32 + threadIdx.x] = sums[k * 32 + ((threadIdx.x + k) & 31)];
}
extern "C" int row_sums(const float* v, const float* r, const int* row, int n, double* out) {
  rows<<<1, 32>>>(v, r, row, n, out);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.mark.parametrize("n", [1, 9, 128])
def test_row_sums(G, tmp_path, n):
    import torch
    from paper_2510_02639_gb300 import build as B
    (tmp_path / "rows.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-o", str(tmp_path / "librows.so"),
                    str(tmp_path / "rows.cu"), "-lcudart"], check=True)
    rng = np.random.default_rng(41)
    v = (rng.standard_normal((n, 32, 12)) * 10.0 ** rng.uniform(-4, 4, (n, 32, 12))).astype(np.float32)
    r = rng.uniform(0.2, 2.0, (n, 32)).astype(np.float32)
    row = rng.integers(0, 4096, (n, 32)).astype(np.int32)
    dev = [torch.tensor(x, device="cuda") for x in (v, r, row)]
    out = torch.empty((15, 32), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(x.data_ptr()) for x in dev]
    assert ctypes.CDLL(str(tmp_path / "librows.so")).row_sums(*p, n, ctypes.c_void_p(out.data_ptr())) == 0
    from fractions import Fraction as F
    got = out.cpu().numpy()
    for lane in range(0, 32, 5):
        for k in range(15):
            a = {0: 0, 1: 0, 2: 0, 3: 1, 4: 1}.get(k, k - 3)
            terms = []
            for i in range(n):
                x, rr, h = F(float(v[i, lane, a])), F(float(r[i, lane])), F(int(row[i, lane])) + F(1, 2)
                terms.append(x if k == 0 else x * h if k == 1 else x * rr * h if k == 4 else x * rr)
            bound = (2 if k == 4 else 1) * n * F(1, 2 ** 53) * sum(abs(t) for t in terms)
            assert abs(F(float(got[k, lane])) - sum(terms)) <= bound, (n, k, lane)
