"""The network's SiLU and its derivative against CUDA's own division, and what
infinite pre-activations give.

Bounds.  q + r (z - q d) and r + r (1 - d r) leave an error below 2^-44 of the
quotient before the last rounding, so each is within one ulp of the rounded division
and differs from it only where the quotient is within 2^-20 ulp of a midpoint,
on average in fewer than 2^-19 of all values.  In the derivative s (1 + z (1 -
s)) an ulp of s, 2^-23 s, moves the result by at most (1 + |z|) times that, and
its three operations round once more each.
"""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.test_gpu_parity import G  # noqa: F401
from tests.test_gpu_surrogate import rand_features

pytestmark = pytest.mark.gpu

SOURCE = """
#include "icrs_silu.cuh"
__global__ void both(const float* z, float* s, float* p, float* sd, float* pd) {
  const size_t i = 16 * ((size_t)blockIdx.x * blockDim.x + threadIdx.x);
  float x[16], y[16], v[16];
  for (int j = 0; j < 16; ++j) { x[j] = y[j] = z[i + j]; v[j] = 1.0f; }
  icrs::silu_n<16>(y);
  icrs::silu_prime_n<16>(x, v);
  for (int j = 0; j < 16; ++j) {
    const float d = 1.0f + expf(-x[j]), g = 1.0f / d;
    s[i + j] = y[j]; p[i + j] = v[j];
    sd[i + j] = x[j] / d; pd[i + j] = g * (1.0f + x[j] * (1.0f - g));
  }
}
extern "C" int silu_both(const float* z, float* s, float* p, float* sd, float* pd, int blocks) {
  both<<<blocks, 256>>>(z, s, p, sd, pd);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
"""


@pytest.fixture(scope="module")
def silu_both(tmp_path_factory):
    import torch
    from paper_2510_02639_gb300 import build as B
    d = tmp_path_factory.mktemp("silu")
    (d / "silu.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-shared", "-o", str(d / "libsilu.so"), str(d / "silu.cu"), "-lcudart"],
                   check=True)
    lib = ctypes.CDLL(str(d / "libsilu.so"))

    def run(z):
        assert z.size % 4096 == 0
        zt = torch.tensor(z, device="cuda")
        out = [torch.empty_like(zt) for _ in range(4)]
        torch.cuda.synchronize()
        assert lib.silu_both(*[ctypes.c_void_p(x.data_ptr()) for x in (zt, *out)], z.size // 4096) == 0
        return [x.cpu().numpy() for x in out]
    return run


def keys(x):
    """Integers in the order of the floats, neighbouring floats one apart (+0 and -0 the same)."""
    b = x.view(np.int32).astype(np.int64)
    return np.where(b < 0, -(b & 0x7fffffff), b)


def test_against_the_division(silu_both):
    rng = np.random.default_rng(31)
    n = 1 << 23
    lin = np.sort(rng.uniform(-85.0, 85.0, n)).astype(np.float32)
    log = np.sort((10.0 ** rng.uniform(-40.0, 1.9, n) * rng.choice([-1.0, 1.0], n)).astype(np.float32))
    for z in (lin, log):
        s, p, sd, pd = silu_both(z)
        du = np.abs(keys(s) - keys(sd))
        assert du.max() <= 1, (z[du.argmax()], du.max())
        normal = np.abs(sd) >= 2.0 ** -120
        share = 2.0 ** -19 * normal.sum()
        assert np.count_nonzero(du[normal]) <= share + 5.0 * np.sqrt(share)
        z64, sg = z.astype(np.float64), 1.0 / (1.0 + np.exp(-z.astype(np.float64)))
        bound = 2.0 ** -23 * sg * (1.0 + np.abs(z64)) * 4.0 + 2.0 ** -148
        assert np.all(np.abs(p.astype(np.float64) - pd) <= bound)
        far = np.abs(z) > 81.0  # (a thread with such a value divides)
        assert np.array_equal(s[far], sd[far])


def test_other_values(silu_both):
    """Infinities, NaN and the largest finite values, alone among ordinary ones:
    what the division gives."""
    special = np.array([np.inf, -np.inf, np.nan, 3.4e38, -3.4e38, 88.7, -88.7, -104.0, 80.0, -80.0, 79.99, -79.99,
                        0.0, 1e-45, -1e-45, -87.5], dtype=np.float32)
    z = np.tile(np.linspace(-3.0, 3.0, 16, dtype=np.float32), 256).reshape(256, 16)
    z[np.arange(256), np.arange(256) % 16] = special[np.arange(256) // 16]
    s, p, sd, pd = silu_both(z.reshape(-1))
    assert np.array_equal(np.isnan(s), np.isnan(sd)) and np.array_equal(np.isnan(p), np.isnan(pd))
    ok = ~np.isnan(sd)
    assert np.all(np.isinf(s[ok]) == np.isinf(sd[ok])) and np.abs(keys(s[ok]) - keys(sd[ok])).max() <= 1


def test_infer_infinite_pre_activation(G):
    """A hidden unit at -inf is NaN (-inf / inf), and so is the query's answer."""
    import torch
    th = np.zeros(G.MLP_NPARAM, dtype=np.float32)
    th[7 * 128:] = np.random.default_rng(32).standard_normal(th.size - 7 * 128).astype(np.float32) * 0.05
    th[0] = -3.0e38          # W0[0][0]
    th[7 * 128] = -3.0e38    # b0[0]
    f = rand_features(200, 33)
    f[:, 0] = 0.0
    f[::7, 0] = 1.0
    tt = torch.tensor(th, device="cuda")
    out = G.mlp_infer(G.mlp_pack(tt), tt, torch.tensor(f, device="cuda")).cpu().numpy()
    hit = np.arange(200) % 7 == 0
    assert np.all(np.isnan(out[hit])) and np.all(np.isfinite(out[~hit]))
