"""The network kernels' bounded waits.

A library is built in which every first wait runs out at once (its limit is 0
tries).  Each kernel then reports an error, waits (with the ordinary limit) for
the copies and contractions that it has in flight, gives its tensor memory back
and returns; the ordinary library's results are the same before and after.
"""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.test_gpu_parity import G  # noqa: F401
from tests.test_gpu_surrogate import rand_features, theta_for_test

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def impatient(tmp_path_factory):
    from paper_2510_02639_gb300 import build as B
    out = str(tmp_path_factory.mktemp("icrs") / "libicrs_impatient.so")
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-DICRS_MLP_WAIT_TRIES=0", "-shared", "-o", out,
                    f"{B.CSRC}/icrs_surrogate.cu", "-lcudart"], check=True)
    return ctypes.CDLL(out)


def test_waits_that_run_out(G, impatient):
    import torch
    n = 3 * 152 * 128 + 5
    f = torch.tensor(rand_features(n, 21), device="cuda")
    y = torch.tensor(np.random.default_rng(22).standard_normal(n).astype(np.float32), device="cuda")
    th = torch.tensor(theta_for_test(23), device="cuda")
    pack = G.mlp_pack(th)

    def both():
        g, err = torch.zeros_like(th), torch.zeros(1, dtype=torch.int32, device="cuda")
        out = G.mlp_infer(pack, th, f, err=err)
        G.mlp_train_step(th, None, None, pack, 1, 0.0, f, y, grad=g, err=err)
        torch.cuda.synchronize()
        assert int(err.item()) == 0
        return out, g
    out, g = both()
    vp, st = ctypes.c_void_p, torch.cuda.current_stream().cuda_stream
    ws = G.mlp_workspace(n)
    for _ in range(3):
        err = torch.zeros(2, dtype=torch.int32, device="cuda")
        o2 = torch.empty_like(out)
        assert impatient.icrs_mlp_infer(vp(pack.data_ptr()), vp(th.data_ptr()), vp(f.data_ptr()), n, vp(o2.data_ptr()),
                                        vp(err.data_ptr()), vp(st)) == 0
        assert impatient.icrs_mlp_train_step(vp(th.data_ptr()), None, None, vp(pack.data_ptr()), 1, ctypes.c_float(0.0),
                                             vp(f.data_ptr()), vp(y.data_ptr()), n, None, None, vp(ws.data_ptr()),
                                             ctypes.c_size_t(ws.numel()), vp(err.data_ptr() + 4), vp(st)) == 0
        torch.cuda.synchronize()
        assert err.tolist() == [1, 1]
    again = both()
    assert torch.equal(again[0], out) and torch.equal(again[1], g)
