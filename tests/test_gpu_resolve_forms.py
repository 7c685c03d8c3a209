"""The three forms of the FP64 root re-solve, with the number of queued limb
points known: in these lenses (a wide binary, a triple of comparable masses) no
FP32 image set is trusted, so the counter of FP64 solves is N_limb at every epoch.

Up to 16 points take a warp each; up to 16 x (32 / N_deg), 96 binary and 48
triple, share warps; more take a thread each.  An odd number leaves warps partly filled.
"""
import numpy as np
import pytest

from paper_2510_02639_gb300 import inputs as I
from tests.test_gpu_parity import G, assert_parity, assert_status  # noqa: F401

pytestmark = pytest.mark.gpu

LENSES = {
    2: (I.binary(q=0.5, s=300.0, rho=1e-2, t0=-(200.0 - 1.0 / 450.0), tE=1.0, u0=0.2, alpha=0.0),
        np.linspace(-0.5, 0.5, 5)),
    3: (I.triple(q2=0.3, q3=0.25, s2=3.0, s3=2.5, rho=1e-3, tE=1.0, u0=1e-4, alpha=0.7), np.linspace(-4e-3, 4e-3, 5)),
}


@pytest.mark.parametrize("n_lens,n_limb", [(2, 16), (2, 17), (2, 95), (2, 96), (2, 97), (2, 500),
                                           (3, 16), (3, 17), (3, 47), (3, 48), (3, 49), (3, 300)])
def test_every_limb_point_resolved(G, oracle_mod, n_lens, n_limb):
    import torch
    p, t = LENSES[n_lens]
    g = I.grid(n_limb=n_limb)
    A, st, _, cnt, _ = G.magnification_diag(G.params_to_device([p]), torch.tensor(t[None], device="cuda"),
                                            G.grid_from_dict(g, n_lens))
    Ao, so = oracle_mod.magnification([p], t[None], g)
    assert np.all(cnt[0, :, 1].cpu().numpy() == n_limb), cnt[0, :, 1]
    assert_parity(A.cpu().numpy(), Ao)
    assert_status(st.cpu().numpy(), so)
    assert not np.any(st.cpu().numpy() & 1)


@pytest.mark.parametrize("law", [dict(u1=0.0, a1=0.6, a2=0.3, a3=-0.2, a4=0.1), dict(u2=0.2, a3=0.2),
                                 dict(u1=0.0, a1=0.4, spot_x=0.3, spot_y=-0.2, spot_r=0.4, spot_c=0.7)])
def test_power_series_on_the_triple_lens(G, oracle_mod, law):
    from tests.test_gpu_parity import run_gpu
    params, t = I.triple_curve()
    params, t = [dict(params[0], **law)], t[:, 700:1300:120]
    g = I.grid(n_r=97, n_theta=1029, n_limb=200)
    A, st = run_gpu(G, params, t, g)
    Ao, so = oracle_mod.magnification(params, t, g)
    assert_parity(A, Ao)
    assert_status(st, so)
