"""Parameters that make a lens mass negative (q2 + q3 > 1, q < 0), as a sampler that steps out of its
prior asks for: the method has a value there, and the kernels' error bounds and
superblock tests, which are sums over the masses, have to hold.
"""
import numpy as np
import pytest

from paper_2510_02639_gb300 import inputs as I
from tests.test_gpu_adjoint import assert_dA, gpu_dA
from tests.test_gpu_parity import G, assert_parity, assert_status, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu

TRIPLE = I.triple(q2=0.0173472, q3=0.9874713, s2=0.7904591, s3=2.9867487, psi=0.1671148, rho=0.00258421, u0=0.125525,
                  alpha=6.007382, tE=1.0, u1=0.6, u2=0.2)
GRIDS = [(165, 392), (97, 1029), (200, 2100)]
BINARIES = {q: I.binary(q=q, s=s, rho=0.02, u0=0.3, alpha=0.7, tE=1.0) for q, s in ((-1e-3, 1.0), (-0.2, 1.3), (-0.5, 0.8))}


# (not q = -0.001 at 165 x 392: 165 rows put a row's centre on the edge of every
# image, and the oracle's own A moves by 1.5e-5 there when the margin moves by 2e-6)
@pytest.mark.parametrize("p,n_r,n_theta", [(TRIPLE, *g) for g in GRIDS] +
                         [(p, *g) for q, p in BINARIES.items() for g in GRIDS if (q, g[0]) != (-1e-3, 165)])
def test_forward(G, oracle_mod, p, n_r, n_theta):
    t = np.linspace(-0.95, 0.95, 12)
    g = I.grid(n_r=n_r, n_theta=n_theta, n_limb=333)
    A, st = run_gpu(G, [p], t, g)
    Ao, so = oracle_mod.magnification([p], t[None], g)
    assert_parity(A, Ao)
    assert_status(st, so)


@pytest.mark.parametrize("q,s", [(-1e-3, 1.0), (-0.2, 1.3)])
def test_gradient(G, oracle_mod, q, s):
    p, t = I.binary(q=q, s=s, rho=0.02, u0=0.3, alpha=0.7, tE=1.0), np.linspace(-0.95, 0.95, 7)
    g = I.grid(n_r=97, n_theta=1029, n_limb=333)
    A, dA, _, _ = gpu_dA(G, [p], t[None], g)
    Ao, dAo, _ = oracle_mod.magnification_fwd([p], t[None], g)
    assert np.all(np.abs(A / Ao - 1) <= 1e-5)
    assert_dA(dA, dAo, str(q), Ao)
