"""Tasks of the forward ray stage with more boundary points than places.

On a grid of 4096 rows a task takes whole rows (32 of them).  A sector with a ring or two
images has four points a row, 128 a task; 64 have a place of their own.  Tasks
go to whichever warp is free, so a repeated call must still give the same bits.
"""
import numpy as np
import pytest

from paper_2510_02639_gb300 import inputs as I
from tests.test_gpu_parity import G, assert_parity, assert_status, run_gpu  # noqa: F401

pytestmark = pytest.mark.gpu

SPOT = dict(spot_x=0.3, spot_y=-0.2, spot_r=0.4, spot_c=0.7)


@pytest.mark.parametrize("n_r,n_theta,p,law", [
    (4096, 512, I.binary(rho=0.3, u0=0.1, s=1.0, q=0.5), {}),     # 94 of 128 tasks with 128 points
    (4096, 512, I.binary(rho=0.05, u0=0.01, s=1.0, q=1e-3), {}),  # a ring: 17 of 128
    (2048, 1024, I.binary(rho=0.3, u0=0.1, s=1.0, q=0.5), {}),    # 25 of 128 with 96
    (4096, 512, I.binary(rho=0.3, u0=0.1, s=1.0, q=0.5), SPOT),
    (4096, 256, I.triple(rho=0.1, u0=0.02), {}),
])
def test_more_points_than_places(G, oracle_mod, n_r, n_theta, p, law):
    params, t = [dict(p, **law)], np.linspace(0.0, 0.3, 6)
    g = I.grid(n_r=n_r, n_theta=n_theta, n_limb=200)
    A, st = run_gpu(G, params, t, g)
    Ao, so = oracle_mod.magnification(params, t.reshape(1, -1), g)
    assert_parity(A, Ao)
    assert_status(st, so)
    for _ in range(20):
        A2, st2 = run_gpu(G, params, t, g)
        assert np.array_equal(A, A2) and np.array_equal(st, st2), A2 - A
