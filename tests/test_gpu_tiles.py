"""Sizes at which the tiled kernels change shape: remainders of the ray stage's
row blocks and column chunks, its superblocks, the FP64 root re-solve's three
forms, and the row tiles of the surrogate's network, against the FP64 oracle.

Tolerances.  Forward: 1e-5, the parity tolerance, on grids of at least 2,048
rays a sector.  A crossing's weight f(delta) has a slope of at most 40 (just
above delta_c = 0.02) and delta an FP32 error of a few 1e-6, so a single limb
ray is off by about 1e-4 of itself, and where a grid has only a few rays that is
an error of A: 1e-3 there, of max(A, 1).  Derivative: the bound of
test_gpu_adjoint.  Network: the bounds of test_gpu_surrogate.
"""
import numpy as np
import pytest

from paper_2510_02639_gb300 import inputs as I
from tests.test_gpu_adjoint import assert_dA, gpu_dA
from tests.test_gpu_parity import G, assert_parity, assert_status, run_gpu  # noqa: F401
from tests.test_gpu_surrogate import rand_features, theta_for_test

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_r,n_theta,n_limb", [
    (1, 8, 16), (3, 15, 40), (31, 16, 100),           # one row block, chunks of 16 columns or the whole row
    (32, 64, 100), (33, 255, 100), (65, 999, 100),    # remainders of both
    (97, 1025, 200), (40, 2049, 200),                 # superblocks of 32 and 64 columns, ragged ends
    (1023, 530, 100), (4062, 64, 1024),               # many row blocks; the most tasks a sector has, largest N_limb
])
def test_forward_grids(G, oracle_mod, n_r, n_theta, n_limb):
    params, t = I.caustic_crossing_binary(n_epochs=500)
    t = t[:, 30:470:80]
    g = I.grid(n_r=n_r, n_theta=n_theta, n_limb=n_limb)
    A, st = run_gpu(G, params, t, g)
    Ao, so = oracle_mod.magnification(params, t, g)
    if n_r * n_theta >= 2048:
        assert_parity(A, Ao, what=str((n_r, n_theta)))
    else:
        assert np.all(np.abs(A - Ao) <= 1e-3 * np.maximum(Ao, 1.0)), (A, Ao)
    assert_status(st, so, what=str((n_r, n_theta)))


@pytest.mark.parametrize("law", ["quadratic", "powers", "spot", "uniform", "triple", "triple spot"])
def test_forward_laws_on_ragged_superblocks(G, oracle_mod, law):
    """Every instantiation of the sweep on a grid with superblocks and
    remainders (97 x 1029)."""
    n_limb = 200
    if law.startswith("triple"):
        params, t = I.triple_curve()
        t = t[:, 700:1300:120]
        if law == "triple spot":
            n_limb = 580  # the largest that fits
            params = [dict(params[0], spot_x=0.3, spot_y=-0.2, spot_r=0.4, spot_c=0.7)]
    else:
        params, t = I.caustic_crossing_binary(n_epochs=500)
        t = t[:, 40:470:100]
        if law == "quadratic":
            params = [dict(params[0], u2=0.2)]
        elif law == "powers":
            params = [dict(params[0], a1=0.3, a2=0.2, a3=-0.1, a4=0.05)]
        elif law == "spot":
            params = [dict(params[0], spot_x=0.3, spot_y=-0.2, spot_r=0.4, spot_c=0.7)]
    g = I.grid(n_r=97, n_theta=1029, n_limb=n_limb, uniform=1 if law == "uniform" else 0)
    A, st = run_gpu(G, params, t, g)
    Ao, so = oracle_mod.magnification(params, t, g)
    assert_parity(A, Ao, what=law)
    assert_status(st, so, what=law)


@pytest.mark.parametrize("n_limb", [16, 100, 500, 1024])
def test_root_resolve_queues(G, oracle_mod, n_limb):
    """q = 1e-5: the FP32 images of many limb points are not trusted, from a few
    points a epoch (a warp for each) to most of them (a thread for each)."""
    p = I.binary(q=1e-5, s=1.0, rho=1e-3, u1=0.5, t0=0.0, tE=1.0, u0=1e-4, alpha=0.7)
    t = np.linspace(-4e-3, 4e-3, 9)
    g = I.grid(n_limb=n_limb)
    A, st = run_gpu(G, [p], t, g)
    Ao, so = oracle_mod.magnification([p], t.reshape(1, -1), g)
    assert_parity(A, Ao, what=str(n_limb))


@pytest.mark.parametrize("n_r,n_theta,n_limb", [
    (33, 255, 100), (63, 1025, 200),                  # remainders, without and with superblocks
    (257, 521, 200), (64, 2049, 500),                 # more row blocks than warps; superblocks of 64
    (16, 8192, 900),                                  # no room for the table of column angles
])
def test_derivative_grids(G, oracle_mod, n_r, n_theta, n_limb):
    params, t = I.caustic_crossing_binary(n_epochs=500)
    t = t[:, 30:470:80]
    g = I.grid(n_r=n_r, n_theta=n_theta, n_limb=n_limb)
    A, dA, st, _ = gpu_dA(G, params, t, g)
    Ao, dAo, so = oracle_mod.magnification_fwd(params, t, g)
    assert np.all(np.abs(A / Ao - 1) <= 1e-5)
    assert_dA(dA, dAo, str((n_r, n_theta)), Ao)


@pytest.mark.parametrize("n", [1, 127, 128, 129, 3 * 152 * 128 + 1, 2 * 3 * 152 * 128 + 77])
def test_infer_row_tiles(G, n):
    import torch
    from oracle import mlp as M
    f = rand_features(n, 11)
    th = theta_for_test(12)
    tt = torch.tensor(th, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    out = G.mlp_infer(G.mlp_pack(tt), tt, torch.tensor(f, device="cuda"), err=err).cpu().numpy()
    assert int(err.item()) == 0 and out.shape[0] == n and np.all(np.isfinite(out))
    rows = np.arange(n) if n <= 1000 else np.unique(np.r_[np.arange(200), np.arange(n - 300, n), np.arange(0, n, 97)])
    Yr, bound = M.inference_bound(th, f[rows][:, :7].astype(np.float64))
    ratio = np.abs(out[rows] - Yr) / (1.5 * bound + 1e-30)
    assert np.all(ratio <= 1.0), (np.argwhere(ratio > 1.0)[:5], ratio.max())


def test_infer_non_finite_features(G):
    """A query with a NaN or an infinite feature comes back NaN, the others of
    its tile untouched."""
    import torch
    f = rand_features(300, 16)
    tt = torch.tensor(theta_for_test(17), device="cuda")
    pack = G.mlp_pack(tt)
    ref = G.mlp_infer(pack, tt, torch.tensor(f, device="cuda")).cpu().numpy()
    f[5, 0], f[130, 6], f[299, 3] = np.nan, np.inf, -np.inf
    out = G.mlp_infer(pack, tt, torch.tensor(f, device="cuda")).cpu().numpy()
    bad = np.zeros(300, dtype=bool)
    bad[[5, 130, 299]] = True
    assert np.all(np.isnan(out[bad])) and np.array_equal(out[~bad], ref[~bad])


@pytest.mark.parametrize("n", [127, 128, 129, 152 * 128 + 1])
def test_train_row_tiles(G, n):
    """Gradient and loss, and the weights repacked by the same step."""
    import torch
    from oracle import mlp as M
    f = rand_features(n, 13)
    y = np.random.default_rng(14).standard_normal(n).astype(np.float32)
    th = theta_for_test(15)
    tt = torch.tensor(th, device="cuda")
    m, v = torch.zeros_like(tt), torch.zeros_like(tt)
    pack = G.mlp_pack(tt)
    grad = torch.zeros_like(tt)
    loss = torch.zeros(1, dtype=torch.float32, device="cuda")
    err = torch.zeros(1, dtype=torch.int32, device="cuda")
    G.mlp_train_step(tt, m, v, pack, 1, 1e-3, torch.tensor(f, device="cuda"), torch.tensor(y, device="cuda"),
                     grad=grad, loss=loss, err=err)
    assert int(err.item()) == 0
    X = f[:, :7].astype(np.float64)
    gr, scale, Lr = M.gradient_term_scale(th, X, y.astype(np.float64))
    Yr, bY = M.inference_bound(th, X)
    _, dY = M.nll(Yr, y.astype(np.float64))
    assert abs(float(loss.item()) - Lr) <= 1.5 * float(np.sum(np.abs(dY) * bY)) + 1e-6 * abs(Lr)
    ratio = np.abs(grad.cpu().numpy() - gr) / (4.0 * M.U_BF16 * scale + 1e-12)
    assert np.all(ratio <= 1.0), (np.argwhere(ratio > 1.0)[:5], ratio.max())
    assert torch.equal(pack, G.mlp_pack(tt))


def test_train_single_row(G):
    """One row.  (The bound above, relative to the sum of |terms|, needs many
    rows: a single row's term can itself be a sum that cancels, and the network
    with every rounding mirrored in FP64 is then off by as much.)  The mean
    gradient of 128 copies of the row is the same number: its terms are the
    row's divided by 128, exactly, so only the FP32 sum of 128 equal terms
    rounds, by 128 2^-24 of it at most."""
    import torch
    f, y = rand_features(1, 13), np.random.default_rng(14).standard_normal(1).astype(np.float32)
    tt = torch.tensor(theta_for_test(15), device="cuda")
    pack = G.mlp_pack(tt)

    def grad(n):
        g = torch.zeros_like(tt)
        G.mlp_train_step(tt, None, None, pack, 1, 0.0, torch.tensor(np.repeat(f, n, 0), device="cuda"),
                         torch.tensor(np.repeat(y, n), device="cuda"), grad=g)
        return g.cpu().numpy().astype(np.float64)
    one, many = grad(1), grad(128)
    assert np.count_nonzero(one) > one.size // 2
    assert np.all(np.abs(one - many) <= 128 * 2.0 ** -24 * np.abs(one) + 1e-30)
