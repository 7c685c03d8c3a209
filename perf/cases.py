"""Workloads on which this library's speed is measured.

Each case is one call (or one short sequence of calls) through the public entry
points of ``paper_2510_02639_gb300`` with the sizes of the package's own
workloads (``inputs``): light curves of one binary or triple lens, batches of
parameter sets, chi^2 and marginal-likelihood gradients, the preselected light
curves and the surrogate network.

A case is a dict of plain values.  ``kind`` names the call; the other keys are
its sizes and options.  ``exact`` evaluates the same quantities in 64 bits with
numpy, independently of the library, where that takes seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2510_02639_gb300 import icrs, surrogate
from paper_2510_02639_gb300 import inputs as I

LAWS = ("linear", "quadratic", "power4", "spot")


def listed():
    return [
        # a handful of epochs of one light curve, the default grid: what an
        # interactive user or a single likelihood term asks for; latency
        dict(name="curve_24", kind="curve", sets=1, epochs=24, n_r=64, n_theta=256, n_limb=500, law="linear"),
        # the package's caustic-crossing light curve, default grid
        dict(name="curve_500", kind="curve", sets=1, epochs=500, n_r=64, n_theta=256, n_limb=500, law="linear"),
        # the 64-set binary batch at the default grid: model grids, samplers
        # that run many chains at once
        dict(name="batch", kind="batch", sets=64, epochs=500, n_r=64, n_theta=256, n_limb=500, law="linear"),
        # the same batch at the grid whose error is below 1e-4 everywhere: the
        # package's headline workload, and the data of the surrogate
        dict(name="batch_fine", kind="batch", sets=64, epochs=400, n_r=1024, n_theta=2048, n_limb=500, law="linear"),
        # sets whose sources follow different brightness laws (linear,
        # quadratic, power series, a spot), odd sizes throughout
        dict(name="laws_ragged", kind="batch", sets=13, epochs=77, n_r=251, n_theta=999, n_limb=401, law="mixed"),
        # the triple-lens light curve
        dict(name="triple", kind="triple", sets=1, epochs=2000, n_r=64, n_theta=256, n_limb=500, law="linear"),
        # chi^2 and its gradient over a cloud of sets around one binary, as a
        # sampler or an optimiser steps through it, default grid
        dict(name="chi2", kind="chi2", sets=32, epochs=500, n_r=64, n_theta=256, n_limb=500, law="linear"),
        # the same at the fine grid
        dict(name="chi2_fine", kind="chi2", sets=8, epochs=250, n_r=1024, n_theta=2048, n_limb=500, law="linear"),
        # the flux-marginalised likelihood and its gradient, odd sizes
        dict(name="nll_ragged", kind="nll", sets=7, epochs=333, n_r=200, n_theta=777, n_limb=500, law="quadratic"),
        # light curves that run ray shooting near caustics only: features,
        # preselection, indexed magnification
        dict(name="preselected", kind="preselected", sets=50, epochs=1000, n_r=512, n_theta=1024, n_limb=500,
             law="linear"),
        # inference of the surrogate network on a million queries
        dict(name="mlp_infer", kind="mlp_infer", n=1 << 20),
        # one training step of it on a mini-batch (gather, forward, backward, Adam)
        dict(name="mlp_train", kind="mlp_train", n=8192),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# Rays of the largest listed case per sector; drawn cases stay below it.  An
# epoch's work before the rays (root finding) weighs about as much as EPOCH
# rays, a derivative about 4 times its magnification.
EPOCH = 400_000
MAX_COST = 64 * 400 * (1024 * 2048 + EPOCH)
WEIGHT = {"curve": 1, "batch": 1, "triple": 8, "chi2": 8, "nll": 8, "preselected": 1}


def draw(rng):
    kind = rng.choice(["curve", "curve", "batch", "batch", "batch", "triple", "chi2", "chi2", "nll", "preselected",
                       "mlp_infer", "mlp_train"])
    if kind == "mlp_infer":
        return dict(kind=kind, n=_log_int(rng, 1, 1 << 21))
    if kind == "mlp_train":
        return dict(kind=kind, n=_log_int(rng, 100, 1 << 16))
    n_r = _log_int(rng, 32, 1024)
    n_theta = min(2048, max(96, int(n_r * rng.uniform(1.5, 4.5))))
    sets = 1 if kind in ("curve", "triple") else _log_int(rng, 2, 64)
    law = "linear"
    if kind in ("curve", "batch", "chi2", "nll"):
        law = rng.choice(["linear", "linear", "quadratic", "power4", "spot", "mixed"])
        if sets == 1 and law == "mixed":
            law = "quadratic"
    most = MAX_COST / (WEIGHT[kind] * (n_r * n_theta + EPOCH) * sets * (4 if law in ("spot", "mixed") else 1))
    epochs = min(_log_int(rng, 8, 2000), max(4, int(0.5 * most)))
    return dict(kind=kind, sets=sets, epochs=epochs, n_r=n_r, n_theta=n_theta, n_limb=rng.choice([500, 500, 256, 333]),
                law=law)


# ---------------------------------------------------------------- inputs
def _params(case, seed):
    """Parameter dicts and times [S][E] (host) of a magnification case."""
    rng = np.random.default_rng([seed, 77])
    S, E, kind = case["sets"], case["epochs"], case["kind"]
    if kind == "curve":
        # the caustic-crossing binary, each parameter within a percent
        p0, _ = I.caustic_crossing_binary(2)
        params = [dict(p0[0]) for _ in range(S)]
        for p in params:
            for k in ("u0", "alpha", "rho", "u1", "s", "q"):
                p[k] *= 1.0 + 0.01 * rng.standard_normal()
        t = np.sort(rng.uniform(-0.5, 0.5, (S, E)), axis=1)
    elif kind == "triple":
        p0, _ = I.triple_curve(2)
        params = [dict(p0[0]) for _ in range(S)]
        for p in params:
            for k in ("u0", "alpha", "rho", "u1", "q2", "q3", "s2", "s3"):
                p[k] *= 1.0 + 0.01 * rng.standard_normal()
        t = np.sort(rng.uniform(-3.0, 3.0, (S, E)), axis=1)
    elif kind in ("chi2", "nll"):
        params, t, _, _ = I.adjoint_batch(S, E, seed=1000 + seed)
        t = np.sort(t + rng.uniform(-0.5, 0.5, t.shape) * 100.0 / E, axis=1)
    else:
        params, t = I.binary_batch(S, E, seed=1000 + seed)
    for i, p in enumerate(params):
        p.update(I.SOURCE_LAWS[LAWS[i % 4] if case["law"] == "mixed" else case["law"]])
    return params, t


def _grid(case):
    return I.grid(n_r=case["n_r"], n_theta=case["n_theta"], n_limb=case["n_limb"])


def _features(n, seed, rows):
    """Rows of network inputs in the ranges of the batch distribution."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    u = torch.rand((n, rows), generator=g, device="cuda")
    f = torch.empty((n, 8), device="cuda")
    f[:, 0:2] = 4.0 * u[:, 0:2] - 2.0
    f[:, 2] = u[:, 2] - 0.52
    f[:, 3] = 2.0 * u[:, 3] - 1.0
    f[:, 4] = 2.0 * u[:, 4] - 1.0
    f[:, 5] = 2.0 * u[:, 5] - 1.0
    f[:, 6] = torch.log10(1.0 - 0.9 * u[:, 6])
    f[:, 7] = 20.0 * u[:, 7] - 10.0
    return f, u


def prepare(case, seed):
    kind = case["kind"]
    if kind == "mlp_infer":
        theta = torch.tensor(surrogate.init_theta(seed), device="cuda")
        feat, _ = _features(case["n"], seed, 8)
        return dict(kind=kind, theta=theta, pack=icrs.mlp_pack(theta), feat=feat,
                    err=torch.zeros(1, dtype=torch.int32, device="cuda"))
    if kind == "mlp_train":
        n = case["n"]
        theta = torch.tensor(surrogate.init_theta(seed), device="cuda")
        feat, u = _features(4 * n, seed, 9)
        target = torch.sin(3.0 * feat[:, 0]) * feat[:, 3] + feat[:, 6] + 0.2 * (u[:, 8] - 0.5)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        idx = torch.randperm(4 * n, generator=g, device="cuda")[:n].to(torch.int32)
        m = 1e-3 * torch.randn(theta.shape, generator=g, device="cuda")
        v = 1e-5 * torch.rand(theta.shape, generator=g, device="cuda") + 1e-6
        return dict(kind=kind, theta=theta, m=m, v=v, pack=icrs.mlp_pack(theta), feat=feat, target=target, idx=idx,
                    fb=torch.empty((n, 8), device="cuda"), yb=torch.empty(n, device="cuda"),
                    ws=icrs.mlp_workspace(n), loss=torch.zeros(1, device="cuda"), step=100,
                    err=torch.zeros(1, dtype=torch.int32, device="cuda"))
    params, t = _params(case, seed)
    st = dict(kind=kind, pd=icrs.params_to_device(params), t=torch.tensor(t, device="cuda"),
              grid=icrs.grid_from_dict(_grid(case), 3 if kind == "triple" else 2), sets=case["sets"])
    if kind in ("chi2", "nll"):
        rng = np.random.default_rng([seed, 78])
        # data about a light curve of the cloud's centre: a single-lens curve
        # is near enough for the size of the residuals
        u = np.hypot(t / 25.0, 0.02)
        y = (u * u + 2.0) / (u * np.sqrt(u * u + 4.0)) * (1.0 + 0.01 * rng.standard_normal(t.shape))
        st["y"] = torch.tensor(y, device="cuda")
        st["sigma"] = torch.tensor(0.01 * y * rng.uniform(0.5, 2.0, t.shape), device="cuda")
    if kind == "nll":
        st["prior"] = torch.tensor(np.tile([1.0, 1.0, 100.0, 100.0], (case["sets"], 1)), device="cuda")
        nb = int(icrs.lib.icrs_marginal_nll_workspace_bytes(case["sets"], case["epochs"]))
        st["ws"] = torch.empty(nb, dtype=torch.uint8, device="cuda")
    return st


def run(st):
    kind = st["kind"]
    if kind in ("curve", "batch", "triple"):
        A, status = icrs.magnification(st["pd"], st["t"], st["grid"])
        return dict(A=A, status=status)
    if kind == "chi2":
        chi2, grad, A, status = icrs.chi2_grad(st["pd"], st["t"], st["grid"], st["y"], st["sigma"])
        return dict(chi2=chi2, grad=grad, A=A, status=status)
    if kind == "nll":
        nll, grad, fluxes, A, status = icrs.marginal_nll_grad(st["pd"], st["t"], st["grid"], st["y"], st["sigma"],
                                                              st["prior"], workspace=st["ws"])
        return dict(nll=nll, grad=grad, fluxes=fluxes, A=A, status=status)
    if kind == "preselected":
        feat, A_ps, flags = icrs.surrogate_features(st["pd"], st["t"], st["grid"])
        A, k = surrogate.preselected_magnification(st["pd"], st["t"], st["grid"], caustic_min=-6.0, b_max=100.0,
                                                   feat=feat, A_ps=A_ps, st=flags)
        return dict(A=A, routed=k, feat=feat, A_ps=A_ps, flags=flags)
    if kind == "mlp_infer":
        return dict(out=icrs.mlp_infer(st["pack"], st["theta"], st["feat"], err=st["err"]), err=st["err"])
    if kind == "mlp_train":
        icrs.surrogate_batch(st["feat"], st["target"], st["idx"], st["fb"], st["yb"])
        st["step"] += 1
        icrs.mlp_train_step(st["theta"], st["m"], st["v"], st["pack"], st["step"], 1e-3, st["fb"], st["yb"],
                            workspace=st["ws"], loss=st["loss"], err=st["err"])
        return dict(theta=st["theta"], m=st["m"], v=st["v"], pack=st["pack"].view(torch.bfloat16), loss=st["loss"],
                    err=st["err"])
    raise ValueError(kind)


def work(case):
    """The path's own arithmetic and traffic: an image sector's rays (30
    operations each for a binary lens, 40 for a triple, and their gradients
    about 100 more; about 3 sectors an epoch, 5 for a triple), the limb points'
    polynomial roots (about 3 sweeps of Ehrlich-Aberth), the network's layers."""
    kind = case["kind"]
    if kind in ("mlp_infer", "mlp_train"):
        n, layers = case["n"], 2 * (7 * 128 + 3 * 128 * 128 + 2 * 128)
        if kind == "mlp_infer":
            return dict(bytes=n * 40 + 4 * icrs.MLP_NPARAM, flops=float(n * layers))
        return dict(bytes=n * 40 + 24 * icrs.MLP_NPARAM + icrs.MLP_PACK_BYTES, flops=float(3 * n * layers))
    S, E = case["sets"], case["epochs"]
    n = S * E
    triple, der = kind == "triple", kind in ("chi2", "nll")
    rays = (5 if triple else 3) * case["n_r"] * case["n_theta"]
    flops = rays * ((40 if triple else 30) + (100 if der else 0)) + case["n_limb"] * (24000 if triple else 3500)
    nbytes = S * 192 + n * 20 + (n * 16 + S * 72 if der else 0)
    if kind == "preselected":
        # every epoch's 33 point-source solves; about an eighth of them go on
        return dict(bytes=nbytes + n * 48, flops=float(n * 33 * 3500 + 0.125 * n * flops))
    return dict(bytes=nbytes, flops=float(n * flops))


# ---------------------------------------------------------------- 64 bits
def _lens(p):
    q, s = p["q"], p["s"]
    return np.array([1.0 / (1.0 + q), q / (1.0 + q)]), np.array([-q * s / (1.0 + q), s / (1.0 + q)], dtype=complex)


def _centre(p, t):
    tau = (t - p["t0"]) / p["tE"]
    return (tau + 1j * p["u0"]) * np.exp(1j * p["alpha"])


def _images(p, w, tol=1e-3):
    """Roots of the binary lens polynomial at the source positions w [n]
    (companion matrices, then Newton on the lens equation) and which of them
    are images."""
    eps, a = _lens(p)
    ll = int(np.argmin(eps))
    c = a - a[ll]                       # frame of the lightest lens
    wl = w - a[ll]
    D = np.poly(c)[::-1]                # low -> high
    F = eps[0] * np.array([-c[1], 1.0]) + eps[1] * np.array([-c[0], 1.0])
    n = w.size
    G = np.zeros((2, n, 3), complex)
    for k in range(2):
        G[k] = np.conj(wl - c[k])[:, None] * D[None, :]
        G[k, :, :2] += F[None, :]

    def mul(x, y):
        out = np.zeros((n, x.shape[1] + y.shape[1] - 1), complex)
        for i in range(x.shape[1]):
            out[:, i:i + y.shape[1]] += x[:, i:i + 1] * y
        return out

    PG = mul(G[0], G[1])
    DS = mul(np.broadcast_to(D, (n, 3)), eps[0] * G[1] + eps[1] * G[0])
    b = np.zeros((n, 6), complex)
    b[:, 1:] = PG
    b[:, :5] -= wl[:, None] * PG + DS
    M = np.zeros((n, 5, 5), complex)
    M[:, 0, :] = -b[:, 4::-1] / b[:, 5:]
    for i in range(4):
        M[:, i + 1, i] = 1.0
    z = np.linalg.eigvals(M)
    for _ in range(3):                  # Newton on the polynomial
        v, d = b[:, 5:] + 0 * z, 0 * z
        for k in range(4, -1, -1):
            d = d * z + v
            v = v * z + b[:, k:k + 1]
        z = z - np.where(np.abs(d) > 0, v / np.where(d == 0, 1, d), 0)
    f = z - sum(eps[i] / np.conj(z - c[i]) for i in range(2)) - wl[:, None]
    ok = np.abs(f) <= tol
    for _ in range(3):                  # and, for the images, on the lens equation
        f = z - sum(eps[i] / np.conj(z - c[i]) for i in range(2)) - wl[:, None]
        g = sum(eps[i] / (z - c[i]) ** 2 for i in range(2))
        dz = (np.conj(g) * np.conj(f) - f) / (1.0 - np.abs(g) ** 2)
        z = np.where(ok & (np.abs(dz) < 1e-3), z + dz, z)
    return z + a[ll], ok


def _point_source(p, w):
    z, ok = _images(p, w)
    eps, a = _lens(p)
    g = sum(eps[i] / (z - a[i]) ** 2 for i in range(2))
    return np.sum(np.where(ok, 1.0 / np.abs(1.0 - np.abs(g) ** 2), 0.0), axis=1)


def _sectors(z, inside, g):
    """Image-centred sectors (r_lo, r_hi, th_lo, width, full) of the image-limb
    points z; inside(z): does a lens-plane point map into the source."""
    BT, BR, mar, tp = g["n_bins_theta"], g["n_bins_r"], g["margin"], 2 * math.pi
    ht = tp / BT
    r, th = np.abs(z), np.angle(z)
    tb = np.clip(np.floor((th + math.pi) / ht).astype(int), 0, BT - 1)
    occ = np.zeros(BT, bool)
    occ[tb] = True
    full = bool(occ.all())
    run = np.full(BT, -1)
    start = []
    if full:
        run[:], start = 0, [0]
    else:
        t0 = int(np.argmin(occ))
        for k in range(1, BT + 1):
            t = (t0 + k) % BT
            if occ[t]:
                if occ[t - 1]:
                    run[t] = run[t - 1]
                else:
                    run[t] = len(start)
                    start.append(t)
    origin = bool(inside(np.array([0j]))[0])
    boxes = []
    for T in range(len(start)):
        sel = run[tb] == T
        rs, bs, ts = r[sel], tb[sel], th[sel]
        lo, h = rs.min(), (rs.max() - rs.min()) / BR
        rb = np.clip(np.floor((rs - lo) / h).astype(int), 0, BR - 1) if h > 0 else np.zeros(rs.size, int)
        hist = np.zeros((BR, BT), bool)
        hist[rb, bs] = True
        ro = hist.any(axis=1)
        fill = np.zeros(BR, bool)
        b = 1
        while b < BR:
            if ro[b] or not ro[b - 1]:
                b += 1
                continue
            e = b
            while e < BR and not ro[e]:
                e += 1
            if e >= BR:
                break
            both = np.nonzero(hist[:b].any(axis=0) & hist[e:].any(axis=0))[0]
            rg = lo + h * 0.5 * (b + e)
            if both.size and inside(rg * np.exp(1j * (-math.pi + (both + 0.5) * ht))).any():
                fill[b:e] = True
            b = e
        ro |= fill
        cell = np.cumsum(ro & ~np.concatenate([[False], ro[:-1]])) - 1
        ts = np.where(bs < start[T], ts + tp, ts)
        for c in range(int(cell[-1]) + 1):
            m = cell[rb] == c
            if not m.any():
                continue
            r0, r1, a0, a1 = rs[m].min(), rs[m].max(), ts[m].min(), ts[m].max()
            rl = 0.0 if origin and c == 0 else max(0.0, r0 - mar * (r1 - r0))
            wd = (a1 - a0) * (1 + 2 * mar)
            if full or wd >= tp:
                boxes.append([rl, r1 + mar * (r1 - r0), -math.pi, tp, True])
            else:
                x = (a0 - mar * (a1 - a0) + math.pi) % tp - math.pi
                boxes.append([rl, r1 + mar * (r1 - r0), x, wd, False])

    def overlap(a, b):
        if not (a[0] < b[1] and b[0] < a[1]):
            return False
        if a[4] or b[4]:
            return True
        d = (b[2] - a[2]) % tp
        return d < a[3] or d + b[3] > tp

    def unite(a, b):
        u = [min(a[0], b[0]), max(a[1], b[1]), -math.pi, tp, True]
        if a[4] or b[4]:
            return u
        d = (b[2] - a[2]) % tp
        s, w = (a[2], max(a[3], d + b[3])) if d < a[3] else (a[2] + d - tp, max(a[3] + tp - d, b[3]))
        return u if w >= tp else u[:2] + [(s + math.pi) % tp - math.pi, w, False]

    more = True
    while more:
        more = False
        for i in range(len(boxes)):
            for j in range(i + 1, len(boxes)):
                if not more and overlap(boxes[i], boxes[j]):
                    boxes[i] = unite(boxes[i], boxes[j])
                    del boxes[j]
                    more = True
                    break
            if more:
                break
    return boxes if len(boxes) <= 5 else None


def _magnification(p, t, g):
    """The discrete method in 64 bits at the times t (linear or quadratic
    limb darkening); nan where it needs more sectors than the cap."""
    eps, a = _lens(p)
    rho, u1, u2, K = p["rho"], p["u1"], p["u2"], g["n_limb"]
    I0 = 1.0 / (math.pi * (1.0 - u1 / 3.0 - u2 / 6.0))
    limb = np.exp(2j * math.pi * np.arange(K) / K)
    out = []
    for w in _centre(p, t):
        def dist(z):
            return np.abs(z - eps[0] / np.conj(z - a[0]) - eps[1] / np.conj(z - a[1]) - w)

        z, ok = _images(p, w + rho * limb, g["img_tol"])
        boxes = _sectors(z[ok], lambda z: dist(z) < rho, g)
        if boxes is None:
            out.append(math.nan)
            continue
        tot = 0.0
        for r0, r1, th0, wd, per in boxes:
            dr, dth, n = (r1 - r0) / g["n_r"], wd / g["n_theta"], g["n_theta"]
            r = r0 + (np.arange(g["n_r"]) + 0.5) * dr
            th = th0 + (np.arange(-2, n + 2) + 0.5) * dth      # two halo columns a side
            col = np.arange(-2, n + 2) % n if per else np.arange(-2, n + 2)
            d = dist(r[:, None] * np.exp(1j * (th0 + (np.clip(col, 0, n - 1) + 0.5) * dth))[None, :])
            if not per:
                d[:, :2] = d[:, -2:] = math.inf
            chi = d < rho
            mu = np.sqrt(np.clip(1.0 - (d / rho) ** 2, 0.0, None))
            bright = I0 * (1.0 - u1 * (1.0 - mu) - u2 * (1.0 - mu) ** 2)
            c = chi[:, 2:-2]
            f = {}                             # f(delta) of the points whose left, right neighbour is outside
            for side in (-1, 1):
                i, l = np.nonzero(c & ~chi[:, 2 + side:n + 2 + side])
                offs = np.array([-2, -1, 0, 1] if side < 0 else [-1, 0, 1, 2])
                y = np.stack([d[i, l + 2 + o] for o in offs], axis=1)
                delta = np.full(i.size, 0.5)
                edge = ~np.isfinite(y[:, 1 if side < 0 else 2])
                for k in np.nonzero(~edge)[0]:
                    fin = np.isfinite(y[k])
                    cf = np.polyfit(offs[fin], y[k][fin] - rho, int(fin.sum()) - 1)
                    lo, hi = 0.0, float(side)
                    x = 0.5 * side
                    for _ in range(60):
                        gx = np.polyval(cf, x)
                        if gx < 0:
                            lo = x
                        else:
                            hi = x
                        s = np.polyval(np.polyder(cf), x)
                        xn = x - gx / s if s != 0 else 0.5 * (lo + hi)
                        if not min(lo, hi) < xn < max(lo, hi):
                            xn = 0.5 * (lo + hi)
                        if abs(xn - x) < 1e-13:
                            x = xn
                            break
                        x = xn
                    delta[k] = abs(x)
                f[side] = np.ones(c.shape)
                f[side][i, l] = np.where(delta >= g["delta_c"],
                                         (0.5 + delta) * (2.0 / 3.0) * np.sqrt(1.0 + 0.5 / np.maximum(delta, 1e-300)),
                                         2.0 / 3.0 * delta + 0.5)
            L, R = chi[:, 1:-3], chi[:, 3:-1]
            W = np.where(L & R, 1.0, np.where(L, f[1], np.where(R, f[-1], np.clip(f[-1] + f[1] - 1.0, 0.0, None))))
            tot += float(((bright[:, 2:-2] * W * c).sum(axis=1) * r).sum() * dr * dth)
        out.append(tot / rho ** 2)
    return np.array(out)


def _mlp(theta, f):
    """(mu, s) of the network in 64 bits, and the layers."""
    shapes = [(128, 7), (128, 128), (128, 128), (128, 128), (2, 128)]
    x, o, W = f.double(), 0, []
    for n, (i, j) in enumerate(shapes):
        w, b = theta[o:o + i * j].reshape(i, j), theta[o + i * j:o + i * j + i]
        o += i * j + i
        W.append((w, b))
        x = x @ w.T + b
        if n < 4:
            x = torch.nn.functional.silu(x)
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "mlp_infer":
        st = prepare(case, seed)
        out = torch.cat([_mlp(st["theta"].double(), x) for x in st["feat"][:, :7].split(1 << 16)])
        return dict(out=out, err=None)
    if kind == "mlp_train":
        st = prepare(case, seed)
        th = st["theta"].double().requires_grad_()
        f, y = st["feat"][st["idx"].long()], st["target"][st["idx"].long()].double()
        o = _mlp(th, f[:, :7])
        loss = 0.5 * ((y - o[:, 0]) ** 2 * torch.exp(-o[:, 1]) + o[:, 1]).mean()
        g, = torch.autograd.grad(loss, th)
        k = st["step"] + 1
        m = 0.9 * st["m"].double() + 0.1 * g
        v = 0.999 * st["v"].double() + 0.001 * g * g
        new = th.detach() - 1e-3 * (m / (1 - 0.9 ** k)) / (torch.sqrt(v / (1 - 0.999 ** k)) + 1e-8)
        return dict(theta=new, m=m, v=v, pack=None, loss=loss.detach().reshape(1), err=None)
    params, t = _params(case, seed)
    if kind == "preselected" and case["sets"] * case["epochs"] <= 100_000:
        A_ps = np.concatenate([_point_source(p, _centre(p, t[i])) for i, p in enumerate(params)])
        return dict(A=None, routed=None, feat=None, A_ps=A_ps, flags=None)
    # the light curves that a few seconds of numpy can follow
    if kind in ("curve", "batch") and case["law"] in ("linear", "quadratic") and \
            case["sets"] * case["epochs"] * (case["n_r"] * case["n_theta"] + EPOCH) <= 12 * EPOCH * 24:
        g = _grid(case)
        return dict(A=np.stack([_magnification(p, t[i], g) for i, p in enumerate(params)]), status=None)
    return None
