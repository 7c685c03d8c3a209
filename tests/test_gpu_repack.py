"""A training step writes the whole of `pack`, its padding included."""
import numpy as np
import pytest

from tests.test_gpu_parity import G  # noqa: F401
from tests.test_gpu_surrogate import rand_features, theta_for_test

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("noalloc", [False, True])
def test_step_writes_the_padding(G, noalloc):
    import torch
    n = 300
    th = torch.tensor(theta_for_test(51), device="cuda")
    f = torch.tensor(rand_features(n, 52), device="cuda")
    y = torch.tensor(np.random.default_rng(53).standard_normal(n).astype(np.float32), device="cuda")
    weights = G.mlp_pack(torch.ones_like(th)).view(torch.int16) != 0
    step = G.mlp_train_step_noalloc if noalloc else G.mlp_train_step

    def run(pad):
        t, m, v = th.clone(), torch.zeros_like(th), torch.zeros_like(th)
        pack = G.mlp_pack(t)
        pack.view(torch.int16)[~weights] = pad
        step(t, m, v, pack, 1, 1e-3, f, y)
        return t, pack
    t0, p0 = run(0)
    assert torch.equal(p0, G.mlp_pack(t0))
    # (finite padding meets zeros only: the step itself is the same)
    t1, p1 = run(0x3f80)
    assert torch.equal(t1, t0) and torch.equal(p1, p0)
