"""The output layer's weight gradient dW_4 = sum over a tile's samples of X_4 dZ_4
against exact sums: no further off, in the root mean square, than additions of the products in FP32.

With zero weights the prediction is (0, 0) for every sample, so dZ_4 is known
exactly, and X_4 is the SiLU of the biases b_3.
"""
import numpy as np
import pytest

from tests.test_gpu_parity import G  # noqa: F401

pytestmark = pytest.mark.gpu
H = 128


def bf16(x):
    import torch
    return torch.tensor(np.asarray(x, dtype=np.float32)).to(torch.bfloat16).to(torch.float32).numpy()


def test_dw4_is_as_good_as_fp32_additions(G):
    import torch
    b3 = G.MLP_NPARAM - 2 - 2 * H - H
    n, got_e, f32_e = 128, [], []
    for seed in range(24):
        rng = np.random.default_rng(seed)
        y = rng.standard_normal(n).astype(np.float32)
        th = np.zeros(G.MLP_NPARAM, dtype=np.float32)
        th[b3:b3 + H] = rng.uniform(0.5, 3.0, H)
        tt = torch.tensor(th, device="cuda")
        g = torch.zeros_like(tt)
        G.mlp_train_step(tt, None, None, G.mlp_pack(tt), 1, 0.0, torch.zeros((n, 8), device="cuda"),
                         torch.tensor(y, device="cuda"), grad=g)
        g = g.cpu().numpy().astype(np.float64)
        d0 = bf16(-y / np.float32(n))
        assert g[-2] == d0.astype(np.float64).sum()  # db_4: exact here, and shows that dZ_4 is
        z = th[b3:b3 + H].astype(np.float64)
        x = bf16(z / (1.0 + np.exp(-z)))
        s = np.zeros(H, dtype=np.float32)
        for m in range(n):
            s = s + x * d0[m]  # (the product of two BF16 numbers is exact in FP32)
        ref, scale = x.astype(np.float64) * d0.astype(np.float64).sum(), np.abs(x) * np.abs(d0.astype(np.float64)).sum()
        got_e.append((g[b3 + H:b3 + 2 * H] - ref) / scale)
        f32_e.append((s.astype(np.float64) - ref) / scale)
    got, f32 = np.concatenate(got_e), np.concatenate(f32_e)
    assert np.abs(got).max() <= 128 * 2.0 ** -24
    assert np.sqrt((got ** 2).mean()) <= np.sqrt((f32 ** 2).mean()), (np.sqrt((got ** 2).mean()), np.sqrt((f32 ** 2).mean()))
