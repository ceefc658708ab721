"""Tile edges of the screen's network kernels (16 samples a tile and CTA in the gradient, 8
samples a tile and warp in the prediction, up to the grid, then a loop) and parameter vectors
without 16-byte alignment, against the NumPy FP64 oracle.  Tolerances as in test_gpu_mlp.py:
FP32 accumulation over chains of 64 terms and three layers stays below 2e-4 in norm (gradient)
and 1e-4 of the largest prediction."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


def _problem(n, seed):
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(n, 9)).astype(np.float32) * 2 + 1
    y = (0.3 * x[:, 0] - 0.2 * x[:, 5] + 0.5 * rng.normal(size=n)).astype(np.float32)
    theta = omlp.init(seed).astype(np.float32)
    mean, std = x.mean(0) + 0.1, x.std(0) + 0.5
    return x, y, theta, mean.astype(np.float32), std.astype(np.float32)


def _dev(a, dt=torch.float32, shift=0):
    """Device copy whose first element lies `shift` elements past a 16-byte boundary."""
    a = np.ascontiguousarray(a)
    t = torch.empty(a.size + shift, dtype=dt, device="cuda")
    t[shift:].copy_(torch.as_tensor(a.reshape(-1), dtype=dt))
    return t[shift:].view(a.shape)


@pytest.mark.parametrize("n,shift", [(1, 0), (15, 0), (16, 0), (17, 1), (63, 0), (65, 3),
                                     (152 * 16, 0), (152 * 16 + 5, 0), (3 * 152 * 64 + 1, 0)])
def test_tile_edges(n, shift):
    x, y, theta, mean, std = _problem(n, n)
    idx = np.random.default_rng(n).permutation(n).astype(np.int32)
    tb = omlp.bf16_round(theta)
    xf, mf, sf = x.astype(np.float64), mean.astype(np.float64), std.astype(np.float64)
    W, X, Y, M, S = (_dev(a, shift=shift) for a in (theta, x, y, mean, std))
    ref, _ = omlp.forward(tb, xf, mf, sf)
    p = rimp2.mlp_predict(W, X, M, S).cpu().numpy()
    assert p.shape == (n,) and np.max(np.abs(p - ref)) <= 1e-4 * (1 + np.max(np.abs(ref)))
    want = omlp.grad(tb, xf, y.astype(np.float64), mf, sf)
    for rows in (None, _dev(idx, torch.int32)):
        g, loss = rimp2.mlp_grad(W, X, Y, rows, n, M, S)
        assert np.linalg.norm(g.cpu().numpy() - want) <= 2e-4 * np.linalg.norm(want)
        assert float(loss.item()) == pytest.approx(omlp.loss(tb, xf, y.astype(np.float64), mf, sf), rel=1e-4)
