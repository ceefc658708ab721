"""The gradient's rounding error on large minibatches: the CTAs' sums meet in at most 36 additions
per parameter (one a cluster).  A chain of m FP32 additions of like terms errs by u sqrt(m) / 3
(u = 2^-24, errors uniform): 2 u for 36, which bounds the mean over several networks."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2048, 4096, 20000])
def test_mean_error(n):
    errs = []
    for seed in range(8):
        rng = np.random.default_rng(seed)
        x = (rng.normal(size=(n, 9)) * 2 + 1).astype(np.float32)
        y = (0.3 * x[:, 0] - 0.2 * x[:, 5] + 0.5 * rng.normal(size=n)).astype(np.float32)
        theta = omlp.init(seed).astype(np.float32)
        mean, std = x.mean(0).astype(np.float32), (x.std(0) + 0.5).astype(np.float32)
        dev = [torch.as_tensor(a, device="cuda") for a in (theta, x, y, mean, std)]
        g, _ = rimp2.mlp_grad(dev[0], dev[1], dev[2], None, n, dev[3], dev[4])
        want = omlp.grad(omlp.bf16_round(theta), x.astype(np.float64), y.astype(np.float64),
                         mean.astype(np.float64), std.astype(np.float64))
        errs.append(np.linalg.norm(g.cpu().numpy().astype(np.float64) - want) / np.linalg.norm(want))
    assert np.mean(errs) <= 2 * 2.0 ** -24, errs
