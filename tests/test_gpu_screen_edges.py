"""Edges of the screen's prediction pass.  Features: distances and pair corrections over the
range of FP64, next to 1, zero, infinite and NaN, against NumPy's FP64 functions rounded to
FP32; both sides are FP64 values with relative errors far below 2^-40 before the rounding, so
they differ by one unit in the last place at most.  Network: inputs, weights and biases that are
not finite give the values that FP32 arithmetic gives, finite ones the 1e-4 of
test_gpu_mlp.py."""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


def _dev(a, dt):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt).cuda()


def _sort3(a, b, c):
    lt = lambda x, y: np.where(x > y, y, x)          # the kernel's exchanges: only where x > y
    gt = lambda x, y: np.where(x > y, x, y)
    a, b = lt(a, b), gt(a, b)
    b, c = lt(b, c), gt(b, c)
    return lt(a, b), gt(a, b), c


@pytest.mark.parametrize("n", [3, 40, 257])
def test_features(n):
    rng = np.random.default_rng(n)
    cen = rng.normal(size=(n, 3)) * 10.0 ** rng.uniform(-3, 3, size=(n, 1))
    nocc = rng.integers(1, 30, size=n)
    de = rng.normal(size=(n, n)) * 10.0 ** rng.uniform(-14, 2, size=(n, n))
    special = [0.0, -0.0, 1.0, -1.0, 1e-16, 1e-300, 1e300, 3e-17, 0.1, 10.0, 2.0, np.inf, -np.inf, np.nan]
    special += [s * (1 + d * 2.0 ** -k) for k in range(1, 53, 3) for d in (1, -1) for s in (1.0, 4.0)]
    if n > 3:
        de.reshape(-1)[rng.permutation(n * n)[:len(special)]] = special
        cen[1], cen[2], cen[3], cen[4], cen[5] = cen[0], 1e25, 1e-25, cen[6] + 1e-18, -1e16
        cen[7, 1] = np.inf
    tri = np.stack([rng.permutation(n)[:3] for _ in range(5000)]).astype(np.int32)
    with np.errstate(all="ignore"):
        I, J, K = tri.T
        d = lambda a, b: np.sqrt(((cen[a] - cen[b]) ** 2).sum(1)).astype(np.float32)
        lg = lambda a, b: np.log10(np.abs(de[a, b]) + 1e-16).astype(np.float32)
        ref = np.stack([*_sort3(d(I, J), d(I, K), d(J, K)),
                        *_sort3(*(nocc[x].astype(np.float32) for x in (I, J, K))),
                        *_sort3(lg(I, J), lg(I, K), lg(J, K))], 1)
    got = rimp2.screen_features(_dev(cen, torch.float64), _dev(nocc, torch.int32), _dev(tri, torch.int32),
                                _dev(de, torch.float64)).cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    ok = np.isfinite(ref)
    assert np.array_equal(got[~ok & ~np.isnan(ref)], ref[~ok & ~np.isnan(ref)])
    assert np.all(np.abs(got[ok] - ref[ok]) <= np.spacing(np.abs(ref[ok])))


@pytest.mark.parametrize("where,value", [(3, np.inf), (600, np.inf), (2000, -np.inf), (4700, np.nan),
                                         (580, np.inf), (4800, 3.395e38), (9000, -np.inf), (None, None)])
def test_network_not_finite(where, value):
    n = 333
    rng = np.random.default_rng(7)
    x = rng.normal(size=(n, 9)).astype(np.float32)
    x[5, 2], x[17, 8], x[18, 0], x[100, 4] = np.inf, -np.inf, np.nan, 3e38
    theta = omlp.init(3).astype(np.float32)
    if where is not None:
        theta[where] = value
    mean, std = np.zeros(9, np.float32), np.ones(9, np.float32)
    p = rimp2.mlp_predict(*(_dev(a, torch.float32) for a in (theta, x, mean, std))).cpu().numpy()
    with np.errstate(all="ignore"):
        h, tb = x, omlp.bf16_round(theta).astype(np.float32)
        off = 0
        for width in (9, 64, 64):
            W, off = tb[off:off + 64 * width].reshape(64, width), off + 64 * width
            b, off = tb[off:off + 64], off + 64
            z = (h[:, None, :] * W).sum(2, dtype=np.float32) + b
            h = z * (np.float32(1) / (np.float32(1) + np.exp(-z)))
        ref = (h * tb[off:off + 64]).sum(1, dtype=np.float32) + tb[off + 64]
    ok = np.isfinite(ref)
    assert np.array_equal(np.isnan(p), np.isnan(ref))
    assert np.array_equal(p[~ok & ~np.isnan(ref)], ref[~ok & ~np.isnan(ref)])
    small = ok & (np.abs(ref) < 1e6)
    assert np.max(np.abs(p[small] - ref[small]), initial=0.0) <= 1e-4 * (1 + np.max(np.abs(ref[small]), initial=0.0))
