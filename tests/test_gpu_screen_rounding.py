"""The screen's features are FP64 results rounded once: distances and logarithms that lie 2^-50 to
2^-46 (relative) from the middle between two FP32 numbers take the nearer one, which an error of
a few FP64 units in the last place (2^-52) cannot change and a coarser one would."""
from decimal import Decimal, getcontext

import numpy as np
import pytest
import torch

from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu
getcontext().prec = 40
LN10 = Decimal(10).ln()
K = 700


def _log10(x):
    return Decimal(float(x)).ln() / LN10


def _middle(f):
    """The middle between FP32 f and the next FP32 away from zero, exact in FP64, and that one."""
    g = np.nextafter(f, np.float32(np.copysign(np.inf, f)))
    return (float(f) + float(g)) / 2, g


def _logs(rng, lo, hi, sign):
    """FP64 arguments x and the FP32 numbers nearest to log10(x)."""
    xs, want = [], []
    while len(xs) < K:
        f = np.float32(sign * np.exp(rng.uniform(np.log(lo), np.log(hi))))
        t, g = _middle(f)
        x = float((Decimal(t) * LN10).exp())
        x *= 1 + int(rng.integers(-48, 49)) * 2.0 ** -52 * min(1.0, abs(t))
        off = (_log10(x) - Decimal(t)) / Decimal(abs(t))
        if not 2.0 ** -50 <= abs(off) <= 2.0 ** -46:
            continue
        xs.append(x)
        want.append(max(f, g) if off > 0 else min(f, g))
    return np.array(xs), np.array(want, dtype=np.float32)


def _features(cen, de):
    n = 3 * K
    tri = np.arange(n, dtype=np.int32).reshape(K, 3)
    nocc = torch.ones(n, dtype=torch.int32, device="cuda")
    return rimp2.screen_features(torch.as_tensor(cen).cuda(), nocc, torch.as_tensor(tri).cuda(),
                                 torch.as_tensor(de).cuda()).cpu().numpy()


@pytest.mark.parametrize("lo,hi,sign", [(0.002, 0.05, 1), (0.002, 0.05, -1), (0.1, 2, 1), (0.1, 14, -1)])
def test_logarithms(lo, hi, sign):
    xs, want = _logs(np.random.default_rng(int(100 * hi) + sign), lo, hi, sign)
    # |de| + 1e-16 = x to the bit
    de = xs - 1e-16
    for step in (-1, 1):
        miss = de + 1e-16 != xs
        de[miss] = np.nextafter(xs[miss] - 1e-16, step * np.inf)
    use = de + 1e-16 == xs
    assert use.sum() > K // 2
    m = np.zeros((3 * K, 3 * K))
    for a, b in ((0, 1), (0, 2), (1, 2)):
        m[np.arange(K) * 3 + a, np.arange(K) * 3 + b] = de
    got = _features(np.zeros((3 * K, 3)), m)
    assert np.array_equal(got[use, 6], want[use]) and np.array_equal(got[use, 8], want[use])


def test_distances():
    rng = np.random.default_rng(0)
    cen, want = np.zeros((3 * K, 3)), np.zeros(K, dtype=np.float32)
    for k in range(K):
        f = np.float32(np.exp(rng.uniform(np.log(0.5), np.log(200))))
        t, g = _middle(f)
        up = rng.integers(2)
        cen[3 * k + 1:3 * k + 3, k % 3] = t * (1 + (1 if up else -1) * 2.0 ** -rng.integers(46, 51))
        want[k] = g if up else f
    got = _features(cen, np.zeros((3 * K, 3 * K)))
    assert np.array_equal(got[:, 1], want) and np.array_equal(got[:, 2], want)
