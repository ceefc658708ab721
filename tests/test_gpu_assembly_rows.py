"""Row lengths of the assembly kernel (32 lanes x 8 elements at a time) and its three ways to
start an element: accumulating, from a first contribution (coefficient 1 or not), and from
none (a block whose fragments have no Gamma offset), against index loops in NumPy.  The
gather adds the same FP64 products in the same order: equal to the last rounding."""
import itertools

import numpy as np
import pytest
import torch

from paper_2410_21888_gb300 import rimp2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nocc,nvir,naux", [
    ((1, 2), (1, 3), (1, 31)), ((3, 1), (9, 8), (33, 32)),
    ((2, 2), (7, 1), (256, 257)), ((1, 1), (300, 5), (511, 600)),
])
@pytest.mark.parametrize("accumulate", [False, True])
def test_rows(nocc, nvir, naux, accumulate):
    frags, coeff = [(0,), (1,), (0, 1), (1, 0)], [-2, 3, 1, 1]
    rng = np.random.default_rng(sum(naux))
    off, at = [[], [], []], [1, 0, 3]          # odd offsets: rows start on 8-byte boundaries only
    dims = [[sum(s[m] for m in f) for s in (nocc, nvir, naux)] for f in frags]
    for k, (o, v, x) in enumerate(dims):
        for q, n in enumerate((o * v * x, o * o, v * v)):
            off[q].append(at[q])
            at[q] += n + 1
    off[0][3] = -1                             # the last fragment gives no Gamma
    pools = [rng.normal(size=n) for n in at]
    asm = rimp2.MBEAssembly(nocc, nvir, naux, frags, coeff, *off)
    out = [torch.full_like(t, 0.5 if accumulate else np.nan) for t in asm.outputs()]
    asm.run(*(torch.as_tensor(p, device="cuda") for p in pools), *out, accumulate=accumulate)
    start = 0.5 if accumulate else 0.0
    cum = [[0, s[0], s[0] + s[1]] for s in (nocc, nvir, naux)]
    want = [np.full((cum[k][2],) * 2, start) for k in (0, 1)]
    blocks = {(I, J, K): np.full((nocc[I], nvir[J], naux[K]), start)
              for I, J, K in itertools.product((0, 1), repeat=3)}
    for k, f in enumerate(frags):
        o, v, x = dims[k]
        r = [[0] + list(np.cumsum([s[m] for m in f])) for s in (nocc, nvir, naux)]
        mats = [pools[1][off[1][k]:off[1][k] + o * o].reshape(o, o),
                pools[2][off[2][k]:off[2][k] + v * v].reshape(v, v)]
        for (a, I), (b, J) in itertools.product(enumerate(f), repeat=2):
            for q in (0, 1):
                want[q][cum[q][I]:cum[q][I + 1], cum[q][J]:cum[q][J + 1]] += \
                    coeff[k] * mats[q][r[q][a]:r[q][a + 1], r[q][b]:r[q][b + 1]]
            if off[0][k] >= 0:
                g = pools[0][off[0][k]:off[0][k] + o * v * x].reshape(o, v, x)
                for c, K in enumerate(f):
                    blocks[I, J, K] += coeff[k] * g[r[0][a]:r[0][a + 1], r[1][b]:r[1][b + 1],
                                                    r[2][c]:r[2][c + 1]]
    for got, ref in zip(out[1:], want):
        assert np.allclose(got.cpu().numpy(), ref, rtol=1e-15, atol=1e-14)
    for key, ref in blocks.items():
        got = asm.block(out[0], *key, nocc, nvir, naux).cpu().numpy()
        assert np.allclose(got, ref, rtol=1e-15, atol=1e-14), key
