"""P_ij and P_ab through the slice-stacked contraction kernel at the edges of its tiles: 4-row
padding, one or two row groups of 128 rows (6 slices: 20 | 24 rows), one or two tiles a side
(40 | 41, 80), the first extents that go to the 128-row tiles (81; FP8, 10 slices: 25), K shorter than a stage, several fragments of different widths in one launch.  Against
the CPU oracle, tolerances of test_gpu_split.py (the split path's accuracy target)."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu

BF16 = [(1, 1, 3), (2, 4, 9), (4, 21, 30), (20, 24, 31), (21, 25, 40), (24, 40, 50), (40, 41, 33),
        (41, 9, 28), (3, 80, 17), (80, 6, 20), (5, 81, 22), (81, 5, 18)]
FP8 = [(3, 5, 9), (12, 16, 25), (13, 24, 30), (24, 25, 26), (25, 12, 20), (48, 8, 19), (49, 7, 18),
       (6, 49, 21)]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _check(out, ref):
    assert abs(float(out["energy"]) - ref["energy"]) <= 1e-8
    for k in ("gamma", "pij", "pab", "epair"):
        assert rel(out[k].cpu().numpy(), ref[k]) <= 1e-9, k
    for k in ("pij", "pab"):
        g = out[k].cpu().numpy()
        assert np.array_equal(g, g.T) or rel(g, g.T) <= 1e-13, k


@pytest.mark.parametrize("precision,dims", [("bf16", d) for d in BF16] + [("fp8", d) for d in FP8])
def test_stacked_extents(precision, dims):
    f = synth.fragment_inputs(*dims, seed=sum(dims))
    _check(rimp2.energy_grad(f.B, f.eo, f.ev, precision=precision), oracle.fragment(f.B, f.eo, f.ev))


@pytest.mark.parametrize("precision,dims,opts", [("bf16", BF16, {}), ("fp8", FP8, {}),
                                                 ("bf16", BF16, {"slices_t": 7}), ("bf16", BF16, {"slices_t": 8})])
def test_mixed_widths_in_one_launch(precision, dims, opts):
    frags = [synth.fragment_inputs(*d, seed=sum(d)) for d in dims]
    eng = rimp2.Engine(dims, precision=precision, **opts)
    eng.set_inputs(frags)
    for _ in range(2):   # the second call replays the graph
        eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    for k, f in enumerate(frags):
        _check(eng.views(k), oracle.fragment(f.B, f.eo, f.ev))
