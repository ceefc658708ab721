"""Edges of the FP64 GEMM's tiles (64, 32 or 16 wide, trimmed to 16 rows or columns) and K
pieces (multiples of 16 of the flat K index): fragments whose nocc nvir, nvir, nocc and naux
lie on, just below and just above them, against the CPU oracle, alone and as one uneven
batch (whose plan picks other tile widths and piece lengths).  Tolerance as in
test_gpu_fp64.py: both sides are FP64 in different summation orders."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu

TOL = 1e-11
DIMS = [
    (1, 15, 16), (1, 17, 15), (4, 4, 17),      # one tile, one K block more or less
    (3, 21, 33), (5, 13, 64), (8, 8, 63),      # ov 63, 65, 64
    (16, 3, 20), (17, 2, 9), (33, 1, 40),      # nocc at the tile width, K0 = nvir below 16
    (2, 127, 31), (20, 65, 47),                # nvir 65 and 127: trimmed diagonal tiles
]


def _check(out, ref):
    assert abs(float(out["energy"]) - ref["energy"]) <= TOL * abs(ref["energy"])
    for k in ("gamma", "pij", "pab", "epair"):
        g = out[k].cpu().numpy()
        assert np.linalg.norm(g - ref[k]) <= TOL * np.linalg.norm(ref[k]), k
    for k in ("pij", "pab"):                   # both triangles are written
        g = out[k].cpu().numpy()
        assert np.linalg.norm(g - g.T) <= TOL * np.linalg.norm(g), k


@pytest.mark.parametrize("dims", DIMS)
def test_tile_edges(dims):
    f = synth.fragment_inputs(*dims, seed=sum(dims))
    _check(rimp2.energy_grad(f.B, f.eo, f.ev, precision="fp64"), oracle.fragment(f.B, f.eo, f.ev))


def test_tile_edges_in_one_batch():
    frags = [synth.fragment_inputs(*d, seed=sum(d)) for d in DIMS]
    eng = rimp2.Engine(DIMS, precision="fp64")
    eng.set_inputs(frags)
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    for k, f in enumerate(frags):
        _check(eng.views(k), oracle.fragment(f.B, f.eo, f.ev))
