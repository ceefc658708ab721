"""The cooperative conjugate-gradient kernel at the edges of its work split (32-row items,
256-column items, grids of one CTA up to two per SM), against the dense oracle, and a
right-hand side of zero.  Tolerances as in test_gpu_zvector.py."""
import numpy as np
import pytest
import torch

from oracle import oracle, zvector
from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(1, 1, 300), (2, 3, 1), (1, 40, 257), (4, 8, 256), (33, 5, 20),
                                  (3, 67, 31), (24, 96, 360)])
def test_dai_matches_dense_solve(dims):
    o, v, X = dims
    f = synth.full_mo_inputs(o, v, X, seed=o + v)
    ref = oracle.fragment(f.frag.B, f.frag.eo, f.frag.ev)
    want = zvector.solve_dai(f.Bf, f.eps, ref["gamma"], ref["pij"], ref["pab"], f.jmh, o)
    got = rimp2.zvector(f.Bf, f.eps, ref["gamma"], ref["pij"], ref["pab"])
    info = got["info"].cpu().numpy()
    assert 1 <= info[0] <= 100 and info[1] <= 1e-12 and info[2] > 0, info
    d = got["dai"].cpu().numpy() - want
    assert np.linalg.norm(d) <= 1e-10 * np.linalg.norm(want)
    # the same workspace again: every counter and flag starts from zero
    again = rimp2.zvector(f.Bf, f.eps, ref["gamma"], ref["pij"], ref["pab"],
                          workspace=got["_keep"][-1])
    assert again["info"][0].item() == info[0]
    assert np.linalg.norm(again["dai"].cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)


def test_zero_rhs_takes_no_iteration():
    f = synth.full_mo_inputs(5, 9, 12, seed=1)
    out = rimp2.zvector(f.Bf, f.eps, np.zeros((5, 9, 12)), np.zeros((5, 5)), np.zeros((9, 9)))
    assert out["info"].cpu().tolist() == [0.0, 0.0, 0.0]
    assert torch.count_nonzero(out["dai"]).item() == 0
