"""Failure detection in the conjugate-gradient kernel without a GPU fault: with the barrier limit set
to zero by the test hook its CTAs give up while the others are still on their way, every one of
them leaves the kernel, and the call reports info[0] = -1, not the max_iter + 1 of a solve that
did not converge.  With the normal limit the next solve on the same workspace is correct again.
"""
import ctypes

import numpy as np
import pytest
import torch

from oracle import oracle, zvector
from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def test_expired_barrier_is_reported_and_the_next_solve_is_right():
    set_limit = rimp2.load().rimp2_testing_set_zvec_wait_limit
    set_limit.argtypes, set_limit.restype = [ctypes.c_int64], ctypes.c_int
    o, v, X = 12, 40, 150
    f = synth.full_mo_inputs(o, v, X, seed=4)
    ref = oracle.fragment(f.frag.B, f.frag.eo, f.frag.ev)
    want = zvector.solve_dai(f.Bf, f.eps, ref["gamma"], ref["pij"], ref["pab"], f.jmh, o)

    def solve(**kw):
        return rimp2.zvector(f.Bf, f.eps, ref["gamma"], ref["pij"], ref["pab"], **kw)

    good = solve()
    ws = good["_keep"][-1]
    try:
        assert set_limit(0) == 0
        assert solve(workspace=ws)["info"][0].item() == -1
        torch.cuda.synchronize()
    finally:
        assert set_limit(-1) == 0
    assert solve(workspace=ws, max_iter=2)["info"][0].item() == 3    # not converged
    again = solve(workspace=ws)
    assert again["info"][0].item() == good["info"][0].item()
    assert np.linalg.norm(again["dai"].cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
