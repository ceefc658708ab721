"""Few pairs on the FP64 path: pairs cut over several amplitude CTAs, Gamma in two K pieces that
are added into a zeroed output, energies summed beside the contractions.  Sizes around the
shortest K that is cut (nocc nvir = 128), one and several 32-wide tiles, one pair and more pairs
than CTAs.  A second run on new inputs must start from clean outputs and counters, and agree with
the first call of a fresh plan to the bit (two Gamma pieces add in either order to the same sum).
Tolerance as in test_gpu_fp64.py: FP64 in different summation orders."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.mark.parametrize("dims", [[(1, 127, 16)], [(1, 128, 16)], [(1, 129, 17)], [(1, 1, 1)], [(2, 33, 5)],
                                  [(10, 40, 30)], [(33, 8, 20)], [(2, 65, 40), (0, 4, 4), (1, 32, 9), (5, 31, 64)]])
def test_second_run_starts_clean(dims):
    eng = rimp2.Engine(dims, precision="fp64")
    for seed in (1, 2):
        frags = [synth.fragment_inputs(*d, seed=10 * seed + k) for k, d in enumerate(dims)]
        eng.set_inputs(frags)
        eng.run()
        torch.cuda.synchronize()
        eng.check_status()
    new = rimp2.Engine(dims, precision="fp64")
    new.set_inputs(frags)
    new.run()
    torch.cuda.synchronize()
    for k, (f, (o, v, X)) in enumerate(zip(frags, dims)):
        out, one = eng.views(k), new.views(k)
        assert float(out["energy"]) == float(one["energy"]) and torch.equal(out["gamma"], one["gamma"])
        if o == 0:
            continue
        ref = oracle.fragment(f.B, f.eo, f.ev)
        assert abs(float(out["energy"]) - ref["energy"]) <= TOL * abs(ref["energy"])
        for n in ("gamma", "pij", "pab", "epair"):
            assert np.linalg.norm(out[n].cpu().numpy() - ref[n]) <= TOL * np.linalg.norm(ref[n]), n
