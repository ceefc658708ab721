"""Results of small fragments on the split path do not depend on the order in which the pieces of
a contraction end: below the lengths from which K is cut for speed (24,576 for Gamma, whose
slabs hold about 16,384) an element is the sum of at most two pieces added to zero, so repeated
calls give the same bits.  Work entries: a plan's minus those of the same plan without the
output."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def _engine(dims, precision, **want):
    eng = rimp2.Engine([dims], precision=precision, **want)
    eng.set_inputs([synth.fragment_inputs(*dims, seed=5)])
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    return eng


def _same_bits(eng, names, calls=24):
    first = {n: getattr(eng, n).clone() for n in names}
    for _ in range(calls):
        eng.run()
        torch.cuda.synchronize()
        for n in names:
            assert torch.equal(first[n], getattr(eng, n)), n


def _entries(eng):
    return eng.plan.stats().tiles_per_call


# one and two tiles of rows, auxiliary extents on both sides of a tile's 80 columns, K from a
# few stages to many
@pytest.mark.parametrize("dims", [(4, 16, 60), (10, 40, 80), (10, 40, 150), (14, 56, 210),
                                  (17, 68, 81)])
def test_gamma(dims):
    o, v, X = dims
    energies = _engine(dims, "bf16", want_gamma=False, want_p=False)
    eng = _engine(dims, "bf16", want_p=False)
    tiles = -(-o * v // 128) * -(-X // 80)
    assert tiles <= _entries(eng) - _entries(energies) <= 2 * tiles
    _same_bits(eng, ["gamma", "energy", "epair"])
