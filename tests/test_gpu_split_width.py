"""V's tile width follows the amount of work: every width gives the same bits (the sums of an
element do not depend on its tile), on both sides of the rule's lines, and a pinned width stays
pinned."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def _run(dims, n, precision, **kw):
    eng = rimp2.Engine([dims] * n, precision=precision, want_gamma=False, want_p=False, **kw)
    eng.set_inputs([synth.fragment_inputs(*dims, seed=k) for k in range(n)])
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    return eng.plan.stats().n_tile[0], eng.epair.clone(), eng.energy.clone()


@pytest.mark.parametrize("dims,n,precision,slices,width", [
    ((6, 21, 50), 1, "bf16", 0, 48), ((10, 90, 70), 3, "bf16", 0, 48),     # few tiles
    ((10, 90, 70), 14, "bf16", 0, 64), ((10, 90, 576), 14, "bf16", 0, 80),
    ((10, 90, 575), 14, "bf16", 0, 64), ((10, 90, 1025), 14, "bf16", 0, 80),
    ((10, 90, 1025), 14, "bf16", 8, 64), ((6, 21, 50), 1, "bf16", 8, 48),
    ((6, 21, 50), 1, "fp8", 0, 48), ((10, 90, 600), 14, "fp8", 0, 64)])
def test_width(dims, n, precision, slices, width):
    got, ep, e = _run(dims, n, precision, slices_v=slices)
    assert got == width
    for nt in (48, 64, 80):
        pinned, ep2, e2 = _run(dims, n, precision, slices_v=slices, n_tile=nt)
        assert pinned == nt or (nt == 80 and (slices == 8 or precision == "fp8"))
        assert torch.equal(ep, ep2) and torch.equal(e, e2)
