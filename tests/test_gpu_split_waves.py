"""V's tile width follows the work of each launch: a batch whose launches are small because the
workspace budget cuts it into waves takes the narrow tiles of a small launch, with the results
of the single wave to the bit."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def _run(dims, budget, **kw):
    eng = rimp2.Engine(dims, precision="bf16", want_gamma=False, want_p=False,
                       max_workspace_bytes=budget, **kw)
    eng.set_inputs([synth.fragment_inputs(*d, seed=k) for k, d in enumerate(dims)])
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    st = eng.plan.stats()
    return st.waves, st.n_tile[0], eng.epair.clone(), eng.energy.clone()


@pytest.mark.parametrize("dims,width,narrow", [
    ([(10, 90, 70)] * 14, 64, 48), ([(10, 90, 576)] * 14, 80, 48),
    # one fragment with enough tiles of its own among small ones: its wave keeps the wide tiles
    ([(30, 90, 70)] + [(6, 21, 50)] * 2, 64, 64)])
def test_width_follows_the_wave(dims, width, narrow):
    waves, one, ep, e = _run(dims, 0)
    assert waves == 1 and one == width
    waves, many, ep2, e2 = _run(dims, 1)
    assert waves == len(dims) and many == narrow
    assert torch.equal(ep, ep2) and torch.equal(e, e2)
    assert _run(dims, 1, n_tile=64)[1] == 64      # pinned
