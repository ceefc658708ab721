"""The split path's pair energies carry no bias: with eight slices for V (72 bits) the energies
and their opposite-spin parts differ from the FP64 path's by rounding alone.  Limit: a unit in
the last place of either path's FP64 sum, 2^-52, for the mean signed difference over the
fragments (the double-float products' own errors, 2^-48 an element and of either sign, average
out over more than 10^6 elements)."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(20, 80, 300), (24, 97, 130)])
def test_mean_difference(dims):
    frags = [synth.fragment_inputs(*dims, seed=s) for s in range(6)]
    out = []
    for precision, opts in (("fp64", {}), ("bf16", {"slices_v": 8})):
        eng = rimp2.Engine([dims] * len(frags), precision=precision, want_gamma=False, want_p=False, **opts)
        eng.set_inputs(frags)
        eng.run()
        torch.cuda.synchronize()
        eng.check_status()
        out.append([t.clone() for t in (eng.energy, eng.energy_os, eng.energy_scs)])
    for ref, got in zip(*out):
        assert abs(((got - ref) / ref).mean().item()) <= 2.0 ** -52
