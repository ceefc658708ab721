"""What the split path's merged small launches took over: the checks of B and the orbital
energies (same codes as the FP64 path, both zeros equal, NaN not taken for an order), energies
and zeroed outputs of fragments without occupied or virtual orbitals inside a batch, and
plans without the checks."""
import numpy as np
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def _code(f, precision, **kw):
    try:
        rimp2.energy_grad(f.B, f.eo, f.ev, precision=precision, **kw)
    except rimp2.Rimp2Error as e:
        return e.code
    return 0


@pytest.mark.parametrize("precision", ["fp64", "bf16", "fp8"])
def test_checks(precision):
    def frag(**kw):
        f = synth.fragment_inputs(3, 5, 40, seed=1)
        for k, (i, x) in kw.items():
            getattr(f, k)[i] = x
        return f

    assert _code(frag(), precision) == 0
    assert _code(frag(eo=(1, 0.0), ev=(2, 0.1)), precision) == 0
    for x in (np.nan, np.inf, -np.inf):
        assert _code(frag(B=((2, 4, 39), x)), precision) == -4
    assert _code(frag(eo=(0, np.nan)), precision) == -4
    assert _code(frag(ev=(4, np.nan)), precision) == -4
    assert _code(frag(ev=(4, np.inf)), precision) == -4
    assert _code(frag(eo=(2, -np.inf)), precision) == -4
    assert _code(frag(eo=(1, -0.0), ev=(2, 0.0)), precision) == -3      # equal: not negative
    assert _code(frag(eo=(1, 0.0), ev=(2, -0.0)), precision) == -3
    assert _code(frag(eo=(1, 0.3), ev=(2, 0.25)), precision) == -3
    assert _code(frag(eo=(1, 0.3), ev=(2, 0.25)), precision, check_inputs=False) == 0


@pytest.mark.parametrize("precision", ["fp64", "bf16"])
@pytest.mark.parametrize("grad", [True, False])
def test_empty_fragments_in_a_batch(precision, grad):
    dims = [(0, 3, 7), (2, 4, 9), (3, 0, 5), (0, 0, 0), (3, 4, 0), (6, 9, 20)]
    eng = rimp2.Engine(dims, precision=precision, want_gamma=grad, want_p=grad)
    for t in (eng.energy, eng.energy_os, eng.energy_scs, eng.gamma, eng.pij, eng.pab, eng.epair):
        if t is not None:
            t.fill_(7.0)                        # outputs are overwritten, never accumulated
    eng.set_inputs([synth.fragment_inputs(*d, seed=k) for k, d in enumerate(dims)])
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    for k, (o, v, X) in enumerate(dims):
        out = eng.views(k)
        if o * v * X == 0:
            assert all(torch.count_nonzero(out[n]).item() == 0 for n in out if out[n].numel()), (k, dims[k])
        else:
            one = rimp2.energy_grad(*[getattr(synth.fragment_inputs(o, v, X, seed=k), a) for a in ("B", "eo", "ev")],
                                    precision=precision, want_gamma=grad, want_p=grad)
            for n in out:
                a, b = out[n].cpu().numpy(), one[n].cpu().numpy()
                assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b), (k, n)
