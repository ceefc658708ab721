"""The P launches and Gamma's overlap (each may start on SMs that the one before leaves): a
call still ends with all of them.  Outputs read on the stream right behind a call, without a
synchronisation, and overwritten there before the next one, alone, replayed as the plan's graph
and inside a caller's graph; batches with P only stacked, only tiled, both, and without Gamma.
Both sides are the same engine, whose P and Gamma sums may differ in their order of additions
only (test_gpu_split.py bounds their error): 1e-12 of the norm."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu

BATCHES = [[(4, 9, 30)], [(10, 40, 150)], [(12, 90, 100)], [(3, 7, 20), (30, 70, 90), (5, 60, 64)]]


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("gamma", [True, False])
@pytest.mark.parametrize("dims", BATCHES)
@pytest.mark.parametrize("how", ["launches", "graph", "captured"])
def test_outputs_behind_the_call(dims, gamma, precision, how):
    eng = rimp2.Engine(dims, precision=precision, want_gamma=gamma, use_graph=how == "graph")
    eng.set_inputs([synth.fragment_inputs(*d, seed=k) for k, d in enumerate(dims)])
    outs = [t for t in (eng.gamma, eng.pij, eng.pab, eng.energy) if t is not None]
    eng.run()
    torch.cuda.synchronize()
    eng.check_status()
    ref = [t.clone() for t in outs]
    got = [torch.empty_like(t) for t in outs]

    def call():
        for t in outs:
            t.fill_(3.0)
        eng.run()
        for t, g in zip(outs, got):
            g.copy_(t)
        for t in outs:
            t.fill_(5.0)

    run = call
    if how == "captured":
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call()
        run = graph.replay
    for _ in range(20):
        run()
        run()
        torch.cuda.synchronize()
        for t, r in zip(got, ref):
            assert torch.linalg.vector_norm(t - r).item() <= 1e-12 * torch.linalg.vector_norm(r).item()


@pytest.mark.parametrize("precision", ["bf16", "fp8"])
@pytest.mark.parametrize("dims", [[(24, 9, 30)], [(25, 9, 30)], [(1, 1, 1)], [(24, 33, 40), (0, 3, 5), (7, 0, 4), (2, 130, 20)],
                                  [(24, 5, 9), (25, 5, 9)]])
def test_energies_beside_and_in_the_amplitude_kernel(dims, precision):
    """Both sides of the rule (24 occupied orbitals) against the FP64 path.  With V's widest
    digits and T in double-float (2^-46 a term) the pair energies agree to 1e-11 of the norm."""
    frags = [synth.fragment_inputs(*d, seed=k) for k, d in enumerate(dims)]
    outs = []
    for kw in (dict(precision="fp64"), dict(precision=precision, slices_v=8 if precision == "bf16" else 12)):
        eng = rimp2.Engine(dims, **kw)
        for t in (eng.energy, eng.energy_os, eng.energy_scs, eng.epair):
            t.fill_(7.0)
        eng.set_inputs(frags)
        eng.run()
        torch.cuda.synchronize()
        eng.check_status()
        outs.append([t.clone() for t in (eng.energy, eng.energy_os, eng.energy_scs, eng.epair)])
    for a, b in zip(*outs):
        assert torch.linalg.vector_norm(a - b).item() <= 1e-11 * torch.linalg.vector_norm(a).item()
