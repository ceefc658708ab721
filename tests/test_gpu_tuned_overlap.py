"""A tuned plan runs without stage events (they keep its launches from overlapping): stage_ms is
reported by the trials and with profile_stages only, and a tuned call is not slower than the
untuned default.  The events alone cost these small calls half of their time again; the limit
of a quarter leaves room for another choice of shapes and the spread of the timer."""
import pytest
import torch

from paper_2410_21888_gb300 import rimp2, synth

pytestmark = pytest.mark.gpu


def _engine(dims, precision, **kw):
    eng = rimp2.Engine([dims], precision=precision, **kw)
    eng.set_inputs([synth.fragment_inputs(*dims, seed=2)])
    return eng


def _call_ms(eng, n=50):
    best = float("inf")
    for _ in range(6):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda.synchronize()
        a.record()
        for _ in range(n):
            eng.run()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / n)
    return best


@pytest.mark.parametrize("dims,precision", [((10, 40, 150), "bf16"), ((10, 40, 150), "fp8"),
                                            ((6, 24, 90), "fp64")])
def test_tuned_plan_has_no_stage_events(dims, precision, tmp_path):
    cache = str(tmp_path / "tune.txt")
    tuned = _engine(dims, precision, autotune=True, autotune_cache=cache)
    for k in range(tuned.plan.stats().tune_trials):
        tuned.run()
        assert sum(tuned.plan.stats().stage_ms) > 0      # a trial
    tuned.run()
    cached = _engine(dims, precision, autotune=True, autotune_cache=cache)
    cached.run()
    for eng in (tuned, cached):
        st = eng.plan.stats()
        assert st.tune_done == 1 and sum(st.stage_ms) == 0 and sum(st.launch_ms) == 0
    ref = _call_ms(_engine(dims, precision))
    assert _call_ms(tuned) <= 1.25 * ref and _call_ms(cached) <= 1.25 * ref


def test_profiled_plan_reports_stages_after_tuning():
    eng = _engine((6, 24, 90), "bf16", autotune=True, profile_stages=True)
    for _ in range(eng.plan.stats().tune_trials + 2):
        eng.run()
    st = eng.plan.stats()
    assert st.tune_done == 1 and sum(st.stage_ms) > 0
