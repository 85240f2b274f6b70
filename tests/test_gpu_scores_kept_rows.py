"""Which runs have their scores computed from a copy of the kept rows: those where it pays by the images' mean length, not every
run of a plan that allows long images.  The profiling record names the instance.  Marked gpu."""
import pytest

from paper_2605_00392_b200 import binding, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths,most,params,kernel", [
    ([400] * 64, 4512, dict(r_fixed=0.25), "scores"),                                              # a plan for far longer images
    ([100] * 64, 4512, dict(dynamic=1, phi_lo=0.0, phi_hi=0.5, r_max=0.5), "scores"),
    ([1000] * 2, 4512, dict(r_fixed=0.4), "scores_kept"),                                           # few CTAs either way
    ([1400] * 40, 1400, dict(dynamic=1, phi_lo=0.0, phi_hi=0.5, r_max=0.5), "scores"),               # prunes too little for a copy
    ([1400] * 40, 1400, dict(r_fixed=0.47), "scores_kept"),
    ([2700, 1200, 2500] * 5, 2700, dict(r_fixed=0.4), "scores_kept")])
def test_which_runs_copy_the_kept_rows(lengths, most, params, kernel):
    import parity
    w = synth.ragged(lengths, params=dict(iters=10, **params))
    plan = binding.Plan(w.d, w.X.dtype, w.batch, w.total_tokens, most)
    try:
        plan.profile_enable(True)
        parity.check_workload(w, plan=plan, images=[0, w.batch - 1])
        names = [n for n, _ in plan.profile_read()]
        assert kernel in names, names
        plan.profile_enable(False)
    finally:
        plan.close()
