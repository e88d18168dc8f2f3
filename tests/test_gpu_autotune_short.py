"""The batch autotuner with trials of one step weighs launches of two steps too: on
large lattices they are faster by a third."""
import pytest

pytestmark = pytest.mark.gpu


def test_one_trial_step_finds_the_two_step_launches():
    from paper_1908_06742_gb300 import ddflb as D
    cfgs = [D.Config(nx=1024, ny=1024, bc="cavity", u_lid=0.05, check_every=1000)
            for _ in range(16)]
    b, rec = D.Batch(cfgs).autotune(trial_steps=1, cache=False)
    assert b.schedule() == 1
    long = D.Batch(cfgs).autotune(trial_steps=20, cache=False)[1]
    # time per step, not per trial (a trial of two steps is timed with its launch)
    assert 0.5 * long["ms_per_step"] < rec["ms_per_step"] < 2.0 * long["ms_per_step"]
