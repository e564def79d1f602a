"""A plan set with lbm_batch_set_plan is the one lbm_batch_step runs on, also in a
batch large enough for two steps per launch (csrc/lbm_batch.cu)."""
import numpy as np
import pytest

from paper_2011_15073_gb300 import inputs, lbm

pytestmark = pytest.mark.gpu

# 502,500 nodes: above the 300,000 from which steps go two to a launch
CASES = [dict(nx=a, ny=b, n=0.7, Da=1e-2, Ra=1e5, Pr=6.2, porosity=0.6) for a, b in ((500, 400), (401, 500), (204, 500))]


def test_a_set_plan_is_in_effect():
    """Seen by its barrier: with a budget of a few cycles the persistent plan's
    blocks give it up, which only that plan can (tests/test_batch_gpu.py)."""
    with lbm.Batch(CASES, prec="f32d") as b:
        b.set_wait_budget(4)
        b.step(20)   # two steps per launch: no barrier
        b.set_plan("persistent", 128, 4)
        with pytest.raises(lbm.LBMError) as e:
            b.step(20)
        assert e.value.code == -6


def test_plans_and_two_step_launches_agree():
    """set_plan takes the two-step launches away, tune gives them back; the
    states are the same."""
    states = []
    for change in (lambda b: None, lambda b: b.set_plan("per_step", 64, 8), lambda b: b.set_plan("persistent", 128, 4),
                   lambda b: (b.set_plan("per_step", 64, 8), b.tune(4))):
        with lbm.Batch(CASES, prec="f32d") as b:
            for i, c in enumerate(CASES):
                st = lbm.get_state_f64(b.case_ctx(i), c["nx"], c["ny"])
                lbm.set_state_f64(b.case_ctx(i), *inputs.perturbed_state(st, seed=i, amp=1e-2))
            change(b)
            b.step(7)
            b.step(6)
            out = [np.empty(lbm.state_bytes(b.case_ctx(i)), np.uint8) for i in range(len(CASES))]
            for i, h in enumerate(out):
                lbm.get_state(b.case_ctx(i), h)
            states.append(out)
    for other in states[1:]:
        for x, y in zip(states[0], other):
            assert np.array_equal(x, y)
