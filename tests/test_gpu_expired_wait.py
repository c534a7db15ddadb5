"""A device wait that expired (here: its error word, set without one) ends the call that meets it
with FMDP_ERR_TIMEOUT and leaves nothing behind: training takes no step on the gradient of
such a batch, reports it, and trains as if nothing had been the next time. Known plans do not
come from a rollout, and are stored whatever an earlier call left.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import FmdpError, Scheduler  # noqa: E402

TIMEOUT = -4


def test_training_reports_it_and_takes_no_step():
    sc = S.c1_plain_small()
    with Scheduler.from_scenario(sc) as s:
        s.learned_collect(sc.requests[:4])
        s.learned_init(seed=3)
        p0 = s.learned_get_params()
        s.selftest_expired_wait()
        with pytest.raises(FmdpError) as e:
            s.learned_train(epochs=2, batch=64, lr=1e-3, seed=1)
        assert e.value.status == TIMEOUT
        np.testing.assert_array_equal(s.learned_get_params(), p0)
        s.learned_init(seed=3)
        losses = s.learned_train(epochs=2, batch=64, lr=1e-3, seed=1)
        assert losses[1] < losses[0] and not np.array_equal(s.learned_get_params(), p0)
        assert s.schedule(sc.requests[0])["n_points"] > 1  # (no error is left for the next call)


@pytest.mark.parametrize("n", [1, 8, 9, 40])
def test_known_plans_are_stored_whatever_an_earlier_call_left(n):
    """Up to eight plans are appended to the index's rows, more rebuild them."""
    sc = S.c1_plain_small()
    plans = [(p.t0, p.xyz) for p in sc.plans[:n]]
    reports = []
    for left in (False, True):
        with Scheduler.from_scenario(sc, add_plans=False) as s:
            if left:
                s.selftest_expired_wait()
            ids = s.add_plans(plans)
            for i, (t0, xyz) in zip(ids, plans):
                g0, g = s.get_plan(i)
                assert g0 == t0
                np.testing.assert_array_equal(g, xyz)
            reports.append([s.sep_check(t0, xyz + np.float32(20.0)) for t0, xyz in plans])
    assert reports[0] == reports[1] and all(r["conflicts"] > 0 for r in reports[0])
