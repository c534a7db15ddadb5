"""A device wait that expired (here: its error word, set without one) ends the call that meets it
with FMDP_ERR_TIMEOUT and leaves nothing behind: training takes no step on the gradient of
such a batch, reports it, and trains as if nothing had been the next time.
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
