"""Proposals do not depend on the form of the rollout that makes them: clusters with 16 to 64 rows,
their queue refilled, and CTAs that stream the weights (more than six fifths of the clusters' rows).
The network steers for the goal, so that proposals get there in numbers of steps of their own, and
depends on the traffic around it.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import MLP_PARAMS, Scheduler  # noqa: E402

N = 5003


def steering(actions, seed):
    """Weights that carry the goal's bearing and height (features 6, 7 and 4) through the layers to
    the turns and climbs that follow them, and noise on all of them."""
    rng = np.random.default_rng(seed)
    dims = ((128, 256), (256, 256), (256, 256), (256, 256), (256, 25))
    W = [rng.normal(0.0, 0.06 * math.sqrt(2.0 / i), (i, o)) for i, o in dims]
    b = [np.zeros(o) for _, o in dims]
    for j, (f, sign) in enumerate([(6, 1.0), (6, -1.0), (7, 1.0), (7, -1.0), (4, 1.0), (4, -1.0)]):
        W[0][f, j] += sign
        for layer in W[1:4]:
            layer[j, j] += 1.0
    for a, (turn, climb) in enumerate(actions):
        c, s = math.cos(math.radians(turn)), math.sin(math.radians(turn))
        for j, w in enumerate((30.0 * c, -30.0 * c, 30.0 * s, -30.0 * s, climb, -climb)):
            W[4][j, a] += w
        b[4][a] -= 0.1 * climb * climb
    return np.concatenate([np.concatenate([w.ravel(), v]) for w, v in zip(W, b)]).astype(np.float32)


@pytest.fixture(scope="module")
def proposals():
    sc = S.c1_plain_small()
    rng = np.random.default_rng(2)
    reqs = S.make_requests(rng, sc.box, N, zlo=50.0, zhi=450.0, tlo=0, thi=600, horizon=900)
    reqs["horizon"][11] = 0
    with Scheduler.from_scenario(sc) as s:
        params = steering(sc.actions, 4)
        assert params.size == MLP_PARAMS
        s.learned_set_params(params)

        def evaluate(r):
            rep, accepted, steps, _ = s.learned_evaluate(r, slack=0.2)
            return rep["proposals_captured"], np.asarray(accepted), np.asarray(steps)

        parts = [evaluate(reqs[i:i + 40]) for i in range(0, N, 40)]
        yield evaluate, reqs, sum(p[0] for p in parts), *(np.concatenate([p[k] for p in parts]) for k in (1, 2))


def test_the_proposals_tell_rows_apart(proposals):
    """Over a thousand of them reach their goal, each after its own number of steps; the others fly to
    their horizon."""
    _, reqs, captured, accepted, steps = proposals
    assert captured > 1000 and 0 < accepted.sum() < captured
    assert (steps < reqs["horizon"]).sum() >= 1000 and len(np.unique(steps)) > 200


@pytest.mark.parametrize("n", [1, 17, 609, 1825, 2433, 2918, 2919, 4864, 4865, N])
def test_every_form_gives_the_same_proposals(proposals, n):
    evaluate, reqs, _, accepted, steps = proposals
    _, got_accepted, got_steps = evaluate(reqs[:n])
    np.testing.assert_array_equal(got_steps, steps[:n])
    np.testing.assert_array_equal(got_accepted, accepted[:n])
