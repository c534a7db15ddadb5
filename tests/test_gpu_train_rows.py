"""Loss and gradient at row counts around the kernels' tiles: one row, a block of 16 rows and
its neighbours, the first batch that is split over stretches, ragged stretches, the largest.

Up to 1025 rows against the oracle with the same bf16 roundings, with the bounds of the proposal network's
gradient test: an activation or output gradient may land on the other side of a bf16 rounding
boundary (2^-8 relative), so 2e-2 relative plus 2e-3 of a block's largest element. With 8192 x 1024
activations some lie within an fp32 rounding of zero, on the other side of the ReLU than the
oracle's FP64 sums, which moves an element by a row's whole share; so the largest batch is
compared with its eighths instead: rows are independent and division by 8 is exact, so every
bf16 value is the same and only the fp32 sums over rows differ (1e-4 covers them; a stretch
left out moves elements by their eighth).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import learned as OL  # noqa: E402
from paper_2008_03518_gb300 import scenarios as S  # noqa: E402
from paper_2008_03518_gb300.fmdp import Scheduler  # noqa: E402
from test_gpu_learned import _bias_blocks, _weight_blocks, bf16  # noqa: E402


@pytest.fixture(scope="module")
def net():
    sc = S.c1_plain_small()
    with Scheduler.from_scenario(sc) as s:
        s.learned_init(seed=5)
        yield s, len(sc.actions)


@pytest.mark.parametrize("rows", [1, 15, 16, 17, 127, 128, 129, 1025])
def test_gradient(net, rows):
    s, A = net
    rng = np.random.default_rng(rows)
    p = s.learned_get_params()
    X = rng.normal(0.0, 0.7, size=(rows, 128)).astype(np.float32)  # rounded to bf16 on the GPU
    y = rng.integers(0, A, size=rows).astype(np.uint8)
    loss, g = s.learned_loss_grad(X, y)
    again = s.learned_loss_grad(X, y)
    assert again[0] == loss and np.array_equal(again[1], g)  # sums in a fixed order
    q = p.astype(np.float64).copy()
    for o, n in _weight_blocks():
        q[o:o + n] = bf16(p[o:o + n])
    r_loss, r_g = OL.loss_and_grad(q, bf16(X).astype(np.float64), y, n_valid=A, round_fn=OL.bf16)
    assert abs(loss - r_loss) <= 1e-4 * r_loss
    for o, n in list(_weight_blocks()) + list(_bias_blocks()):
        scale = float(np.abs(r_g[o:o + n]).max())
        np.testing.assert_allclose(g[o:o + n], r_g[o:o + n], rtol=2e-2, atol=2e-3 * scale, err_msg=f"block at {o}")


def test_the_largest_batch_is_the_mean_of_its_parts(net):
    s, A = net
    rng = np.random.default_rng(8192)
    X = rng.normal(0.0, 0.7, size=(8192, 128)).astype(np.float32)
    y = rng.integers(0, A, size=8192).astype(np.uint8)
    loss, g = s.learned_loss_grad(X, y)
    parts = [s.learned_loss_grad(X[i:i + 1024], y[i:i + 1024]) for i in range(0, 8192, 1024)]
    assert abs(loss - np.mean([p[0] for p in parts])) <= 1e-5 * loss
    want = np.mean([p[1].astype(np.float64) for p in parts], axis=0)
    for o, n in list(_weight_blocks()) + list(_bias_blocks()):
        scale = float(np.abs(want[o:o + n]).max())
        np.testing.assert_allclose(g[o:o + n], want[o:o + n], rtol=1e-4, atol=1e-4 * scale, err_msg=f"block at {o}")
