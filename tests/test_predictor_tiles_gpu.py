"""The predictor's products at the size from which a warp takes the wider tile
(8,192 rows by 128 columns) and around its edges: the same k order, so the rows of
one large call equal those of small calls bit by bit, and the gradient of a large
batch is the mean of its parts'."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


@pytest.mark.parametrize("rows", [8_176, 8_177, 8_191, 8_192, 8_193, 20_001])
def test_wide_tiles_equal_small_tiles(rows):
    rng = np.random.default_rng(rows)
    x = torch.from_numpy(rng.normal(size=(rows, ae.MLP_IN)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=(rows, ae.MLP_OUT)).astype(np.float32)).cuda()
    m = ae.Mlp(5)
    m.set_norm(np.linspace(-1, 1, ae.MLP_IN), np.linspace(0.5, 2, ae.MLP_IN), [0.1, -0.2], [1.5, 0.7])
    y = torch.empty(rows, ae.MLP_OUT, device="cuda")
    m.forward(x.data_ptr(), rows, y.data_ptr())
    part = torch.empty_like(y)
    loss, grad = m.loss_grad(x.data_ptr(), t.data_ptr(), rows)
    sum_loss, sum_grad = 0.0, np.zeros(ae.MLP_PARAMS)
    for r in range(0, rows, 1_000):
        n = min(1_000, rows - r)
        m.forward(x[r:].data_ptr(), n, part[r:].data_ptr())
        pl, pg = m.loss_grad(x[r:].data_ptr(), t[r:].data_ptr(), n)
        sum_loss += pl * n
        sum_grad += pg.astype(np.float64) * n
    assert torch.equal(y, part)
    # fp32 sums of `rows` products of bf16 values in another order, and the scale 1 / rows of the
    # output gradient rounded to bf16 with it: 2^-8 of the mean magnitude of a term at most
    assert abs(loss - sum_loss / rows) <= 1e-5 * abs(loss)
    want = sum_grad / rows
    assert np.abs(grad - want).max() <= 2.0 ** -8 * np.abs(want).max()
