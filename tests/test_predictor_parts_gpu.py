"""The predictor's features where a query's parts can go wrong: lengths around
one part of 256 positions and many parts, empty queries between others, many
short queries, and a training step whose products split their sums (128 rows)
beside ones that do not."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo
from workloads import dna_scale_query, dna_scale_text

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_1208_0274_gb300 import ae  # noqa: E402


@pytest.mark.parametrize("lengths", [
    (0, 255, 0, 0, 256, 257, 0),
    (258, 511, 513, 30_000, 1),
    tuple([3, 20, 0, 40] * 100),
])
def test_features_of_parts(lengths):
    text = dna_scale_text(seed=31, n=50_000)
    idx = ae.ae_index_build(text, ae.AE_DNA)
    rng = np.random.default_rng(len(lengths))
    qs = [dna_scale_query(text, m, rng)[0] if m else np.zeros(0, np.uint8) for m in lengths]
    off = np.concatenate([[0], np.cumsum([q.size for q in qs])]).astype(np.int64)
    seq = torch.from_numpy(np.concatenate(qs)).cuda()
    feat = torch.full((len(qs), ae.MLP_IN), 9.0, device="cuda")
    ae.ae_mlp_features(idx, seq.data_ptr(), off, feat.data_ptr())
    got = feat.cpu().numpy()
    idx.close()
    some = [k for k, q in enumerate(qs) if q.size]
    want = mo.features(text, [qs[k] for k in some])
    assert np.allclose(got[some][:, :65], want[:, :65], rtol=1e-6, atol=1e-7)
    assert np.allclose(got[some][:, 65], want[:, 65], rtol=1e-5, atol=1e-6)
    assert not got[[k for k, q in enumerate(qs) if not q.size]].any()


@pytest.mark.parametrize("rows,batch", [(128, 128), (257, 128), (100, 112)])
def test_training_steps_equal_gradient_steps(rows, batch):
    # one epoch without weight decay from a training call equals Adam on the gradients of
    # the same batches only up to the batches' order: a single batch has none
    rng = np.random.default_rng(rows)
    X = rng.normal(size=(rows, ae.MLP_IN)).astype(np.float32)
    T = rng.normal(size=(rows, ae.MLP_OUT)).astype(np.float32)
    dx, dt = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    m = ae.Mlp(3)
    m.set_norm(np.zeros(ae.MLP_IN), np.ones(ae.MLP_IN), np.zeros(ae.MLP_OUT), np.ones(ae.MLP_OUT))
    p0 = m.get_params()
    _, g = m.loss_grad(dx.data_ptr(), dt.data_ptr(), rows)
    m.set_params(p0)
    m.train(dx.data_ptr(), dt.data_ptr(), rows, 1, rows, 1e-3, 0.0, 1)
    p1 = m.get_params()
    # Adam's first step moves every parameter by lr * g / (|g| + eps)
    big = np.abs(g) > 1e-4
    assert big.sum() > 1000
    assert np.allclose((p0 - p1)[big], 1e-3 * np.sign(g)[big], rtol=2e-3)
    m.set_params(p0)
    m.train(dx.data_ptr(), dt.data_ptr(), rows, 1, batch, 1e-3, 0.0, 1)
    assert np.isfinite(m.get_params()).all()
