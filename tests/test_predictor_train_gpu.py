"""A training run against its restatement on the host: the same permutation of the
rows, the batches' gradients (ae_mlp_loss_grad, tested against the oracle) and Adam,
with normalisations that matter, a last batch of one row, several epochs and weight
decay."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from oracle import mlp_oracle as mo  # noqa: E402
from paper_1208_0274_gb300 import ae  # noqa: E402

M64 = (1 << 64) - 1


def _splitmix(state):
    state = (state + 0x9E3779B97F4A7C15) & M64
    z = state
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & M64
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & M64
    return state, z ^ (z >> 31)


@pytest.mark.parametrize("rows,batch,epochs,wd", [(257, 128, 1, 0.0), (100, 33, 2, 0.05), (65, 64, 1, 0.1), (1, 8, 3, 0.0)])
def test_training_run(rows, batch, epochs, wd):
    rng = np.random.default_rng(rows)
    x_mu, x_sd = rng.normal(size=ae.MLP_IN), rng.uniform(0.3, 3.0, size=ae.MLP_IN)
    X = (x_mu + x_sd * rng.normal(size=(rows, ae.MLP_IN))).astype(np.float32)
    T = rng.normal(loc=4.0, size=(rows, ae.MLP_OUT)).astype(np.float32)
    lr, seed = 1e-3, 17
    m = ae.Mlp(3)
    m.set_norm(x_mu, x_sd, [3.5, 4.5], [1.5, 0.7])
    p0 = m.get_params()
    dx, dt = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    loss = m.train(dx.data_ptr(), dt.data_ptr(), rows, epochs, batch, lr, wd, seed)
    got = m.get_params()

    ref = ae.Mlp(3)
    ref.set_norm(x_mu, x_sd, [3.5, 4.5], [1.5, 0.7])
    p = p0.astype(np.float64)
    am, av, t, state = np.zeros_like(p), np.zeros_like(p), 0, seed
    for _ in range(epochs):
        perm = np.arange(rows)
        for i in range(rows - 1, 0, -1):
            state, z = _splitmix(state)
            j = z % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        losses = []
        for r in range(0, rows, batch):
            b = perm[r:r + batch]
            bx, bt = torch.from_numpy(X[b]).cuda(), torch.from_numpy(T[b]).cuda()
            ref.set_params(p.astype(np.float32))
            bl, g = ref.loss_grad(bx.data_ptr(), bt.data_ptr(), len(b))
            losses.append(bl)
            t += 1
            g = g.astype(np.float64)
            am = 0.9 * am + 0.1 * g
            av = 0.999 * av + 0.001 * g * g
            p = p - lr * ((am / (1 - 0.9 ** t)) / (np.sqrt(av / (1 - 0.999 ** t)) + 1e-8) + wd * p)
    # a weight that rounds to another bf16 value moves a gradient by up to 2^-8 of one of its terms,
    # and Adam's step by as much of lr where that term is all there is; another batch or another
    # normalisation moves most parameters by lr itself
    d = np.abs(got - p)
    assert np.quantile(d, 0.99) <= 0.05 * lr and np.abs(got - p0).max() > 0.5 * lr
    assert abs(loss - np.mean(losses)) <= 1e-3 * abs(loss)
    assert mo.n_params() == got.size
