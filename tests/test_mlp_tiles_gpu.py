"""The network kernels at the edges of their tiles: row tiles of 64 and 16 and
their remainders, widths that are no multiple of 4 or 32, an output layer on
either side of the narrow form (8 outputs), one to seven hidden layers; more
rows than max_batch in predict; a training step that uses the copy of the
weights the step before renewed.

Tolerances as in test_mlp_gpu: FP32 sums of up to 128 products against FP64,
1e-5 of the largest output; gradients, sums over the minibatch of such
products, 1e-4 of the largest component."""
import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members,shape,batch", [
    (1, (1, 1, 1, 1), 1),        # smallest of everything
    (3, (5, 128, 3, 2), 65),     # 64 + 1 rows, 16 x 4 + 1
    (160, (5, 40, 2, 2), 63),    # enough members for the 64-row tiles
    (2, (7, 33, 2, 8), 17),      # odd widths, widest narrow output
    (2, (3, 100, 1, 9), 16),     # first output count of the tiled form
    (80, (6, 66, 2, 12), 130),   # 64-row tiles, tiled output
    (1, (128, 128, 7, 128), 50),  # the largest shape (shared memory)
])
def test_forward_gradient_and_step(members, shape, batch):
    from paper_2311_15242_gb300 import Mlp
    rng = np.random.default_rng(members + batch)
    d = M.dims(*shape)
    m = Mlp(members, *shape, max_batch=batch)
    th = rng.normal(0, 1.0 / np.sqrt(shape[1]), (members, m.P)).astype(np.float32)
    m.set_params(th)
    x = rng.normal(size=(members, batch, d[0])).astype(np.float32)
    t = rng.normal(size=(members, batch, d[-1])).astype(np.float32)
    y = m.forward(x)
    loss, g = m.gradient(x, t)
    for e in (0, members - 1):
        yo, _, _ = M.forward(th[e].astype(np.float64), d, x[e])
        assert np.abs(y[e] - yo).max() <= 1e-5 * np.abs(yo).max()
        Lo, go = M.gradient(th[e].astype(np.float64), d, x[e], t[e])
        assert loss[e] == pytest.approx(Lo, rel=1e-5)
        assert np.abs(g[e] - go).max() <= 1e-4 * np.abs(go).max()
    # one training step on a data set of one row is Adam's step on that row
    # repeated; the forward pass that follows uses the renewed weights
    m.set_data(x[0, :1], t[0, :1])
    m.train(1, batch, 1e-3, seed=1)
    p = m.params()
    rows = np.repeat(x[0, :1], batch, 0)
    e = members - 1
    _, go = M.gradient(th[e].astype(np.float64), d, rows, np.repeat(t[0, :1], batch, 0))
    ref, _, _ = M.adam(th[e].astype(np.float64), go, 0 * go, 0 * go, 1, 1e-3)
    # (the first step is lr g / (|g| + eps): only where g is clear of rounding)
    clear = np.abs(go) > 1e-3 * np.abs(go).max()
    assert np.abs(p[e] - ref)[clear].max() <= 2e-6
    assert np.array_equal(m.forward(x)[e], fresh_forward(m, shape, batch, p, x)[e])


def fresh_forward(m, shape, batch, p, x):
    from paper_2311_15242_gb300 import Mlp
    n = Mlp(m.E, *shape, max_batch=batch)
    n.set_params(p)
    return n.forward(x)


@pytest.mark.parametrize("n", [1, 64, 65, 1000, 70000])
def test_predict_chunks(n):
    """Rows in one launch, or in chunks when there are more than max_batch
    (65,536 a chunk): the same outputs as a network that takes them whole."""
    from paper_2311_15242_gb300 import Mlp
    shape, E = (5, 32, 2, 2), 3
    rng = np.random.default_rng(n)
    m = Mlp(E, *shape, max_batch=64)
    th = rng.normal(0, 0.2, (E, m.P)).astype(np.float32)
    m.set_params(th)
    x = rng.normal(size=(n, 5)).astype(np.float32)
    mean, sd = m.predict(x, bf16=False)
    d = M.dims(*shape)
    mu, s = M.ensemble_stats([M.forward(th[e].astype(np.float64), d, x)[0] for e in range(E)])
    assert np.abs(mean - mu).max() <= 1e-5 * np.abs(mu).max()
    assert np.abs(sd - s).max() <= 1e-5 * np.abs(mu).max()
