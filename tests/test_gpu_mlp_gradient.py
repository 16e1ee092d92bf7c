"""The gradient kernel at the edges of its tiles (32 samples) and of its grid
(304 blocks, then several tiles per block), against the FP64 backward pass."""
import numpy as np
import pytest

import oracle.mlp as M
from paper_1005_5384_gb300 import octgrav as G

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("n", [1, 31, 32, 33, 304 * 32, 304 * 32 + 1, 2 * 304 * 32 + 45])
def test_gradient_at_tile_and_grid_edges(n):
    """Every entry is an FP32 sum of at most n / blocks + 304 terms below the
    row's largest, so 2e-5 of the largest entry covers its rounding; the sum
    over blocks has a fixed order, so a second call gives the same bits."""
    rng = np.random.default_rng(n)
    w = M.init(3).astype(np.float32)
    x = rng.standard_normal((n, 12)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    g, loss = G.mlp_grad(w, x, t)
    loss64, g64 = M.loss_and_grad(w.astype(np.float64), x.astype(np.float64), t.astype(np.float64))
    assert np.abs(g - g64).max() <= 2e-5 * np.abs(g64).max()
    assert abs(loss - loss64) <= 2e-5 * abs(loss64)
    g2, loss2 = G.mlp_grad(w, x, t)
    assert np.array_equal(g.view(np.uint32), g2.view(np.uint32)) and loss == loss2


@pytest.mark.parametrize("batch,steps", [(40, 3), (1000, 513), (20000, 20)])
def test_training_is_reproducible_and_lowers_the_loss(batch, steps):
    """Few blocks with many parameters each, a launch boundary (512 steps), and
    several tiles per block: the same record twice, a loss below the first's."""
    rng = np.random.default_rng(5)
    f = rng.standard_normal((30000, 12)).astype(np.float32)
    label = (10.0 ** (-3.0 + 0.3 * f[:, 0] - 0.2 * f[:, 3])).astype(np.float32)
    first = G.mlp_train(f, label, steps=1, batch=batch, seed=7)
    a = G.mlp_train(f, label, steps=steps, batch=batch, seed=7)
    b = G.mlp_train(f, label, steps=steps, batch=batch, seed=7)
    assert np.array_equal(a[0].view(np.uint32), b[0].view(np.uint32)) and a[1] == b[1]
    assert np.all(np.isfinite(a[0])) and a[1] < first[1]
