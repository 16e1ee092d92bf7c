"""The level kernel of the GPU build where its rules change: cells on both sides
of 128 particles (all keys at once, or a search), trees on both sides of four
million particles (one range of a level a block, or several), levels that take
up to a dozen of them, and a level that overflows the cell capacity in them.
Byte equality with the host build throughout."""
import numpy as np
import pytest

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


def _same(pos, m, n_leaf, n_group):
    A, B = G.Tree.build(pos, m, n_leaf, n_group), G.Tree.build_gpu(pos, m, n_leaf, n_group)
    assert A.stats == B.stats
    assert np.array_equal(A.perm(), B.perm()) and np.array_equal(A.cell_keys(), B.cell_keys())
    a, b = A.cell_props(), B.cell_props()
    for k in a:
        assert np.array_equal(a[k].view(np.uint64), b[k].view(np.uint64)), k
    return B


@pytest.mark.parametrize("n_leaf", [1, 31, 64, 127, 128])
@pytest.mark.parametrize("count", [33, 64, 65, 96, 97, 127, 128, 129, 130, 160])
def test_cells_at_the_bounds_of_the_keys_loaded_at_once(count, n_leaf):
    """Cells of `count` particles side by side, so that one's keys are loaded while
    another is split, among cells above and below the bounds."""
    rng = np.random.default_rng(count)
    corners = np.array([[x, y, z] for x in (0, 1) for y in (0, 1) for z in (0, 1)], float)
    sizes = [count, 1, count, 129, count, 33, count, 500]
    pos = np.concatenate([c + 0.4 * rng.random((k, 3)) for c, k in zip(corners, sizes)])
    _same(pos, rng.random(len(pos)), n_leaf, 4 * n_leaf)


@pytest.mark.parametrize("n,n_leaf,clustered", [(3999999, 16, False), (4000000, 16, False), (4200001, 1, True)])
def test_trees_at_the_bound_of_several_ranges(n, n_leaf, clustered):
    pos, m = W.clustered(n, seed=n_leaf) if clustered else W.plummer(n, seed=n_leaf)
    _same(pos, m, n_leaf, 64)


def test_a_level_of_several_ranges_that_overflows(monkeypatch):
    """The capacity ends on a level of some hundred thousand cells; the build enlarges
    it and starts again."""
    pos, m = W.plummer(4000000, seed=1)
    monkeypatch.setenv("OCTGRAV_GPU_CELL_CAP", "300000")
    B = _same(pos, m, 16, 64)
    assert B.stats["n_cells"] > 4 * 150000
