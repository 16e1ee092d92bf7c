"""The level and node kernels of the GPU build where their rules change: cells
of 32 and 33 particles (one probe per particle or a search), levels that end at
the depth limit, trees of one block and of many, more nodes on a level than
eight-lane groups take, the most chunks that are sorted in one launch, and groups
and items on both sides of a block's range. Byte equality with the host build throughout."""
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


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 34, 255, 256, 257, 4095, 4097])
@pytest.mark.parametrize("n_leaf", [1, 8])
def test_small_trees(n, n_leaf):
    pos, m = W.uniform_cube(n, seed=n)
    _same(pos, m, n_leaf, 8 * n_leaf)


@pytest.mark.parametrize("count", [32, 33, 1057, 1088, 1089])
def test_cells_at_the_probe_bounds(count):
    """One octant holds all but one particle: the first cells hold `count` and
    fewer particles, on both sides of one round (32) and two (33 x 32 + 32)."""
    rng = np.random.default_rng(count)
    pos = rng.random((count, 3)) * 0.25
    pos[0] = 1.0
    _same(pos, np.full(count, 1.0 / count), 1, 4)


def test_depth_limit_and_massless_nodes():
    """Coincident particles below the depth limit (every level has one node),
    and nodes whose children have no mass."""
    rng = np.random.default_rng(3)
    pos = rng.random((3000, 3))
    pos[:40] = pos[0]
    m = np.full(3000, 1e-3)
    m[pos[:, 0] < 0.5] = 0.0
    B = _same(pos, m, 4, 16)
    assert B.stats["depth"] == G.MAX_DEPTH


def test_more_nodes_on_a_level_than_eight_lane_groups_take():
    """N_leaf = 1: tens of thousands of nodes on a level take the kernel's
    lane-per-node form, the levels above it the eight-lane form."""
    pos, m = W.plummer(120000, seed=6)
    B = _same(pos, m, 1, 32)
    depth = np.floor(np.log2(B.cell_keys().astype(np.float64)) / 3)
    counts = B.cell_props()["count"]
    assert max(int(np.sum((depth == d) & (counts > 1))) for d in range(22)) > 4 * 4 * 608


@pytest.mark.parametrize("n", [1023, 1025, 3073, 8 * 4096, 8 * 4096 + 1, 64 * 4096, 64 * 4096 + 1])
def test_sort_in_one_launch_and_in_passes(n):
    """The last sizes that one launch sorts with four and with two blocks a chunk
    and the first that they do not, and chunks whose last blocks are empty."""
    rng = np.random.default_rng(n)
    _same(rng.random((n, 3)) ** 3, rng.random(n), 16, 64)


@pytest.mark.parametrize("sizes", [[1, 4096, 4097, 2, 9000], [1, 1, 4096, 4097, 2], [64] * 64, [64] * 65])
def test_sort_of_several_systems(sizes):
    """Every system is sorted by itself, whatever its number of chunks; 64 chunks
    take the one launch and 65 do not."""
    rng = np.random.default_rng(len(sizes))
    systems = [(rng.random((k, 3)), rng.random(k)) for k in sizes]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    A = G.Tree.build_batch(systems, 8, 32)
    B = G.Tree.build_gpu(np.concatenate([p for p, _ in systems]), np.concatenate([m for _, m in systems]), 8, 32,
                         offsets=offs)
    assert A.stats == B.stats
    assert np.array_equal(A.perm(), B.perm()) and np.array_equal(A.cell_keys(), B.cell_keys())


def _same_items(A, B):
    a, b = A.item_info(), B.item_info()
    assert A.stats == B.stats and a.keys() == b.keys()
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("n", [1, 255, 256, 257, 608 * 256, 608 * 256 + 1])
@pytest.mark.parametrize("n_group", [1, 8, 300])
def test_groups_and_items(n, n_group):
    """One particle range per block of the group kernel and two, groups of one
    particle and of more than an item holds, and items cut anew."""
    pos, m = W.plummer(n, seed=n)
    A, B = G.Tree.build(pos, m, min(8, n_group), n_group), G.Tree.build_gpu(pos, m, min(8, n_group), n_group)
    _same_items(A, B)
    for ppl in (1, 2):
        A.set_launch(ppl)
        B.set_launch(ppl)
        _same_items(A, B)


def test_groups_of_several_systems_and_of_coincident_particles():
    rng = np.random.default_rng(8)
    systems = [(rng.random((k, 3)), rng.random(k)) for k in (700, 1, 3000, 257)]
    systems[2][0][:900] = systems[2][0][0]
    offs = np.array([0, 700, 701, 3701, 3958], np.int64)
    A = G.Tree.build_batch(systems, 8, 64)
    B = G.Tree.build_gpu(np.concatenate([p for p, _ in systems]), np.concatenate([m for _, m in systems]), 8, 64,
                         offsets=offs)
    _same_items(A, B)
