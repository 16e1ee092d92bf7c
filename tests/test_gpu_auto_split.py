"""The list split that launches of small trees choose themselves: the number of
parts on both sides of the rule's bounds in items and particles, every staging mode, the
allocation-free call and a user's own stream capture; and source chunks whose
leaves are shorter and longer than a chunk."""
import numpy as np
import pytest

import oracle as O
from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL_RMS = 1e-5


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()
    return t


def _dev(torch, T, eps=0.01, theta=0.6):
    out = torch.empty((T.n, 4), dtype=torch.float32, device="cuda")
    T.forces_device(eps, theta, out)
    torch.cuda.synchronize()
    assert T.status() == G.OK
    return out.cpu().numpy()


def _clumps(items, per_item, seed):
    """`items` clumps of `per_item` particles: one work item each."""
    rng = np.random.default_rng(seed)
    c = rng.random((items, 3)) * 100
    return (np.repeat(c, per_item, 0) + 1e-4 * rng.random((items * per_item, 3))), rng.random(items * per_item)


@pytest.mark.parametrize("items,per_item,parts", [
    (49, 20, 1), (50, 20, 8), (580, 20, 8), (581, 20, 4), (1300, 20, 4), (1301, 20, 2), (3200, 20, 2), (3201, 20, 1),
    (111, 9, 1), (112, 9, 8), (170, 6, 8), (200, 6, 4), (500, 6, 2), (1010, 6, 2), (1011, 6, 1), (500, 5, 1)])
def test_parts_by_number_and_size_of_items(torch, items, per_item, parts):
    """Both sides of the rule's bounds: the launch equals that of the number of
    parts that the rule states, and the unsplit one within FP32 rounding."""
    pos, m = _clumps(items, per_item, 2 * items + per_item)
    n_leaf = per_item
    T = G.Tree.build_gpu(pos, m, n_leaf, n_leaf)
    assert T.stats["n_items"] == items
    auto = _dev(torch, T)
    c = T.interaction_counts()
    T.set_split(parts)
    assert np.array_equal(_dev(torch, T).view(np.uint32), auto.view(np.uint32))
    T.set_split(1)
    one = _dev(torch, T)
    assert T.interaction_counts() == c
    ref = O.Tree(pos, m, n_leaf, n_leaf).forces(0.01, 0.6)
    for a in (auto, one):
        acc, pot = np.empty((len(m), 3)), np.empty(len(m))
        acc[T.perm()], pot[T.perm()] = a[:, :3], a[:, 3]
        assert O.rel_rms(acc, ref[0]) <= TOL_RMS
        assert np.linalg.norm(pot - ref[1]) <= TOL_RMS * np.linalg.norm(ref[1])


def test_small_systems_of_a_batch_are_not_split(torch):
    systems = [_clumps(40, 20, k) for k in range(3)]
    T = G.Tree.build_batch(systems, 20, 20)
    assert T.stats["n_items"] == 120
    auto = _dev(torch, T)
    T.set_split(1)
    assert np.array_equal(_dev(torch, T).view(np.uint32), auto.view(np.uint32))


def test_staging_modes_and_noalloc_agree(torch):
    pos, m = W.plummer(5000, seed=4)
    T = G.Tree.build_gpu(pos, m, 16, 64)
    ref = _dev(torch, T)
    for stage in (0, 2):
        T.set_staging(stage)
        assert np.array_equal(_dev(torch, T).view(np.uint32), ref.view(np.uint32))
    T.set_staging(1)
    arena = torch.empty(T.noalloc_arena_bytes(), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        out = torch.full((T.n, 4), float("nan"), dtype=torch.float32, device="cuda")
        T.forces_noalloc(0.01, 0.6, out, arena)
        assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("ppl", [2, 1])
def test_first_launch_inside_a_stream_capture(torch, ppl):
    """A new tree's first launch may be one that a program captures itself: it
    allocates nothing (the launch configuration comes from another tree)."""
    pos, m = W.plummer(5000, seed=5)
    first = G.Tree.build_gpu(pos, m, 16, 64)
    first.set_launch(ppl)
    ref = _dev(torch, first)
    T = G.Tree.build_gpu(pos, m, 16, 64)
    T.set_launch(ppl)
    out = torch.zeros((T.n, 4), dtype=torch.float32, device="cuda")
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=st):
        T.forces_device(0.01, 0.6, out, stream=torch.cuda.current_stream())
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.view(np.uint32))


@pytest.mark.parametrize("n_leaf", [1, 31, 32, 33, 100])
def test_leaves_shorter_and_longer_than_a_source_chunk(n_leaf):
    pos, m = W.clustered(6000, 5, seed=n_leaf)
    T = G.Tree.build(pos, m, n_leaf, max(64, n_leaf))
    acc, pot = T.forces(0.01, 0.6)
    R = O.Tree(pos, m, n_leaf, max(64, n_leaf))
    ra, rp, npp, npc, _ = R.forces(0.01, 0.6)
    assert O.rel_rms(acc, ra) <= TOL_RMS
    assert np.linalg.norm(pot - rp) <= TOL_RMS * np.linalg.norm(rp)
    c = T.interaction_counts()
    assert c["n_pp"] == int(npp.sum()) and c["n_pc"] == int(npc.sum())
