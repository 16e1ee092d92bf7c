"""The list split that launches of small trees choose themselves: the number of
parts on both sides of the rule's bounds, every staging mode, the
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


@pytest.mark.parametrize("items,parts", [(1, 8), (637, 8), (638, 4), (1275, 4), (1276, 2), (2550, 2), (2551, 1)])
def test_parts_by_number_of_items(torch, items, parts):
    """One particle per leaf and group on a line: one work item per particle."""
    pos = np.zeros((items, 3))
    pos[:, 0] = np.arange(items) + 0.25 * np.sin(np.arange(items))
    m = np.full(items, 1.0 / items)
    T = G.Tree.build_gpu(pos, m, 1, 1)
    assert T.stats["n_items"] == items
    auto = _dev(torch, T)
    c = T.interaction_counts()
    T.set_split(parts)
    assert np.array_equal(_dev(torch, T).view(np.uint32), auto.view(np.uint32))
    T.set_split(1)
    one = _dev(torch, T)
    assert T.interaction_counts() == c
    ref = O.Tree(pos, m, 1, 1).forces(0.01, 0.6)
    for a in (auto, one):
        acc, pot = np.empty((items, 3)), np.empty(items)
        acc[T.perm()], pot[T.perm()] = a[:, :3], a[:, 3]
        if items > 1:
            assert O.rel_rms(acc, ref[0]) <= TOL_RMS
            assert np.linalg.norm(pot - ref[1]) <= TOL_RMS * np.linalg.norm(ref[1])


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
