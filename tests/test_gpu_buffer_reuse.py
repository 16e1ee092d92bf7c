"""Trees that take over a freed tree's device buffers: other sizes, other
kinds of tree, a criterion set before the upload, several threads and streams.
Forces must be bit for bit those of the first, fresh tree of each input."""
import threading

import numpy as np
import pytest

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()
    return t


def _forces(torch, pos, m, gpu, stream=None):
    T = (G.Tree.build_gpu if gpu else G.Tree.build)(pos, m, 16, 64)
    out = torch.empty((T.n, 4), dtype=torch.float32, device="cuda")
    T.forces_device(0.01, 0.6, out, stream=stream)
    (stream or torch.cuda.current_stream()).synchronize()
    assert T.status() == G.OK
    return out.cpu().numpy()


def test_sizes_and_kinds_in_turn(torch):
    inputs = [W.plummer(n, seed=n) for n in (30000, 700, 12001, 50000)]
    first = [_forces(torch, *i, gpu=True) for i in inputs]
    for gpu in (True, False, True):
        for i, ref in zip(inputs[::-1], first[::-1]):
            assert np.array_equal(_forces(torch, *i, gpu=gpu).view(np.uint32), ref.view(np.uint32))


def test_criterion_set_before_the_upload_survives(torch):
    """A host-built tree whose criterion is set before its first launch, once
    with no idle buffers for it and once with a freed tree's."""
    import oracle.mlp as M
    pos, m = W.plummer(20000, seed=8)
    rec = np.concatenate([np.zeros(12), np.full(12, 3.0), np.full(12, -1e3), np.full(12, 1e3), M.init(5)]).astype(np.float32)

    def run():
        T = G.Tree.build(pos, m, 16, 128)
        T.set_criterion(rec, tau=0.0, theta_lo=0.5, theta_hi=1.2, theta_fb=0.8)
        return T.forces(0.01, 0.6)[0]
    ref = run()
    _forces(torch, pos, m, gpu=True)
    assert np.array_equal(run(), ref)


def test_a_live_tree_keeps_its_buffers(torch):
    """A freed tree's buffers go to one new tree only; trees alive at the same
    time, on several threads with their own streams, do not share any."""
    inputs = [W.plummer(4000 + 500 * k, seed=k) for k in range(4)]
    ref = [_forces(torch, *i, gpu=True) for i in inputs]
    bad = []

    def work(k):
        st = torch.cuda.Stream()
        for _ in range(8):
            if not np.array_equal(_forces(torch, *inputs[k], gpu=True, stream=st), ref[k]):
                bad.append(k)
    threads = [threading.Thread(target=work, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad


def test_a_refused_build_gives_its_buffers_back(torch):
    pos, m = W.plummer(200000, seed=2)
    bad = pos.copy()
    bad[5, 1] = np.nan
    free = []
    for _ in range(6):
        with pytest.raises(G.OctgravError) as e:
            G.Tree.build_gpu(bad, m, 16, 64)
        assert e.value.code == G.ERR_NONFINITE
        torch.cuda.synchronize()
        free.append(torch.cuda.mem_get_info()[0])
    assert free[-1] >= free[1] - (32 << 20)
