"""A tree freed on one thread while another thread captures a stream: the
capture ends and replays, and the tree's buffers serve the next tree."""
import threading

import numpy as np
import pytest

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
def test_a_tree_freed_during_another_threads_capture(mode):
    torch = pytest.importorskip("torch")
    G.load()
    pos, m = W.plummer(20000, seed=2)
    T, other = (G.Tree.build_gpu(pos, m, 16, 64) for _ in range(2))
    ref, out = (torch.zeros((T.n, 4), dtype=torch.float32, device="cuda") for _ in range(2))
    T.forces_device(0.01, 0.6, ref)
    other.forces_device(0.01, 0.6, out)
    torch.cuda.synchronize()
    out.zero_()
    st = torch.cuda.Stream()
    st.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()

    def free():
        torch.cuda.set_device(0)
        other.free()
    with torch.cuda.graph(g, stream=st, capture_error_mode=mode):
        t = threading.Thread(target=free)
        t.start()
        t.join()
        T.forces_device(0.01, 0.6, out, stream=torch.cuda.current_stream())
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint32), ref.cpu().numpy().view(np.uint32))
    again = torch.zeros_like(ref)
    G.Tree.build_gpu(pos, m, 16, 64).forces_device(0.01, 0.6, again)
    assert torch.equal(again.view(torch.int32), ref.view(torch.int32))
