"""Builds and training on one stream while a kernel of one block runs on another:
their cooperative launches leave it its place and do not wait for it."""
import numpy as np
import pytest

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CYCLES = 4_000_000_000  # about two seconds; the calls take milliseconds


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()
    return t


def _beside(torch, call):
    """call(), once alone and once beside the other stream's kernel; both results."""
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(mine):
        alone = call()                      # what it keeps is allocated now
        torch.cuda.synchronize()
        with torch.cuda.stream(other):
            torch.cuda._sleep(CYCLES)
        beside = call()
    mine.synchronize()
    assert not other.query()
    torch.cuda.synchronize()
    return alone, beside


@pytest.mark.parametrize("n,systems", [(5000, 1), (200000, 1), (300000, 1), (2000000, 1), (4000000, 1), (500000, 200)])
def test_build(torch, n, systems):
    pos, m = W.plummer(n, seed=1)
    x, w = torch.from_numpy(pos).cuda(), torch.from_numpy(m).cuda()
    off = np.linspace(0, n, systems + 1).astype(np.int64) if systems > 1 else None
    A, B = _beside(torch, lambda: G.Tree.build_gpu(x, w, 16, 64, offsets=off))
    assert A.stats == B.stats and np.array_equal(A.perm(), B.perm())


@pytest.mark.parametrize("batch", [256, 4096, 30000])
def test_training(torch, batch):
    rng = np.random.default_rng(1)
    f, y = rng.standard_normal((30000, 12)).astype(np.float32), rng.random(30000).astype(np.float32)
    (a, _), (b, _) = _beside(torch, lambda: G.mlp_train(f, y, steps=3, batch=batch))
    assert np.array_equal(a, b)
