"""The direct sum's source chunks follow the grid: sizes on both sides of the
rule's bounds (few targets: many small chunks; many targets: few chunks)."""
import numpy as np
import pytest

import oracle as O
from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()


@pytest.mark.parametrize("n,nt", [(255, 1), (257, 256), (77825, 257), (20000, 1025), (20011, 20011)])
def test_direct_sum_at_the_chunk_bounds(n, nt):
    """FP64 sums of positive-mass terms: 1e-12 of the largest result covers
    n roundings of 1.1e-16 with a factor of 100 to spare."""
    pos, m = W.galaxy(n, seed=n)
    samp = W.sample_indices(n, nt, seed=2)
    a, p = G.direct(pos, m, 0.02, targets=None if nt == n else samp)
    check = W.sample_indices(nt, min(nt, 300), seed=4)
    ra, rp = O.direct(pos, m, 0.02, targets=samp[check])
    assert np.abs(a[check] - ra).max() <= 1e-12 * np.abs(ra).max()
    assert np.abs(p[check] - rp).max() <= 1e-12 * np.abs(rp).max()
