"""Forces in other units of length. Scaling every position and eps by a power
of two scales each FP32 operation of the evaluation exactly as long as nothing
leaves the normal range, so the results may differ from those at scale one by
no more than roundings of the reciprocal square root: 1e-6 (FP32 has 6e-8)."""
import numpy as np
import pytest

from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-6


@pytest.fixture(scope="module", autouse=True)
def torch():
    t = pytest.importorskip("torch")
    if not t.cuda.is_available():
        pytest.skip("no CUDA device")
    G.load()
    return t


def _scaled(torch, k, ppl, split):
    """Accelerations and potentials of one system at scale 2^k, in the units of scale one."""
    pos, m = W.plummer(20000, seed=3)
    T = G.Tree.build(pos * 2.0 ** k, m, 16, 64)
    T.set_launch(ppl)
    T.set_split(split)
    out = torch.empty((T.n, 4), dtype=torch.float32, device="cuda")
    T.forces_device(0.01 * 2.0 ** k, 0.5, out)
    assert T.status() == G.OK
    a = out.cpu().numpy().astype(np.float64)
    return a[:, :3] * 4.0 ** k, a[:, 3] * 2.0 ** k


def _close(a, b):
    return np.linalg.norm(a - b) <= TOL * np.linalg.norm(b)


@pytest.mark.parametrize("split", [1, 4])
@pytest.mark.parametrize("ppl", [1, 2])
@pytest.mark.parametrize("k", [-20, -12, 12, 24, 28])
def test_potentials(torch, k, ppl, split):
    assert _close(_scaled(torch, k, ppl, split)[1], _scaled(torch, 0, ppl, split)[1])


@pytest.mark.parametrize("split", [1, 4])
@pytest.mark.parametrize("k", [-20, -12, 12, 24, 28])
def test_accelerations_with_one_particle_per_lane(torch, k, split):
    assert _close(_scaled(torch, k, 1, split)[0], _scaled(torch, 0, 1, split)[0])


@pytest.mark.parametrize("k", [-16, 16])
def test_accelerations_with_two_particles_per_lane(torch, k):
    """The stated range of this layout: softened distances from 1e-7 up, 1e7 at most."""
    assert _close(_scaled(torch, k, 2, 1)[0], _scaled(torch, 0, 2, 1)[0])


@pytest.mark.parametrize("split", [2, 4, 16])
def test_results_beyond_the_largest_number_are_infinite(torch, split):
    """G (finite in FP32: the mass is 16) times a potential that overflows, and
    parts whose sum does."""
    pos, m = W.plummer(5000, seed=3)
    T = G.Tree.build(pos, 16.0 * m, 16, 64)
    T.set_split(1)
    out = torch.empty((T.n, 4), dtype=torch.float32, device="cuda")
    T.forces_device(0.01, 0.5, out)
    phi = out[:, 3].double().cpu().numpy()
    big = 3.4028235e38
    g = 1.2 * big / float(np.abs(phi).max())        # some potentials beyond the range, their parts mostly within
    T.set_split(split)
    T.forces_device(0.01, 0.5, out, G=g)
    got = out[:, 3].cpu().numpy()
    beyond = g * np.abs(phi) > 1.00001 * big
    within = g * np.abs(phi) < 0.99999 * big
    assert g < big and beyond.any() and np.isneginf(got[beyond]).all() and np.isfinite(got[within]).all()
