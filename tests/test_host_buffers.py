"""What the host library does with device buffers, stream captures and launch
settings, on the CPU: its host sources linked with stand-ins for the CUDA
runtime and the kernels (fake_device.cpp). No GPU takes part."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1005_5384_gb300 import build as B
from paper_1005_5384_gb300 import octgrav as G
from paper_1005_5384_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fake")
    srcs = [os.path.join(B.CSRC, s) for s in ("octgrav_host.cpp", "octgrav_host_build.cpp", "octgrav_host_mlp.cpp")]
    srcs.append(os.path.join(HERE, "fake_device.cpp"))
    objs = [str(d / (os.path.basename(s) + ".o")) for s in srcs]
    inc = ["-I", os.path.join(B._cuda_home(), "include"), "-I", B.INCLUDE, "-I", B.CSRC]
    procs = [subprocess.Popen(["g++", "-O1", "-std=c++17", "-fPIC", "-ffp-contract=off", "-pthread", "-Wno-psabi", *inc, "-c", s, "-o", o])
             for s, o in zip(srcs, objs)]
    assert all(p.wait() == 0 for p in procs)
    so = str(d / "libfake.so")
    subprocess.check_call(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so, *objs, "-lpthread", "-ldl"])
    lib = C.CDLL(so)
    for name, (res, args) in G._SIGS.items():
        f = getattr(lib, name)
        f.restype, f.argtypes = res, args
    lib.fake_used.restype = C.c_size_t
    lib.fake_set_limit.argtypes = [C.c_int, C.c_size_t]
    lib.fake_set_context.argtypes = [C.c_int, C.c_ulonglong]
    lib.fake_set_time.argtypes = [C.c_int, C.c_int, C.c_float]
    return lib


@pytest.fixture
def fake(fake_lib, monkeypatch):
    """The package on the stand-in library, with nothing allocated or kept."""
    monkeypatch.setattr(G, "_lib", fake_lib)
    monkeypatch.setattr(G, "_stream_handle", lambda stream: C.c_void_p(1))
    fake_lib.fake_reset()
    yield fake_lib
    for T in _made:
        T.free()
    _made.clear()
    assert fake_lib.fake_bad_frees() == 0


_made = []  # freed while the stand-in library is in place


def _tree(n, seed=1, n_group=64):
    pos, m = W.plummer(n, seed=seed)
    _made.append(G.Tree.build(pos, m, 16, n_group))
    return _made[-1]


def _upload(T):
    G._check(G.load().octgrav_tree_upload(T._h, None))
    return T


def _forces(T, theta=0.5):
    G._check(G.load().octgrav_forces_device(T._h, 0.01, theta, 1.0, C.c_void_p(256), None))


def _last(lib):
    v = (C.c_int * 3)()
    lib.fake_launch(lib.fake_launches() - 1, v)
    return dict(nparts=v[0], stage=v[1], ppl=v[2])


def test_freeing_a_tree_leaves_captures_alone(fake):
    """A tree may be freed while another thread captures a stream (a device-wide
    synchronisation would end that capture)."""
    T = _upload(_tree(2000))
    fake.fake_begin_capture()
    frees = fake.fake_frees()
    T.free()
    assert fake.fake_end_capture() == 0
    assert fake.fake_frees() > frees        # the wait that stands before any reuse


def _one_tree(n=3000, seed=1):
    T = _upload(_tree(n, seed))
    T.free()


def test_a_failed_allocation_leaves_other_devices_buffers(fake):
    """Buffers kept from a tree of device 1 survive an allocation that fails on
    device 0, and serve device 1's next tree."""
    fake.fake_set_device(1)
    _one_tree()
    kept = fake.fake_used(1)
    assert kept > 0
    fake.fake_set_device(0)
    fake.fake_set_limit(0, 1 << 10)
    T = _tree(20000)
    assert fake.octgrav_tree_upload(T._h, None) == G.ERR_OOM
    fake.fake_set_device(1)
    _upload(_tree(3000))
    assert fake.fake_used(1) <= kept + 256          # the smallest buffer had been given back


def test_a_failed_allocation_gives_back_its_own_contexts_buffers_only(fake):
    """Two contexts of one device."""
    first = 1 << 20
    fake.fake_set_context(0, first)
    _one_tree()
    kept = fake.fake_used(0)
    fake.fake_set_context(0, first + 1)
    both = [_upload(_tree(3000, seed)) for seed in (1, 2)]
    for T in both:
        T.free()
    fake.fake_set_limit(0, fake.fake_used(0) + (1 << 10))
    T = _tree(20000)                                # takes one set, needs more: the other one goes back
    assert fake.octgrav_tree_upload(T._h, None) == G.ERR_OOM
    assert fake.fake_used(0) < 3 * kept
    fake.fake_set_limit(0, 1 << 40)
    fake.fake_set_context(0, first)
    before = fake.fake_used(0)
    _upload(_tree(3000))
    assert fake.fake_used(0) <= before + 256


def test_contexts_that_are_gone_do_not_use_up_the_places(fake):
    for k in range(40):                             # as after 40 device resets
        fake.fake_set_context(0, (1 << 21) + k)
        _one_tree()
    before = fake.fake_used(0)
    _one_tree()
    assert fake.fake_used(0) == before


def test_kept_buffers_are_bounded_and_given_back(fake):
    """Two trees of about 0.6 GiB each (256 bytes a particle are the parts'
    outputs of a launch split over 16 warps; nothing writes them here)."""
    both = [_upload(_tree(1900000, n_group=256)) for _ in range(2)]
    for T in both:
        T.set_split(16)
        _forces(T)
    assert fake.fake_used(0) > 1 << 30
    for T in both:
        T.free()
    assert 0 < fake.fake_used(0) <= 1 << 30
    alive = _upload(_tree(3000))
    G.release_buffers()
    left = fake.fake_used(0)
    alive.free()
    G.release_buffers()
    assert fake.fake_used(0) == 0 < left            # a tree in use had kept its own


def test_a_set_goes_to_a_tree_that_it_fits(fake):
    """A small tree leaves a large one's buffers alone, so that the next large
    tree allocates nothing; sets that fit no more make room for new ones."""
    _one_tree(200000)
    large = fake.fake_used(0)
    small = _upload(_tree(2000))
    own = fake.fake_used(0) - large
    assert 0 < own < large // 8
    T = _upload(_tree(200000))
    assert fake.fake_used(0) <= large + own + 256   # the smallest buffer had been given back
    T.free()
    small.free()
    for n in (2000, 200000, 2000, 150000):          # both sets serve again
        before = fake.fake_used(0)
        T = _upload(_tree(n))
        assert fake.fake_used(0) <= before + 512
        T.free()
    for n in (10000, 11000, 12000, 13000):          # each too large for the last
        _one_tree(n)
    assert fake.fake_used(0) < large // 2           # the newest two
    before = fake.fake_used(0)
    _upload(_tree(13000))
    assert fake.fake_used(0) <= before + 256


@pytest.mark.parametrize("own", [False, True])
def test_captured_launches_keep_the_buffer_they_write(fake, own):
    """A launch captured with the parts that a small tree chooses itself, by
    octgrav_graph_capture or by the caller, writes a buffer that is still there
    after launches with more parts."""
    T = _upload(_tree(3000))
    _forces(T)
    auto = _last(fake)["nparts"]
    assert auto > 1
    if own:
        fake.fake_begin_capture()
        _forces(T)
        fake.fake_end_capture()
    else:
        G._check(fake.octgrav_graph_capture(T._h, 0.01, 0.5, 1.0, C.c_void_p(256), C.c_void_p(1)))
    for parts in range(1, 17):
        T.set_split(parts)
        _forces(T)
        assert _last(fake)["nparts"] == parts
        if own:
            assert fake.fake_replay() == 0
        else:
            G._check(fake.octgrav_graph_launch(T._h, None))
    assert fake.fake_dangling() == 0
    T.free()
    G.release_buffers()
    assert fake.fake_used(0) == 0


@pytest.mark.parametrize("stage", [0, 1, 2])
def test_a_split_that_was_asked_for_runs_with_staging_mode_1(fake, stage):
    T = _upload(_tree(3000))
    T.set_staging(stage)
    _forces(T)
    assert _last(fake) == dict(nparts=8, stage=stage, ppl=2)      # the automatic split: any mode
    T.set_split(4)
    _forces(T)
    assert _last(fake) == dict(nparts=4 if stage == 1 else 1, stage=stage, ppl=2)


def _noalloc(lib, T, theta=0.5):
    """Runs octgrav_forces_noalloc in an arena of the size it asks for and returns
    its status."""
    need = C.c_size_t(0)
    G._check(lib.octgrav_forces_noalloc(T._h, None, C.byref(need), 1.0, 0.5, 1.0, None, None))
    arena = np.empty(need.value + 256, np.uint8)
    start = -arena.ctypes.data % 256
    return lib.octgrav_forces_noalloc(T._h, C.c_void_p(arena.ctypes.data + start), C.byref(need), 0.01, theta, 1.0,
                                      C.c_void_p(256), None)


def test_noalloc_arena_holds_the_tree_alone(fake):
    """The arena's size depends on the tree, not on the split that it runs with,
    so one sized for a tree of as many cells and items serves."""
    T = _upload(_tree(3000))
    need = T.noalloc_arena_bytes()
    T.set_split(1)
    assert T.noalloc_arena_bytes() == need
    s = T.stats
    arrays = [32 * s["n"], 16 * s["n_cells"], 8 * s["n_cells"], 64 * s["n_cells"], 16 * s["n_items"], 64 * s["n_items"]]
    assert need == sum(-(-a // 256) * 256 for a in arrays)


def test_noalloc_runs_as_a_launch_does(fake):
    """Split as a launch of the same tree chooses itself, unsplit where that was
    turned off."""
    T = _upload(_tree(3000))
    _forces(T)
    auto = _last(fake)["nparts"]
    assert auto > 1
    for asked, runs in ((None, auto), (4, auto), (1, 1)):
        if asked:
            T.set_split(asked)
        assert _noalloc(fake, T) == G.OK
        assert _last(fake)["nparts"] == runs


def test_autotuner_times_the_staging_modes_unsplit(fake):
    """An unsplit winner's staging modes are tried as it runs: unsplit. (By the
    stand-in clock unsplit launches are the fastest with mode 1, and split ones
    would be faster still with mode 0.)"""
    for stage in (0, 1, 2):
        fake.fake_set_time(1, stage, 0.5 if stage == 1 else 0.75)
        for parts in (2, 4, 8):
            fake.fake_set_time(parts, stage, 0.125 if stage == 0 else 1.0)
    best = G.autotune([W.plummer(3000, seed=5)], 16, 0.01, 0.5, candidates=(64,))
    assert best == dict(n_group=64, particles_per_lane=1, split=1, staging=1, ms=0.5)


def _parts(items, n, theta, ppl):
    """The rule of the automatic split, restated."""
    wide = min(1.0, 0.6 / theta) if theta else 1.0
    if n * wide ** 0.75 < 6 * items or n < 1000:
        return 1
    fill = min(1.0, n / items * wide ** 0.5 / 19)
    if ppl == 1 and theta > 0.5:
        fill *= (0.5 / theta) ** 0.7
    return next((p for p, most in ((8, 4640), (4, 5200), (2, 6400)) if items * p <= fill * most), 1)


@pytest.mark.parametrize("n,n_group,ppl", [(5003, 32, 2), (40000, 64, 2), (40000, 64, 1), (20000, 256, 1), (3000, 64, 2),
                                           (1100, 32, 1)])
def test_parts_by_opening_angle(fake, n, n_group, ppl):
    """The parts that launches choose as theta grows; all of them are reserved with
    the upload, so that a launch in a capture allocates nothing."""
    T = _tree(n, n_group=n_group)
    T.set_launch(ppl)
    _upload(T)
    used = fake.fake_used(0)
    items = T._stats()["n_items"]
    seen = []
    for theta in (2.5, 1.6, 1.2, 1.0, 0.9, 0.8, 0.7, 0.6, 0.5, 0.3, 0.0):
        _forces(T, theta)
        seen.append(_last(fake)["nparts"])
        assert seen[-1] == _parts(items, n, theta, ppl)
        assert _noalloc(fake, T, theta=theta) == G.OK and _last(fake)["nparts"] == seen[-1]
    assert seen == sorted(seen) and fake.fake_used(0) == used
    if n in (5003, 40000):
        assert seen[0] == 1 < seen[-1]              # 8 and 16 particles an item: not split at wide angles


def test_parts_of_a_batch_follow_its_widest_angle(fake):
    systems = [W.plummer(4000, seed=k) for k in (1, 2)]
    _made.append(G.Tree.build_batch(systems, 16, 32))
    T = _upload(_made[-1])
    _forces(T, 0.5)
    narrow = _last(fake)["nparts"]
    for theta, parts in (([0.5, 0.5], narrow), ([0.5, 2.5], 1)):
        T.set_system_params([0.01, 0.01], theta)
        _forces(T, 0.3)
        assert _last(fake)["nparts"] == parts
    assert narrow > 1


def _grad(lib, n):
    x, t, g = np.zeros((n, 12), np.float32), np.zeros(n, np.float32), np.zeros(5057, np.float32)
    return lib.octgrav_mlp_grad(g.ctypes.data, x.ctypes.data, t.ctypes.data, n, g.ctypes.data, None, None)


def _direct(lib, n):
    x, m, a, p = np.zeros((n, 3)), np.zeros(n), np.zeros((2, 3)), np.zeros(2)
    return lib.octgrav_direct(x.ctypes.data, m.ctypes.data, n, None, 2, 0.01, 1.0, a.ctypes.data, p.ctypes.data, None)


def test_scratch_is_kept_and_bounded(fake):
    """A thread's direct sums, gradients and training calls allocate once; large ones
    give their buffer back; another context gets its own. (The kernels are not
    imitated, so every call ends with an error here.)"""
    G.release_buffers()
    _grad(fake, 5000)
    kept, frees = fake.fake_used(0), fake.fake_frees()
    assert 0 < kept <= 32 << 20
    for n in (5000, 1, 700):
        assert _grad(fake, n) == G.ERR_CUDA and _direct(fake, n + 1) == G.ERR_CUDA
    assert fake.fake_used(0) == kept and fake.fake_frees() == frees
    _grad(fake, 1000000)
    _direct(fake, 1200000)
    assert fake.fake_used(0) == kept                # 52 and 38 MB, given back
    fake.fake_set_context(0, 1 << 22)
    _grad(fake, 5000)
    G.release_buffers()
    assert fake.fake_used(0) == kept                # the first context's is not touched
    fake.fake_set_context(0, (1 << 22) + 1)
    _grad(fake, 700)
    assert fake.fake_used(0) == kept


def test_the_automatic_split_can_be_had_back(fake):
    T = _upload(_tree(3000))
    _forces(T)
    auto, used = _last(fake)["nparts"], fake.fake_used(0)
    T.set_split(1)
    _forces(T)
    assert _last(fake)["nparts"] == 1 < auto
    T.auto_split()
    _forces(T)
    assert _last(fake)["nparts"] == auto and fake.fake_used(0) == used
    with pytest.raises(G.OctgravError):
        T.set_split(0)                              # no number of parts
