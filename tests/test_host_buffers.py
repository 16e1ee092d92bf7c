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
