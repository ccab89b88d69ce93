"""What the launchers ask of the CUDA runtime, without a GPU: the library's objects
linked against a runtime that records the launches (fake_cudart.cpp)."""

import ctypes
import os
import subprocess
import threading
import time

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
OUT = 1 << 20  # a device address: nothing is written


@pytest.fixture
def lib(tmp_path):
    """A copy of the library of this test's own, on the recording runtime."""
    from paper_2109_01329_gb300 import _binding, build

    build.build()
    objs = [os.path.join(build.BUILD_DIR, os.path.splitext(s)[0] + ".o") for s in build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    path = str(tmp_path / "libgrng_fake.so")
    # bound to itself: the runtime that torch loads has the same names
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-pthread",
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-o", path], check=True, timeout=300)
    L = ctypes.CDLL(path)
    for name in ("grng_generate", "grng_generate_substreams", "grng_engine_create", "grng_fill_set_geometry"):
        f, g = getattr(L, name), getattr(_binding.load(), name)
        f.argtypes, f.restype = g.argtypes, g.restype
    return L


def _dist(kind, dtype, p0=0.0, p1=1.0):
    from paper_2109_01329_gb300 import Distribution

    return Distribution(kind, dtype, p0, p1)._c()


def _engine(lib, kind, offset):
    e = ctypes.c_void_p()
    assert lib.grng_engine_create(ctypes.byref(e), kind, 1, offset) == 0
    return e


def _launches(lib, first=0):
    """(kernel, grid) of each launch from the first-th on."""
    name = ctypes.create_string_buffer(4096)
    r = []
    for i in range(first, lib.fake_launches()):
        grid = lib.fake_launch(i, name, 4096)
        r.append((name.value.decode(), grid))
    return r


# (distribution, word phase, bytes past a 16-byte boundary): the launchers with a
# kernel for fills inside 2^32 blocks and one for fills that cross a multiple of it
TWO_KERNELS = {"shift": ((0, 0), 1, 0), "split": ((2, 1), 1, 4), "pieces": ((2, 1), 2, 0), "rotate": ((1, 2), 2, 0)}


@pytest.mark.parametrize("name", TWO_KERNELS)
def test_first_fills_from_two_threads(lib, name):
    """Two threads' first fills, one of which crosses a multiple of 2^32 blocks, the
    second while the first is still asking for its kernel's resident CTAs."""
    (kind, dtype), phase, lead = TWO_KERNELS[name]
    d = _dist(kind, dtype)
    inside, crossing = _engine(lib, 0, phase), _engine(lib, 0, (1 << 34) - 40 + phase)
    status = {}

    def fill(key, engine, at):
        time.sleep(at)
        status[key] = lib.grng_generate(ctypes.byref(d), engine, 10001, OUT + lead, None)

    lib.fake_occupancy_delay(200)
    threads = [threading.Thread(target=fill, args=a) for a in (("inside", inside, 0.0), ("crossing", crossing, 0.3))]
    [t.start() for t in threads]
    [t.join() for t in threads]
    assert status == {"inside": 0, "crossing": 0}
    assert len(_launches(lib)) == 2


@pytest.mark.parametrize("n", [1024, 1024 * 2 + 4, 1 << 18])
@pytest.mark.parametrize("kind, dtype", [(0, 0), (2, 1), (2, 2)])
def test_tuned_geometry_reaches_long_aligned_substreams(lib, kind, dtype, n):
    """Substreams long enough for a CTA per tile of a stream: a tuned geometry still
    caps the CTAs (the recording runtime has 152 SMs of 4 resident CTAs)."""
    d, e, streams = _dist(kind, dtype), _engine(lib, 0, 0), 16384

    def grid():
        first = lib.fake_launches()
        assert lib.grng_generate_substreams(ctypes.byref(d), e, n, streams, 1 << 40, 0, OUT, None) == 0
        (_, g), = _launches(lib, first)
        return g

    built_in = grid()
    for geometry, ctas in ((1, 152), (3, 3 * 152), (16, 4 * 152), (18, 8 * 152)):
        assert lib.grng_fill_set_geometry(0, ctypes.byref(d), n * streams, geometry) == 0
        assert grid() == ctas
    assert lib.grng_fill_set_geometry(0, ctypes.byref(d), n * streams, 0) == 0
    assert grid() == built_in


@pytest.mark.parametrize("phase", [0, 1, 2])
def test_pieces_of_a_long_fill_take_its_geometry(lib, phase):
    """A fill launched in pieces of 2^32 elements has one geometry, that of its own
    size: the aligned, the shift and the pieces kernel."""
    d, n = _dist(2, 1), (1 << 33) + (1 << 30)
    assert lib.grng_fill_set_geometry(0, ctypes.byref(d), n, 1) == 0
    assert lib.grng_generate(ctypes.byref(d), _engine(lib, 0, phase), n, OUT, None) == 0
    launches = _launches(lib)
    assert len(launches) == 3 and [g for _, g in launches] == [152] * 3
