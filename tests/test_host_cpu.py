"""The library's host code on a recording CUDA runtime (fake_cudart.cpp): its own
objects, driven through the C ABI, with no GPU."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from paper_1901_08088_gb300 import _lib, build_lib

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    build_lib.build()
    out = str(tmp_path_factory.mktemp("host") / "libqbvh_host.so")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build_lib.nvcc()))), "include")
    objs = [os.path.join(build_lib.BUILD, os.path.splitext(s)[0] + ".o") for s in build_lib.SOURCES]
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-Wl,-Bsymbolic", "-I", include, "-o", out,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs, "-ldl"], check=True)
    L = C.CDLL(out)
    for name, (res, args) in _lib.SIGNATURES.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    L.fake_launched.restype = C.c_char_p
    return L


class Handle:
    """One handle, with 16-byte aligned host arrays as device memory."""

    def __init__(self, L, device=0, **options):
        self.L, self.h = L, C.c_void_p()
        assert L.qbvh_create(C.byref(self.h), device) == 0
        for k, v in options.items():
            assert self.set(k, v) == 0
        self.buf = np.zeros(1 << 20, np.float64)

    def set(self, name, value):
        return self.L.qbvh_set_option(self.h, getattr(_lib, "QBVH_OPT_" + name), value)

    def get(self, name):
        v = C.c_int()
        assert self.L.qbvh_get_option(self.h, getattr(_lib, "QBVH_OPT_" + name), C.byref(v)) == 0
        return v.value

    def build(self, n, T=1):
        return self.L.qbvh_build(self.h, self.buf.ctypes.data, n, 50.0, T, None)

    def query(self, T=1):
        r = np.full((T, T), 3.0, np.float32)
        return self.L.qbvh_query(self.h, r.ctypes.data, 8, 0, None)

    def forces(self, T=1):
        """Names of the kernels of one LJ pass."""
        rc, p, first = np.full((T, T), 2.5, np.float32), self.buf.ctypes.data, self.L.fake_launches()
        assert self.L.qbvh_lj_forward(self.h, p, p, p, rc.ctypes.data, p, p, p, p, p, None) == 0
        return [self.L.fake_launched(k) for k in range(first, self.L.fake_launches())]

    def close(self):
        assert self.L.qbvh_destroy(self.h) == 0


@pytest.mark.parametrize("n", [100, 1500, 3000])
@pytest.mark.parametrize("node_format", [0, 1])
def test_one_block_build_on_every_device(host, n, node_format):
    """More than 48 KB of shared memory is a per-device permission."""
    for device in (0, 1, 0):
        h = Handle(host, device, NODE_FORMAT=node_format)
        assert h.build(n) == 0
        h.close()


@pytest.mark.parametrize("n", [100, 20000, 70000])
def test_traversal_blocks_keep_the_shared_memory_limit(host, n):
    """The limit of a kernel never falls: a thread with a smaller block would take
    it from one that is about to launch a larger one."""
    before = host.fake_limits_lowered()
    for device in (0, 1):
        for block in (256, 224, 128, 256):
            h = Handle(host, device, QUERY_BLOCK=block)
            assert h.build(n) == 0 and h.query() == 0
            h.close()
    assert host.fake_limits_lowered() == before


@pytest.mark.parametrize("T", [1, 2])
def test_lj_tables_outlive_other_lanes(host, T):
    """A recorded LJ launch reads its block tables and writes its block records on
    every replay: a pass with other lanes over the same systems leaves both alone."""
    h = Handle(host)
    assert h.build(70000, T) == 0 and h.query(T) == 0
    host.fake_forget_uploads()
    h.forces(T)
    frees = host.fake_frees()
    assert host.fake_uploads() > 0
    for lanes in (8, 32, 1, 16, 4, 2):
        h.set("LJ_LANES", lanes)
        h.forces(T)
        assert host.fake_uploads_lost() == 0
        assert host.fake_frees() == frees
    h.close()


@pytest.mark.parametrize("n", [100, 20000, 70000])
def test_writing_an_option_back_changes_nothing(host, n):
    """The default of the LJ lanes is the value that get_option returns and that the
    autotuner starts from: setting it leaves the kernel of a pass the same."""
    from paper_1901_08088_gb300.autotune import DEFAULTS

    h = Handle(host)
    assert h.build(n) == 0 and h.query() == 0
    kernels = h.forces()
    assert DEFAULTS[_lib.QBVH_OPT_LJ_LANES] == h.get("LJ_LANES")
    assert h.set("LJ_LANES", 8) == 0 and h.forces() != kernels
    assert h.set("LJ_LANES", DEFAULTS[_lib.QBVH_OPT_LJ_LANES]) == 0
    assert h.forces() == kernels
    h.close()
