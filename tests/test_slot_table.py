"""The slot table when a launch fails: the library's host side (csrc/wk_api.cu) built against stand-ins for the CUDA runtime and
the kernel launchers, so that any of them can be made to fail without a GPU."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2605_22718_b200 import binding
from paper_2605_22718_b200.build import CSRC, ROOT, _nvcc

SLOTS, LAYERS = 3, 2
POSE_BYTES = 8 * 4


class Host:
    def __init__(self, lib):
        self.lib = lib
        vp = C.c_void_p
        cfg = binding.wk_config(LAYERS, 1, 128, 4, 3, 2, SLOTS, SLOTS, 1, 0, 0.0, 0)
        lib.wk_pool_bytes.restype = lib.wk_scratch_bytes.restype = C.c_size_t
        lib.wk_pool_tag.restype = C.c_int64
        pool, scratch = lib.wk_pool_bytes(C.byref(cfg)), lib.wk_scratch_bytes(C.byref(cfg), LAYERS, 1, 1)
        self.ctx = vp()
        assert lib.wk_create(C.byref(cfg), C.byref(self.ctx)) == 0
        self.memory = np.zeros(pool + scratch + 1024, dtype=np.uint8)
        base = (self.memory.ctypes.data + 255) // 256 * 256
        s_base = (base + pool + 255) // 256 * 256
        assert lib.wk_bind(self.ctx, vp(base), C.c_size_t(pool), vp(s_base), C.c_size_t(scratch), LAYERS, 1, 1) == 0
        rows = (LAYERS * SLOTS * 6 * 128 * 2 + 255) // 256 * 256
        off = base - self.memory.ctypes.data + 2 * rows          # poses, then validity flags, each padded to 256 bytes
        self.poses = self.memory[off:off + SLOTS * POSE_BYTES].view(np.float32).reshape(SLOTS, 8)
        self.valid = self.memory[off + 256:off + 256 + SLOTS * 4].view(np.int32)
        self.chunk = np.zeros(LAYERS * 12 * 128 + 8, dtype=np.uint16)
        self.keep = np.zeros(LAYERS * 6, dtype=np.int32)

    def store(self, tag, slot=-1, layer0=0, n=LAYERS, evict=1):
        at = (self.chunk.ctypes.data + 15) // 16 * 16
        pose = (C.c_float * 8)(*[tag] * 8)
        slot_io, evicted = C.c_int32(slot), C.c_int32(-7)
        st = self.lib.wk_pool_compress_append(self.ctx, layer0, n, C.c_void_p(at), C.c_void_p(at), C.c_int64(12 * 128),
                                              C.c_void_p(self.keep.ctypes.data), pose, C.c_int64(tag), evict,
                                              C.byref(slot_io), C.byref(evicted), None)
        return st, slot_io.value, evicted.value

    def fail(self, **which):
        for name in ("compress", "append", "mark"):
            C.c_int.in_dll(self.lib, "fail_" + name).value = which.get(name, 0)

    def tags(self):
        return [self.lib.wk_pool_tag(self.ctx, s) for s in range(SLOTS)]

    def agrees(self):
        """Host and device agree on which slots hold a chunk."""
        tags = self.tags()
        assert [int(v) for v in self.valid] == [int(t >= 0) for t in tags]
        assert self.lib.wk_pool_count(self.ctx) == sum(t >= 0 for t in tags)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    out = str(tmp_path_factory.mktemp("host") / "libwk_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(_nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", cuda, "-I", CSRC, "-x", "c++",
                    os.path.join(CSRC, "wk_api.cu"), os.path.join(ROOT, "tests", "host", "fake_device.cc"), "-o", out], check=True)
    return C.CDLL(out)


@pytest.fixture
def host(lib):
    h = Host(lib)
    h.fail()
    yield h
    lib.wk_destroy(h.ctx)


def test_whole_chunks_replace_the_oldest(host):
    for tag in range(5):
        st, slot, evicted = host.store(tag)
        assert (st, slot, evicted) == (0, tag % SLOTS, tag % SLOTS if tag >= SLOTS else -1)
        assert host.poses[slot, 0] == tag
        host.agrees()
    assert host.tags() == [3, 4, 2]


@pytest.mark.parametrize("which", ["compress", "append"])
@pytest.mark.parametrize("n", [LAYERS, 1])
def test_a_failed_store_leaves_no_mark_on_the_slot_it_freed(host, which, n):
    for tag in range(SLOTS):
        assert host.store(tag)[0] == 0
    host.fail(**{which: 1})
    st, slot, evicted = host.store(10, n=n)
    assert (st, slot, evicted) == (binding.WK_ERR_CUDA, -1, 0)
    assert host.tags() == [-1, 1, 2]
    host.agrees()
    host.fail()
    assert host.store(11)[:2] == (0, 0)
    assert host.tags() == [11, 1, 2]
    host.agrees()


@pytest.mark.parametrize("which", ["compress", "append"])
def test_a_failed_store_into_a_free_or_open_slot(host, which):
    assert host.store(0)[0] == 0
    host.fail(**{which: 1})
    assert host.store(1)[0] == binding.WK_ERR_CUDA
    host.agrees()
    host.fail()
    st, slot, _ = host.store(2, layer0=0, n=1)
    assert (st, slot) == (0, 1)
    host.agrees()
    host.fail(**{which: 1})
    assert host.store(2, slot=1, layer0=1, n=1)[0] == binding.WK_ERR_CUDA
    host.agrees()
    host.fail()
    assert host.store(2, slot=1, layer0=1, n=1)[0] == 0
    assert host.tags() == [0, 2, -1]
    host.agrees()
