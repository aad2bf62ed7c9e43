"""The host runtime (st_runtime.cu) without a GPU, linked with a stand-in for
the CUDA runtime and the kernel launchers (fake_cuda.cpp, fake_launch.cu): what a call leaves
behind when a launch in its middle fails, and what scratch it makes do with."""

import ctypes as C
import os
import subprocess

import pytest

from conftest import ROOT
from paper_2606_14480_gb300 import build, st

FAR = 1 << 40  # a device address that nothing reads


@pytest.fixture(scope="module")
def rt(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("host_runtime"))
    so = os.path.join(d, "libhost.so")
    inc = ["-I", build.INCLUDE, "-I", build.CSRC]
    nvcc = [build.nvcc(), *build.ARCH, "-std=c++17", "-O1", "-Xcompiler", "-fPIC", *inc]
    here = os.path.join(ROOT, "tests")
    for cmd in ([*nvcc, "-c", os.path.join(here, "fake_cuda.cpp"), "-o", "cuda.o"],
                [*nvcc, "-c", os.path.join(here, "fake_launch.cu"), "-o", "launch.o"],
                [*nvcc, "-c", os.path.join(build.CSRC, "st_runtime.cu"), "-o", "runtime.o"],
                ["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, "runtime.o", "launch.o", "cuda.o", "-lpthread"]):
        r = subprocess.run(cmd, capture_output=True, text=True, cwd=d)
        assert r.returncode == 0, r.stdout + r.stderr
    lib = C.CDLL(so)
    for name, sig in st.SIGNATURES.items():
        if hasattr(lib, name):
            fn = getattr(lib, name)
            fn.argtypes, fn.restype = sig
    lib.fake_stream.restype = C.c_void_p
    lib.fake_used.restype = C.c_int64
    lib.fake_launch_name.restype = C.c_char_p
    lib.fake_reset.argtypes = [C.c_int, C.c_int64]
    lib.fake_unjoined.argtypes = lib.fake_elsewhere.argtypes = [C.c_void_p]
    return lib


class Ctx:
    def __init__(self, rt, **over):
        rt.fake_reset(-1, -1)
        cfg = st.StConfig()
        rt.st_config_default(C.byref(cfg))
        for k, v in over.items():
            setattr(cfg, k, v)
        self.rt, self.h = rt, C.c_void_p()
        assert rt.st_create(C.byref(cfg), 0, C.byref(self.h)) == st.ST_OK

    def seeding_run(self, n, max_hits, stream, cap=4096):
        hits = st.StHits(n, FAR, FAR, FAR, None, None, max_hits, 0)
        seeds = st.StSeeds(cap, *[FAR] * 6)
        return self.rt.seeding_run(self.h, C.byref(hits), C.byref(seeds), stream)

    def close(self):
        self.rt.st_destroy(self.h)


def names(rt):
    return [rt.fake_launch_name(k).decode() for k in range(rt.fake_launches())]


def test_split_batch_joins_after_a_failed_launch(rt):
    """Whichever launch of a batch with large events fails, the caller's stream
    waits for what the side stream was given before."""
    ctx = Ctx(rt)
    s = rt.fake_stream()
    assert ctx.seeding_run(500, 16384, s) == st.ST_OK
    chain = names(rt)
    assert chain == ["build_large", "build", "order", "seed_large", "seed", "gather"]
    assert rt.fake_elsewhere(s) == 2 and rt.fake_unjoined(s) == 0
    for k in range(len(chain)):
        rt.fake_reset(k, -1)
        assert ctx.seeding_run(500, 16384, s) == st.ST_ECUDA
        assert names(rt) == chain[:k + 1]
        assert rt.fake_unjoined(s) == 0, chain[k]
    rt.fake_reset(-1, -1)
    assert ctx.seeding_run(500, 16384, s) == st.ST_OK and names(rt) == chain
    ctx.close()


def test_split_batch_without_room_for_its_own_slots(rt):
    """Where device memory has no room for the scratch of the larger CTAs, a
    batch with large events runs as split with what the ordinary CTAs have."""
    used = []
    for max_hits in (6144, 6145):
        ctx = Ctx(rt)
        before = rt.fake_used()
        assert ctx.seeding_run(500, max_hits, None) == st.ST_OK
        used.append(rt.fake_used() - before)
        chain = names(rt)
        ctx.close()
    assert used[1] - used[0] > 50 << 20 and "seed_large" in chain
    ctx = Ctx(rt)
    rt.fake_reset(-1, rt.fake_used() + used[1] - (50 << 20))
    assert ctx.seeding_run(500, 6145, None) == st.ST_OK and names(rt) == chain
    rt.fake_reset(-1, rt.fake_used())  # (nothing more is allocated)
    assert ctx.seeding_run(500, 6145, None) == st.ST_OK
    ctx.close()
    ctx = Ctx(rt)
    rt.fake_reset(-1, rt.fake_used() + used[0] // 2)
    assert ctx.seeding_run(500, 6145, None) == st.ST_ENOMEM
    ctx.close()
