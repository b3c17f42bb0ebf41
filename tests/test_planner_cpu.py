"""Which kernel a call launches, and how: kvs_api.cpp over stand-ins for CUDA (planner_fake.cpp)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2609_35065_gb300 import build, kvs

HERE = os.path.dirname(os.path.abspath(__file__))
LDG, TMA, LINK, LINK_STAGED, LINK_PREFETCH, LINK_SIGNAL, FP8_RETRIEVE, FP8_RETRIEVE_STAGED, FP8_STORE = range(9)
RETRIEVE, STORE = kvs.KVS_DIR_RETRIEVE, kvs.KVS_DIR_STORE
SHORT = (2, 2, 64, 2, 16, 256)           # 4 KiB runs
LONG = (2, 8, 128, 2, 16, 256)           # 32 KiB runs
HBM, HOST = kvs.KVS_SRC_DEVICE, kvs.KVS_SRC_HOST_PINNED


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    if not (shutil.which("g++") and os.path.exists(os.path.join(cuda, "cuda_runtime.h"))):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("planner") / "libplanner.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", build.INCLUDE, "-I", build.CSRC,
                    "-I", cuda, os.path.join(build.CSRC, "kvs_api.cpp"), os.path.join(HERE, "planner_fake.cpp"),
                    "-o", out], check=True)
    L = ctypes.CDLL(out)
    L.fake_set_ms.argtypes = [ctypes.c_int, ctypes.c_float]
    return L


class Planner:
    def __init__(self, lib):
        self.lib = lib

    def speeds(self, **ms):
        for name, t in ms.items():
            self.lib.fake_set_ms(globals()[name], t)

    def _args(self, geom, where, tokens):
        g = kvs._geometry(geom)
        table = np.arange(-(-tokens // geom[4]), dtype=np.int32)
        full, rest = divmod(tokens, geom[5])
        counts = [geom[5]] * full + ([rest] if rest else [])
        req = kvs.RequestArg(table, [kvs.ChunkArg((1 << 40) + (k << 30), n, where) for k, n in enumerate(counts)])
        m = kvs._Marshalled([(1 << 44) + (p << 32) for p in range(2 * geom[0])], len(table), [req])
        return g, m, (ctypes.byref(g), ctypes.byref(m.cache), m.reqs, m.n)

    def _run(self, name, *args):
        n = self.lib.fake_count()
        self.lib.kvs_last_error.restype = ctypes.c_char_p
        assert getattr(self.lib, name)(*args) == 0, self.lib.kvs_last_error()
        out = []
        for k in range(n, self.lib.fake_count()):
            v = (ctypes.c_int * 4)()
            self.lib.fake_launch(k, v)
            out.append(dict(zip(("kernel", "grid", "carried", "early"), v)))
        return out

    def call(self, name, geom, where, tokens=512, flags=0):
        """The launches of one call, in order."""
        g, m, a = self._args(geom, where, tokens)
        return self._run(name, *a, None, ctypes.c_uint32(flags))

    def tune(self, geom, where, direction, tokens=512):
        g, m, a = self._args(geom, where, tokens)
        rep = kvs.kvs_tune_report()
        self._run("kvs_tune", *a, None, ctypes.c_uint32(0), direction, 1, ctypes.byref(rep))
        return rep

    def choice(self):
        rep = kvs.kvs_bw_report()
        self._run("kvs_get_choice", ctypes.byref(rep))
        return rep


@pytest.fixture
def planner(library):
    library.fake_reset()
    yield Planner(library)
    library.kvs_shutdown()


def _kernels(launches):
    return [x["kernel"] for x in launches]


@pytest.mark.parametrize("name,direction", [("kvs_retrieve", RETRIEVE), ("kvs_store", STORE)])
@pytest.mark.parametrize("geom", [SHORT, LONG], ids=["4KiB_runs", "32KiB_runs"])
def test_the_kernel_that_tune_measured_faster_serves_later_calls(planner, geom, name, direction):
    assert _kernels(planner.call(name, geom, HBM)) == [LDG]
    for faster, want in ((TMA, kvs.KVS_KERNEL_TMA), (LDG, kvs.KVS_KERNEL_LDG)):
        planner.speeds(**{"LDG": 2.0, "TMA": 1.0} if faster == TMA else {"LDG": 1.0, "TMA": 2.0})
        rep = planner.tune(geom, HBM, direction)
        assert rep.chosen_kernel_device == want == planner.choice().chosen_kernel_device
        assert _kernels(planner.call(name, geom, HBM)) == [faster]


def test_what_was_measured_on_long_runs_does_not_decide_for_short_ones(planner):
    """TMA moves one run a CTA, so a probe or a tuned call of 32 KiB runs says nothing about 4 KiB ones."""
    planner.speeds(LDG=2.0, TMA=1.0)
    assert planner.tune(LONG, HBM, RETRIEVE).chosen_kernel_device == kvs.KVS_KERNEL_TMA
    assert _kernels(planner.call("kvs_retrieve", LONG, HBM)) == [TMA]
    assert _kernels(planner.call("kvs_retrieve", SHORT, HBM)) == [LDG]
    planner.tune(SHORT, HBM, RETRIEVE)
    assert _kernels(planner.call("kvs_retrieve", SHORT, HBM)) == [TMA]
    planner._run("kvs_query_bw", None, None, ctypes.c_int64(16 << 20))
    assert _kernels(planner.call("kvs_retrieve", LONG, HBM)) == [TMA]
    assert _kernels(planner.call("kvs_retrieve", SHORT, HBM)) == [LDG]


@pytest.mark.parametrize("name", ["kvs_retrieve", "kvs_store", "kvs_retrieve_fp8", "kvs_store_fp8"])
@pytest.mark.parametrize("geom", [SHORT, LONG, (2, 3, 20, 2, 16, 256)], ids=["4KiB_runs", "32KiB_runs", "120B_rows"])
def test_only_uncapped_hbm_kernels_let_the_next_call_in_early(planner, geom, name):
    """The next carried call's CTAs wait on SMs: not beside a copy that the link or the caller's cap bounds."""
    if "fp8" in name and geom[2] % 16:
        pytest.skip("fp8 chunks need head_dim a multiple of 16")
    cap = 4 << 16
    assert kvs.KVS_F_MAX_CTAS(4) == cap
    for where, flags, early in ((HBM, 0, 1), (HBM, cap, 0), (HOST, 0, 0), (HOST, cap, 0)):
        seen = planner.call(name, geom, where, 257, flags)
        assert [x["early"] for x in seen] == [early], (where, flags, seen)
        assert all(x["carried"] for x in seen)


def test_fp8_retrieval_from_the_host_holds_whole_tpcs(planner):
    """Of the 50 CTAs of the built-in cap, 47, on the SMs of 48: four CTAs to the two SMs that a
    GEMM's CTA pair needs, and no common factor with a span's pieces.  Calls of less than 16 MiB
    of codes take an eighth more than the cap."""
    assert planner.choice().hostlink_ctas == 50
    grid = lambda geom, tokens, flags=0: planner.call("kvs_retrieve_fp8", geom, HOST, tokens, flags)[0]["grid"]
    assert grid((32, 8, 128, 2, 16, 256), 256) == grid((32, 8, 128, 2, 16, 256), 2000) == 47
    assert grid(LONG, 512) == grid((32, 8, 128, 2, 16, 256), 255) == 56
    assert grid(LONG, 512, kvs.KVS_F_MAX_CTAS(50)) == 50
