"""Small calls in a row on one stream, each reading or overwriting what the one before moves.

Calls whose tables travel in the launch's parameters are launched programmatically: on HBM
chunks a call's CTAs may be in place while the call before it still runs, and wait for it.
Nothing here synchronises or validates between the calls, and every round moves other
values, so a kernel that did not wait would leave an earlier round's bytes.  The results
are compared with the CPU oracle, exactly.
"""
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import pytest
import torch

import oracle
from paper_2609_35065_gb300 import kvs

pytestmark = pytest.mark.gpu

ROUNDS = 5
L = 9                                    # layer by layer: more launches than carry their tables


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    kvs.kvs_shutdown()                   # the built-in defaults
    yield
    torch.cuda.synchronize()


# name: (fp8, H, D, B, C, tokens of the requests, flags)
CASES = {
    "ldg_pieces": (False, 8, 128, 16, 256, (512, 512), 0),
    "tma_pieces": (False, 8, 128, 16, 256, (512, 512), kvs.KVS_F_FORCE_TMA),
    "tma_short_runs": (False, 2, 64, 16, 256, (1024, 700), kvs.KVS_F_FORCE_TMA),
    "spans": (False, 2, 64, 16, 256, (2048, 1801), 0),
    "spans_and_narrow": (False, 5, 36, 8, 256, (1024, 777), 0),
    "narrow": (False, 3, 5, 4, 256, (1024, 999), 0),
    "capped": (False, 8, 128, 16, 256, (512, 300), kvs.KVS_F_MAX_CTAS(7)),
    "fp8_units": (True, 8, 128, 16, 256, (512, 512), 0),
    "fp8_wide_units": (True, 6, 80, 16, 256, (512, 300), 0),
    "fp8_clusters": (True, 3, 256, 16, 256, (512, 300), 0),
    "fp8_capped": (True, 8, 128, 16, 256, (256, 200), kvs.KVS_F_MAX_CTAS(7)),
    "fp8_clusters_capped": (True, 3, 256, 16, 256, (256, 200), kvs.KVS_F_MAX_CTAS(9)),
    "fp8_wide_units_capped": (True, 6, 80, 16, 256, (256, 200), kvs.KVS_F_MAX_CTAS(9)),
}


class Chain:
    """Requests over one block table; any number of planes and of chunk sets for them."""

    def __init__(self, name):
        self.fp8, self.H, self.D, self.B, self.C, self.tokens, self.flags = CASES[name]
        self.geom = (L, self.H, self.D, 2, self.B, self.C)
        per = [-(-t // self.B) for t in self.tokens]
        self.nb = sum(per) + 5
        ids = np.random.default_rng(7).permutation(self.nb).astype(np.int32)
        self.tables, at = [], 0
        for n in per:
            self.tables.append(ids[at:at + n].copy())
            at += n
        self.counts = [[self.C] * (t // self.C) + ([t % self.C] if t % self.C else []) for t in self.tokens]
        self.stream = torch.cuda.Stream()
        entries = sum(map(len, self.counts))
        assert 2 * L * 8 + entries * (16 + self.C // self.B * 4) + 8 <= 3584      # tables that a launch carries

    def planes(self, seed=None):
        n = self.nb * self.B * self.H * self.D
        if seed is None:
            return torch.zeros(2 * L, n, dtype=torch.int16, device="cuda")
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return torch.randn(2 * L, n, device="cuda", generator=gen).bfloat16().view(torch.int16)

    def chunk_bytes(self, n):
        codes = 2 * L * n * self.H * self.D
        return (2 * L * self.H * 4 + 255) // 256 * 256 + codes if self.fp8 else 2 * codes

    def chunks(self):
        return [[torch.zeros(self.chunk_bytes(n), dtype=torch.uint8, device="cuda") for n in c] for c in self.counts]

    def call(self, op, planes, chunks, uploaded=False, **kw):
        reqs = [kvs.RequestArg(t, [kvs.ChunkArg(x, n, kvs.KVS_SRC_DEVICE) for x, n in zip(mine, c)])
                for t, mine, c in zip(self.tables, chunks, self.counts)]
        ptrs = [int(p.data_ptr()) for p in planes]
        fn = "kvs_" + op + ("_fp8" if self.fp8 else "")
        if uploaded:
            getattr(kvs, fn + "_layers")(self.geom, ptrs, self.nb, reqs, 1, None, self.stream, self.flags)
        elif kw:
            getattr(kvs, fn + "_layers")(self.geom, ptrs, self.nb, reqs, kw["lps"], None, self.stream, self.flags,
                                         ready_events=kw["ready"])
        else:
            getattr(kvs, fn)(self.geom, ptrs, self.nb, reqs, self.stream, self.flags)

    # ---- the same by the oracle, on numpy arrays -----------------------------------------
    def _each_plane(self, op, planes, chunks):
        def one(p):
            mine = [None] * (2 * L)
            mine[p] = planes[p]
            for t, c, n in zip(self.tables, chunks, self.counts):
                a = (L, self.H, self.D, self.B, mine, self.nb, 0)
                if self.fp8:
                    rc = getattr(oracle, op + "_fp8")(*a, c, n, t, p0=p, p1=p + 1)
                else:
                    rc = getattr(oracle, op)(*a, [x.view(np.uint16) for x in c], t, p0=p, p1=p + 1)
                assert rc == 0, rc
        with ThreadPoolExecutor(8) as ex:
            list(ex.map(one, range(2 * L)))

    def stored(self, planes):
        out = [[np.zeros(self.chunk_bytes(n), np.uint8) for n in c] for c in self.counts]
        self._each_plane("store", planes, out)
        return out

    def retrieved(self, chunks):
        out = [np.zeros(self.nb * self.B * self.H * self.D, np.uint16) for _ in range(2 * L)]
        self._each_plane("retrieve", out, chunks)
        return out


def _np(planes):
    return [p.cpu().numpy().view(np.uint16) for p in planes]


def _sleep(stream):
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        torch.cuda._sleep(20_000_000)                  # the whole chain is queued meanwhile


@pytest.mark.parametrize("name", sorted(CASES))
def test_store_then_retrieve_of_the_same_chunks(name):
    """Each retrieval reads the chunks that the call before it writes, and the next round's store
    overwrites the chunks that the call before it reads."""
    c = Chain(name)
    src = [c.planes(seed) for seed in range(ROUNDS)]
    dst = [c.planes() for _ in range(ROUNDS)]
    chunks = c.chunks()
    _sleep(c.stream)
    for r in range(ROUNDS):
        c.call("store", src[r], chunks, uploaded=r == 2)
        c.call("retrieve", dst[r], chunks, uploaded=r == 3)
    c.stream.synchronize()
    assert kvs.kvs_check_errors(None) == kvs.KVS_OK
    for r in range(ROUNDS):
        want = c.retrieved(c.stored(_np(src[r])))
        for p, (got, exp) in enumerate(zip(_np(dst[r]), want)):
            assert np.array_equal(got, exp), (name, r, p)


@pytest.mark.parametrize("name", sorted(CASES))
def test_retrieve_then_store_of_the_same_planes(name):
    """Each store reads the planes that the call before it writes, and the next round's retrieval
    overwrites the planes that the call before it reads."""
    c = Chain(name)
    src = [c.chunks() for _ in range(ROUNDS)]
    want = []
    for r in range(ROUNDS):
        x = c.stored(_np(c.planes(r)))
        want.append(c.stored(c.retrieved(x)))
        for mine, data in zip(src[r], x):
            for t, v in zip(mine, data):
                t.copy_(torch.from_numpy(v))
    dst = [c.chunks() for _ in range(ROUNDS)]
    planes = c.planes()
    _sleep(c.stream)
    for r in range(ROUNDS):
        c.call("retrieve", planes, src[r], uploaded=r == 2)
        c.call("store", planes, dst[r], uploaded=r == 3)
    c.stream.synchronize()
    assert kvs.kvs_check_errors(None) == kvs.KVS_OK
    for r in range(ROUNDS):
        for mine, data in zip(dst[r], want[r]):
            for t, v in zip(mine, data):
                assert np.array_equal(t.cpu().numpy(), v), (name, r)


@pytest.mark.parametrize("name", ["ldg_pieces", "tma_pieces", "spans", "fp8_units", "fp8_clusters"])
def test_store_groups_that_carry_their_tables_wait_for_their_ready_events(name):
    """A producer on another stream rewrites each layer group's planes late; between two carried
    launches lies only the wait for its event."""
    c = Chain(name)
    planes, fresh, other = c.planes(1), c.planes(2), c.planes(3)
    chunks, spare = c.chunks(), c.chunks()
    lps = 3
    ready = [torch.cuda.Event() for _ in range(-(-L // lps))]
    producer = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(producer):
        for k, ev in enumerate(ready):
            torch.cuda._sleep(10_000_000)
            planes[2 * k * lps:2 * (k + 1) * lps].copy_(fresh[2 * k * lps:2 * (k + 1) * lps])
            ev.record(producer)
    c.call("store", other, spare)
    c.call("store", planes, chunks, lps=lps, ready=ready)
    torch.cuda.synchronize()
    want = c.stored(_np(fresh))
    for mine, data in zip(chunks, want):
        for t, v in zip(mine, data):
            assert np.array_equal(t.cpu().numpy(), v), name
