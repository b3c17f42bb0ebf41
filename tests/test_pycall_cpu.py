"""The binding's marshalling extension against its numpy marshalling, without a GPU.

A callback of the C functions' signature stands in for the library and writes down the
structs it is given: both paths must hand over the same ones, and the extension must
leave alone (return None for) whatever is not an ordinary form.
"""
import ctypes
import gc
import sys

import numpy as np
import pytest

from paper_2609_35065_gb300 import build, kvs

GEOM = (2, 4, 64, 2, 16, 256)
PLANES = [0x7F00_0000_0000 + 4096 * p for p in range(4)]


class Buffer:
    """Anything with data_ptr()."""

    def __init__(self, at):
        self.at = at

    def data_ptr(self):
        return self.at


@pytest.fixture(scope="module")
def call():
    fn = build.load_pycall()
    if fn is None:
        pytest.skip("no Python headers: the binding marshals with numpy")
    return fn


def _requests():
    t = np.arange(100, dtype=np.int32)
    return [kvs.RequestArg(t[:40], [kvs.ChunkArg(Buffer(1 << 40), 256), kvs.ChunkArg(2 << 40, 7, kvs.KVS_SRC_DEVICE)]),
            kvs.RequestArg(t[40:], [], first_token=256, num_tokens=0),
            kvs.RequestArg(t, [kvs.ChunkArg((1 << 64) - 16, 1)] * 70, first_token=512, num_tokens=3)]


def _read(geom, cache, reqs, n, num_planes):
    r = []
    for k in range(n):
        q = reqs[k]
        r.append((q.first_token, q.num_tokens, [(q.chunks[i].base, q.chunks[i].num_tokens, q.chunks[i].residency)
                                                for i in range(q.num_chunks)],
                  [q.block_table[i] for i in range(q.block_table_len)]))
    g = geom.contents
    return ([getattr(g, f) for f, _ in g._fields_], [cache.contents.kv_planes[p] for p in range(num_planes)],
            cache.contents.num_blocks, r)


def _whole(num_planes, seen, status=0):
    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.POINTER(kvs.kvs_geometry), ctypes.POINTER(kvs.kvs_paged_cache),
                      ctypes.POINTER(kvs.kvs_request), ctypes.c_int32, ctypes.c_void_p, ctypes.c_uint32)
    def fn(geom, cache, reqs, n, stream, flags):
        seen.append((_read(geom, cache, reqs, n, num_planes), stream, flags))
        return status
    return fn, ctypes.cast(fn, ctypes.c_void_p).value


@pytest.mark.parametrize("geom", [GEOM, kvs.kvs_geometry(*GEOM)], ids=["tuple", "struct"])
@pytest.mark.parametrize("planes", [PLANES, tuple(PLANES), [Buffer(p) for p in PLANES]], ids=["list", "tuple", "objects"])
def test_same_structs_as_the_numpy_path(call, geom, planes):
    for reqs in (_requests(), tuple(_requests()), []):
        seen = []
        fn, at = _whole(4, seen, -3)
        assert call(at, geom, planes, 1000, reqs, 0xABC, 0xFFFF0001) == -3
        m = kvs._Marshalled(planes, 1000, reqs)
        fn(ctypes.byref(kvs._geometry(geom)), ctypes.byref(m.cache), m.reqs, m.n, 0xABC, 0xFFFF0001)
        assert seen[0] == seen[1] and len(seen) == 2


def test_layer_calls_pass_their_events(call):
    seen = []

    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32,
                      ctypes.POINTER(ctypes.c_void_p), ctypes.c_void_p, ctypes.c_uint32)
    def retrieve(g, c, r, n, lps, events, stream, flags):
        seen.append((n, lps, [events[k] for k in range(2)] if events else None, stream, flags))
        return 0

    @ctypes.CFUNCTYPE(ctypes.c_int, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int32, ctypes.c_int32,
                      ctypes.POINTER(ctypes.c_void_p), ctypes.POINTER(ctypes.c_void_p), ctypes.c_void_p, ctypes.c_uint32)
    def store(g, c, r, n, lps, ready, events, stream, flags):
        seen.append((n, lps, [ready[k] for k in range(2)] if ready else None,
                     [events[k] for k in range(2)] if events else None, stream, flags))
        return 0

    at = [ctypes.cast(f, ctypes.c_void_p).value for f in (retrieve, store)]
    args = (GEOM, PLANES, 10, _requests(), 0, 5)
    assert call(at[0], *args, 1, 1, None, [11, 0]) == 0
    assert call(at[0], *args, 1, 2, None, None) == 0
    assert call(at[1], *args, 2, 1, [7, 8], [0, 12]) == 0
    assert call(at[1], *args, 2, 1, None, None) == 0
    assert seen == [(3, 1, [11, None], None, 5), (3, 2, None, None, 5), (3, 1, [7, 8], [None, 12], None, 5),
                    (3, 1, None, None, None, 5)]


class Index:
    def __index__(self):
        return 256


def _odd():
    t = np.arange(64, dtype=np.int32)
    ok = [kvs.ChunkArg(1 << 40, 256)]
    yield "geometry of five", dict(geom=GEOM[:5])
    yield "geometry out of range", dict(geom=(1 << 40,) + GEOM[1:])
    yield "geometry list", dict(geom=list(GEOM))
    yield "planes array", dict(planes=np.array(PLANES, dtype=np.uint64))
    yield "no planes", dict(planes=[])
    yield "too few planes", dict(planes=PLANES[:3])
    yield "negative plane", dict(planes=[-1] + PLANES[1:])
    yield "plane of None", dict(planes=[None] + PLANES[1:])
    yield "num_blocks float", dict(num_blocks=10.0)
    yield "num_blocks too large", dict(num_blocks=1 << 70)
    yield "requests iterator", dict(requests=iter([]))
    yield "flags numpy", dict(flags=np.uint32(1))
    yield "flags negative", dict(flags=-1)
    for name, c in (("float tokens", kvs.ChunkArg(1 << 40, 256.0)), ("numpy tokens", kvs.ChunkArg(1 << 40, np.int32(256))),
                    ("index tokens", kvs.ChunkArg(1 << 40, Index())), ("bool residency", kvs.ChunkArg(1 << 40, 256, True)),
                    ("huge tokens", kvs.ChunkArg(1 << 40, 1 << 40)), ("numpy base", kvs.ChunkArg(np.zeros(4), 256)),
                    ("negative base", kvs.ChunkArg(-16, 256)), ("float pointer", kvs.ChunkArg(Buffer(1.5), 256))):
        yield name, dict(requests=[kvs.RequestArg(t, [c])])
    yield "int64 table", dict(requests=[kvs.RequestArg(t.astype(np.int64), ok)])
    yield "uint32 table", dict(requests=[kvs.RequestArg(t.astype(np.uint32), ok)])
    yield "strided table", dict(requests=[kvs.RequestArg(t[::2], ok)])
    yield "list table", dict(requests=[kvs.RequestArg([1, 2, 3], ok)])
    yield "chunks generator", dict(requests=[kvs.RequestArg(t, (c for c in ok))])
    yield "float first token", dict(requests=[kvs.RequestArg(t, ok, first_token=0.0)])
    yield "not a request", dict(requests=[object()])


@pytest.mark.parametrize("name,odd", list(_odd()), ids=[n for n, _ in _odd()])
def test_other_forms_are_left_to_numpy(call, name, odd):
    seen = []
    fn, at = _whole(4, seen)
    a = dict(geom=GEOM, planes=PLANES, num_blocks=10, requests=_requests(), stream=0, flags=0)
    a.update(odd)
    assert call(at, a["geom"], a["planes"], a["num_blocks"], a["requests"], a["stream"], a["flags"]) is None
    assert seen == []


def test_exceptions_of_data_ptr_come_through_and_nothing_leaks(call):
    class Bad:
        def data_ptr(self):
            raise RuntimeError("no storage")
    seen = []
    fn, at = _whole(4, seen)
    table = np.arange(8, dtype=np.int32)
    good, bad = kvs.ChunkArg(Buffer(64), 256), kvs.ChunkArg(Bad(), 256)
    before = [sys.getrefcount(x) for x in (table, good, bad)]
    for _ in range(50):
        with pytest.raises(RuntimeError, match="no storage"):
            call(at, GEOM, PLANES, 10, [kvs.RequestArg(table, [good]), kvs.RequestArg(table, [good, bad])], 0, 0)
        assert call(at, GEOM, PLANES, 10, [kvs.RequestArg(table, [good])], 0, 0) == 0
        assert call(at, GEOM, PLANES, 10, [kvs.RequestArg(table, [good]), object()], 0, 0) is None
    gc.collect()
    assert [sys.getrefcount(x) for x in (table, good, bad)] == before
    table.resize(16, refcheck=False)              # no view of it is still held
