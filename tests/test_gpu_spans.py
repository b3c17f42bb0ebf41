"""Span pieces against the CPU oracle: runs shorter than a 32 KiB piece, runs that are no
whole number of pieces, and rows, chunks and planes that are no multiple of 16 bytes.

Exact equality: the path only copies bytes.
"""
import pytest
import torch

import gpu_check as gc
from paper_2609_35065_gb300 import buffers, kvs, synth

pytestmark = pytest.mark.gpu

# (L, H, D, element bytes, B, C, tokens of the requests)
GEOMETRIES = {
    "4KiB_runs": (3, 2, 64, 2, 16, 256, (700, 256, 1)),
    "1KiB_runs_two_pieces": (2, 1, 64, 2, 8, 512, (1024, 513)),
    "16B_runs": (2, 1, 8, 2, 1, 256, (300, 255)),
    "20KiB_runs": (2, 5, 128, 2, 16, 256, (512, 259)),
    "run_ends_mid_vector_row": (3, 3, 20, 2, 16, 256, (900, 133, 255)),     # 120-byte rows, whole runs aligned
    "odd_chunk_spans": (3, 5, 36, 2, 8, 256, (777, 255)),                   # 360-byte rows, odd last chunks
    "odd_bytes": (2, 1, 20, 1, 8, 256, (403, 257)),
    "unaligned_runs": (2, 3, 5, 2, 4, 64, (130, 63)),                       # 30-byte rows
    "long_odd_rows": (2, 7, 333, 2, 1, 64, (70, 33)),                       # 4662-byte runs, block-wise
    "long_runs": (1, 5, 300, 2, 16, 64, (200, 64)),                         # 48000-byte runs, two a piece
    "long_runs_odd_chunk": (1, 7, 333, 2, 16, 64, (197,)),                  # 74592-byte runs
    "one_vector": (1, 1, 8, 2, 1, 1, (1,)),
    "all_chunks_short": (3, 2, 64, 2, 16, 256, (42, 17, 33)),
    "all_chunks_short_32KiB_runs": (2, 8, 128, 2, 16, 256, (40, 1, 48)),
}


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    yield
    torch.cuda.synchronize()


def _workload(name, residency, **kw):
    L, H, D, e, B, C, tokens = GEOMETRIES[name]
    nb = sum(-(-t // B) for t in tokens) + 3
    return synth.custom(L, H, D, B, C, nb, list(tokens), kw.pop("matched", list(tokens)), seed=11,
                        elem_bytes=e, residency=residency, **kw)


@pytest.mark.parametrize("cap", [0, 1, 5], ids=["uncapped", "1_cta", "5_ctas"])
@pytest.mark.parametrize("residency", ["host", "device"])
@pytest.mark.parametrize("name", sorted(GEOMETRIES))
def test_span_pieces(name, residency, cap):
    flags = kvs.KVS_F_MAX_CTAS(cap)
    w = _workload(name, residency)
    buf = buffers.allocate(w)
    kvs.kvs_retrieve(w.geom, buf.plane_ptrs, w.num_blocks, buf.requests, None, flags)
    torch.cuda.synchronize()
    gc.check_retrieve(buf)
    tokens = list(GEOMETRIES[name][-1])
    w = _workload(name, residency, matched=[0] * len(tokens), store_tokens=tokens)
    buf = buffers.allocate(w, store=True, store_residency=residency, plane_init="random")
    kvs.kvs_store(w.geom, buf.plane_ptrs, w.num_blocks, buf.store_requests, None, flags)
    kvs.kvs_check_errors(None)
    torch.cuda.synchronize()
    gc.check_store(buf)


@pytest.mark.parametrize("name", ["4KiB_runs", "run_ends_mid_vector_row", "odd_chunk_spans", "unaligned_runs"])
@pytest.mark.parametrize("entry", ["noalloc", "layers", "hbmcopy"])
def test_span_pieces_by_every_entry(name, entry):
    """The other calls that reach the span kernels: the allocation-free retrieval, layer
    groups (a plane range that starts past 0), and the copy-engine ring's scatter."""
    w = _workload(name, ["device", "host", "device"][:len(GEOMETRIES[name][-1])])
    buf = buffers.allocate(w)
    args = (w.geom, buf.plane_ptrs, w.num_blocks, buf.requests)
    if entry == "noalloc":
        kvs.kvs_retrieve_noalloc(*args, None)
    elif entry == "layers":
        kvs.kvs_retrieve_layers(*args, 1, None, None)
    else:
        kvs.kvs_retrieve(*args, None, kvs.KVS_F_FORCE_HBMCOPY)
    torch.cuda.synchronize()
    gc.check_retrieve(buf)


def test_span_pieces_skip_blocks_another_request_writes():
    """Shared blocks inside a span piece: the dropped writer's bytes differ and must not land."""
    L, H, D, B, C = 2, 2, 64, 16, 256
    w = synth.custom(L, H, D, B, C, 60, [256, 256, 160], [256, 256, 160], seed=4, residency="device")
    for k in (3, 4, 9):                                  # middle blocks of request 1 and 2 are request 0's
        for r in (1, 2):
            w.requests[r].block_table[k] = w.requests[0].block_table[k]
    buf = buffers.allocate(w)
    kvs.kvs_retrieve(w.geom, buf.plane_ptrs, w.num_blocks, buf.requests, None)
    torch.cuda.synchronize()
    # request 0 wins every tie, so the result is requests 2, 1, 0 written in that order
    w.requests.reverse()
    buf.chunks.reverse()
    gc.check_retrieve(buf)
