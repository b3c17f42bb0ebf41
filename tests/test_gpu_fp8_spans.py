"""fp8 retrieval by span pieces against the CPU oracle, bit for bit: runs shorter than a
piece of 16 KiB of codes, runs that are no whole number of pieces, heads that change
inside a piece, and planes that are 16- but not 32-byte aligned.

The conversions are defined to the last bit, so the comparison is exact.
"""
import pytest
import torch

import gpu_check as gc
from paper_2609_35065_gb300 import buffers, kvs, synth

pytestmark = pytest.mark.gpu

# (L, H, D, B, C, matched tokens of the requests)
SHAPES = {
    "2KiB_runs": (3, 2, 64, 16, 256, (700, 256, 1)),
    "512B_runs": (2, 1, 64, 8, 512, (1024, 513)),
    "16B_runs": (2, 1, 16, 1, 256, (300, 255)),
    "20KiB_runs": (2, 10, 128, 16, 256, (512, 259)),
    "24KiB_runs_head_96": (2, 16, 96, 16, 128, (300,)),
    "head_80": (2, 3, 80, 16, 256, (257, 40)),
    "head_176_rows_cross_pieces": (2, 5, 176, 3, 48, (200, 47)),
    "one_vector": (1, 1, 16, 1, 1, (1,)),
    "all_chunks_short": (3, 2, 64, 16, 256, (42, 17, 33)),
    "rows_of_512_vectors": (1, 64, 128, 4, 64, (130, 3)),    # a thread's vectors are still of one head
    "rows_of_1024_vectors": (1, 128, 128, 2, 32, (73,)),
}


def _buffers(name, residency):
    L, H, D, B, C, tokens = SHAPES[name]
    nb = sum(-(-t // B) for t in tokens) + 3
    return buffers.allocate_fp8(synth.custom(L, H, D, B, C, nb, list(tokens), list(tokens), seed=D, residency=residency))


@pytest.mark.parametrize("cap", [0, 1, 5], ids=["uncapped", "1_cta", "5_ctas"])
@pytest.mark.parametrize("residency", ["host", "device"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_fp8_span_pieces(name, residency, cap):
    buf = _buffers(name, residency)
    w = buf.workload
    kvs.kvs_retrieve_fp8(w.geom, buf.plane_ptrs, w.num_blocks, buf.requests, None, kvs.KVS_F_MAX_CTAS(cap))
    kvs.kvs_check_errors(None)
    torch.cuda.synchronize()
    gc.check_retrieve_fp8(buf)


@pytest.mark.parametrize("residency", ["host", "device"])
def test_fp8_planes_aligned_to_16_bytes(residency):
    """Plane bases at odd multiples of 16 bytes: neighbouring lanes' stores meet sectors halfway."""
    buf = _buffers("2KiB_runs", residency)
    w = buf.workload
    P, n = buf.planes.shape
    shifted = torch.empty(P * (n + 16) + 8, dtype=torch.int16, device="cuda")
    planes = [shifted[8 + p * (n + 16):][:n] for p in range(P)]
    for p in range(P):
        planes[p].copy_(buf.planes[p])
    assert any(t.data_ptr() % 32 for t in planes) and not any(t.data_ptr() % 16 for t in planes)
    torch.cuda.synchronize()
    kvs.kvs_retrieve_fp8(w.geom, [t.data_ptr() for t in planes], w.num_blocks, buf.requests, None)
    torch.cuda.synchronize()
    for p in range(P):
        buf.planes[p].copy_(planes[p])
    gc.check_retrieve_fp8(buf)
