"""fp8 store-back into HBM chunks against the CPU oracle, byte for byte, at the shapes
where its units change: several heads a unit, one, and one over a cluster of CTAs.

The conversions are defined to the last bit, so the comparison is exact.
"""
import pytest
import torch

import gpu_check as gc
from paper_2609_35065_gb300 import buffers, kvs, synth

pytestmark = pytest.mark.gpu

# (L, H, D, B, C, tokens stored by each request)
SHAPES = {
    "one_head_64KiB": (3, 4, 128, 16, 256, (700, 256, 1)),
    "pairs_of_80": (2, 6, 80, 16, 256, (512, 300)),          # 104 KiB units, idle threads
    "fours_of_48": (2, 8, 48, 8, 256, (512, 257)),
    "odd_heads_of_112": (2, 3, 112, 16, 256, (300, 256)),
    "one_head_of_192": (2, 2, 192, 16, 256, (400,)),
    "all_heads_of_16": (3, 5, 16, 1, 64, (130, 64)),
    "128_heads": (1, 128, 16, 4, 64, (100,)),
    "cluster_of_2": (2, 3, 256, 16, 256, (600, 255, 1)),
    "cluster_of_4": (2, 2, 512, 32, 256, (300, 512)),
    "cluster_of_2_odd_rows": (2, 1, 208, 1, 260, (520, 7)),
    "all_chunks_short": (2, 8, 128, 16, 256, (42, 17, 33)),
    "above_every_unit": (1, 1, 1024, 16, 256, (300,)),       # falls to the two-pass kernel
}


def _fill(buf, seed, infinities):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    for p in range(buf.planes.shape[0]):
        synth.fill_values(buf.planes[p], "normal", gen)
        if infinities:                                       # and NaNs, in some heads
            at = torch.randint(0, buf.planes[p].numel(), (5,), device="cuda", generator=gen)
            buf.planes[p][at] = torch.tensor([0x7F80, 0xFF80 - 65536, 0x7FC1, 0xFFC0 - 65536, 0x7F80],
                                             dtype=torch.int16, device="cuda")
    torch.cuda.synchronize()


@pytest.mark.parametrize("cap,infinities", [(0, False), (0, True), (1, False), (5, True)],
                         ids=["plain", "infinities", "1_cta", "5_ctas_infinities"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_store_units(name, cap, infinities):
    L, H, D, B, C, tokens = SHAPES[name]
    nb = sum(-(-t // B) for t in tokens) + 3
    w = synth.custom(L, H, D, B, C, nb, list(tokens), [0] * len(tokens), seed=D, store_tokens=list(tokens))
    buf = buffers.allocate_fp8(w, store=True, store_residency="device")
    _fill(buf, D + cap, infinities)
    kvs.kvs_store_fp8(w.geom, buf.plane_ptrs, w.num_blocks, buf.store_requests, None,
                      kvs.KVS_F_VALIDATE | kvs.KVS_F_MAX_CTAS(cap))
    torch.cuda.synchronize()
    gc.check_store_fp8(buf)


@pytest.mark.parametrize("name", sorted(SHAPES))
def test_store_units_with_carried_tables(name):
    """The ordinary small call: its tables in the launch's parameters (validated calls upload them)."""
    L, H, D, B, C, tokens = SHAPES[name]
    nb = sum(-(-t // B) for t in tokens) + 3
    w = synth.custom(L, H, D, B, C, nb, list(tokens), [0] * len(tokens), seed=D, store_tokens=list(tokens))
    buf = buffers.allocate_fp8(w, store=True, store_residency="device")
    _fill(buf, D, True)
    kvs.kvs_store_fp8(w.geom, buf.plane_ptrs, w.num_blocks, buf.store_requests, None)
    assert kvs.kvs_check_errors(None) == kvs.KVS_OK
    gc.check_store_fp8(buf)
