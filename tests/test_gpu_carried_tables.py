"""Calls whose tables travel in the launches' parameters, beside calls that upload them.

Tables of up to 3584 bytes are carried; the sizes here lie on both sides of that, and
calls of both kinds alternate without waiting, so that a table reused too early would
show.  Exact equality with the CPU oracle.
"""
import pytest
import torch

import gpu_check as gc
from paper_2609_35065_gb300 import buffers, kvs, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    torch.cuda.set_device(0)
    yield
    torch.cuda.synchronize()


def _table_bytes(w):
    g = w.geom
    entries = sum(len(w.chunk_counts(r)) for r in w.requests)
    return 2 * g.layers * 8 + entries * 16 + entries * (g.chunk_tokens // g.block_size) * 4 + 8


def _workload(requests, seed, residency, tokens=500):
    return synth.custom(3, 2, 64, 16, 256, 600, [tokens] * requests, [tokens] * requests, seed=seed, residency=residency)


@pytest.mark.parametrize("residency", ["host", "device", "mixed"])
def test_tables_around_the_limit(residency):
    """11, 21, 22 and 23 requests of two chunks (160 bytes a request): below, at and above."""
    sizes = []
    for n in (11, 21, 22, 23):
        res = residency if residency != "mixed" else ["host", "device"] * (n // 2) + ["host"] * (n % 2)
        w = synth.custom(3, 2, 64, 16, 256, n * 20, [300] * n, [300] * n, seed=n, residency=res)
        sizes.append(_table_bytes(w))
        buf = buffers.allocate(w)
        kvs.kvs_retrieve(w.geom, buf.plane_ptrs, w.num_blocks, buf.requests, None)
        torch.cuda.synchronize()
        gc.check_retrieve(buf)
    assert sizes[0] < 3584 < sizes[-1]


@pytest.mark.parametrize("residency", ["host", "device"])
def test_many_calls_in_flight(residency):
    """Forty calls of different tables queued behind a sleeping kernel, every third uploaded."""
    bufs = [buffers.allocate(_workload(24 if k % 3 == 0 else 1 + k % 4, k, residency, 280 + k)) for k in range(40)]
    assert any(_table_bytes(b.workload) > 3584 for b in bufs) and any(_table_bytes(b.workload) < 3584 for b in bufs)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        torch.cuda._sleep(20_000_000)
    for b in bufs:
        kvs.kvs_retrieve(b.workload.geom, b.plane_ptrs, b.workload.num_blocks, b.requests, s)
    s.synchronize()
    for b in bufs:
        gc.check_retrieve(b)


@pytest.mark.parametrize("lps", [1, 2])
def test_layer_groups_that_carry_and_that_upload(lps):
    """20 layers: 20 launches upload, 10 with two layers each too; 3 layers carry."""
    for L in (3, 20):
        w = synth.custom(L, 2, 64, 16, 256, 60, [300], [300], seed=L, residency="device")
        buf = buffers.allocate(w)
        kvs.kvs_retrieve_layers(w.geom, buf.plane_ptrs, w.num_blocks, buf.requests, lps, None, None)
        torch.cuda.synchronize()
        gc.check_retrieve(buf)


@pytest.mark.parametrize("flags", [0, kvs.KVS_F_VALIDATE], ids=["carried", "uploaded"])
@pytest.mark.parametrize("shape", [(3, 8, 128, 16), (2, 2, 64, 16), (2, 5, 256, 16)],
                         ids=["32KiB_runs", "4KiB_runs", "40KiB_runs"])
def test_forced_tma_small_calls(shape, flags):
    """TMA pieces with their tables in the launch's parameters, and uploaded."""
    L, H, D, B = shape
    w = synth.custom(L, H, D, B, 256, 80, [600, 256], [512, 256], seed=D, residency="device", store_tokens=[88, 0])
    buf = buffers.allocate(w, store=True, store_residency="device")
    assert _table_bytes(w) < 3584
    args = (w.geom, buf.plane_ptrs, w.num_blocks)
    kvs.kvs_retrieve(*args, buf.requests, None, kvs.KVS_F_FORCE_TMA | flags)
    kvs.kvs_store(*args, buf.store_requests, None, kvs.KVS_F_FORCE_TMA | flags)
    assert kvs.kvs_check_errors(None) == kvs.KVS_OK
    gc.check_retrieve(buf)
    gc.check_store(buf)
