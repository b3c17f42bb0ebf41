#!/usr/bin/env python
"""Prefix-KV retrieval benchmark on GB300 (fast tier -> paged GPU KV cache).

Default workload: Llama-3-8B-shaped KV (32 layers, 8 KV heads, head_dim 128,
bf16, 128 KiB/token), 16 requests of 4096-token prompts at 50% prefix hit
(2048 matched tokens each, 8 chunks of 256 tokens), 20,000-block paged cache
with a seeded random block assignment, chunks in pinned host memory.  One step
= one kvs_retrieve of the whole batch (4 GiB of KV).

Prints ONE JSON line.  ``--impl reference`` times the CPU oracle instead (the
plain element loop, on the host cores), on the same workload.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "prefix-KV retrieval GB/s and tokens/s on 1 GB300; % of HBM / host-link roofline"
MEASURED_PEAKS = os.path.join(ROOT, "MEASURED_PEAKS.json")
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "traffic.json")
# the copy kernels and the async-copy helpers they inline
KERNEL_SRCS = [os.path.join(ROOT, "paper_2609_35065_gb300", "csrc", f) for f in ("kvs_kernels.cu", "kvs_async.cuh", "kvs_job.cuh")]
HBM_FALLBACK_GBS = 6800.0


def parse_args(argv=None):
    ap = argparse.ArgumentParser(description=__doc__.splitlines()[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--config", default="llama8b",
                    help="llama8b | sweep25 | sweep50 | sweep75 | qwen14b | llama70b[_25|_50|_100]")
    ap.add_argument("--variant", choices=["auto", "hostlink", "hbmcopy", "few_sms"], default="auto",
                    help="host-chunk variant; few_sms: KVS_F_FEW_SMS (staged host-link kernel, its own cap)")
    ap.add_argument("--kernel", choices=["auto", "ldg", "tma"], default="auto")
    ap.add_argument("--max-ctas", type=int, default=0)
    ap.add_argument("--probe-bytes", type=int, default=1 << 30)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--skip-probe", action="store_true",
                    help="skip kvs_query_bw (profiling runs): built-in variant defaults, no host-link peak")
    ap.add_argument("--overlap", action="store_true", help="llama70b: retrieval beside a bf16 GEMM loop")
    ap.add_argument("--layerwise", action="store_true",
                    help="llama8b: layer-wise retrieval pipelined with a per-layer prefill GEMM")
    ap.add_argument("--tempokv", action="store_true",
                    help="TempoKV control-plane model driven by the retrieval rate measured in this run")
    ap.add_argument("--sizes", action="store_true",
                    help="llama8b shape: retrieval rate against call size (1 to 128 chunks)")
    ap.add_argument("--tier", action="store_true",
                    help="llama8b: claims staged into the fast-tier ledger's pinned arena, retrieved from its slots")
    ap.add_argument("--duplex", action="store_true",
                    help="llama8b: retrieval (host->GPU) and store-back (GPU->host) at the same time")
    ap.add_argument("--side-priority", choices=["normal", "high"], default="high",
                    help="priority of the retrieval stream in --overlap runs")
    ap.add_argument("--fp8", action="store_true",
                    help="the workload's chunks as fp8 (E4M3 + per-head scales): retrieve and store-back rates")
    ap.add_argument("--no-extras", action="store_true",
                    help="default line without its extra legs (no-alloc, store to host, sweep50, overlap)")
    return ap.parse_args(argv)


# ---------------------------------------------------------------------------
def workload(name: str):
    from paper_2609_35065_gb300 import synth
    if name == "llama8b":
        return synth.llama8b()
    if name == "llama8b_small":          # profiling case: 512 MiB payload, 2.1 GB of planes
        return synth.llama8b(requests=2, num_blocks=1024)
    if name.startswith("sweep"):
        return synth.sweep(int(name[5:]) / 100.0)
    if name == "qwen14b":
        return synth.qwen14b()
    if name == "qwen14b_small":          # profiling case: 2.25 GiB retrieved, 768 MiB stored, 3.2 GB planes
        return synth.qwen14b(requests=1, num_blocks=1024)
    if name.startswith("llama70b"):
        frac = int(name.split("_")[1]) / 100.0 if "_" in name else 1.0
        return synth.llama70b(buffer_frac=frac)
    if name == "tiny":
        return synth.tiny()
    raise SystemExit(f"unknown config {name}")


def describe(w) -> str:
    g = w.geom
    m = w.matched_tokens
    return (f"{w.name}: L{g.layers} H{g.kv_heads} D{g.head_dim} bf16 B{g.block_size} C{g.chunk_tokens}, "
            f"{len(w.requests)} requests, {m} matched tokens, NB {w.num_blocks}")


def token_bytes(g) -> int:
    return 2 * g.layers * g.row_elems * g.elem_bytes


def measured_peaks() -> dict:
    try:
        with open(MEASURED_PEAKS) as f:
            return json.load(f)
    except (OSError, ValueError):
        return {}


def kernel_hash(src: str | None = None) -> str:
    """Hash of the kernel source with comments and whitespace removed: it changes
    with the code, not with its commentary."""
    import re
    if src is None:
        src = ""
        for path in KERNEL_SRCS:
            with open(path) as f:
                src += f.read() + "\n"
    src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
    src = re.sub(r"//[^\n]*", " ", src)
    return hashlib.sha256(" ".join(src.split()).encode()).hexdigest()[:16]


def recorded_traffic(kernel: str, config: str):
    """(per-launch DRAM bytes, provenance) from an ncu capture recorded for the current
    kernel source, else (None, why).  The bytes are a stored record, not measured in
    this run: the provenance says which capture and source hash they come from."""
    try:
        with open(TRAFFIC_FILE) as f:
            rec = json.load(f)
    except (OSError, ValueError):
        return None, {"kind": "none", "why": "no recorded capture"}
    ent = rec.get(f"{config}/{kernel}")
    sha = kernel_hash()
    if not ent:
        return None, {"kind": "none", "why": f"no recorded capture of {kernel} on {config}"}
    if ent.get("kernel_sha") != sha:
        return None, {"kind": "stale", "why": "kernel source changed since the capture",
                      "capture_kernel_sha": ent.get("kernel_sha"), "kernel_sha": sha}
    prov = {"kind": "recorded", "kernel_sha": sha, "capture": ent.get("capture", "profiles/traffic.json")}
    if "scaled_from" in ent:
        prov["scaled_from"] = ent["scaled_from"]
    return ent.get("dram_bytes_per_launch"), prov


class ClockSampler:
    """nvidia-smi clocks and throttle reasons, timestamped on arrival."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.samples = []
        self.proc = None
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(index), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "50"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            return
        self.thread = threading.Thread(target=self._read, daemon=True)
        self.thread.start()

    def _read(self):
        for line in self.proc.stdout:
            self.samples.append((time.time(), [x.strip() for x in line.split(",")]))

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self, t0: float, t1: float):
        if not self.samples:
            return None
        inside = [s for t, s in self.samples if t0 - 0.06 <= t <= t1 + 0.06] or \
                 [min(self.samples, key=lambda ts: abs(ts[0] - (t0 + t1) / 2))[1]]
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        reasons = set()
        sm, mx, pw = [], [], []
        for s in inside:
            try:
                sm.append(float(s[0]))
                mx.append(float(s[1]))
            except (ValueError, IndexError):
                continue
            try:
                pw.append(float(s[2]))
            except (ValueError, IndexError):
                pass
            for k, nm in enumerate(names):
                if len(s) > 4 + k and s[4 + k].lower().startswith("active"):
                    reasons.add(nm)
        if not sm:
            return None
        out = {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
               "samples": len(sm)}
        if pw:
            out["power_w"] = round(statistics.median(pw), 1)
        return out


# ---------------------------------------------------------------------------
# CPU oracle (baseline / reference arm)
# ---------------------------------------------------------------------------
def oracle_inputs_from_buffers(buf):
    from paper_2609_35065_gb300.buffers import NP_DTYPES
    npd = NP_DTYPES[buf.workload.geom.elem_bytes]
    return [[(t.numpy() if t.device.type == "cpu" else t.cpu().numpy()).view(npd) for t in mine]
            for mine in buf.chunks]


def oracle_pass(w, chunks_np, threads: int, planes=None) -> float:
    """One pass of the workload through the CPU oracle (planes [lo, hi) or all);
    each thread owns one reusable host plane.  Returns seconds."""
    import numpy as np
    from concurrent.futures import ThreadPoolExecutor
    import oracle

    g = w.geom
    P = 2 * g.layers
    planes = list(range(P)) if planes is None else list(planes)
    n = w.num_blocks * g.block_size * g.row_elems
    local = threading.local()

    def one(p):
        buf = getattr(local, "buf", None)
        if buf is None:
            buf = local.buf = np.empty(n, dtype=np.uint16)
        ps = [None] * P
        ps[p] = buf
        for r, req in enumerate(w.requests):
            if chunks_np[r]:
                oracle.retrieve(g.layers, g.kv_heads, g.head_dim, g.block_size, ps, w.num_blocks,
                                req.first_token, chunks_np[r], req.block_table, p0=p, p1=p + 1)

    with ThreadPoolExecutor(threads) as ex:
        list(ex.map(lambda p: None, range(threads)))     # start threads before timing
        t = time.perf_counter()
        list(ex.map(one, planes))
        return time.perf_counter() - t


def cpu_chunks(w):
    """Chunk buffers of ``w`` on the host (seeded, torch CPU generator)."""
    import numpy as np
    import torch
    from paper_2609_35065_gb300 import buffers
    buf = buffers.allocate(w, device="cpu", with_planes=False)
    return [[t.numpy().view(np.uint16) for t in mine] for mine in buf.chunks]


def max_over_ranks(x: float, dist=None, device: str = "cpu") -> float:
    """Largest value over all ranks (the slowest replica sets the job's time)."""
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(units_per_step: float, steps: int, world: int, total_ms: float) -> float:
    """Units all replicas processed per second: each rank runs its own copy of the
    workload (weak scaling), the time is the slowest rank's."""
    return units_per_step * steps * world / (total_ms / 1e3)


def moved_bytes(w):
    """Bytes each source class actually moves in one step: a physical block named by
    several requests is written once (by the writer covering most tokens)."""
    g = w.geom
    B = g.block_size
    row = 2 * g.layers * g.row_elems * g.elem_bytes // 1        # bytes per token, all planes
    best = {}
    for r in w.requests:
        for t0 in range(r.first_token, r.first_token + r.matched_tokens, B):
            blk = int(r.block_table[t0 // B])
            n = min(B, r.first_token + r.matched_tokens - t0)
            if blk not in best or n > best[blk][0]:
                best[blk] = (n, r.residency)
    out = {"host": 0, "device": 0}
    for n, res in best.values():
        out[res] += n * row
    return out


def host_cores() -> int:
    return len(os.sched_getaffinity(0))


def run_reference(args):
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    w = workload(args.config)
    chunks_np = cpu_chunks(w)
    cores = host_cores()
    payload = w.matched_tokens * token_bytes(w.geom)
    for _ in range(args.warmup):
        oracle_pass(w, chunks_np, cores)
    total = 0.0
    for _ in range(args.steps):
        total += oracle_pass(w, chunks_np, cores)
    gbs = payload * args.steps / total / 1e9
    line = {
        "metric": METRIC, "value": round(gbs, 3), "unit": "GB/s", "impl": "reference",
        "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": round(total / args.steps * 1e3, 3), "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16 (copied as u16)", "data": "synthetic",
        "config": {"workload": describe(w), "source": "host memory (oracle reads numpy buffers)"},
        "tokens_per_s": round(w.matched_tokens * args.steps / total, 1),
        "cpu_baseline": {"value": round(gbs, 3), "unit": "GB/s", "cores": cores, "kind": "oracle",
                         "sample": f"every step = the whole workload ({payload} bytes), all {2 * w.geom.layers} planes"},
        "e2e": {"value": round(gbs, 3), "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
def run_ours(args):
    import numpy as np
    import torch
    from paper_2609_35065_gb300 import buffers, kvs

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    else:
        torch.cuda.set_device(0)
    dev = torch.cuda.current_device()

    def barrier():
        if dist is not None:
            dist.barrier()
        torch.cuda.synchronize()

    kvs.lib()
    stream = torch.cuda.Stream()
    bw = kvs.kvs_get_choice() if args.skip_probe else kvs.kvs_query_bw(stream, args.probe_bytes)
    host_peak = max(bw["h2d_copy_engine_gbs"], bw["zero_copy_read_gbs"]) or float("nan")

    w = workload(args.config)
    g = w.geom
    buf = buffers.allocate(w)
    payload = buf.payload_bytes
    tokens = w.matched_tokens
    flags = 0
    if args.variant == "hostlink":
        flags |= kvs.KVS_F_FORCE_HOSTLINK
    elif args.variant == "hbmcopy":
        flags |= kvs.KVS_F_FORCE_HBMCOPY
    elif args.variant == "few_sms":
        flags |= kvs.KVS_F_FEW_SMS
    if args.kernel == "ldg":
        flags |= kvs.KVS_F_FORCE_LDG
    elif args.kernel == "tma":
        flags |= kvs.KVS_F_FORCE_TMA
    if args.max_ctas:
        flags |= kvs.KVS_F_MAX_CTAS(args.max_ctas)
    choice = kvs.kvs_get_choice()
    host_variant = {"hostlink": 1, "hbmcopy": 2, "few_sms": 1}.get(args.variant, choice["chosen_retrieve_host"])

    def step(requests, f=flags):
        kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, requests, stream, f)

    # correctness gate before timing: one validated call
    step(buf.requests, flags | kvs.KVS_F_VALIDATE)
    for _ in range(args.warmup):
        step(buf.requests)
    barrier()

    sampler = ClockSampler(dev)
    time.sleep(0.15)
    K = args.steps
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(K)]
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    launches0 = kvs.kvs_stat_launches()
    barrier()
    wall0 = time.time()
    t_start.record(stream)
    for k in range(K):
        ev[k][0].record(stream)
        step(buf.requests)
        ev[k][1].record(stream)
    t_end.record(stream)
    torch.cuda.synchronize()
    wall1 = time.time()
    barrier()
    launches = kvs.kvs_stat_launches() - launches0
    total_ms = max_over_ranks(t_start.elapsed_time(t_end), dist, "cuda")
    per_call_ms = [a.elapsed_time(b) for a, b in ev]
    call_ms = statistics.mean(per_call_ms)
    value = whole_job_rate(payload, K, world, total_ms) / 1e9
    tokens_per_s = whole_job_rate(tokens, K, world, total_ms)
    kernel_name = ("kvs_link_staged_kernel" if args.variant == "few_sms" else "kvs_link_kernel") if host_variant == 1 \
        else "hbmcopy_pipeline"

    # e2e: the public API from host arguments (request objects built anew each step),
    # each step's status word read back to the host.  Pipelined as a serving loop
    # runs: step k's 4-byte status is read while step k+1 already runs.
    e2e_steps = max(3, min(K, 20))
    desc_bytes = 8 * 2 * g.layers + sum(len(r.chunks) * (16 + 4 * (g.chunk_tokens // g.block_size))
                                        for r in buf.requests)
    words = torch.zeros(2, dtype=torch.int32, pin_memory=True)
    landed = [torch.cuda.Event(), torch.cuda.Event()]

    def status(k):
        landed[k % 2].synchronize()
        if int(words[k % 2]):
            raise RuntimeError(f"step {k}: device status {int(words[k % 2])}")

    barrier()
    t0 = time.perf_counter()
    for k in range(e2e_steps):
        reqs = [kvs.RequestArg(r.block_table, r.chunks, r.first_token) for r in buf.requests]
        kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, reqs, stream, flags)
        kvs.kvs_enqueue_error_read(stream, words[k % 2])   # 4-byte device->host read of the status
        landed[k % 2].record(stream)
        if k:
            status(k - 1)
    status(e2e_steps - 1)
    e2e_s = (time.perf_counter() - t0) / e2e_steps
    # the same with a synchronising status read after every step
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        reqs = [kvs.RequestArg(r.block_table, r.chunks, r.first_token) for r in buf.requests]
        kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, reqs, stream, flags)
        kvs.kvs_check_errors(stream)
    sync_s = (time.perf_counter() - t0) / e2e_steps
    e2e = {"value": round(payload * world / e2e_s / 1e9, 3), "unit": "GB/s",
           "h2d_bytes_per_step": int(payload + desc_bytes), "d2h_bytes_per_step": 4,
           "ms_per_step": round(e2e_s * 1e3, 3),
           "loop": "pipelined: step k's status read (kvs_enqueue_error_read) while step k+1 runs",
           "synchronous_value": round(payload * world / sync_s / 1e9, 3)}

    # device-resident (HBM staging) source, same workload: the HBM roofline
    hbm = hbm_store = None
    if rank == 0 and w.name.startswith("llama8b"):
        dpool = torch.empty_like(buf.host_pool, device="cuda")
        dpool.copy_(buf.host_pool)
        per_tok = 2 * g.layers * g.row_elems
        dreqs = []
        at = 0
        for r in buf.requests:
            cs = []
            for c in r.chunks:
                cs.append(kvs.ChunkArg(dpool[at:at + c.num_tokens * per_tok], c.num_tokens, kvs.KVS_SRC_DEVICE))
                at += c.num_tokens * per_tok
            dreqs.append(kvs.RequestArg(r.block_table, cs, r.first_token))
        dflags = flags & ~(kvs.KVS_F_FORCE_HOSTLINK | kvs.KVS_F_FORCE_HBMCOPY)
        step(dreqs, dflags | kvs.KVS_F_VALIDATE)
        for _ in range(3):
            step(dreqs, dflags)
        torch.cuda.synchronize()
        nd = max(5, min(K, 20))
        dev_ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nd)]
        for a, b in dev_ev:                       # back to back: planning overlaps the previous copy
            a.record(stream)
            step(dreqs, dflags)
            b.record(stream)
        torch.cuda.synchronize()
        dev_ms = [a.elapsed_time(b) for a, b in dev_ev]
        dms = statistics.mean(dev_ms)
        peaks = measured_peaks()
        # the roofline is the faster of the driver's copy measurement and our own
        # flat copy kernel in this run (both count read + write bytes)
        drv_pk = peaks.get("hbm_gbs", HBM_FALLBACK_GBS)
        hpk = max(drv_pk, bw["hbm_copy_gbs"])
        hpk_src = ("in-run flat copy kernel (kvs_query_bw hbm_copy_gbs, read+write bytes)" if hpk > drv_pk else
                   "MEASURED_PEAKS.json hbm_gbs (copy, read+write bytes)" if peaks else "fallback")
        ach = 2 * payload / (dms / 1e3) / 1e9
        tma = args.kernel == "tma" or (args.kernel == "auto" and choice["chosen_kernel_device"] == 2)
        if args.max_ctas:
            kname = "kvs_tma_kernel" if tma else "kvs_span_kernel"
        else:
            kname = "kvs_tma_piece_kernel" if tma else "kvs_ldg_piece_kernel"
        tr, tr_src = recorded_traffic(kname, "llama8b_device")
        hbm = {"bound": "hbm", "achieved": round(ach, 1), "peak": round(hpk, 1), "unit": "GB/s",
               "frac": round(ach / hpk, 4), "traffic": tr, "traffic_source": tr_src,
               "kernel": kname, "payload_gbs": round(payload / (dms / 1e3) / 1e9, 1),
               "peak_source": hpk_src, "measured_peaks_hbm_gbs": drv_pk,
               "frac_of_measured_peaks": round(ach / drv_pk, 4),
               "bytes_counted": "2 x payload (read + write)"}

        # store-back (gather) of the same blocks into the HBM-resident chunks
        def sstep(f=dflags):
            kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, dreqs, stream, f)
        sstep(dflags | kvs.KVS_F_VALIDATE)
        for _ in range(3):
            sstep()
        torch.cuda.synchronize()
        st_ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(nd)]
        for a, b in st_ev:
            a.record(stream)
            sstep()
            b.record(stream)
        torch.cuda.synchronize()
        sms = statistics.mean(a.elapsed_time(b) for a, b in st_ev)
        sach = 2 * payload / (sms / 1e3) / 1e9
        tr, tr_src = recorded_traffic(kname, "llama8b_device_store")
        hbm_store = {"bound": "hbm", "achieved": round(sach, 1), "peak": round(hpk, 1), "unit": "GB/s",
                     "frac": round(sach / hpk, 4), "traffic": tr, "traffic_source": tr_src,
                     "peak_source": hpk_src, "measured_peaks_hbm_gbs": drv_pk,
                     "frac_of_measured_peaks": round(sach / drv_pk, 4),
                     "kernel": kname,
                     "payload_gbs": round(payload / (sms / 1e3) / 1e9, 1),
                     "bytes_counted": "2 x payload (read + write)"}
        del dpool

    def timed_calls(fn, n):
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n)]
        fn()
        torch.cuda.synchronize()
        for a, b in evs:
            a.record(stream)
            fn()
            b.record(stream)
        torch.cuda.synchronize()
        return statistics.mean(a.elapsed_time(b) for a, b in evs) / 1e3

    extras = {}
    classes = {r.residency for r in w.requests}
    if len(classes) > 1:                      # report each source class separately
        per_tok_b = token_bytes(g)
        for cls in sorted(classes):
            sub = [ra for ra, r in zip(buf.requests, w.requests) if r.residency == cls]
            nbytes = sum(r.matched_tokens for r in w.requests if r.residency == cls) * per_tok_b
            sec = timed_calls(lambda: step(sub), max(3, min(K, 10)))
            extras[f"class_{cls}"] = {"gbs": round(nbytes / sec / 1e9, 2), "bytes": nbytes,
                                      "rw_gbs": round((2 if cls == "device" else 1) * nbytes / sec / 1e9, 2)}
    if any(r.store_tokens for r in w.requests):
        sbuf = buffers.allocate(w, store=True, with_planes=False)
        nbytes = sum(r.store_tokens for r in w.requests) * token_bytes(g)
        sec = timed_calls(lambda: kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, sbuf.store_requests, stream, 0),
                          max(3, min(K, 10)))
        d2h_peak = max(bw["d2h_copy_engine_gbs"], bw["zero_copy_write_gbs"]) or float("nan")
        extras["store_host"] = {"gbs": round(nbytes / sec / 1e9, 2), "bytes": nbytes,
                                "frac_of_d2h_link": round(nbytes / sec / 1e9 / d2h_peak, 4),
                                "variant": {1: "hostlink", 2: "hbmcopy"}[choice["chosen_store_host"]]}
        del sbuf

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        chunks_np = oracle_inputs_from_buffers(buf)
        cores = host_cores()
        secs = oracle_pass(w, chunks_np, cores)
        sub = list(range(min(4, 2 * g.layers)))
        secs1 = oracle_pass(w, chunks_np, 1, sub)
        cpu = {"value": round(payload / secs / 1e9, 3), "unit": "GB/s", "cores": cores, "kind": "oracle",
               "sample": f"one full pass of the workload ({payload} bytes, all {2 * g.layers} planes), "
                         f"threads split by plane",
               "single_thread": {"value": round(payload * len(sub) / (2 * g.layers) / secs1 / 1e9, 3),
                                 "unit": "GB/s", "cores": 1,
                                 "sample": f"planes 0-{len(sub) - 1} of {2 * g.layers} (same bytes per plane)"}}

    if rank == 0 and world == 1 and w.name == "llama8b" and not args.no_extras:
        extras.update(default_line_legs(args, buf, bw, stream, sampler, flags))
    time.sleep(0.1)
    sampler.stop()
    clocks = sampler.summary(wall0, wall1)
    mv = moved_bytes(w)
    hbm_peak = measured_peaks().get("hbm_gbs", HBM_FALLBACK_GBS)
    if mv["device"] == 0:
        achieved = mv["host"] / (call_ms / 1e3) / 1e9
        tr, tr_src = recorded_traffic(kernel_name, w.name)
        roofline = {"bound": "host_link", "achieved": round(achieved, 2), "peak": round(host_peak, 2),
                    "unit": "GB/s", "frac": round(achieved / host_peak, 4),
                    "traffic": tr, "traffic_source": tr_src, "kernel": kernel_name,
                    "peak_source": "measured in this run: max(copy-engine pinned H2D, zero-copy read kernel)",
                    "bytes_counted": f"bytes moved over the host link per step ({mv['host']})"}
    else:
        # both classes run concurrently: the step cannot beat the slower of the two
        ideal_s = max(mv["host"] / (host_peak * 1e9), 2 * mv["device"] / (hbm_peak * 1e9))
        achieved = payload / (call_ms / 1e3) / 1e9
        peak = payload / ideal_s / 1e9
        roofline = {"bound": "host_link+hbm", "achieved": round(achieved, 2), "peak": round(peak, 2),
                    "unit": "GB/s", "frac": round(achieved / peak, 4), "traffic": None,
                    "kernel": "kvs_link_kernel (host) + device-class kernel on a second stream",
                    "peak_source": "payload / max(host bytes / in-run host-link peak, "
                                   "2 x device bytes / MEASURED_PEAKS hbm_gbs)",
                    "bytes_counted": f"host {mv['host']} over the link, device {mv['device']} read+written in HBM"}
    if rank == 0:
        line = {
            "metric": METRIC, "value": round(value, 3), "unit": "GB/s", "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": round(total_ms / K, 4), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16 (copied as u16)", "data": "synthetic",
            "config": {"workload": describe(w), "source": "pinned host memory (fast-tier stand-in)",
                       "variant": {1: "hostlink", 2: "hbmcopy"}[host_variant],
                       "l2": f"inputs ({payload >> 20} MiB per step) larger than L2; no flush",
                       "parallelism": f"replicas x{world}"},
            "tokens_per_s": round(tokens_per_s, 1),
            "per_step": {"best_ms": round(min(per_call_ms), 4), "median_ms": round(statistics.median(per_call_ms), 4),
                         "best_gbs": round(payload / min(per_call_ms) / 1e6, 3),
                         "median_gbs": round(payload / statistics.median(per_call_ms) / 1e6, 3)},
            "roofline": roofline,
            "roofline_hbm": hbm,
            "roofline_hbm_store": hbm_store,
            "extras": extras or None,
            "cpu_baseline": cpu,
            "e2e": e2e,
            "gpu_launches": int(launches),
            "clocks": clocks,
            "bw_probe": {k: (round(v, 2) if isinstance(v, float) else v) for k, v in bw.items()},
        }
        print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


COPY_ENGINE_ONLY = -1          # overlap variant: plain copy-engine copy of the pinned buffer, no scatter


def FP8(flags: int = 0):
    """Overlap variant: the same tokens retrieved from fp8 chunks (kvs_retrieve_fp8)."""
    return ("fp8", flags)


def overlap_measure(w, bw, side, variants, sampler=None):
    """Retrieval of workload ``w`` on the ``side`` stream while the current stream runs a
    bf16 8192 x 8192 GEMM loop, for each (name, flags) of ``variants``, alone and beside the
    GEMM.  The pinned fast-tier buffer holds ``w.notes['buffer_frac']`` of the batch and is
    refilled between passes (untimed).  Returns {name: {"alone": ..., "with_gemm": ...}},
    with the clocks of each GEMM window when ``sampler`` is given."""
    import torch
    from paper_2609_35065_gb300 import kvs, synth

    g = w.geom
    frac = w.notes.get("buffer_frac", 1.0)
    passes = max(1, int(round(1 / frac)))
    per_pass = len(w.requests) // passes
    per_tok = 2 * g.layers * g.row_elems
    main = torch.cuda.current_stream()
    host_peak = max(bw["h2d_copy_engine_gbs"], bw["zero_copy_read_gbs"])
    n = w.num_blocks * g.block_size * g.row_elems
    planes = torch.full((2 * g.layers, n), synth.SENTINEL_BF16, dtype=torch.int16, device="cuda")
    ptrs = [int(planes[p].data_ptr()) for p in range(2 * g.layers)]
    tokens_pass = sum(r.matched_tokens for r in w.requests[:per_pass])
    pinned = torch.empty(tokens_pass * per_tok, dtype=torch.int16, pin_memory=True)
    src = torch.empty(tokens_pass * per_tok, dtype=torch.int16, device="cuda")
    synth.fill_values(src, w.dist, torch.Generator(device="cuda").manual_seed(w.seed))
    pinned.copy_(src)
    del src
    refill_src = pinned.clone() if passes > 1 else None      # stands in for the next pass's KV
    C = g.chunk_tokens
    fp8_chunk_bytes = 2 * g.layers * C * g.row_elems + (2 * g.layers * g.kv_heads * 4 + 255) // 256 * 256

    fp8 = {}

    def fp8_requests(k):
        """The pass's tokens as fp8 chunks in one pinned pool (built on first use)."""
        from paper_2609_35065_gb300 import buffers
        if "pool" not in fp8:
            cb = (buffers.fp8_chunk_bytes(g, C) + 255) // 256 * 256
            fp8["cb"] = cb
            fp8["pool"] = torch.empty((tokens_pass // C) * cb, dtype=torch.uint8, pin_memory=True)
            gen = torch.Generator(device="cuda").manual_seed(w.seed)
            for j in range(tokens_pass // C):
                buffers.fill_fp8_chunk(fp8["pool"][j * cb:(j + 1) * cb], g, gen)
            fp8["refill"] = fp8["pool"].clone() if passes > 1 else None
        cb, pool = fp8["cb"], fp8["pool"]
        reqs, at = [], 0
        for r in w.requests[k * per_pass:(k + 1) * per_pass]:
            cs = []
            for j in range(r.matched_tokens // C):
                cs.append(kvs.ChunkArg(pool[at:at + buffers.fp8_chunk_bytes(g, C)], C))
                at += cb
            reqs.append(kvs.RequestArg(r.block_table, cs))
        return reqs

    def pass_requests(k):
        reqs, at = [], 0
        for r in w.requests[k * per_pass:(k + 1) * per_pass]:
            cs = []
            for j in range(r.matched_tokens // C):
                cs.append(kvs.ChunkArg(pinned[at:at + C * per_tok], C))
                at += C * per_tok
            reqs.append(kvs.RequestArg(r.block_table, cs))
        return reqs

    a = torch.randn(8192, 8192, dtype=torch.bfloat16, device="cuda")
    b = torch.randn(8192, 8192, dtype=torch.bfloat16, device="cuda")
    c = torch.empty(8192, 8192, dtype=torch.bfloat16, device="cuda")

    def ev():
        return torch.cuda.Event(enable_timing=True)

    # The GEMM loop runs at the power cap, where the clock settles only after a
    # few hundred milliseconds: every measured window follows ~0.5 s of GEMMs,
    # and the GEMM rate beside a retrieval is compared with the same loop
    # alone over a window of the same length, measured right after it.
    for _ in range(5):
        torch.matmul(a, b, out=c)
    torch.cuda.synchronize()
    e0, e1 = ev(), ev()
    e0.record(main)
    for _ in range(50):
        torch.matmul(a, b, out=c)
    e1.record(main)
    torch.cuda.synchronize()
    gemm_ms = e0.elapsed_time(e1) / 50
    preheat = max(1, int(500 / gemm_ms))

    def gemm_window(iters, side_work=None):
        """Preheat, then `iters` GEMMs from g0 (side_work starts on the side
        stream at g0 too); returns (g0, per-GEMM end events, side's end event)."""
        for _ in range(preheat):
            torch.matmul(a, b, out=c)
        g0 = ev()
        g0.record(main)
        end = None
        if side_work is not None:
            side.wait_event(g0)
            side_work()
            end = ev()
            end.record(side)
        gev = []
        for _ in range(iters):
            torch.matmul(a, b, out=c)
            e = ev()
            e.record(main)
            gev.append(e)
        torch.cuda.synchronize()
        return g0, gev, end

    def rate_within(g0, gev, window_ms):
        done = [t for t in (g0.elapsed_time(e) for e in gev) if t <= window_ms]
        return (2 * 8192 ** 3 * len(done) / (done[-1] / 1e3) / 1e12) if done else float("nan")

    scratch = {}

    def copy(reqs, flags):
        """One retrieval of ``reqs``; KVS_F_LAYER_LAUNCHES here means one launch per layer
        (a layer-wise call without events), which hands SMs back between layers.  The
        flags value COPY_ENGINE_ONLY instead copies the pass's pinned buffer into one HBM
        buffer with a plain cudaMemcpyAsync: the copy engine's rate with no scatter."""
        if isinstance(flags, tuple):
            kvs.kvs_retrieve_fp8(g, ptrs, w.num_blocks, reqs, side, flags[1])
            return
        if flags == COPY_ENGINE_ONLY:
            if "dst" not in scratch:
                scratch["dst"] = torch.empty_like(pinned, device="cuda")
            with torch.cuda.stream(side):
                scratch["dst"].copy_(pinned, non_blocking=True)
            return
        if flags & kvs.KVS_F_LAYER_LAUNCHES:
            kvs.kvs_retrieve_layers(g, ptrs, w.num_blocks, reqs, 1, None, side, flags)
        else:
            kvs.kvs_retrieve(g, ptrs, w.num_blocks, reqs, side, flags)

    def retrieval(flags, with_gemm):
        total_ms, gemm_during, gemm_alone = 0.0, [], []
        wall = [time.time(), None]
        is_fp8 = isinstance(flags, tuple)
        for k in range(passes):
            reqs = fp8_requests(k) if is_fp8 else pass_requests(k)
            if k:                                        # refill between passes (untimed)
                if is_fp8:
                    fp8["pool"].copy_(fp8["refill"])
                else:
                    pinned.copy_(refill_src)
            copy(reqs, flags)                            # warm
            torch.cuda.synchronize()
            if not with_gemm:
                r0, r1 = ev(), ev()
                r0.record(side)
                copy(reqs, flags)
                r1.record(side)
                torch.cuda.synchronize()
                total_ms += r0.elapsed_time(r1)
                continue
            # GEMMs queued so that they outlast the retrieval
            iters = int(1.3 * (tokens_pass * per_tok * 2 / (host_peak * 1e9)) / (gemm_ms / 1e3)) + 4
            g0, gev, r1 = gemm_window(iters, lambda: copy(reqs, flags))
            r_ms = g0.elapsed_time(r1)
            total_ms += r_ms
            gemm_during.append(rate_within(g0, gev, r_ms))
            a0, aev, _ = gemm_window(iters)
            gemm_alone.append(rate_within(a0, aev, r_ms))
        wall[1] = time.time()
        moved = tokens_pass // C * fp8_chunk_bytes if is_fp8 else tokens_pass * per_tok * 2
        gbs = passes * moved / (total_ms / 1e3) / 1e9
        out = {"retrieval_gbs": round(gbs, 2), "frac_of_host_link": round(gbs / host_peak, 4),
               "tokens_per_s": round(passes * tokens_pass / (total_ms / 1e3), 1)}
        if with_gemm:
            during, alone = statistics.mean(gemm_during), statistics.mean(gemm_alone)
            out.update({"gemm_tflops_during": round(during, 1), "gemm_tflops_alone_same_window": round(alone, 1),
                        "gemm_kept": round(during / alone, 4)})
            if sampler is not None:
                out["clocks"] = sampler.summary(*wall)
        return out

    results = {}
    for name, fl in variants:
        results[name] = {"alone": retrieval(fl, False), "with_gemm": retrieval(fl, True)}
    info = {"buffer_frac": frac, "passes": passes, "host_link_peak_gbs": round(host_peak, 2),
            "gemm": "bf16 8192x8192x8192 torch.matmul loop on the main stream",
            "gemm_tflops_short_burst": round(2 * 8192 ** 3 / (gemm_ms / 1e3) / 1e12, 1)}
    del planes, pinned, refill_src, a, b, c
    scratch.clear()
    fp8.clear()
    torch.cuda.empty_cache()
    return results, info


def default_line_legs(args, buf, bw, stream, sampler, flags):
    """Extra legs of the default line, each a short window with its own clock record:

    * ``noalloc``: the same 4 GiB batch through kvs_retrieve_noalloc (allocation-free
      entry point), next to kvs_retrieve's rate;
    * ``store_host``: the batch stored back from the paged cache into its pinned host
      chunks (the store-back direction over the host link);
    * ``sweep50``: the mixed-residency sweep at 50% prefix hit (32 requests x 4096
      matched tokens, half in HBM staging, half in pinned host memory) into the same
      20,000-block cache, with each source class alone;
    * ``overlap``: the 70B-shaped batch (pinned buffer of 25%, 4 passes, refilled
      between passes) retrieved on a high-priority side stream beside a bf16 8192^3
      GEMM loop: at the default CTA cap, with KVS_F_FEW_SMS (the staged kernel on its
      measured cap), from fp8 chunks of the same tokens (``tokens_per_s`` compares them;
      default grid and KVS_F_FEW_SMS), and as a plain copy-engine copy.
    """
    import torch
    from paper_2609_35065_gb300 import buffers, kvs, synth

    w = buf.workload
    g = w.geom
    payload = buf.payload_bytes
    host_peak = max(bw["h2d_copy_engine_gbs"], bw["zero_copy_read_gbs"])
    d2h_peak = max(bw["d2h_copy_engine_gbs"], bw["zero_copy_write_gbs"])
    hbm_peak = max(measured_peaks().get("hbm_gbs", HBM_FALLBACK_GBS), bw["hbm_copy_gbs"])
    n = max(5, min(args.steps, 20))
    legs = {}

    def timed(fn):
        """Mean and best seconds of n back-to-back calls of fn (CUDA events on `stream`),
        and the wall-clock window they ran in."""
        fn()
        torch.cuda.synchronize()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n)]
        t0 = time.time()
        for a, b in evs:
            a.record(stream)
            fn()
            b.record(stream)
        torch.cuda.synchronize()
        t1 = time.time()
        ms = [a.elapsed_time(b) for a, b in evs]
        return statistics.mean(ms) / 1e3, min(ms) / 1e3, (t0, t1)

    # the allocation-free entry point on the same batch (host chunks: the link kernel on
    # kvs_retrieve's cap), and kvs_retrieve again over the same window length
    kvs.kvs_retrieve_noalloc(g, buf.plane_ptrs, w.num_blocks, buf.requests, stream, kvs.KVS_F_VALIDATE)
    sec, best, win = timed(lambda: kvs.kvs_retrieve_noalloc(g, buf.plane_ptrs, w.num_blocks, buf.requests,
                                                            stream, flags & 0xFFFF0000))
    ref, _, _ = timed(lambda: kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, buf.requests, stream, flags))
    legs["noalloc"] = {"gbs": round(payload / sec / 1e9, 2), "best_gbs": round(payload / best / 1e9, 2),
                       "frac_of_host_link": round(payload / sec / 1e9 / host_peak, 4),
                       "kvs_retrieve_gbs_same_window": round(payload / ref / 1e9, 2), "calls": n,
                       "kernel": "kvs_link_kernel (host chunks, kvs_retrieve's CTA cap)",
                       "clocks": sampler.summary(*win)}

    # store-back of the same blocks into the pinned host chunks
    kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, buf.requests, stream, kvs.KVS_F_VALIDATE)
    sec, best, win = timed(lambda: kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, buf.requests, stream, 0))
    choice = kvs.kvs_get_choice()
    legs["store_host"] = {"gbs": round(payload / sec / 1e9, 2), "best_gbs": round(payload / best / 1e9, 2),
                          "frac_of_d2h_link": round(payload / sec / 1e9 / d2h_peak, 4),
                          "d2h_link_peak_gbs": round(d2h_peak, 2), "bytes": payload, "calls": n,
                          "variant": {1: "hostlink", 2: "hbmcopy"}[choice["chosen_store_host"]],
                          "ctas": choice["store_ctas"], "clocks": sampler.summary(*win)}

    # mixed residency at 50% prefix hit, into the same cache (same geometry and block pool)
    ws = synth.sweep(0.5)
    sb = buffers.allocate(ws, with_planes=False)
    mv = moved_bytes(ws)
    spay = mv["host"] + mv["device"]

    def sweep_call(reqs, f=0):
        kvs.kvs_retrieve(g, buf.plane_ptrs, ws.num_blocks, reqs, stream, f)

    sweep_call(sb.requests, kvs.KVS_F_VALIDATE)
    sec, best, win = timed(lambda: sweep_call(sb.requests))
    ideal = max(mv["host"] / (host_peak * 1e9), 2 * mv["device"] / (hbm_peak * 1e9))
    leg = {"gbs": round(spay / sec / 1e9, 2), "tokens_per_s": round(ws.matched_tokens / sec, 1),
           "frac_of_roofline": round(ideal / sec, 4), "bytes": spay, "calls": n,
           "roofline": "max(host bytes / host-link peak, 2 x device bytes / HBM peak)",
           "clocks": sampler.summary(*win)}
    for cls in ("host", "device"):
        sub = [ra for ra, r in zip(sb.requests, ws.requests) if r.residency == cls]
        csec, _, _ = timed(lambda: sweep_call(sub))
        cb = mv[cls]
        leg[f"class_{cls}"] = {"gbs": round(cb / csec / 1e9, 2), "bytes": cb,
                               "frac": round(cb / csec / 1e9 / host_peak, 4) if cls == "host"
                               else round(2 * cb / csec / 1e9 / hbm_peak, 4)}
    legs["sweep50"] = leg
    del sb
    torch.cuda.empty_cache()

    # fp8 chunks (E4M3 + per-head scales) of the same batch: half the bytes over the link
    import copy
    w8 = copy.deepcopy(w)
    for r in w8.requests:                   # store the retrieved tokens back into fresh fp8 chunks
        r.store_tokens, r.store_first = r.matched_tokens, r.first_token
    fb = buffers.allocate_fp8(w8, store=True, with_planes=False)
    fbytes = fb.payload_bytes
    kvs.kvs_retrieve_fp8(g, buf.plane_ptrs, w.num_blocks, fb.requests, stream, kvs.KVS_F_VALIDATE)
    sec, best, win = timed(lambda: kvs.kvs_retrieve_fp8(g, buf.plane_ptrs, w.num_blocks, fb.requests, stream, 0))
    kvs.kvs_store_fp8(g, buf.plane_ptrs, w.num_blocks, fb.store_requests, stream, kvs.KVS_F_VALIDATE)
    ssec, sbest, swin = timed(lambda: kvs.kvs_store_fp8(g, buf.plane_ptrs, w.num_blocks, fb.store_requests,
                                                        stream, 0))
    legs["fp8"] = {"retrieve": {"link_gbs": round(fbytes / sec / 1e9, 2),
                                "frac_of_host_link": round(fbytes / sec / 1e9 / host_peak, 4),
                                "tokens_per_s": round(w.matched_tokens / sec, 1),
                                "bf16_bytes_delivered_gbs": round(payload / sec / 1e9, 2),
                                "kernel": "kvs_fp8_retrieve_kernel", "clocks": sampler.summary(*win)},
                   "store": {"link_gbs": round(fbytes / ssec / 1e9, 2),
                             "frac_of_d2h_link": round(fbytes / ssec / 1e9 / d2h_peak, 4),
                             "tokens_per_s": round(w.matched_tokens / ssec, 1),
                             "kernel": "kvs_fp8_store_head_kernel", "clocks": sampler.summary(*swin)},
                   "chunk_bytes": fbytes, "format": "OCP OFP8 rev 1.0 E4M3 codes + binary32 scale per "
                                                    "(chunk, layer, K/V, head)", "calls": n}
    del fb
    torch.cuda.empty_cache()

    # retrieval beside a bf16 GEMM loop (70B shape, 25% buffer), default cap
    side = torch.cuda.Stream(priority=-1)
    w70 = synth.llama70b(buffer_frac=0.25)
    results, info = overlap_measure(w70, bw, side, [
        ("default", 0),
        ("few_sms", kvs.KVS_F_FEW_SMS),
        ("fp8", FP8()),
        ("fp8_few_sms", FP8(kvs.KVS_F_FEW_SMS)),
        ("copy_engine_only", COPY_ENGINE_ONLY)], sampler)
    choice = kvs.kvs_get_choice()
    legs["overlap"] = {"workload": describe(w70), **info, "hostlink_ctas": choice["hostlink_ctas"],
                       "few_sm_ctas": choice["few_sm_ctas"], "side_stream": "high priority", **results}
    return legs


def run_fp8(args):
    """Retrieval from, and store-back into, fp8 chunks (E4M3 codes with one binary32 scale
    per chunk, layer, K/V and head) of the workload, host-resident as in its config:
    link GB/s (fp8 bytes), prefix tokens/s, and the BF16 line's tokens/s for comparison."""
    import copy
    import torch
    from paper_2609_35065_gb300 import buffers, kvs

    torch.cuda.set_device(0)
    kvs.lib()
    stream = torch.cuda.Stream()
    bw = kvs.kvs_get_choice() if args.skip_probe else kvs.kvs_query_bw(stream, args.probe_bytes)
    host_peak = max(bw["h2d_copy_engine_gbs"], bw["zero_copy_read_gbs"]) or float("nan")
    d2h_peak = max(bw["d2h_copy_engine_gbs"], bw["zero_copy_write_gbs"]) or float("nan")
    w = copy.deepcopy(workload(args.config))
    for r in w.requests:
        r.store_tokens, r.store_first = r.matched_tokens, r.first_token
    g = w.geom
    fb = buffers.allocate_fp8(w, store=True)
    fbytes = fb.payload_bytes
    flags = kvs.KVS_F_MAX_CTAS(args.max_ctas) if args.max_ctas else 0
    if args.variant == "few_sms":
        flags |= kvs.KVS_F_FEW_SMS

    def timed(fn, k):
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(k)]
        for a, b in evs:
            a.record(stream)
            fn()
            b.record(stream)
        torch.cuda.synchronize()
        return [a.elapsed_time(b) / 1e3 for a, b in evs]

    def ret():
        kvs.kvs_retrieve_fp8(g, fb.plane_ptrs, w.num_blocks, fb.requests, stream, flags)

    def sto():
        kvs.kvs_store_fp8(g, fb.plane_ptrs, w.num_blocks, fb.store_requests, stream, flags)

    kvs.kvs_retrieve_fp8(g, fb.plane_ptrs, w.num_blocks, fb.requests, stream, flags | kvs.KVS_F_VALIDATE)
    kvs.kvs_store_fp8(g, fb.plane_ptrs, w.num_blocks, fb.store_requests, stream, flags | kvs.KVS_F_VALIDATE)
    for _ in range(args.warmup):
        ret()
        sto()
    torch.cuda.synchronize()
    sampler = ClockSampler(torch.cuda.current_device())
    time.sleep(0.15)
    t0 = time.time()
    rs = timed(ret, args.steps)
    t1 = time.time()
    ss = timed(sto, args.steps)
    t2 = time.time()
    time.sleep(0.1)
    sampler.stop()
    rm, sm = statistics.mean(rs), statistics.mean(ss)
    line = {"metric": METRIC + " (fp8 chunks)", "unit": "GB/s", "value": round(fbytes / rm / 1e9, 3),
            "steps": args.steps, "warmup": args.warmup, "dtype": "fp8 e4m3 chunks -> bf16 planes",
            "config": {"workload": describe(w), "source": "pinned host memory" if w.requests[0].residency == "host"
                       else "HBM", "chunk_bytes": fbytes,
                       "format": "OCP OFP8 rev 1.0 E4M3 + binary32 scale per (chunk, layer, K/V, head)"},
            "retrieve": {"link_gbs": round(fbytes / rm / 1e9, 2), "frac_of_host_link": round(fbytes / rm / 1e9 / host_peak, 4),
                         "tokens_per_s": round(w.matched_tokens / rm, 1), "ms": round(rm * 1e3, 4),
                         "clocks": sampler.summary(t0, t1)},
            "store": {"link_gbs": round(fbytes / sm / 1e9, 2), "frac_of_d2h_link": round(fbytes / sm / 1e9 / d2h_peak, 4),
                      "tokens_per_s": round(w.matched_tokens / sm, 1), "ms": round(sm * 1e3, 4),
                      "clocks": sampler.summary(t1, t2)},
            "host_link_peak_gbs": round(host_peak, 2), "d2h_link_peak_gbs": round(d2h_peak, 2)}
    # the same chunks staged in HBM: retrieve reads the codes (half the BF16 bytes) and writes
    # BF16 planes, store reads the planes and writes codes; 1.5 x the BF16 payload either way
    if not args.no_extras:
        hbm_peak = max(measured_peaks().get("hbm_gbs", HBM_FALLBACK_GBS), bw["hbm_copy_gbs"])
        dev = {}
        for name, pool in (("chunks", fb.pools[0]), ("store", fb.pools[-1])):
            dev[name] = pool.to("cuda")
        def dev_reqs(reqs, pool, dpool):
            base = int(pool.data_ptr())
            return [kvs.RequestArg(r.block_table, [kvs.ChunkArg(int(dpool.data_ptr()) + (kvs._addr(c.base) - base),
                                                               c.num_tokens, kvs.KVS_SRC_DEVICE) for c in r.chunks],
                                   r.first_token) for r in reqs]
        dreq = dev_reqs(fb.requests, fb.pools[0], dev["chunks"])
        dsto = dev_reqs(fb.store_requests, fb.pools[-1], dev["store"])
        payload16 = w.matched_tokens * token_bytes(g)
        kvs.kvs_retrieve_fp8(g, fb.plane_ptrs, w.num_blocks, dreq, stream, kvs.KVS_F_VALIDATE)
        kvs.kvs_store_fp8(g, fb.plane_ptrs, w.num_blocks, dsto, stream, kvs.KVS_F_VALIDATE)
        rd = statistics.mean(timed(lambda: kvs.kvs_retrieve_fp8(g, fb.plane_ptrs, w.num_blocks, dreq, stream, 0),
                                   args.steps))
        sd = statistics.mean(timed(lambda: kvs.kvs_store_fp8(g, fb.plane_ptrs, w.num_blocks, dsto, stream, 0),
                                   args.steps))
        line["hbm_source"] = {
            "retrieve": {"gbs_rw": round(1.5 * payload16 / rd / 1e9, 1), "frac_of_hbm": round(1.5 * payload16 / rd / 1e9 / hbm_peak, 4),
                         "tokens_per_s": round(w.matched_tokens / rd, 1), "ms": round(rd * 1e3, 4)},
            "store": {"gbs_rw": round(1.5 * payload16 / sd / 1e9, 1), "frac_of_hbm": round(1.5 * payload16 / sd / 1e9 / hbm_peak, 4),
                      "tokens_per_s": round(w.matched_tokens / sd, 1), "ms": round(sd * 1e3, 4)},
            "bytes_counted": "1.5 x BF16 payload (codes read + BF16 written, or BF16 read + codes written)",
            "hbm_peak_gbs": round(hbm_peak, 1)}
    print(json.dumps(line), flush=True)
    return 0


def run_overlap(args):
    """Retrieval of the 70B-shaped batch on a side stream while the main stream runs a
    bf16 8192 x 8192 GEMM loop; the pinned fast-tier buffer holds buffer_frac of the
    batch and is refilled between passes (untimed)."""
    import torch
    from paper_2609_35065_gb300 import kvs

    torch.cuda.set_device(0)
    kvs.lib()
    w = workload(args.config)
    side = torch.cuda.Stream(priority=-1 if args.side_priority == "high" else 0)
    bw = kvs.kvs_query_bw(side, 1 << 30)
    variants = [("default", 0), ("hostlink_full", kvs.KVS_F_FORCE_HOSTLINK | kvs.KVS_F_MAX_CTAS(bw["num_sms"] * 3)),
                ("hostlink_8ctas", kvs.KVS_F_FORCE_HOSTLINK | kvs.KVS_F_MAX_CTAS(8)),
                ("hostlink_12ctas", kvs.KVS_F_FORCE_HOSTLINK | kvs.KVS_F_MAX_CTAS(12)),
                ("hostlink_24ctas", kvs.KVS_F_FORCE_HOSTLINK | kvs.KVS_F_MAX_CTAS(24)),
                ("hbmcopy", kvs.KVS_F_FORCE_HBMCOPY),
                ("dma", kvs.KVS_F_FORCE_DMA),
                ("few_sms", kvs.KVS_F_FEW_SMS),
                ("few_sms_12ctas", kvs.KVS_F_FEW_SMS | kvs.KVS_F_MAX_CTAS(12)),
                ("few_sms_16ctas", kvs.KVS_F_FEW_SMS | kvs.KVS_F_MAX_CTAS(16)),
                ("few_sms_24ctas", kvs.KVS_F_FEW_SMS | kvs.KVS_F_MAX_CTAS(24)),
                ("fp8", FP8()), ("fp8_few_sms", FP8(kvs.KVS_F_FEW_SMS)),
                ("fp8_few_sms_12ctas", FP8(kvs.KVS_F_FEW_SMS | kvs.KVS_F_MAX_CTAS(12))),
                ("fp8_few_sms_8ctas", FP8(kvs.KVS_F_FEW_SMS | kvs.KVS_F_MAX_CTAS(8))),
                ("fp8_48ctas", FP8(kvs.KVS_F_MAX_CTAS(48))),
                ("fp8_24ctas", FP8(kvs.KVS_F_MAX_CTAS(24))), ("fp8_12ctas", FP8(kvs.KVS_F_MAX_CTAS(12))),
                ("prefetch_l2_12ctas", kvs.KVS_F_PREFETCH_L2 | kvs.KVS_F_MAX_CTAS(12)),
                ("prefetch_l2_24ctas", kvs.KVS_F_PREFETCH_L2 | kvs.KVS_F_MAX_CTAS(24)),
                ("copy_engine_only", COPY_ENGINE_ONLY),
                ("layer_launches", kvs.KVS_F_LAYER_LAUNCHES),
                ("layer_launches_96ctas", kvs.KVS_F_LAYER_LAUNCHES | kvs.KVS_F_MAX_CTAS(96))]
    sampler = ClockSampler(torch.cuda.current_device())
    results, info = overlap_measure(w, bw, side, variants, sampler)
    sampler.stop()
    line = {"metric": METRIC + " (overlap with a bf16 GEMM loop)", "unit": "GB/s",
            "config": {"workload": describe(w), **info},
            "side_stream_priority": args.side_priority, "hostlink_ctas_default": bw["hostlink_ctas"],
            "few_sm_ctas_default": bw["few_sm_ctas"],
            "variants": results}
    print(json.dumps(line), flush=True)
    return 0


def run_layerwise(args):
    """Prefill of the uncached suffix with the matched prefix retrieved layer by
    layer: layer l's compute (one bf16 GEMM sized like a Llama-3-8B layer over the
    suffix tokens) waits only for layer l's retrieval event.  Compared with
    retrieving everything first, and with the compute alone.

    The GEMM loop runs at the GPU's power cap, where the SM clock settles only
    after a few hundred milliseconds; single runs of ~0.27 s mostly measure
    that transient.  Each schedule is therefore timed as a sustained stretch of
    back-to-back repetitions, and the schedules are interleaved in two passes
    (A B C ... A B C ...) so that slow drift of the power state cancels."""
    import torch
    from paper_2609_35065_gb300 import buffers, kvs

    torch.cuda.set_device(0)
    kvs.lib()
    side = torch.cuda.Stream(priority=-1 if args.side_priority == "high" else 0)
    main = torch.cuda.current_stream()
    kvs.kvs_query_bw(side, 1 << 30)
    w = workload(args.config)
    g = w.geom
    for r in w.requests:                  # the computed suffix is stored back into chunks
        r.store_tokens = r.prompt_tokens - r.matched_tokens
    buf = buffers.allocate(w, store=True)
    # the same prefix and suffix as fp8 chunks (E4M3 + per-head scales), into the same planes
    fb = buffers.allocate_fp8(w, store=True, with_planes=False)
    suffix = sum(r.prompt_tokens - r.matched_tokens for r in w.requests)
    # per-layer prefill work of the suffix: q/k/v + o + gated MLP widths of Llama-3-8B
    M, K, N = suffix, 4096, (4096 + 2 * 1024) + 4096 + 3 * 14336
    a = torch.randn(M, K, dtype=torch.bfloat16, device="cuda")
    b = torch.randn(K, N, dtype=torch.bfloat16, device="cuda") * 0.01
    c = torch.empty(M, N, dtype=torch.bfloat16, device="cuda")
    L = g.layers

    def ev():
        return torch.cuda.Event(enable_timing=True)

    def copies(fp8):
        """The four copy calls, BF16 or fp8 chunks."""
        if fp8:
            return (lambda: kvs.kvs_retrieve_fp8(g, buf.plane_ptrs, w.num_blocks, fb.requests, side, 0),
                    lambda: kvs.kvs_store_fp8(g, buf.plane_ptrs, w.num_blocks, fb.store_requests, side, 0),
                    lambda lps, evs, fl: kvs.kvs_retrieve_fp8_layers(g, buf.plane_ptrs, w.num_blocks, fb.requests,
                                                                     lps, evs, side, fl),
                    lambda lps, fl, ready: kvs.kvs_store_fp8_layers(g, buf.plane_ptrs, w.num_blocks,
                                                                    fb.store_requests, lps, None, side, fl,
                                                                    ready_events=ready))
        return (lambda: kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, buf.requests, side, 0),
                lambda: kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, buf.store_requests, side, 0),
                lambda lps, evs, fl: kvs.kvs_retrieve_layers(g, buf.plane_ptrs, w.num_blocks, buf.requests,
                                                             lps, evs, side, fl),
                lambda lps, fl, ready: kvs.kvs_store_layers(g, buf.plane_ptrs, w.num_blocks, buf.store_requests,
                                                            lps, None, side, fl, ready_events=ready))

    def one(mode, lps=1, ctas=0):
        """Enqueue one prefill under schedule `mode` ("fp8_" + mode: fp8 chunks); the main
        stream ends after it."""
        fp8 = mode.startswith("fp8_")
        mode = mode[4:] if fp8 else mode
        retrieve_all, store_all, retrieve_layers, store_layers = copies(fp8)
        start = ev()
        start.record(main)
        side.wait_event(start)
        if mode == "compute":
            for _ in range(L):
                torch.matmul(a, b, out=c)
        elif mode == "serial":
            retrieve_all()
            done = ev()
            done.record(side)
            main.wait_event(done)
            for _ in range(L):
                torch.matmul(a, b, out=c)
        elif mode == "retrieve":
            retrieve_all()
            done = ev()
            done.record(side)
            main.wait_event(done)
        elif mode == "store_serial":
            for _ in range(L):
                torch.matmul(a, b, out=c)
            computed = ev()
            computed.record(main)
            side.wait_event(computed)
            store_all()
            done = ev()
            done.record(side)
            main.wait_event(done)
        elif mode == "store_layer":
            ready = []
            for _ in range(L):
                torch.matmul(a, b, out=c)
                ready.append(ev())
                ready[-1].record(main)
            store_layers(lps, kvs.KVS_F_MAX_CTAS(ctas), ready[lps - 1::lps] if lps > 1 else ready)
            done = ev()
            done.record(side)
            main.wait_event(done)
        else:
            groups = -(-L // lps)
            evs = [ev() for _ in range(groups)]
            fl = ((kvs.KVS_F_LAYER_SIGNAL if mode == "signal" else kvs.KVS_F_FEW_SMS if mode == "layer_few" else 0)
                  | kvs.KVS_F_MAX_CTAS(ctas))
            retrieve_layers(lps, evs, fl)
            for l in range(L):
                if l % lps == 0:
                    main.wait_event(evs[l // lps])
                torch.matmul(a, b, out=c)

    # "layer": the default (one launch per layer group); "signal": one resident
    # launch that signals each group (KVS_F_LAYER_SIGNAL); "layer_few": one launch
    # per group on the staged few-SM kernel (KVS_F_FEW_SMS)
    schedules = [("compute_only", "compute", 1, 0), ("serial", "serial", 1, 0),
                 ("layerwise_lps1", "layer", 1, 0), ("layerwise_lps4", "layer", 4, 0),
                 ("layerwise_lps8", "layer", 8, 0), ("layerwise_lps1_ctas4", "layer", 1, 4),
                 ("layerwise_signal_lps1", "signal", 1, 0), ("layerwise_signal_lps1_ctas4", "signal", 1, 4),
                 ("layerwise_signal_lps1_ctas16", "signal", 1, 16),
                 ("layerwise_few_sms_lps1", "layer_few", 1, 0), ("layerwise_few_sms_lps1_ctas8", "layer_few", 1, 8),
                 # store-back of the computed suffix: after the whole prefill, or layer by layer
                 ("store_serial", "store_serial", 1, 0), ("store_layerwise_lps1", "store_layer", 1, 0),
                 ("store_layerwise_lps1_ctas4", "store_layer", 1, 4),
                 # the same with fp8 chunks: half the bytes over the link
                 ("fp8_serial", "fp8_serial", 1, 0), ("fp8_layerwise_lps1", "fp8_layer", 1, 0),
                 ("fp8_store_serial", "fp8_store_serial", 1, 0), ("fp8_store_layerwise_lps1", "fp8_store_layer", 1, 0),
                 ("fp8_store_layerwise_lps1_ctas4", "fp8_store_layer", 1, 4),
                 ("fp8_store_layerwise_lps1_ctas32", "fp8_store_layer", 1, 32)]
    reps = max(3, min(args.steps, 10))
    sampler = ClockSampler(0)
    time.sleep(0.2)
    times = {name: [] for name, *_ in schedules}
    clocks = {name: [] for name, *_ in schedules}
    one("retrieve")
    torch.cuda.synchronize()
    retrieve_alone = []
    for _ in range(3):
        t0, t1 = ev(), ev()
        t0.record(main)
        one("retrieve")
        t1.record(main)
        torch.cuda.synchronize()
        retrieve_alone.append(t0.elapsed_time(t1))
    def block(mode, lps, ctas):
        one(mode, lps, ctas)                              # settle into this schedule
        t0, t1 = ev(), ev()
        t0.record(main)
        w0 = time.time()
        for _ in range(reps):
            one(mode, lps, ctas)
        t1.record(main)
        torch.cuda.synchronize()
        return t0.elapsed_time(t1) / reps, sampler.summary(w0 + 0.3, time.time())

    # compute-only blocks bracket every schedule (C S1 C S2 C ...); a schedule's
    # exposed copy time is taken against the mean of its two neighbours, which
    # cancels the slow drift of the power-capped clock
    exposed = {name: [] for name, *_ in schedules if name != "compute_only"}
    for _pass in range(2):
        before, clk = block("compute", 1, 0)
        times["compute_only"].append(before)
        clocks["compute_only"].append(clk)
        for name, mode, lps, ctas in schedules:
            if name == "compute_only":
                continue
            t, clk = block(mode, lps, ctas)
            after, _ = block("compute", 1, 0)
            times[name].append(t)
            clocks[name].append(clk)
            times["compute_only"].append(after)
            exposed[name].append(t - (before + after) / 2)
            before = after
    time.sleep(0.1)
    sampler.stop()
    res = {name: round(statistics.mean(v), 3) for name, v in times.items()}
    exp_ms = {k: round(statistics.mean(v), 3) for k, v in exposed.items()}
    best_lw = min((k for k in exp_ms if k.startswith("layerwise")), key=lambda k: exp_ms[k])
    store_gbs = []
    for _ in range(3):
        t0, t1 = ev(), ev()
        t0.record(side)
        kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, buf.store_requests, side, 0)
        t1.record(side)
        torch.cuda.synchronize()
        store_gbs.append(suffix * token_bytes(g) / (t0.elapsed_time(t1) / 1e3) / 1e9)
    line = {"metric": METRIC + " (layer-wise retrieval and store-back pipelined with prefill compute)",
            "unit": "ms per prefill", "higher_is_better": False,
            "config": {"workload": describe(w), "compute": f"per layer one bf16 GEMM {M}x{K}x{N} "
                       "(Llama-3-8B q/k/v/o/MLP widths over the uncached suffix tokens)",
                       "store": f"the {suffix}-token computed suffix to pinned host chunks",
                       "retrieval_stream_priority": args.side_priority,
                       "timing": f"{reps} back-to-back prefills per schedule, each schedule bracketed by "
                                 "compute-only blocks, two passes, mean"},
            "ms_per_prefill": res,
            "exposed_copy_ms": exp_ms,
            "exposed_copy_ms_per_pass": {k: [round(x, 3) for x in v] for k, v in exposed.items()},
            "retrieve_alone_ms": round(min(retrieve_alone), 3),
            "retrieval_gbs_alone": round(buf.payload_bytes / (min(retrieve_alone) / 1e3) / 1e9, 2),
            "store_alone_gbs": round(max(store_gbs), 2),
            "best_layerwise": best_lw,
            "speedup_vs_serial": round(res["serial"] / res[best_lw], 4),
            "clocks": {k: v[-1] for k, v in clocks.items()}}
    print(json.dumps(line), flush=True)
    return 0


def run_tempokv(args):
    """The control-plane model (12 synthetic documents, prefix ratios 50/75/100%,
    100 GiB fast tier, 50 GiB protected budget, 11 GiB/s staging) with the
    fast-tier -> GPU rate measured now by kvs_query_bw, and with the ~16.8 GB/s
    effective rate implied by the paper's own H100 PCIe measurement."""
    import time as _time

    import numpy as np
    from paper_2609_35065_gb300 import kvs, tempokv
    measured = None
    try:
        import torch
        if torch.cuda.is_available():
            torch.cuda.set_device(0)
            rep = kvs.kvs_query_bw(None, 1 << 30)
            measured = max(rep["retrieve_gbs"])
    except Exception:                                   # no GPU: the model alone
        measured = None
    rates = {"pcie_context_16.8": 16.8}
    if measured:
        rates["gb300_measured"] = round(measured, 2)
    # fp8 chunks (E4M3 codes + one binary32 scale per layer, K/V and head per 256-token chunk):
    # 64 KiB + 8 bytes per token at the 8B geometry, moved at the same link rate (the fp8
    # kernel holds 99% of the link, bench.py --fp8)
    scenarios = {name: (gbs, 128 * 1024) for name, gbs in rates.items()}
    if measured:
        scenarios["gb300_measured_fp8_chunks"] = (round(measured, 2), 64 * 1024 + 2 * 32 * 8 * 4 // 256)
    out = {}
    t0 = _time.perf_counter()
    for name, (gbs, per_tok) in scenarios.items():
        cal = tempokv.Calibration(retrieval_gbs=gbs, kv_bytes_per_token=per_tok)
        for ratio in (0.5, 0.75, 1.0):
            res = tempokv.simulate(tempokv.workload(ratio, cal=cal), cal)
            out[f"{name}/ratio{int(ratio * 100)}"] = {
                "p95_ttft_s": round(res.p95_ttft, 3), "throughput_tok_s": round(res.throughput_tok_s, 2),
                "C_gib_s_per_req": round(res.cost_gib_s_per_req, 3), "blocked_commit_attempts": res.blocked_attempts,
                "ordinary_retrievals": res.ordinary,
                "mean_commit_lead_s": round(float(np.mean(res.commit_lead_s)), 3) if res.commit_lead_s else None}
    line = {"metric": "TempoKV control-plane model: p95 TTFT, throughput and protected-capacity cost C",
            "unit": "s / tok/s / GiB.s per request", "config": {
                "workload": "12 synthetic documents, 16,078-67,744 tokens, arrivals every 0.5 s, <= 128 output tokens",
                "fast_tier": "100 GiB, protected budget 50 GiB, 11 GiB/s staging, FCFS <= 4 active",
                "retrieval_gbs": rates,
                "kv_bytes_per_token": {k: v[1] for k, v in scenarios.items()}}, "results": out,
            "model_seconds": round(_time.perf_counter() - t0, 2)}
    print(json.dumps(line), flush=True)
    return 0


def run_duplex(args):
    """Retrieval of the matched prefix and store-back of the computed suffix (4 GiB each,
    pinned host chunks) on two streams at once, against each alone: how much of the two
    host-link directions can be used together."""
    import torch
    from paper_2609_35065_gb300 import buffers, kvs

    torch.cuda.set_device(0)
    kvs.lib()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    bw = kvs.kvs_query_bw(s1, 1 << 30)
    w = workload(args.config)
    g = w.geom
    for r in w.requests:
        r.store_tokens = r.prompt_tokens - r.matched_tokens
    buf = buffers.allocate(w, store=True)
    rbytes = buf.payload_bytes
    sbytes = sum(r.store_tokens for r in w.requests) * token_bytes(g)

    def ev():
        return torch.cuda.Event(enable_timing=True)

    def run(retrieve, store, caps):
        torch.cuda.synchronize()
        t0 = ev()
        t0.record(s1)
        s2.wait_event(t0)
        if retrieve:
            kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, buf.requests, s1, kvs.KVS_F_MAX_CTAS(caps[0]))
        if store:
            kvs.kvs_store(g, buf.plane_ptrs, w.num_blocks, buf.store_requests, s2, kvs.KVS_F_MAX_CTAS(caps[1]))
        e1, e2 = ev(), ev()
        e1.record(s1)
        e2.record(s2)
        torch.cuda.synchronize()
        return t0.elapsed_time(e1), t0.elapsed_time(e2)

    reps = max(3, min(args.steps, 10))
    res = {}
    for name, r, st, caps in (("retrieve_alone", True, False, (0, 0)), ("store_alone", False, True, (0, 0)),
                              ("both_default_caps", True, True, (0, 0)), ("both_64_64", True, True, (64, 64)),
                              ("both_96_96", True, True, (96, 96))):
        run(r, st, caps)
        ts = [run(r, st, caps) for _ in range(reps)]
        r_ms = statistics.median(t[0] for t in ts)
        s_ms = statistics.median(t[1] for t in ts)
        d = {}
        if r:
            d["retrieve_gbs"] = round(rbytes / r_ms / 1e6, 2)
        if st:
            d["store_gbs"] = round(sbytes / s_ms / 1e6, 2)
        if r and st:
            d["aggregate_gbs"] = round((rbytes + sbytes) / max(r_ms, s_ms) / 1e6, 2)
        res[name] = d
    # the copy engines in both directions at once (1 GiB each way, pinned host memory)
    n = 1 << 30
    h_in = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    h_out = torch.empty(n, dtype=torch.uint8, pin_memory=True)
    d_in = torch.empty(n, dtype=torch.uint8, device="cuda")
    d_out = torch.zeros(n, dtype=torch.uint8, device="cuda")
    ce = {}
    for name, h2d, d2h in (("h2d_alone", True, False), ("d2h_alone", False, True), ("both", True, True)):
        ts = []
        for _ in range(reps + 1):
            torch.cuda.synchronize()
            t0 = ev()
            t0.record(s1)
            s2.wait_event(t0)
            if h2d:
                with torch.cuda.stream(s1):
                    d_in.copy_(h_in, non_blocking=True)
            if d2h:
                with torch.cuda.stream(s2):
                    h_out.copy_(d_out, non_blocking=True)
            e1, e2 = ev(), ev()
            e1.record(s1)
            e2.record(s2)
            torch.cuda.synchronize()
            ts.append(max(t0.elapsed_time(e1) if h2d else 0.0, t0.elapsed_time(e2) if d2h else 0.0))
        ce[name] = round((n * (h2d + d2h)) / statistics.median(ts[1:]) / 1e6, 2)
    res["copy_engines_gbs"] = ce
    line = {"metric": METRIC + " (retrieval and store-back concurrently)", "unit": "GB/s",
            "config": {"workload": describe(w), "store": "computed suffix to pinned host chunks",
                       "timing": f"median of {reps} runs"},
            "host_link_probe": {"h2d_gbs": round(bw["h2d_copy_engine_gbs"], 2),
                                "d2h_gbs": round(bw["d2h_copy_engine_gbs"], 2)},
            "hostlink_ctas": bw["hostlink_ctas"], "store_ctas": bw["store_ctas"], **res}
    print(json.dumps(line), flush=True)
    return 0


def run_sizes(args):
    """Retrieval rate against call size, host and HBM sources: the GPU time of back-to-back
    calls (CUDA events) and the latency of one synchronous call through the API
    (marshalling, planning, upload, launch, completion), for 1 to 128 chunks of 32 MiB."""
    import torch
    from paper_2609_35065_gb300 import buffers, kvs

    torch.cuda.set_device(0)
    kvs.lib()
    stream = torch.cuda.Stream()
    kvs.kvs_query_bw(stream, 1 << 30)
    w = workload("llama8b")
    g = w.geom
    buf = buffers.allocate(w)
    per_tok = 2 * g.layers * g.row_elems
    dpool = torch.empty_like(buf.host_pool, device="cuda")
    dpool.copy_(buf.host_pool)
    chunk_bytes = g.chunk_tokens * token_bytes(g)

    def requests(n, device):
        out, at, left = [], 0, n
        for r in buf.requests:
            if left == 0:
                break
            cs = []
            for c in r.chunks[:left]:
                base = dpool[at:at + c.num_tokens * per_tok] if device else c.base
                cs.append(kvs.ChunkArg(base, c.num_tokens, kvs.KVS_SRC_DEVICE if device else c.residency))
                at += c.num_tokens * per_tok
            at += sum(c.num_tokens for c in r.chunks[left:]) * per_tok
            left -= len(cs)
            out.append(kvs.RequestArg(r.block_table, cs, r.first_token))
        return out

    reps = max(5, min(args.steps, 20))
    res = {}
    for source in ("host", "device"):
        rows = {}
        for n in (1, 2, 4, 8, 16, 32, 64, 128):
            reqs = requests(n, source == "device")
            for _ in range(3):
                kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, reqs, stream, 0)
            torch.cuda.synchronize()
            t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            t0.record(stream)
            for _ in range(reps):
                kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, reqs, stream, 0)
            t1.record(stream)
            torch.cuda.synchronize()
            gpu_ms = t0.elapsed_time(t1) / reps
            lat = []
            for _ in range(reps):
                h0 = time.perf_counter()
                kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, reqs, stream, 0)
                stream.synchronize()
                lat.append((time.perf_counter() - h0) * 1e3)
            nbytes = n * chunk_bytes
            lat_ms = statistics.median(lat)
            rows[str(n)] = {"bytes": nbytes, "gpu_ms": round(gpu_ms, 4), "gpu_gbs": round(nbytes / gpu_ms / 1e6, 1),
                            "call_latency_ms": round(lat_ms, 4), "latency_gbs": round(nbytes / lat_ms / 1e6, 1)}
        res[source] = rows
    line = {"metric": METRIC + " (call size sweep)", "unit": "GB/s",
            "config": {"workload": "llama8b geometry, 1-128 chunks of 256 tokens (32 MiB each)",
                       "timing": f"gpu: {reps} back-to-back calls, CUDA events; latency: median of {reps} "
                                 "synchronous calls through the Python API"},
            **res}
    print(json.dumps(line), flush=True)
    return 0


def run_tier(args):
    """The 8B-shaped batch retrieved from the fast tier's own pinned arena: each request's
    chunks are committed as one claim (its ordered manifest), staged into arena slots (a
    host copy stands in for the SSD read), retrieved from the slots the ledger hands out,
    and released.  The planes must equal those of a retrieval from the ordinary pinned
    pool.  Reports the arena retrieval rate against the host link, the staging copy
    rate, the ledger's cost per operation and the protected byte-time C."""
    import ctypes
    import numpy as np
    import torch
    from paper_2609_35065_gb300 import buffers, kvs, synth

    torch.cuda.set_device(0)
    kvs.lib()
    stream = torch.cuda.Stream()
    bw = kvs.kvs_query_bw(stream, 1 << 30)
    host_peak = max(bw["h2d_copy_engine_gbs"], bw["zero_copy_read_gbs"])
    w = workload("llama8b")
    g = w.geom
    buf = buffers.allocate(w)
    chunk_bytes = g.chunk_tokens * token_bytes(g)
    n_obj = sum(len(r.chunks) for r in buf.requests)
    tier = kvs.Tier(n_obj + 32, n_obj + 8, chunk_bytes, arena=True)
    keys = {r: [r * 1000 + j for j in range(len(q.chunks))] for r, q in enumerate(buf.requests)}
    clock0 = time.perf_counter()

    def now():
        return time.perf_counter() - clock0

    op_us = {"commit": [], "staged": [], "begin_retrieval": [], "end_retrieval": []}

    def timed(name, fn, *a):
        t = time.perf_counter()
        out = fn(*a)
        op_us[name].append((time.perf_counter() - t) * 1e6)
        return out

    stage_s = 0.0
    for r, q in enumerate(buf.requests):
        for k in timed("commit", tier.commit, r + 1, keys[r], now()):
            dst = tier.slot_address(tier.object(k)["slot"])
            t = time.perf_counter()
            ctypes.memmove(dst, q.chunks[k % 1000].base.data_ptr(), chunk_bytes)   # the "SSD read"
            stage_s += time.perf_counter() - t
            timed("staged", tier.staged, k, now())
    areqs = []
    for r, q in enumerate(buf.requests):
        slots = timed("begin_retrieval", tier.begin_retrieval, r + 1, now(), len(keys[r]))
        areqs.append(kvs.RequestArg(q.block_table, [kvs.ChunkArg(tier.slot_address(sl), c.num_tokens)
                                                    for sl, c in zip(slots, q.chunks)], q.first_token))
    # bit-exact against a retrieval of the same batch from the ordinary pinned pool
    kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, buf.requests, stream, kvs.KVS_F_VALIDATE)
    ref = buf.planes.clone()
    buf.planes.fill_(int(np.array([synth.SENTINEL_BF16], dtype=np.uint16).view(np.int16)[0]))
    torch.cuda.synchronize()
    kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, areqs, stream, kvs.KVS_F_VALIDATE)
    torch.cuda.synchronize()
    equal = bool(torch.equal(ref, buf.planes))
    del ref
    reps = max(3, min(args.steps, 20))
    for _ in range(3):
        kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, areqs, stream, 0)
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record(stream)
    for _ in range(reps):
        kvs.kvs_retrieve(g, buf.plane_ptrs, w.num_blocks, areqs, stream, 0)
    t1.record(stream)
    torch.cuda.synchronize()
    ms = t0.elapsed_time(t1) / reps
    for r in range(len(buf.requests)):
        timed("end_retrieval", tier.end_retrieval, r + 1, now())
    st = tier.stats(now())
    gbs = buf.payload_bytes / (ms / 1e3) / 1e9
    line = {"metric": METRIC + " (retrieval from the fast tier's arena, claims through the ledger)",
            "unit": "GB/s", "value": round(gbs, 2),
            "config": {"workload": describe(w), "tier": f"{n_obj + 32} slots of {chunk_bytes >> 20} MiB, "
                       f"budget {n_obj + 8} objects, pinned arena", "claims": len(buf.requests),
                       "timing": f"{reps} back-to-back retrievals while every claim is Transferring"},
            "bit_exact_vs_pool": equal,
            "frac_of_host_link": round(gbs / host_peak, 4),
            "staging_copy_gbs": round(n_obj * chunk_bytes / stage_s / 1e9, 2),
            "ledger_us_per_op": {k: round(statistics.median(v), 1) for k, v in op_us.items()},
            "tier_stats": st,
            "cost_C_gib_s_per_request": round(st["protected_object_seconds"] * chunk_bytes / 2 ** 30
                                              / max(1, st["completed"]), 4)}
    print(json.dumps(line), flush=True)
    tier.close()
    return 0 if equal else 1


def main(argv=None):
    args = parse_args(argv)
    if args.tempokv:
        return run_tempokv(args)
    if args.impl == "reference":
        return run_reference(args)
    if args.overlap:
        return run_overlap(args)
    if args.fp8:
        return run_fp8(args)
    if args.layerwise:
        return run_layerwise(args)
    if args.duplex:
        return run_duplex(args)
    if args.sizes:
        return run_sizes(args)
    if args.tier:
        return run_tier(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
