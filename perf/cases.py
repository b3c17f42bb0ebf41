"""Performance cases: retrieval of matched prefix KV into a paged cache, and store-back.

Every case is one call of the package's public functions, on buffers that a
serving program has in hand: the paged planes, the block tables, the chunk
buffers of the fast tier (pinned host memory, or a staging copy in HBM).

Keys of a case
  op        "retrieve" (chunks -> planes) or "store" (planes -> chunks)
  fmt       "kv" (chunks hold the planes' bytes) or "fp8" (E4M3 codes with per-head scales)
  where     residency of the chunks: "host", "hbm", or "mixed" (requests alternate)
  L H D e   layers, KV heads, head dim, bytes per cache element (2: BF16, 1: opaque bytes)
  B         tokens per paged block; C tokens per full chunk
  requests  requests in the call, `tokens` matched (or newly computed) tokens in each; a
            count that C does not divide leaves a partial last chunk
  shared    leading blocks that all requests of the call share (a common prefix)
  lps       layers per group of the layer-wise call, 0 for the whole call at once
  entry     "plain", or "noalloc" for the allocation-free retrieval
"""
import numpy as np
import torch

from paper_2609_35065_gb300 import kvs

# The largest payload (bytes in the planes) of a drawn case: calls that touch host
# memory run at the host link's rate, about a sixteenth of HBM's.
MOST_HBM = 4 << 30
MOST_HOST = 640 << 20


def _case(name, op, fmt, where, L, H, D, requests, tokens, e=2, B=16, C=256, shared=0, lps=0, entry="plain"):
    return {"name": name, "op": op, "fmt": fmt, "where": where, "L": L, "H": H, "D": D, "e": e, "B": B, "C": C,
            "requests": requests, "tokens": tokens, "shared": shared, "lps": lps, "entry": entry}


def listed():
    return [
        # The smallest call: two chunks of a small model, 1 MiB over the host link; what counts is
        # the time until the call's kernel has run.
        _case("tiny_host", "retrieve", "kv", "host", 2, 4, 64, 1, 512),
        # One cached chunk of the 8B-shaped model (32 layers, 8 KV heads) from its HBM staging
        # copy: a short system prompt that most requests hit.
        _case("one_chunk_hbm", "retrieve", "kv", "hbm", 32, 8, 128, 1, 256),
        # A whole batch of the same shape from HBM: 16 requests, 2048 matched tokens each, 4 GiB.
        _case("batch_hbm", "retrieve", "kv", "hbm", 32, 8, 128, 16, 2048),
        # The 14B-shaped model (48 layers) from pinned host memory, requests with a common prefix:
        # 15 of each one's 96 blocks are the same physical blocks.
        _case("shared_prefix_host", "retrieve", "kv", "host", 48, 8, 128, 2, 1536, shared=15),
        # New KV leaves for the fast tier after a prefill of odd length: into host memory, ...
        _case("suffix_to_host", "store", "kv", "host", 32, 8, 128, 2, 1413),
        # ... and into HBM chunks, 14B-shaped, four requests.
        _case("suffix_to_hbm", "store", "kv", "hbm", 48, 8, 128, 4, 1811),
        # fp8 chunks: a batch read from HBM and dequantised, ...
        _case("fp8_batch_hbm", "retrieve", "fp8", "hbm", 32, 8, 128, 8, 2048),
        # ... quantised on store-back into HBM, ...
        _case("fp8_suffix_to_hbm", "store", "fp8", "hbm", 32, 8, 128, 8, 1900),
        # ... and read over the host link layer group by layer group, as a model that starts on its
        # first layers while the rest is still on the way has it.
        _case("fp8_layers_host", "retrieve", "fp8", "host", 32, 8, 128, 2, 2048, lps=8),
        # A head dim that is no power of two (80), quantised on store-back.
        _case("fp8_head80_to_hbm", "store", "fp8", "hbm", 32, 8, 80, 4, 1024),
        # A small model with two KV heads of 64: one block of one plane is 4 KiB.
        _case("few_heads_hbm", "retrieve", "kv", "hbm", 24, 2, 64, 16, 2000),
        # Rows of 120 bytes, no multiple of 16: three heads of 20, half of the requests' chunks in
        # host memory and half in HBM.
        _case("odd_rows_mixed", "retrieve", "kv", "mixed", 12, 3, 20, 6, 900),
    ]


def _spread(rng, lo, hi):
    """A whole number in [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))


def draw(rng):
    op = rng.choice(["retrieve", "retrieve", "store"])
    fmt = rng.choice(["kv", "kv", "fp8"])
    where = rng.choice(["host", "hbm", "hbm", "mixed"])
    L = _spread(rng, 2, 80)
    H = rng.choice([1, 2, 3, 4, 5, 8, 8, 16])
    if fmt == "fp8":
        D, e = rng.choice([48, 64, 80, 96, 128, 128, 192]), 2
    else:
        D, e = rng.choice([20, 64, 64, 72, 80, 96, 128, 128, 128, 192, 256]), rng.choice([2, 2, 2, 1])
    B = rng.choice([8, 16, 16, 16, 32])
    C = rng.choice([128, 256, 256, 256])
    requests = _spread(rng, 1, 32)
    per_token = 2 * L * H * D * e
    most = (MOST_HBM if where == "hbm" else MOST_HOST) // per_token
    tokens = _spread(rng, min(40, max(1, most // requests)), max(1, min(8192, most // requests)))
    shared, lps, entry = 0, 0, "plain"
    if op == "retrieve" and fmt == "kv" and requests > 1 and rng.random() < 0.25:
        shared = min(tokens // B, 1 + rng.randrange(16))
    if rng.random() < 0.2:
        lps = 1 + rng.randrange(L)
    elif op == "retrieve" and fmt == "kv" and rng.random() < 0.15:
        entry = "noalloc"
    return {"op": op, "fmt": fmt, "where": where, "L": L, "H": H, "D": D, "e": e, "B": B, "C": C,
            "requests": requests, "tokens": tokens, "shared": shared, "lps": lps, "entry": entry}


# ---- sizes ------------------------------------------------------------------
def _counts(case):
    """Tokens of each chunk of one request."""
    full, rest = divmod(case["tokens"], case["C"])
    return [case["C"]] * full + ([rest] if rest else [])


def _scale_bytes(case):
    return (2 * case["L"] * case["H"] * 4 + 255) // 256 * 256


def _chunk_bytes(case, n):
    """Bytes of a chunk of n tokens."""
    row = case["H"] * case["D"]
    if case["fmt"] == "fp8":
        return _scale_bytes(case) + 2 * case["L"] * n * row
    return 2 * case["L"] * n * row * case["e"]


def _where(case, r):
    return case["where"] if case["where"] != "mixed" else ("host" if r % 2 == 0 else "hbm")


def _unique_tokens(case):
    """Tokens of distinct physical slots that the call's requests name."""
    return case["requests"] * case["tokens"] - (case["requests"] - 1) * case["shared"] * case["B"]


def work(case):
    planes = 2 * case["L"] * case["H"] * case["D"] * case["e"] * _unique_tokens(case)
    if case["fmt"] == "fp8":
        chunks = case["requests"] * sum(_chunk_bytes(case, n) for n in _counts(case))
    else:
        chunks = planes                  # a shared block is read from one of its chunks
    return {"bytes": planes + chunks, "flops": 0}


def tolerance(case):
    # Bytes are copied, and the fp8 conversions are defined to the last bit.
    return "exact"


# ---- inputs -----------------------------------------------------------------
class State:
    pass


def _values(n, e, gen):
    """n seeded cache elements on the GPU: BF16 of a unit normal, or random bytes."""
    if e == 1:
        return torch.randint(0, 256, (n,), dtype=torch.uint8, device="cuda", generator=gen)
    out = torch.empty(n, dtype=torch.bfloat16, device="cuda")
    for at in range(0, n, 1 << 28):
        m = min(1 << 28, n - at)
        out[at:at + m].normal_(generator=gen)
    return out


def _fp8_chunk(case, n, gen):
    """A quantised chunk of n tokens of unit-normal KV: its scale block, then its codes."""
    P, H, D = 2 * case["L"], case["H"], case["D"]
    x = _values(P * n * H * D, 2, gen).view(P, n, H, D)
    amax = x.abs().amax(dim=(1, 3)).float().clamp_min(1e-20)                        # [P, H]
    codes = (x.float() * (448.0 / amax)[:, None, :, None]).clamp_(-448, 448).to(torch.float8_e4m3fn)
    head = torch.zeros(_scale_bytes(case), dtype=torch.uint8, device="cuda")
    head[:P * H * 4] = (amax / 448.0).reshape(-1).view(torch.uint8)
    return torch.cat([head, codes.view(torch.uint8).reshape(-1)])


def prepare(case, seed):
    P, H, D, B, e = 2 * case["L"], case["H"], case["D"], case["B"], case["e"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    perm = np.random.default_rng(seed)
    st = State()
    st.case = case
    st.geom = (case["L"], H, D, e, B, case["C"])

    # block tables: blocks of a pool that holds a quarter more than the call needs, in random order
    per = -(-case["tokens"] // B)
    need = case["requests"] * (per - case["shared"]) + case["shared"]
    st.num_blocks = need + need // 4 + 1
    ids = perm.permutation(st.num_blocks).astype(np.int32)
    common, own = ids[:case["shared"]], ids[case["shared"]:]
    st.tables = [np.concatenate([common, own[r * (per - case["shared"]):(r + 1) * (per - case["shared"])]])
                 for r in range(case["requests"])]

    # the paged cache: one allocation, 2L equally spaced planes
    dt = torch.bfloat16 if e == 2 else torch.uint8
    n_plane = st.num_blocks * B * H * D
    if case["op"] == "store":
        st.planes = _values(P * n_plane, e, gen).view(P, n_plane)
    else:
        st.planes = torch.zeros(P, n_plane, dtype=dt, device="cuda")
    base, step = st.planes.data_ptr(), n_plane * e
    st.plane_ptrs = [base + p * step for p in range(P)]

    # the chunk buffers, 256-byte aligned in one pool per residency
    counts = _counts(case)
    room = [-(-_chunk_bytes(case, n) // 256) * 256 for n in counts]
    st.pools = {}
    for where in ("host", "hbm"):
        k = sum(_where(case, r) == where for r in range(case["requests"]))
        if k:
            st.pools[where] = torch.empty(k * sum(room), dtype=torch.uint8, pin_memory=where == "host",
                                          device="cpu" if where == "host" else "cuda").zero_()
    at = {"host": 0, "hbm": 0}
    st.chunks, st.requests, shared = [], [], []
    cdt = torch.uint8 if case["fmt"] == "fp8" else dt
    for r in range(case["requests"]):
        where, mine = _where(case, r), []
        for j, n in enumerate(counts):
            t = st.pools[where][at[where]:at[where] + _chunk_bytes(case, n)].view(cdt)
            at[where] += room[j]
            if case["op"] == "retrieve" and case["fmt"] == "fp8":
                t.copy_(_fp8_chunk(case, n, gen))
            elif case["op"] == "retrieve":
                v = _values(P * n * H * D, e, gen)
                k = min(n, case["shared"] * B - j * case["C"])     # leading tokens that request 0 holds too
                if k > 0 and r == 0:
                    shared.append(v.view(P, n, H * D)[:, :k].clone())
                elif k > 0:
                    v.view(P, n, H * D)[:, :k] = shared[j]
                t.copy_(v)
            mine.append(t)
        st.chunks.append(mine)
        res = kvs.KVS_SRC_HOST_PINNED if where == "host" else kvs.KVS_SRC_DEVICE
        st.requests.append(kvs.RequestArg(st.tables[r], [kvs.ChunkArg(t, n, res) for t, n in zip(mine, counts)]))
    groups = -(-case["L"] // case["lps"]) if case["lps"] else 0
    st.events = [torch.cuda.Event() for _ in range(groups)]
    for ev in st.events:
        ev.record()
    torch.cuda.synchronize()          # the library's own streams read these buffers too
    return st


# ---- one pass ---------------------------------------------------------------
def run(state):
    c = state.case
    args = (state.geom, state.plane_ptrs, state.num_blocks, state.requests)
    stream = torch.cuda.current_stream()
    if c["lps"]:
        call = {("retrieve", "kv"): kvs.kvs_retrieve_layers, ("store", "kv"): kvs.kvs_store_layers,
                ("retrieve", "fp8"): kvs.kvs_retrieve_fp8_layers, ("store", "fp8"): kvs.kvs_store_fp8_layers}
        call[c["op"], c["fmt"]](*args, c["lps"], state.events, stream)
    elif c["entry"] == "noalloc":
        kvs.kvs_retrieve_noalloc(*args, stream)
    else:
        call = {("retrieve", "kv"): kvs.kvs_retrieve, ("store", "kv"): kvs.kvs_store,
                ("retrieve", "fp8"): kvs.kvs_retrieve_fp8, ("store", "fp8"): kvs.kvs_store_fp8}
        call[c["op"], c["fmt"]](*args, stream)
    if c["op"] == "retrieve":
        return state.planes
    if c["fmt"] == "kv" and c["e"] == 2:
        return {where: pool.view(torch.bfloat16) for where, pool in state.pools.items()}
    return dict(state.pools)


# ---- the same in 64 bits ----------------------------------------------------
def exact(case, seed):
    if case["e"] != 2 or (case["op"] == "store" and case["fmt"] == "fp8"):
        return None                    # bytes, not numbers
    st = prepare(case, seed)
    P, H, D, B = 2 * case["L"], case["H"], case["D"], case["B"]
    planes = st.planes.double().view(P, st.num_blocks * B, H * D)
    pools = {w: torch.zeros(p.numel() // 2, dtype=torch.float64, device="cuda") for w, p in st.pools.items()}
    for r, mine in enumerate(st.chunks):
        first, where = 0, _where(case, r)
        table = torch.from_numpy(st.tables[r].astype(np.int64)).cuda()
        for t, n in zip(mine, _counts(case)):
            tok = torch.arange(first, first + n, device="cuda")
            slot = table[tok // B] * B + tok % B
            first += n
            if case["op"] == "store":
                at = (t.data_ptr() - st.pools[where].data_ptr()) // 2
                pools[where][at:at + t.numel()] = planes[:, slot].reshape(-1)
            elif case["fmt"] == "kv":
                planes[:, slot] = t.cuda().double().view(P, n, H * D)
            else:
                sb = _scale_bytes(case)
                scale = t[:P * H * 4].cuda().view(torch.float32).double().view(P, 1, H, 1)
                codes = t[sb:].cuda().view(torch.float8_e4m3fn).to(torch.float32).double().view(P, n, H, D)
                planes[:, slot] = (codes * scale).view(P, n, H * D)
    return pools if case["op"] == "store" else planes.view(P, -1)
