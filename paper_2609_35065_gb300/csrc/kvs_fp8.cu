// kvs_fp8.cu -- retrieval from, and store-back into, fp8 chunks on sm_103a.
//
// A compressed fast-tier format (the paper keeps BF16 KV, Sec. 5 setup): a
// chunk holds E4M3 codes of the OCP 8-bit floating point specification
// (revision 1.0) and one binary32 scale per (layer, K/V, head), so a
// retrieval moves half the bytes of a BF16 chunk over the host link:
//
//   chunk  [scales: 2L*H binary32 at (2l+kv)*H + h, padded to scale_bytes]
//          [codes:  [L][2][n][H][D] E4M3 bytes]
//   plane  BF16 [NB][B][H][D] per (layer, K/V)
//
//   retrieve  plane = bf16_rn(fp32(code) *rn scale); a NaN product gives 0x7FFF
//   store     per (chunk, layer, K/V, head): amax over the finite elements,
//             scale = amax /rn 448 (stored), inv = 448 /rn amax (both 1 when
//             amax is 0), code = e4m3 of x *rn inv, rounded to nearest even
//             and saturated at +-448; NaN gives the code 0x7F
//
// Every element conversion uses the hardware conversions of sm_89+ (E4M3 <->
// f16 pairs, f32 -> bf16 / E4M3 pairs, round to nearest even, the E4M3 one
// saturating) and IEEE round-to-nearest multiplies.  The conversions
// themselves give the canonical NaN patterns the format defines: 0x7FFF for a
// NaN product on retrieval, 0x7F for a NaN input of either sign on store (the
// special-values parity test plants NaN codes, NaN scales and NaN inputs of
// both signs and compares with the oracle).
//
// Retrieval is bound by the host link (or HBM for device chunks): a persistent
// grid of 512-thread CTAs walks span pieces of 16 KiB of codes; each thread keeps two
// pieces' worth of 16-byte code vectors in registers, so the next piece's loads
// are in flight while the current one is converted and stored.  HBM chunks run one
// CTA per piece instead, and KVS_F_FEW_SMS runs a kernel that also stages pieces in
// shared memory so that fewer SMs hold the link beside other kernels.
// Store-back to pinned host runs one 256-thread CTA per (chunk, plane, head):
// the head's BF16 elements are loaded into registers at once, reduced to the
// amax and quantised from registers (heads too large for that take a two-pass
// kernel, one CTA per (chunk, plane)).  Into HBM chunks persistent CTAs, two per
// SM, hold one unit of heads in shared memory and refill it with the next unit's
// loads while they convert.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "kvs.h"
#include "kvs_async.cuh"
#include "kvs_internal.h"
#include "kvs_job.cuh"

namespace kvs {
namespace {

// Threads, 16-code vectors per thread per piece, and CTAs per SM of the retrieval
// kernels: host chunks (two pieces in registers each), HBM chunks.
constexpr int kRtLink = 512, kRtLinkVec = 2, kRtLinkCtas = 2;
constexpr int kRtHbm = 256, kRtHbmVec = 4, kRtHbmCtas = 6;
static_assert(kRtLink * kRtLinkVec * 16 == kFp8PieceCodes && kRtHbm * kRtHbmVec * 16 == kFp8PieceCodes,
              "a piece is one vector set per CTA");
constexpr int kStThreads = 256;

struct Fp8Piece {
    uint64_t codes;      // first code of the piece
    uint64_t out;        // first BF16 element of the piece in the plane
    uint64_t scales;     // scale block row of the piece's plane: H binary32
    uint32_t len;        // codes in the piece (a multiple of 16)
    uint32_t vec0;       // index of the piece's first vector within its run
};

// Piece q -> addresses; false for pieces with nothing to move.  Runs are
// (entry, plane, block) as for BF16 copies; a run holds ntok rows of H*D codes.
__device__ __forceinline__ uint32_t fp8_div(uint32_t n, uint32_t m, uint32_t p) {
    return (uint32_t)(((uint64_t)n * m) >> p);
}

__device__ __forceinline__ bool fp8_piece(const Fp8Job& f, uint32_t q, Fp8Piece& pc) {
    const Job& j = f.job;
    const uint32_t hd = f.heads * f.head_dim;
    const uint32_t per_entry = j.num_planes * j.blocks_per_chunk;
    const uint32_t run = fp8_div(q, f.ppr_m, f.ppr_p);
    const uint32_t k = q - run * j.pieces_per_run;
    const uint32_t e = fp8_div(run, f.pe_m, f.pe_p);
    const uint32_t rem = run - e * per_entry;
    const uint32_t pr = fp8_div(rem, f.bpc_m, f.bpc_p);
    const uint32_t i = rem - pr * j.blocks_per_chunk;
    const uint32_t p = j.plane_begin + pr;
    const int32_t blk = __ldg(j.blocks + (size_t)(j.entry_base + e) * j.blocks_per_chunk + i);
    const Entry en = j.entries[e];
    const int64_t first = (int64_t)i * j.block_size;
    const int64_t ntok = min((int64_t)j.block_size, (int64_t)en.n_tok - first);
    if (ntok <= 0 || blk < 0) return false;
    if (blk >= j.num_blocks) {
        atomicCAS(j.err, 0, KVS_ERR_BOUNDS);
        return false;
    }
    const uint64_t run_codes = (uint64_t)ntok * hd;
    const uint64_t off = (uint64_t)k * kFp8PieceCodes;
    if (off >= run_codes) return false;
    pc.len = (uint32_t)min((uint64_t)kFp8PieceCodes, run_codes - off);
    pc.vec0 = (uint32_t)(off / 16);
    pc.codes = en.chunk + f.scale_bytes + ((uint64_t)p * (uint64_t)en.n_tok + (uint64_t)first) * hd + off;
    pc.out = j.planes[p] + ((uint64_t)blk * j.block_size) * hd * 2 + off * 2;
    pc.scales = en.chunk + (uint64_t)p * f.heads * 4;
    return true;
}

// Coherent, not .nc: a programmatic launch exists while the call before it still writes.
__device__ __forceinline__ uint4 ld_stream16(uint64_t a) {
    uint4 r;
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "l"(a));
    return r;
}

__device__ __forceinline__ void st_cs16(uint64_t a, const uint4& v) {
    asm volatile("st.global.cs.v4.u32 [%0], {%1,%2,%3,%4};"
                 :: "l"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

// Two E4M3 codes (low byte first) times `s` -> two BF16 (low half first).
__device__ __forceinline__ uint32_t e4m3x2_to_bf16x2(uint32_t two, float s) {
    const __half2_raw hr = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(two & 0xFFFFu), __NV_E4M3);
    __half2 h;
    *reinterpret_cast<__half2_raw*>(&h) = hr;
    const float2 v = __half22float2(h);                          // exact
    const float a = __fmul_rn(v.x, s), b = __fmul_rn(v.y, s);
    const __nv_bfloat162 r = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t*>(&r);
}

// 16 codes -> 32 bytes of BF16.
__device__ __forceinline__ void dequant16(const uint4& c, float s, uint4& lo, uint4& hi) {
    lo.x = e4m3x2_to_bf16x2(c.x, s);
    lo.y = e4m3x2_to_bf16x2(c.x >> 16, s);
    lo.z = e4m3x2_to_bf16x2(c.y, s);
    lo.w = e4m3x2_to_bf16x2(c.y >> 16, s);
    hi.x = e4m3x2_to_bf16x2(c.z, s);
    hi.y = e4m3x2_to_bf16x2(c.z >> 16, s);
    hi.z = e4m3x2_to_bf16x2(c.w, s);
    hi.w = e4m3x2_to_bf16x2(c.w >> 16, s);
}

// ---------------------------------------------------------------------------
// Span pieces, as for BF16 copies: piece_codes of the contiguous codes of one
// (chunk, plane), whatever block boundaries they meet, so that short runs (few KV
// heads, small blocks) still fill a CTA.  Offsets are in codes.  One run a piece
// before: 8000 tokens x 24 layers in runs of 2 KiB of codes 42 -> 27.5 us from HBM
// and 293 -> 241 us from the host (the link's own time: 233), in 512-byte runs 58 ->
// 16.6 and 480 -> 124.5 us.
// ---------------------------------------------------------------------------
struct Fp8Spans {
    Fp8Job   f;
    FastDiv  spp, planes, run;      // pieces per span of a full chunk, planes, run codes B*H*D
    FastDiv  vpr, vph;              // 16-code vectors per token row, and per head
    uint64_t run_codes;
    uint32_t piece_codes, num_pieces;
    uint32_t long_runs;             // runs longer than a piece: a piece meets at most two
    uint32_t far_spans;             // spans of 2^31 codes or more: divide in 64 bits
};

struct Fp8Span {
    uint64_t       codes;           // first code of the piece
    uint64_t       plane;           // base of the plane; long runs: plus the first code's offset in its run
    uint64_t       scales;          // H binary32 of the plane
    uint32_t       run0;            // index of the block of the run that holds the first code
    uint32_t       off;             // short runs: offset of the first code in its run; long runs:
                                    // codes from it to the end of its run, at most piece_codes
    uint32_t       len;             // codes, a multiple of 16
    uint32_t       col;             // column of the first vector in its token row
};

// Piece q; false for pieces past the end of a short chunk.  Uniform across the CTA.
template <class TAB>
__device__ __forceinline__ bool fp8_span(const Fp8Spans& dc, const TAB& tab, uint32_t q, Fp8Span& sp) {
    const Job& j = dc.f.job;
    const uint32_t ep = fdiv(q, dc.spp), k = q - ep * dc.spp.d, e = fdiv(ep, dc.planes);
    const uint32_t p = j.plane_begin + (ep - e * dc.planes.d);
    const uint64_t at = (uint64_t)k * dc.piece_codes;
    uint64_t i0, row;
    if (dc.far_spans) {
        i0 = at / dc.run_codes;
        row = at / 16 / dc.vpr.d;
    } else {
        i0 = fdiv((uint32_t)at, dc.run);
        row = fdiv((uint32_t)at / 16, dc.vpr);
    }
    const Entry en = tab.entry(j.entry_base + e);
    const uint64_t span = (uint64_t)en.n_tok * (dc.f.heads * dc.f.head_dim);
    if (at >= span) return false;
    const uint64_t off = at - i0 * dc.run_codes;
    sp.len = (uint32_t)min((uint64_t)dc.piece_codes, span - at);
    sp.col = (uint32_t)(at / 16 - row * dc.vpr.d);
    sp.codes = en.chunk + dc.f.scale_bytes + (uint64_t)p * span + at;
    sp.scales = en.chunk + (uint64_t)p * dc.f.heads * 4;
    sp.plane = tab.plane(p) + (dc.long_runs ? off * 2 : 0);
    sp.run0 = (j.entry_base + e) * j.blocks_per_chunk + (uint32_t)i0;
    sp.off = (uint32_t)(dc.long_runs ? min(dc.run_codes - off, (uint64_t)dc.piece_codes) : off);
    return true;
}

// Run of code x, counted from the piece's first; its block's BF16 address of code x.
__device__ __forceinline__ uint32_t fp8_run(const Fp8Spans& dc, const Fp8Span& sp, uint32_t x) {
    return dc.long_runs ? (uint32_t)(x >= sp.off) : fdiv(sp.off + x, dc.run);
}

__device__ __forceinline__ uint64_t fp8_plane(const Fp8Spans& dc, const Fp8Span& sp, uint32_t x, int32_t blk) {
    const uint32_t i = fp8_run(dc, sp, x);
    if (dc.long_runs) return sp.plane + ((uint64_t)((int64_t)blk - (int64_t)i) * dc.run_codes + x) * 2;
    return sp.plane + ((uint64_t)(uint32_t)blk * dc.run_codes + (sp.off + x - i * (uint32_t)dc.run_codes)) * 2;
}

// Head of vector v of a piece.
__device__ __forceinline__ uint32_t fp8_vec_head(const Fp8Spans& dc, const Fp8Span& sp, uint32_t v) {
    const uint32_t c = sp.col + v;
    return fdiv(c - fdiv(c, dc.vpr) * dc.vpr.d, dc.vph);
}

// A vector's 32 bytes of BF16 at `a` (0: nowhere), every lane of the warp together.
// Two 16-byte stores at a lane stride of 32 bytes would each write half of every
// sector, so neighbouring lanes swap halves and each store writes whole sectors.  8B
// shape, 8192 tokens from HBM: 268 us unswapped, 236 swapped (6.8 TB/s read + write);
// 256-bit stores, which need 32-byte aligned planes, take 239.
__device__ __forceinline__ void st_bf16x16(uint64_t a, const uint4& lo, const uint4& hi) {
    const bool odd = threadIdx.x & 1;
    const uint64_t b = __shfl_xor_sync(0xFFFFFFFFu, a, 1);
    uint4 x = odd ? lo : hi;
    x.x = __shfl_xor_sync(0xFFFFFFFFu, x.x, 1);
    x.y = __shfl_xor_sync(0xFFFFFFFFu, x.y, 1);
    x.z = __shfl_xor_sync(0xFFFFFFFFu, x.z, 1);
    x.w = __shfl_xor_sync(0xFFFFFFFFu, x.w, 1);
    const uint64_t first = odd ? b : a, second = odd ? a : b;   // the even lane's vector, the odd one's
    if (first) st_cs16(first + (odd ? 16 : 0), odd ? x : lo);
    if (second) st_cs16(second + (odd ? 16 : 0), odd ? hi : x);
}

// This thread's vectors of a piece in flight: codes, the scales of their heads, blocks
// (after rt_check, -1 where there is nothing to move).
template <int U>
struct RtRegs {
    uint4   c[U];
    float   s[U];
    int32_t blk[U];
};

// ONE: the vectors of a token row divide T, so that a thread's vectors are all of one head.
template <int T, bool ONE, int U, class TAB>
__device__ __forceinline__ void rt_load(const Fp8Spans& dc, const TAB& tab, const Fp8Span& sp, RtRegs<U>& r) {
    const uint32_t nv = sp.len / 16;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const uint32_t v = threadIdx.x + u * T;
        if (v < nv) r.c[u] = ld_stream16(sp.codes + (uint64_t)v * 16);
        r.s[u] = ONE && u ? r.s[0] : reinterpret_cast<const float*>(sp.scales)[fp8_vec_head(dc, sp, min(v, nv - 1))];
        r.blk[u] = tab.block(sp.run0 + fp8_run(dc, sp, min(v, nv - 1) * 16));
    }
}

// Waits for the blocks; one out of range, which the planner has excluded, is reported
// and skipped.  A host-link CTA checks a piece only before it stores it, with the next
// one's loads on the way (24 CTAs: 138 GB/s when it checked at once, 168 so); a CTA of
// one piece checks at once, while its codes are on the way (8 x 2048 tokens from HBM: 464
// us, 474 the other way).
template <int T, int U>
__device__ __forceinline__ void rt_check(const Fp8Spans& dc, const Fp8Span& sp, RtRegs<U>& r) {
    bool bad = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const bool in = (uint32_t)r.blk[u] < (uint32_t)dc.f.job.num_blocks;
        bad |= !in && r.blk[u] >= 0;
        if (!in || threadIdx.x + u * T >= sp.len / 16) r.blk[u] = -1;
    }
    if (bad) atomicCAS(dc.f.job.err, 0, KVS_ERR_BOUNDS);
}

// Every thread of the CTA, converting and storing.
template <int T, int U>
__device__ __forceinline__ void rt_store(const Fp8Spans& dc, const Fp8Span& sp, const RtRegs<U>& r) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
        uint4 lo, hi;
        dequant16(r.c[u], r.s[u], lo, hi);
        st_bf16x16(r.blk[u] < 0 ? 0 : fp8_plane(dc, sp, (threadIdx.x + u * T) * 16, r.blk[u]), lo, hi);
    }
}

template <class TAB>
__device__ __forceinline__ bool rt_next(const Fp8Spans& dc, const TAB& tab, uint32_t& q, Fp8Span& sp) {
    while (q < dc.num_pieces) {
        const uint32_t cur = q;
        q += gridDim.x;
        if (fp8_span(dc, tab, cur, sp)) return true;
    }
    return false;
}

// Host chunks: the next piece's loads are in flight while a piece is converted.  512
// threads, so that a piece's conversion keeps the next one's loads waiting as little as
// possible: 24 CTAs hold 204 GB/s alone, where 256 threads x 4 vectors hold 189 and 128
// x 8 149.  8192 tokens of the 8B shape take 2564 us on the default grid (the link: 2541).
// Beside a GEMM loop (averages of 8 to 12 runs, in turn on one GPU) 100 CTAs of 128 threads
// x 8, four an SM, kept 199 GB/s and 87.7% of the GEMM; 56 of these with a scale per vector
// 198 and 86.8%; 47 or 48 with one scale a thread (ONE) 197.5 and 88.2%.  49 to 52 of them
// keep 199 and 87.0%, 56 200 and 86.7%: the step lies at whole TPCs (fp8_link_ctas).
template <bool ONE, bool INL>
__global__ void __launch_bounds__(kRtLink, kRtLinkCtas)
kvs_fp8_retrieve_kernel(const __grid_constant__ Fp8Spans dc, const __grid_constant__ Tables<INL> tab) {
    if (INL) grid_wait();
    RtRegs<kRtLinkVec> ra, rb;
    Fp8Span pa, pb;
    uint32_t q = blockIdx.x;
    bool ha = rt_next(dc, tab, q, pa);
    if (ha) rt_load<kRtLink, ONE>(dc, tab, pa, ra);
    while (ha) {
        const bool hb = rt_next(dc, tab, q, pb);
        if (hb) rt_load<kRtLink, ONE>(dc, tab, pb, rb);
        rt_check<kRtLink>(dc, pa, ra);
        rt_store<kRtLink>(dc, pa, ra);
        if (!hb) break;
        ha = rt_next(dc, tab, q, pa);
        if (ha) rt_load<kRtLink, ONE>(dc, tab, pa, ra);
        rt_check<kRtLink>(dc, pb, rb);
        rt_store<kRtLink>(dc, pb, rb);
    }
}

// HBM chunks: one CTA per piece, no persistence; six CTAs per SM (four, or 128 threads x 8
// vectors, or 512 x 2: up to 1% slower).  With carried tables the 40 registers spill 16
// bytes; five CTAs do not (8 x 2048 tokens 470.3 -> 471.1 us, one 256-token chunk 12.6 ->
// 11.5).
template <bool INL>
__global__ void __launch_bounds__(kRtHbm, kRtHbmCtas)
kvs_fp8_retrieve_piece_kernel(const __grid_constant__ Fp8Spans dc, const __grid_constant__ Tables<INL> tab) {
    if (INL) {
        grid_wait();
        grid_trigger();
    }
    Fp8Span sp;
    if (!fp8_span(dc, tab, blockIdx.x, sp)) return;              // uniform across the CTA
    RtRegs<kRtHbmVec> r;
    rt_load<kRtHbm, false>(dc, tab, sp, r);
    rt_check<kRtHbm>(dc, sp, r);
    rt_store<kRtHbm>(dc, sp, r);
}

// Head of this thread's vector v of a piece of one run: when pieces start at token
// rows and a row's vpr vectors divide the CTA's thread count T, vector tid + u*T is
// always in head (tid % vpr) / vph, computed once per thread (`h_fixed`).
__device__ __forceinline__ uint32_t fp8_fixed_head(const Fp8Job& f, uint32_t T) {
    const uint32_t vph = f.head_dim / 16, vpr = f.heads * vph;
    return (f.rows_whole && T % vpr == 0) ? (threadIdx.x % vpr) / vph : 0xFFFFFFFFu;
}

__device__ __forceinline__ uint32_t fp8_head(const Fp8Job& f, const Fp8Piece& pc, uint32_t v, uint32_t h_fixed) {
    if (h_fixed != 0xFFFFFFFFu) return h_fixed;
    const uint32_t vph = f.head_dim / 16, vpr = f.heads * vph;
    return ((pc.vec0 + v) % vpr) / vph;
}

__device__ __forceinline__ bool rt_next(const Fp8Job& f, uint32_t n, uint32_t& q, Fp8Piece& pc) {
    while (q < n) {
        const uint32_t cur = q;
        q += gridDim.x;
        if (fp8_piece(f, cur, pc)) return true;
    }
    return false;
}

// Few-SM flavour of the host-chunk retrieval (KVS_F_FEW_SMS): the scheme of
// the host-link BF16 staged kernel.  A 256-thread CTA keeps seven 16 KiB pieces
// of codes in flight: two in registers and five in shared memory, where each
// thread copies, with cp.async, its own 16-code vectors and the binary32 scale
// of each vector's head into slots that only it reads back (no CTA barrier).
// 100 KiB of shared memory per CTA, two CTAs per SM: 224 KiB of codes in flight
// per SM, where kvs_fp8_retrieve_kernel holds 64 KiB.  Piece i of a CTA lives
// in slot i % 7; pieces come in grid-stride order, so once a slot finds none
// left, neither does any slot after it.
constexpr int kFsThreads = 256;
constexpr int kFsVec = kFp8PieceCodes / 16 / kFsThreads;             // vectors per thread per piece
constexpr int kFsRegPieces = 2;
constexpr int kFsSmemPieces = 5;
constexpr int kFsSlots = kFsRegPieces + kFsSmemPieces;
constexpr uint32_t kFsSlotBytes = kFp8PieceCodes + kFp8PieceCodes / 16 * 4;   // codes + a scale per vector
constexpr uint32_t kFsSmemBytes = kFsSmemPieces * kFsSlotBytes;
static_assert(kFsVec * kFsThreads * 16 == kFp8PieceCodes, "a piece is one vector set per CTA");

__device__ __forceinline__ void fs_cp16(uint32_t dst, uint64_t src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void fs_cp4(uint32_t dst, uint64_t src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst), "l"(src) : "memory");
}

__device__ __forceinline__ void fs_commit() {
    asm volatile("cp.async.commit_group;" ::: "memory");
}

template <int N>
__device__ __forceinline__ void fs_wait() {
    asm volatile("cp.async.wait_group %0;" :: "n"(N) : "memory");
}

// Scale address of vector v of piece pc (its head's binary32 scale).
__device__ __forceinline__ uint64_t fs_scale_addr(const Fp8Job& f, const Fp8Piece& pc, uint32_t v, uint32_t h_fixed) {
    return pc.scales + (uint64_t)fp8_head(f, pc, v, h_fixed) * 4;
}

struct FsRegs {
    uint4 c[kFsVec];
    float s[kFsVec];
};

__device__ __forceinline__ void fs_load_regs(const Fp8Job& f, const Fp8Piece& pc, FsRegs& r, uint32_t h_fixed) {
    const uint32_t nv = pc.len / 16;
#pragma unroll
    for (int u = 0; u < kFsVec; ++u) {
        const uint32_t v = threadIdx.x + u * kFsThreads;
        if (v < nv) {
            r.c[u] = ld_stream16(pc.codes + (uint64_t)v * 16);
            r.s[u] = __ldg(reinterpret_cast<const float*>(fs_scale_addr(f, pc, v, h_fixed)));
        }
    }
}

__device__ __forceinline__ void fs_store_regs(const Fp8Piece& pc, const FsRegs& r) {
    const uint32_t nv = pc.len / 16;
#pragma unroll
    for (int u = 0; u < kFsVec; ++u) {
        const uint32_t v = threadIdx.x + u * kFsThreads;
        if (v < nv) {
            uint4 lo, hi;
            dequant16(r.c[u], r.s[u], lo, hi);
            st_cs16(pc.out + (uint64_t)v * 32, lo);
            st_cs16(pc.out + (uint64_t)v * 32 + 16, hi);
        }
    }
}

// Slot layout: codes of vector v at v * 16, its scale at kFp8PieceCodes + v * 4.
__device__ __forceinline__ void fs_stage(const Fp8Job& f, const Fp8Piece& pc, uint32_t slot, uint32_t h_fixed) {
    const uint32_t nv = pc.len / 16;
#pragma unroll
    for (int u = 0; u < kFsVec; ++u) {
        const uint32_t v = threadIdx.x + u * kFsThreads;
        if (v < nv) {
            fs_cp16(slot + v * 16, pc.codes + (uint64_t)v * 16);
            fs_cp4(slot + kFp8PieceCodes + v * 4, fs_scale_addr(f, pc, v, h_fixed));
        }
    }
}

__device__ __forceinline__ void fs_unstage(const Fp8Piece& pc, uint32_t slot) {
    const uint32_t nv = pc.len / 16;
#pragma unroll
    for (int u = 0; u < kFsVec; ++u) {
        const uint32_t v = threadIdx.x + u * kFsThreads;
        if (v < nv) {
            uint4 c;
            float sc;
            asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(c.x), "=r"(c.y), "=r"(c.z), "=r"(c.w) : "r"(slot + v * 16));
            asm volatile("ld.shared.f32 %0, [%1];" : "=f"(sc) : "r"(slot + kFp8PieceCodes + v * 4));
            uint4 lo, hi;
            dequant16(c, sc, lo, hi);
            st_cs16(pc.out + (uint64_t)v * 32, lo);
            st_cs16(pc.out + (uint64_t)v * 32 + 16, hi);
        }
    }
}

__global__ void __launch_bounds__(kFsThreads, 2) kvs_fp8_retrieve_staged_kernel(const Fp8Job f, uint32_t num_pieces) {
    extern __shared__ __align__(128) uint8_t fs_smem[];
    const uint32_t base = smem_u32(fs_smem);
    const uint32_t h_fixed = fp8_fixed_head(f, kFsThreads);
    FsRegs r[kFsRegPieces];
    Fp8Piece pc[kFsSlots];
    bool has[kFsSlots];
    uint32_t q = blockIdx.x;
    // fill slot s with the CTA's next piece; a shared-memory slot always commits
    // one group (empty past the end), so wait_group counts pieces
    auto fill = [&](int s) {
        has[s] = rt_next(f, num_pieces, q, pc[s]);
        if (s < kFsRegPieces) {
            if (has[s]) fs_load_regs(f, pc[s], r[s < kFsRegPieces ? s : 0], h_fixed);
        } else {
            if (has[s]) fs_stage(f, pc[s], base + (s - kFsRegPieces) * kFsSlotBytes, h_fixed);
            fs_commit();
        }
    };
#pragma unroll
    for (int s = 0; s < kFsSlots; ++s) fill(s);
    bool more = true;
    while (more) {
#pragma unroll
        for (int s = 0; s < kFsSlots; ++s) {
            if (more && !has[s]) more = false;
            if (more) {
                if (s < kFsRegPieces) {
                    fs_store_regs(pc[s], r[s < kFsRegPieces ? s : 0]);
                } else {
                    fs_wait<kFsSmemPieces - 1>();    // the younger shared-memory pieces may be in flight
                    fs_unstage(pc[s], base + (s - kFsRegPieces) * kFsSlotBytes);
                }
                fill(s);
            }
        }
    }
    fs_wait<0>();
}

// ---------------------------------------------------------------------------
// Store-back (quantise)
// ---------------------------------------------------------------------------

// Per-halfword running maximum of |x| over the finite BF16 values of a word
// pair.  |x| of a finite BF16 orders like its bits with the sign cleared
// (0x0000..0x7F7F); adding 0x80 to each half moves the finite ones to
// 0x0080..0x7FFF and infinities / NaN (0x7F80..0x7FFF) to 0x8000..0x807F,
// negative as signed 16-bit lanes, so a signed lane maximum that starts from 0
// never takes them (no carry crosses halves: each half stays below 0x10000).
// The running value is offset by 0x80; amax_bits removes the offset.
__device__ __forceinline__ uint32_t amax2(uint32_t m2, uint32_t w) {
    uint32_t r;
    asm("max.s16x2 %0, %1, %2;" : "=r"(r) : "r"(m2), "r"((w & 0x7FFF7FFFu) + 0x00800080u));   // sm_90+
    return r;
}

// Bits of the largest finite |x| (0 when there is none) from a running amax2 value.
__device__ __forceinline__ uint32_t amax_bits(uint32_t m2) {
    return max(max(m2 & 0xFFFFu, m2 >> 16), 0x80u) - 0x80u;
}

__device__ __forceinline__ uint32_t amax_bits8(const uint4& v) {
    return amax_bits(amax2(amax2(amax2(amax2(0u, v.x), v.y), v.z), v.w));
}

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// Two BF16 (one word) times `inv` -> two E4M3 codes (saturating, nearest even).
__device__ __forceinline__ uint32_t e4m3x2_of(uint32_t w, float inv) {
    return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(__fmul_rn(bf16_lo(w), inv), __fmul_rn(bf16_hi(w), inv)),
                                              __NV_SATFINITE, __NV_E4M3);
}

// 8 BF16 (one 16-byte vector) -> 8 codes.
__device__ __forceinline__ uint2 quant8(const uint4& a, float inv) {
    return make_uint2(e4m3x2_of(a.x, inv) | (e4m3x2_of(a.y, inv) << 16),
                      e4m3x2_of(a.z, inv) | (e4m3x2_of(a.w, inv) << 16));
}

// 16 BF16 (two vectors) -> 16 codes.
__device__ __forceinline__ uint4 quant16(const uint4& a, const uint4& b, float inv) {
    const uint2 x = quant8(a, inv), y = quant8(b, inv);
    return make_uint4(x.x, x.y, y.x, y.y);
}

__device__ __forceinline__ void st_cs8(uint64_t a, const uint2& v) {
    asm volatile("st.global.cs.v2.u32 [%0], {%1,%2};" :: "l"(a), "r"(v.x), "r"(v.y) : "memory");
}

// Single pass, one CTA per (entry, plane, head): the head's n x D BF16 elements
// of the chunk (at most kHeadVec * kStThreads * 8, i.e. 64 KiB) are loaded
// into registers at once (kHeadVec 16-byte vectors per thread, all in flight),
// reduced to the head's amax across the CTA, and quantised from registers:
// the planes are read once and the loads of a whole head are in flight together.
// Thread t handles the 16-byte column w = t % (D/8) of tokens t / (D/8) + u *
// step (step = kStThreads / (D/8) tokens), so the column, and with it the
// address arithmetic inside a token row, is fixed per thread.  Needs D/8 to
// divide kStThreads and n, B below 2^16 (checked by the launcher).
constexpr int kHeadVec = 16;
constexpr uint32_t kHeadMaxElems = kHeadVec * kStThreads * 8;

// One segment of the store: FULL when every thread's kHeadVec vectors all lie in
// the chunk (n * D/8 == kHeadVec * kStThreads, e.g. a 256-token chunk of head_dim
// 128), so the loads and stores need no per-vector bounds test.
template <bool FULL, class TAB>
__device__ __forceinline__ void store_head_segment(const Fp8Job& f, const TAB& tab, uint32_t e, uint32_t p, uint32_t h,
                                                   uint32_t* warp_max, float* sm_inv) {
    const Job& j = f.job;
    const uint32_t H = f.heads, D = f.head_dim, vpt = D / 8;
    const uint32_t B = j.block_size, step = kStThreads / vpt;
    const uint32_t w = threadIdx.x % vpt, i0 = threadIdx.x / vpt;
    const uint64_t row2 = (uint64_t)H * D * 2;
    const Entry en = tab.entry(j.entry_base + e);
    const uint32_t n = (uint32_t)en.n_tok;
    const uint32_t block0 = (j.entry_base + e) * j.blocks_per_chunk;
    const uint64_t src0 = tab.plane(p) + (uint64_t)h * D * 2 + (uint64_t)w * 16;
    uint4 v[kHeadVec];
    uint32_t m2 = 0;
    bool bad = false;
#pragma unroll
    for (int u = 0; u < kHeadVec; ++u) {
        const uint32_t i = i0 + u * step;
        v[u] = make_uint4(0, 0, 0, 0);
        if (FULL || i < n) {
            const uint32_t bi = B == 1 ? i : __umulhi(i, f.block_magic), r = i - bi * B;
            const int32_t blk = tab.block(block0 + bi);
            if (blk < 0 || blk >= j.num_blocks) bad = true;
            else v[u] = ld_stream16(src0 + ((uint64_t)blk * B + r) * row2);
        }
    }
#pragma unroll
    for (int u = 0; u < kHeadVec; ++u)
        m2 = amax2(amax2(amax2(amax2(m2, v[u].x), v[u].y), v[u].z), v[u].w);
    if (bad) atomicCAS(j.err, 0, KVS_ERR_BOUNDS);
    const uint32_t m = __reduce_max_sync(0xFFFFFFFFu, amax_bits(m2));
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        uint32_t a = 0;
        for (int k = 0; k < kStThreads / 32; ++k) a = max(a, warp_max[k]);
        const float af = __uint_as_float(a << 16);
        const float sc = af > 0.0f ? __fdiv_rn(af, 448.0f) : 1.0f;
        *sm_inv = af > 0.0f ? __fdiv_rn(448.0f, af) : 1.0f;
        *reinterpret_cast<float*>(en.chunk + ((uint64_t)p * H + h) * 4) = sc;
    }
    __syncthreads();
    const float inv = *sm_inv;
    const uint64_t hd = (uint64_t)H * D;
    const uint64_t codes = en.chunk + f.scale_bytes + (uint64_t)p * n * hd + (uint64_t)h * D + (uint64_t)w * 8 +
                           (uint64_t)i0 * hd;
#pragma unroll
    for (int u = 0; u < kHeadVec; ++u) {
        const uint32_t i = i0 + u * step;
        if (FULL || i < n) st_cs8(codes + (uint64_t)(u * step) * hd, quant8(v[u], inv));
    }
    __syncthreads();                                       // warp_max / sm_inv are reused
}

template <bool INL>
__global__ void __launch_bounds__(kStThreads)
kvs_fp8_store_head_kernel(const __grid_constant__ Fp8Job f, const __grid_constant__ Tables<INL> tab, uint32_t num_segments) {
    if (INL) grid_wait();
    __shared__ uint32_t warp_max[kStThreads / 32];
    __shared__ float sm_inv;
    const Job& j = f.job;
    const uint32_t H = f.heads, full_n = kHeadVec * kStThreads / (f.head_dim / 8);
    for (uint32_t seg = blockIdx.x; seg < num_segments; seg += gridDim.x) {
        const uint32_t eh = seg / H, h = seg - eh * H;
        const uint32_t e = eh / j.num_planes;
        const uint32_t p = j.plane_begin + (eh - e * j.num_planes);
        if ((uint32_t)tab.entry(j.entry_base + e).n_tok == full_n)          // uniform across the CTA
            store_head_segment<true>(f, tab, e, p, h, warp_max, &sm_inv);
        else
            store_head_segment<false>(f, tab, e, p, h, warp_max, &sm_inv);
    }
}

// ---------------------------------------------------------------------------
// Store-back into HBM chunks
// ---------------------------------------------------------------------------
// A unit is g heads of one (chunk, plane), held in the shared memory of a persistent
// 512-thread CTA: thread t owns the 16-byte column w = t % (g * D / 8), which lies in
// one head, of tokens t / (g * D / 8) + u * step, u < VEC (threads past the last whole
// row idle), copied by cp.async into slots that only it reads back.  Two passes over
// the slots: the heads' maxima (one barrier), then conversion; as a slot is converted
// and its codes are stored, it takes the next unit's vector, so a CTA's loads are in
// flight while it converts, and two CTAs per SM cover each other's reductions.
//
// HBM bounds it (1.5 bytes moved per byte of BF16); what is left to the flat copy's
// rate is the loads' latency behind the reduction of a unit.  8 requests of the
// 8B shape (read + write): 2048 tokens 511 -> 495 us (6.5 TB/s), 1900 tokens 482 ->
// 453 us (6.6 TB/s), against a 512-thread CTA per SM with three 64 KiB stages that
// split its units evenly.  Tried without gain: three CTAs per SM (507 us), one 256-
// or 1024-thread shape (+1 to +4%), units in registers with 256-bit loads (497 us),
// tokens split over clusters of eight so that every access is contiguous (670 us:
// the cluster barrier and fewer resident CTAs cost more than the pattern; contiguous
// accesses alone gain 1.5%), bulk copies of 256-byte rows (1170 us: issue rate).
//
// VEC = 8 holds 64 KiB a unit, one head of 128 at 256 tokens.  VEC = 13 (104 KiB) is
// taken where it holds more heads than 8 does: heads of 80 then go in pairs, whose
// codes are whole sectors (99 -> 89 us; the two-pass kernel took 240), 48 by fours
// (84 -> 78 us), and one of 192 still fits (147 us; two-pass 429).  Larger heads
// split their tokens over a cluster, which exchanges maxima (256 tokens of 256: 283
// -> 108 us), on three CTAs per SM of fewer registers (two: 112 us).
constexpr int kUqThreads = 512;
constexpr uint32_t kUqMaxRows = 4096;
constexpr int kUqVec = 8, kUqVecWide = 13;
constexpr uint32_t kUqMaxTeam = 8, kUqMaxCluster = 4;
// What a unit costs beside its bytes (barrier, reduction, latency), in bytes of BF16.
// 16 x 300 tokens, whose last chunks hold 44: 147 us at 24 KiB, 130 at 128 KiB, 135 at
// 256; 8 x 1900: 480, 453 and 453.
constexpr uint32_t kUqUnitBytes = 131072;
__host__ __device__ constexpr int uq_ctas(bool cluster) { return cluster ? 3 : 2; }
__host__ __device__ constexpr uint32_t uq_stage_bytes(int vec) { return vec * kUqThreads * 16; }

// CTAs work in teams of G neighbours (G divides the H / g groups of a plane): a
// team's member m takes groups m, m + G, ... of the same (chunk, plane), so that
// what the members read of a token row, and write of its codes, lies side by side
// in memory and moves at the same time (8 x 2048 tokens: teams of 8 504 us, of 1 520).
// The work of a team is a contiguous range of units (chunk, plane, G groups), walked
// with a cursor: consecutive units share the chunk and its plane rows, and need no
// division to decode.  The ranges weigh a unit by its tokens and kUqUnitBytes, so that
// short last chunks leave no team idle.
struct UqCur {
    uint32_t e, p, group;
};

__device__ __forceinline__ UqCur uq_at(const Fp8Job& f, uint32_t unit, uint32_t groups, uint32_t G, uint32_t member) {
    const Job& j = f.job;
    const uint32_t per = groups / G, eg = unit / per, r = unit - eg * per;
    const uint32_t e = eg / j.num_planes;
    return {e, j.plane_begin + (eg - e * j.num_planes), r * G + member};
}

__device__ __forceinline__ void uq_step(const Fp8Job& f, UqCur& c, uint32_t groups, uint32_t G) {
    c.group += G;
    if (c.group >= groups) {
        c.group -= groups;
        if (++c.p == f.job.plane_begin + f.job.num_planes) {
            c.p = f.job.plane_begin;
            ++c.e;
        }
    }
}

__device__ __forceinline__ void cp_async16(uint32_t dst_smem, uint64_t src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" :: "r"(dst_smem), "l"(src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}

__device__ __forceinline__ uint4 lds16(uint32_t a) {
    uint4 r;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w) : "r"(a));
    return r;
}

// Two BF16 (one word) times `inv` -> two E4M3 codes: two binary32 multiplies
// rounded to nearest, then one saturating nearest-even pair conversion (the
// high element goes to the high byte).  (A packed f32x2 multiply measured 0.5%
// slower here.)
__device__ __forceinline__ uint32_t e4m3x2_of_pk(uint32_t w, uint64_t inv2) {
    const float inv = __uint_as_float((uint32_t)inv2);
    const float lo = __fmul_rn(__uint_as_float(w << 16), inv), hi = __fmul_rn(__uint_as_float(w & 0xFFFF0000u), inv);
    uint32_t r;
    asm("{\n\t.reg .b16 t;\n\tcvt.rn.satfinite.e4m3x2.f32 t, %1, %2;\n\tcvt.u32.u16 %0, t;\n\t}"
        : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ uint2 quant8_pk(const uint4& a, uint64_t inv2) {
    return make_uint2(e4m3x2_of_pk(a.x, inv2) | (e4m3x2_of_pk(a.y, inv2) << 16),
                      e4m3x2_of_pk(a.z, inv2) | (e4m3x2_of_pk(a.w, inv2) << 16));
}

// Running max of |x| over BF16 pairs in one instruction (sm_86+): the result's
// magnitude is the larger magnitude, its sign the XOR of the signs (cleared at
// the end); a NaN input is ignored.  Infinities are not: a head whose maximum
// comes out infinite takes the exact finite amax (amax2) instead.
__device__ __forceinline__ uint32_t absmax2(uint32_t m2, uint32_t w) {
    uint32_t r;
    asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(m2), "r"(w));
    return r;
}

constexpr uint32_t kBf16Inf = 0x7F80u;

__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t rank, uint32_t v) {
    uint32_t ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
    asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(ra), "r"(v) : "memory");
}

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// Team k of T takes the units that begin in [k * W / T, (k + 1) * W / T) of the job's
// W = sum over its chunks of (tokens + extra) x units per chunk.  CLUSTER: the tokens
// of a unit are split over cl CTAs of a cluster, which exchange their maxima.  EARLY is
// Job::early of a carried call; read at run time it cost 0.4% (heads of 80: 82.5 -> 82.8 us).
template <int VEC, bool CLUSTER, bool INL, bool EARLY>
__global__ void __launch_bounds__(kUqThreads, uq_ctas(CLUSTER))
kvs_fp8_store_unit_kernel(const __grid_constant__ Fp8Job f, const __grid_constant__ Tables<INL> tab, uint32_t g, uint32_t G, uint32_t extra, uint32_t cl) {
    if (INL) grid_wait();
    extern __shared__ __align__(128) uint8_t uq_smem[];
    uint32_t* rows = reinterpret_cast<uint32_t*>(uq_smem + uq_stage_bytes(VEC));   // plane row of each of the CTA's tokens
    // Maxima of unit n's heads in third n % 3, cleared before barrier n - 1: the readers of unit
    // n - 3 have passed barrier n - 2, and the writers of unit n wait for barrier n - 1.
    __shared__ uint32_t amax[3][kFp8MaxHeads], exact[kFp8MaxHeads];
    // The cluster's, by rank, in half n % 2: written before cluster barrier n, read after it, and
    // written again after cluster barrier n + 1.
    __shared__ uint32_t all[CLUSTER ? 2 : 1][CLUSTER ? kUqMaxCluster : 1][kFp8MaxHeads];
    __shared__ uint32_t range[2];
    const Job& j = f.job;
    const uint32_t t = threadIdx.x, D = f.head_dim, vph = D / 8, vpt = g * vph, step = kUqThreads / vpt;
    const uint32_t w = t % vpt, i0 = t / vpt, hl = w / vph;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, i0 < step ? hl : 0xFFFFu);   // lanes on the same head
    const bool lead = i0 < step && (t & 31) == (uint32_t)__ffs(peers) - 1;
    const uint32_t rank = CLUSTER ? blockIdx.x % cl : 0, unit_cta = CLUSTER ? blockIdx.x / cl : blockIdx.x;
    const uint32_t groups = f.heads / g, team = unit_cta / G, teams = (CLUSTER ? gridDim.x / cl : gridDim.x) / G;
    for (uint32_t h = t; h < 3 * kFp8MaxHeads; h += kUqThreads) (&amax[0][0])[h] = 0;
    const uint32_t upe = j.num_planes * (groups / G);
    if (f.ragged) {
        const uint64_t W = (f.tokens + (uint64_t)extra * j.num_entries) * upe;
        const uint64_t x[2] = {W * team / teams, W * (team + 1) / teams};
        for (uint32_t e = t; e < j.num_entries; e += kUqThreads) {
            const Entry en = tab.entry(j.entry_base + e);
            const uint64_t at = (en.first_tok + (uint64_t)extra * e) * upe;
            const uint32_t n = (uint32_t)en.n_tok + extra;
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (x[k] >= at && x[k] < at + (uint64_t)n * upe) range[k] = (uint32_t)((uint64_t)e * upe + (x[k] - at + n - 1) / n);
        }
        if (t == 0 && x[1] == W) range[1] = j.num_entries * upe;
    } else if (t < 2) {
        range[t] = (uint32_t)((uint64_t)j.num_entries * upe * (team + t) / teams);
    }
    if (CLUSTER) cluster_sync();                            // the others have started
    else __syncthreads();
    uint32_t left = range[1] - range[0];
    if (left == 0) return;                                  // uniform across the cluster
    UqCur c = uq_at(f, range[0], groups, G, unit_cta % G);
    uint32_t mine = 0, first = 0;                           // the CTA's tokens of the chunk (0 for an idle thread), from `first`
    // the chunk's plane rows; a block out of range, which the planner has excluded, is reported
    auto enter = [&]() {
        const uint32_t n = (uint32_t)tab.entry(j.entry_base + c.e).n_tok, B = j.block_size;
        const uint32_t block0 = (j.entry_base + c.e) * j.blocks_per_chunk;
        const uint32_t per = CLUSTER ? (n + cl - 1) / cl : n;
        first = CLUSTER ? min(rank * per, n) : 0;
        const uint32_t count = min(per, n - first);
        for (uint32_t r = t; r < count; r += kUqThreads) {
            const uint32_t i = first + r, bi = B == 1 ? i : __umulhi(i, f.block_magic);
            uint32_t blk = (uint32_t)tab.block(block0 + bi);
            if (blk >= (uint32_t)j.num_blocks) {
                atomicCAS(j.err, 0, KVS_ERR_BOUNDS);
                blk = 0;
            }
            rows[r] = blk * B + (i - bi * B);
        }
        mine = i0 < step ? count : 0;
        __syncthreads();
    };
    const uint32_t row2 = f.heads * D * 2;
    auto source = [&]() { return tab.plane(c.p) + (uint64_t)(c.group * vpt + w) * 16; };
    enter();
    const uint32_t slot0 = smem_u32(uq_smem) + t * 16;      // this thread's vector u at slot0 + u * kUqThreads * 16
    {
        const uint64_t src = source();
#pragma unroll
        for (int u = 0; u < VEC; ++u)
            if (i0 + u * step < mine) cp_async16(slot0 + u * kUqThreads * 16, src + (uint64_t)rows[i0 + u * step] * row2);
    }
    for (uint32_t k = 0, half = 0;; half ^= 1) {
        const uint32_t k1 = k == 2 ? 0 : k + 1;
        uint32_t x2 = 0;
        cp_async_wait_all();
#pragma unroll
        for (int u = 0; u < VEC; ++u)
            if (i0 + u * step < mine) {
                const uint4 v = lds16(slot0 + u * kUqThreads * 16);
                x2 = absmax2(absmax2(absmax2(absmax2(x2, v.x), v.y), v.z), v.w);
            }
        x2 &= 0x7FFF7FFFu;                                  // never NaN: at most kBf16Inf per half
        const uint32_t m = __reduce_max_sync(peers, max(x2 & 0xFFFFu, x2 >> 16));
        if (lead) atomicMax(&amax[k][hl], m);
        if (t < g) amax[k1][t] = 0;
        __syncthreads();
        uint32_t a = amax[k][hl];
        // The maximum over the cluster's CTAs of what each has in own[].
        auto over_cluster = [&](const uint32_t* own) {
            for (uint32_t x = t; x < g * cl; x += kUqThreads) st_cluster(smem_u32(&all[half][rank][x % g]), x / g, own[x % g]);
            cluster_sync();
            uint32_t r = 0;
            for (uint32_t c2 = 0; c2 < cl; ++c2) r = max(r, all[half][c2][hl]);
            return r;
        };
        if (CLUSTER) a = over_cluster(amax[k]);
        // a head with an infinity: the largest finite magnitudes of the unit's heads instead
        uint32_t top = 0;                                   // uniform across the cluster
        if (g == 1) top = a;
        else for (uint32_t x = t & 31; x < g; x += 32) top = max(top, amax[k][x]);   // a cluster has one head a unit
        if (g > 1) top = __reduce_max_sync(0xFFFFFFFFu, top);
        if (top == kBf16Inf) {
            uint32_t m2 = 0;
            for (int u = 0; u < VEC; ++u)
                if (i0 + u * step < mine) {
                    const uint4 v = lds16(slot0 + u * kUqThreads * 16);
                    m2 = amax2(amax2(amax2(amax2(m2, v.x), v.y), v.z), v.w);
                }
            const uint32_t mf = __reduce_max_sync(peers, amax_bits(m2));
            if (t < g) exact[t] = 0;
            __syncthreads();
            if (lead) atomicMax(&exact[hl], mf);
            __syncthreads();
            a = exact[hl];
            if (CLUSTER) {
                cluster_sync();                             // the first maxima have been read
                a = over_cluster(exact);
            }
        }
        const float af = __uint_as_float(a << 16);
        const float inv = af > 0.0f ? __fdiv_rn(448.0f, af) : 1.0f;
        const Entry en = tab.entry(j.entry_base + c.e);
        const uint32_t h0 = c.group * g, hd = f.heads * D, old = mine;
        if (rank == 0 && i0 == 0 && w % vph == 0)
            reinterpret_cast<float*>(en.chunk)[(uint64_t)c.p * f.heads + h0 + hl] = af > 0.0f ? __fdiv_rn(af, 448.0f) : 1.0f;
        const uint64_t codes = en.chunk + f.scale_bytes + ((uint64_t)c.p * (uint32_t)en.n_tok + first + i0) * hd + (uint64_t)h0 * D + w * 8;
        uint64_t src = 0;
        if (--left) {
            const uint32_t e = c.e;
            uq_step(f, c, groups, G);
            if (c.e != e) enter();                          // every thread has used the old rows
            src = source();
        } else {
            mine = 0;
            if (EARLY) grid_trigger();
        }
        const uint64_t inv2 = ((uint64_t)__float_as_uint(inv) << 32) | __float_as_uint(inv);
#pragma unroll
        for (int u = 0; u < VEC; ++u) {
            const uint32_t i = i0 + u * step;
            if (i < old)
                st_cs8(codes + (uint64_t)(u * step) * hd, quant8_pk(lds16(slot0 + u * kUqThreads * 16), inv2));
            if (i < mine) cp_async16(slot0 + u * kUqThreads * 16, src + (uint64_t)rows[i] * row2);
        }
        if (!left) break;
        k = k1;
    }
}

constexpr int kStUnroll = 4;                         // vectors per thread in flight per step

// One CTA per (entry, plane) segment: the chunk's n tokens of that plane.
template <bool INL>
__global__ void __launch_bounds__(kStThreads)
kvs_fp8_store_kernel(const __grid_constant__ Fp8Job f, const __grid_constant__ Tables<INL> tab, uint32_t num_segments) {
    if (INL) grid_wait();
    __shared__ uint32_t amax[kFp8MaxHeads];
    __shared__ float scale[kFp8MaxHeads];                    // holds 448 / amax per head
    const Job& j = f.job;
    const uint32_t H = f.heads, vph = f.head_dim / 16, vpr = H * vph;
    const uint64_t row2 = (uint64_t)H * f.head_dim * 2;          // BF16 bytes per token row
    for (uint32_t seg = blockIdx.x; seg < num_segments; seg += gridDim.x) {
        const uint32_t e = seg / j.num_planes;
        const uint32_t p = j.plane_begin + (seg - e * j.num_planes);
        const Entry en = tab.entry(j.entry_base + e);
        const uint32_t n = (uint32_t)en.n_tok;
        const uint32_t block0 = (j.entry_base + e) * j.blocks_per_chunk;
        const uint64_t plane = tab.plane(p);
        const uint64_t codes = en.chunk + f.scale_bytes + (uint64_t)p * n * vpr * 16;
        const uint32_t nvec = n * vpr;
        // source address of vector v (16 BF16 = 32 bytes), or 0 for a bad block
        auto src_of = [&](uint32_t v, uint32_t& h) -> uint64_t {
            const uint32_t i = v / vpr, w = v - i * vpr;
            h = w / vph;
            const int32_t blk = tab.block(block0 + i / j.block_size);
            if (blk < 0 || blk >= j.num_blocks) return 0;
            return plane + ((uint64_t)blk * j.block_size + i % j.block_size) * row2 + (uint64_t)w * 32;
        };
        for (uint32_t h = threadIdx.x; h < H; h += blockDim.x) amax[h] = 0;
        __syncthreads();
        // pass 1: per-head amax over the finite elements of this chunk's plane p
        uint32_t cur_h = 0xFFFFFFFFu, m = 0;
        bool bad = false;
        for (uint32_t v0 = threadIdx.x; v0 < nvec; v0 += blockDim.x * kStUnroll) {
            uint4 a[kStUnroll], b[kStUnroll];
            uint32_t hh[kStUnroll];
            bool ok[kStUnroll];
#pragma unroll
            for (int u = 0; u < kStUnroll; ++u) {
                const uint32_t v = v0 + u * blockDim.x;
                ok[u] = false;
                if (v < nvec) {
                    const uint64_t src = src_of(v, hh[u]);
                    if (src) {
                        a[u] = ld_stream16(src);
                        b[u] = ld_stream16(src + 16);
                        ok[u] = true;
                    } else {
                        bad = true;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kStUnroll; ++u) {
                if (!ok[u]) continue;
                const uint32_t lm = max(amax_bits8(a[u]), amax_bits8(b[u]));
                if (hh[u] != cur_h) {
                    if (cur_h != 0xFFFFFFFFu) atomicMax(&amax[cur_h], m);
                    cur_h = hh[u];
                    m = 0;
                }
                m = max(m, lm);
            }
        }
        if (cur_h != 0xFFFFFFFFu) atomicMax(&amax[cur_h], m);
        if (bad) atomicCAS(j.err, 0, KVS_ERR_BOUNDS);
        __syncthreads();
        for (uint32_t h = threadIdx.x; h < H; h += blockDim.x) {
            const float a = __uint_as_float(amax[h] << 16);
            const float s = a > 0.0f ? __fdiv_rn(a, 448.0f) : 1.0f;
            scale[h] = a > 0.0f ? __fdiv_rn(448.0f, a) : 1.0f;        // the inverse, for pass 2
            *reinterpret_cast<float*>(en.chunk + ((uint64_t)p * H + h) * 4) = s;
        }
        __syncthreads();
        // pass 2: quantise
        for (uint32_t v0 = threadIdx.x; v0 < nvec; v0 += blockDim.x * kStUnroll) {
            uint4 a[kStUnroll], b[kStUnroll];
            uint32_t hh[kStUnroll];
            bool ok[kStUnroll];
#pragma unroll
            for (int u = 0; u < kStUnroll; ++u) {
                const uint32_t v = v0 + u * blockDim.x;
                ok[u] = false;
                if (v < nvec) {
                    const uint64_t src = src_of(v, hh[u]);
                    if (src) {
                        a[u] = ld_stream16(src);
                        b[u] = ld_stream16(src + 16);
                        ok[u] = true;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < kStUnroll; ++u)
                if (ok[u]) st_cs16(codes + (uint64_t)(v0 + u * blockDim.x) * 16, quant16(a[u], b[u], scale[hh[u]]));
        }
        __syncthreads();                                   // amax / scale are reused by the next segment
    }
}

constexpr int kMaxDev = 64;
int g_sms[kMaxDev];                      // SM count per device
bool g_fs_attr[kMaxDev];                 // ... of the few-SM retrieval

int sm_count() {
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= kMaxDev) dev = 0;
    if (g_sms[dev] == 0) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        g_sms[dev] = n > 0 ? n : 1;
    }
    return g_sms[dev];
}

}  // namespace

Fp8Spans make_spans(const Fp8Job& fj, uint32_t piece_codes) {
    Fp8Spans dc;
    const uint32_t hd = fj.heads * fj.head_dim;
    dc.f = fj;
    dc.piece_codes = piece_codes;
    dc.run_codes = (uint64_t)fj.job.block_size * hd;
    const uint64_t span = dc.run_codes * fj.job.blocks_per_chunk;          // of a full chunk
    dc.spp = make_fastdiv((uint32_t)((span + piece_codes - 1) / piece_codes));
    dc.planes = make_fastdiv(fj.job.num_planes);
    dc.run = make_fastdiv(dc.run_codes < (1ull << 31) ? (uint32_t)dc.run_codes : 1u);      // longer: never divided by
    dc.vpr = make_fastdiv(hd / 16);
    dc.vph = make_fastdiv(fj.head_dim / 16);
    dc.long_runs = dc.run_codes > piece_codes;
    dc.far_spans = span >= (1ull << 31);
    dc.num_pieces = (uint32_t)((uint64_t)fj.job.num_entries * fj.job.num_planes * dc.spp.d);
    return dc;
}

cudaError_t launch_fp8_retrieve(const Fp8Job& fj, int grid, cudaStream_t s) {
    if (fj.job.num_pieces == 0) return cudaSuccess;
    const bool per_piece = grid == kFp8PerPiece;
    const uint32_t vpr = fj.heads * fj.head_dim / 16;
    // 16 KiB of codes a piece, halved while a launch would leave CTAs without one, down to 4 KiB
    const int full = sm_count() * kRtLinkCtas;
    if (!per_piece && (grid <= 0 || grid > full)) grid = full;
    const uint64_t total = (uint64_t)fj.job.num_entries * fj.job.num_planes * fj.job.blocks_per_chunk * fj.job.block_size * vpr * 16;
    uint32_t piece = kFp8PieceCodes;
    while (piece > kFp8PieceCodes / 4 && total / piece < 2ull * (per_piece ? sm_count() : grid)) piece /= 2;
    const Fp8Spans dc = make_spans(fj, piece);
    // One scale a thread gains beside other work only, and costs the smallest calls 0.1 us.
    const bool one = kRtLink % vpr == 0 && piece == kFp8PieceCodes;
    const uint32_t ctas = per_piece ? dc.num_pieces : std::min<uint32_t>((uint32_t)grid, dc.num_pieces);
    return with_tables(fj.job, [&](const auto& tab) {
        constexpr bool I = std::decay_t<decltype(tab)>::kInline;
        if (per_piece) launch_on(s, tab, kvs_fp8_retrieve_piece_kernel<I>, ctas, kRtHbm, 0, dc, tab);
        else launch_on(s, tab, one ? kvs_fp8_retrieve_kernel<true, I> : kvs_fp8_retrieve_kernel<false, I>, ctas, kRtLink, 0, dc, tab);
    });
}

cudaError_t launch_fp8_retrieve_staged(const Fp8Job& fj, int grid, cudaStream_t s) {
    const uint64_t n = fj.job.num_pieces;
    if (n == 0) return cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= kMaxDev) dev = 0;
    if (!g_fs_attr[dev]) {
        cudaError_t e = cudaFuncSetAttribute(kvs_fp8_retrieve_staged_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFsSmemBytes);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(kvs_fp8_retrieve_staged_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        g_fs_attr[dev] = true;
    }
    const int full = sm_count() * 2;
    if (grid <= 0 || grid > full) grid = full;
    if ((uint64_t)grid > n) grid = (int)n;
    kvs_fp8_retrieve_staged_kernel<<<grid, kFsThreads, kFsSmemBytes, s>>>(fj, (uint32_t)n);
    return cudaGetLastError();
}

// Team size: the divisor of the groups that leaves the fewest CTAs of the grid without a
// team; the larger among equals, kUqMaxTeam at most.
uint32_t uq_team(uint32_t groups, uint32_t ctas) {
    uint32_t best = 1;
    for (uint32_t n = 2; n <= kUqMaxTeam && n <= ctas; ++n)
        if (groups % n == 0 && ctas % n <= ctas % best) best = n;
    return best;
}

// Heads per unit: the most whose tokens fit the vectors of one CTA; 0 where one head does not.
uint32_t uq_heads(const Fp8Job& fj, uint32_t chunk_tokens, uint32_t vec) {
    for (uint32_t g = fj.heads; g >= 1; --g) {
        const uint32_t vpt = g * (fj.head_dim / 8);
        if (fj.heads % g == 0 && vpt <= kUqThreads && vec * (kUqThreads / vpt) >= chunk_tokens) return g;
    }
    return 0;
}

template <int VEC, bool CLUSTER, bool EARLY, bool INL>
cudaError_t launch_unit(const Fp8Job& fj, const Tables<INL>& tab, int grid, cudaStream_t s, uint32_t chunk_tokens, uint32_t g,
                        uint32_t cl) {
    if (fj.job.num_entries == 0) return cudaSuccess;
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= kMaxDev) dev = 0;
    const auto k = kvs_fp8_store_unit_kernel<VEC, CLUSTER, INL, EARLY>;
    static bool attr[kMaxDev];                              // shared-memory limit raised
    if (!attr[dev]) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(uq_stage_bytes(VEC) + kUqMaxRows * 4));
        if (e != cudaSuccess) return e;
        attr[dev] = true;
    }
    int full = sm_count() * uq_ctas(CLUSTER) / (int)cl;
    cudaLaunchConfig_t cfg{};
    cfg.blockDim = dim3(kUqThreads);
    cfg.dynamicSmemBytes = uq_stage_bytes(VEC) + (chunk_tokens + cl - 1) / cl * 4;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    if (CLUSTER) {                                          // as many clusters as the GPCs hold at once
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = cl;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        static struct { uint32_t cl, smem; int most; } seen[kMaxDev];   // the last answer
        auto& known = seen[dev];
        if (known.cl != cl || known.smem != cfg.dynamicSmemBytes) {
            cfg.gridDim = dim3((uint32_t)full * cl);
            const cudaError_t e = cudaOccupancyMaxActiveClusters(&known.most, k, &cfg);
            if (e != cudaSuccess) return e;
            known.cl = cl;
            known.smem = (uint32_t)cfg.dynamicSmemBytes;
        }
        full = std::max(1, std::min(full, known.most));
    }
    int ctas = grid > 0 ? std::max(1, std::min(grid / (int)cl, full)) : full;
    uint64_t units = 0;
    for (;; --g) {                                          // fewer heads a unit while CTAs have none
        if (fj.heads % g) continue;
        units = (uint64_t)fj.job.num_entries * fj.job.num_planes * (fj.heads / g);
        if (g == 1 || units >= (uint64_t)ctas) break;
    }
    if ((uint64_t)ctas > units) ctas = (int)units;
    const uint32_t G = uq_team(fj.heads / g, (uint32_t)ctas);
    cfg.gridDim = dim3((uint32_t)ctas / G * G * cl);
    if (tab.programmatic()) {                               // see launch_on
        at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        at[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
        cfg.attrs = at;
        ++cfg.numAttrs;
    }
    const uint32_t extra = kUqUnitBytes / (g * fj.head_dim * 2);
    return cudaLaunchKernelEx(&cfg, k, fj, tab, g, G, extra, cl);
}

cudaError_t launch_fp8_store(const Fp8Job& fj, int grid, cudaStream_t s, uint32_t chunk_tokens, bool staged) {
    const uint32_t vpt = fj.head_dim / 8;
    // HBM destinations: plane rows below 2^32, block numbers by a reciprocal (chunk and block
    // sizes below 2^16), a row table of at most 16 KiB.
    if (staged && chunk_tokens <= kUqMaxRows && (uint64_t)fj.job.num_blocks * fj.job.block_size <= 0xFFFFFFFFull) {
        const uint32_t g = uq_heads(fj, chunk_tokens, kUqVec), gw = uq_heads(fj, chunk_tokens, kUqVecWide);
        uint32_t cl = 1;
        if (!g && !gw) {
            cl = 2;
            while (cl <= kUqMaxCluster && vpt <= kUqThreads && kUqVec * (kUqThreads / vpt) * cl < chunk_tokens) cl *= 2;
        }
        if (cl <= kUqMaxCluster && vpt <= kUqThreads && (grid <= 0 || grid >= (int)cl)) {
            cudaError_t e = cudaSuccess;
            const cudaError_t last = with_tables(fj.job, [&](const auto& tab) {
                auto go = [&](auto early) {
                    constexpr bool E = decltype(early)::value;
                    return cl > 1   ? launch_unit<kUqVec, true, E>(fj, tab, grid, s, chunk_tokens, 1, cl)
                           : gw > g ? launch_unit<kUqVecWide, false, E>(fj, tab, grid, s, chunk_tokens, gw, 1)
                                    : launch_unit<kUqVec, false, E>(fj, tab, grid, s, chunk_tokens, g, 1);
                };
                constexpr bool I = std::decay_t<decltype(tab)>::kInline;
                e = I && fj.job.early ? go(std::bool_constant<I>{}) : go(std::false_type{});
            });
            return e != cudaSuccess ? e : last;
        }
    }
    if ((uint64_t)chunk_tokens * fj.head_dim <= kHeadMaxElems && kStThreads % vpt == 0 && chunk_tokens < 65536 &&
        fj.job.block_size < 65536) {
        const uint64_t segs = (uint64_t)fj.job.num_entries * fj.job.num_planes * fj.heads;
        if (segs == 0) return cudaSuccess;
        if (grid <= 0 || (uint64_t)grid > segs) grid = (int)std::min<uint64_t>(segs, 1u << 30);
        return with_tables(fj.job, [&](const auto& tab) {
            constexpr bool I = std::decay_t<decltype(tab)>::kInline;
            launch_on(s, tab, kvs_fp8_store_head_kernel<I>, grid, kStThreads, 0, fj, tab, (uint32_t)segs);
        });
    }
    const uint64_t segs = (uint64_t)fj.job.num_entries * fj.job.num_planes;
    if (segs == 0) return cudaSuccess;
    if (grid <= 0 || (uint64_t)grid > segs) grid = (int)segs;
    return with_tables(fj.job, [&](const auto& tab) {
        constexpr bool I = std::decay_t<decltype(tab)>::kInline;
        launch_on(s, tab, kvs_fp8_store_kernel<I>, grid, kStThreads, 0, fj, tab, (uint32_t)segs);
    });
}

}  // namespace kvs
