// kvs_job.cuh -- arithmetic shared by the kernels that walk a Job's pieces.
#pragma once

#include <cstdint>
#include <cstring>

#include "kvs_internal.h"

namespace kvs {
namespace {

// ---------------------------------------------------------------------------
// Division by a launch-invariant divisor d, for dividends below 2^31: with
// p = 31 + ceil(log2 d) and m = ceil(2^p / d), floor(n / d) = (n * m) >> p
// (round-up reciprocal method; the error term n*(m*d - 2^p)/(d*2^p) stays
// below 1/d).  m < 2^32 for every d >= 1.
// ---------------------------------------------------------------------------
struct FastDiv {
    uint32_t d, m, p;
};

inline FastDiv make_fastdiv(uint32_t d) {
    uint32_t l = 0;
    while ((1ull << l) < d) ++l;
    FastDiv f;
    f.d = d;
    f.p = 31 + l;
    f.m = (uint32_t)(((1ull << f.p) + d - 1) / d);
    return f;
}

__device__ __forceinline__ uint32_t fdiv(uint32_t n, const FastDiv& f) {
    return (uint32_t)(((uint64_t)n * f.m) >> f.p);
}

// ---------------------------------------------------------------------------
// How a kernel reads the call's tables: from device memory, where the planner has
// uploaded them, or from its own parameters.  A small call spends most of its time
// on the upload (a copy on another stream, two events, a wait); tables that fit are
// passed by value instead.
// ---------------------------------------------------------------------------
template <bool INL>
struct Tables;

template <>
struct Tables<false> {
    static constexpr bool kInline = false;
    const Entry*    entries;             // entry_base entries before the job's first
    const int32_t*  blocks;
    const uint64_t* planes;
    static constexpr bool programmatic() { return false; }
    __host__ __device__ explicit Tables(const Job& j)
        : entries(j.entries - j.entry_base), blocks(j.blocks), planes(j.planes) {}
    __device__ __forceinline__ Entry entry(uint32_t e) const { return entries[e]; }
    __device__ __forceinline__ int32_t block(uint32_t k) const { return __ldg(blocks + k); }
    __device__ __forceinline__ uint64_t plane(uint32_t p) const { return planes[p]; }
};

template <>
struct Tables<true> {
    static constexpr bool kInline = true;
    uint32_t entries_at, blocks_at, forked;
    bool programmatic() const { return !forked; }
    alignas(16) unsigned char raw[kTableBytes];
    explicit Tables(const HostTables& t) {
        entries_at = (t.num_planes * 8 + 15) / 16 * 16;
        blocks_at = entries_at + t.num_entries * (uint32_t)sizeof(Entry);
        forked = t.forked;
        memcpy(raw, t.planes, t.num_planes * 8);
        memcpy(raw + entries_at, t.entries, t.num_entries * sizeof(Entry));
        memcpy(raw + blocks_at, t.blocks, t.num_blocks * 4);
    }
    __device__ __forceinline__ Entry entry(uint32_t e) const { return reinterpret_cast<const Entry*>(raw + entries_at)[e]; }
    __device__ __forceinline__ int32_t block(uint32_t k) const { return reinterpret_cast<const int32_t*>(raw + blocks_at)[k]; }
    __device__ __forceinline__ uint64_t plane(uint32_t p) const { return reinterpret_cast<const uint64_t*>(raw)[p]; }
};

// launch(tables) with the tables of `job`, by value or by pointer.
template <class F>
cudaError_t with_tables(const Job& job, F&& launch) {
    if (job.tables) launch(Tables<true>(*job.tables));
    else launch(Tables<false>(job));
    return cudaGetLastError();
}

// Launches a kernel that reads its tables through `tab`.  One that carries them (and
// begins with grid_wait) is launched programmatically: behind another small call it
// has its CTAs in place when that call ends (one 32 MiB chunk from HBM: 13.9 -> 11.5
// us a call).  One that reads uploaded tables waits for the upload's event anyway, and
// between the events of a forked call the attribute costs 1%.
template <class TAB, class... P, class... A>
void launch_on(cudaStream_t s, const TAB& tab, void (*kernel)(P...), uint32_t grid, uint32_t threads, uint32_t smem, const A&... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = tab.programmatic() ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace
}  // namespace kvs
