// kvs_job.cuh -- arithmetic shared by the kernels that walk a Job's pieces.
#pragma once

#include <cstdint>

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

}  // namespace
}  // namespace kvs
