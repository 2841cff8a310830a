// Decode steps until a time, ceil(dt / s), from reciprocals that stand beside the steps in the walking and packed kernels' tables.
// Compiles without CUDA.
#pragma once
#include "route.cuh"

namespace maaso {

MAASO_HD inline uint32_t mul_high(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (uint32_t)((uint64_t)a * b >> 32);
#endif
}

MAASO_HD inline uint32_t bits_of(uint32_t v) {  // 0 has none
#ifdef __CUDA_ARCH__
    return 32u - (uint32_t)__clz((int)v);
#else
    return v ? 32u - (uint32_t)__builtin_clz(v) : 0u;
#endif
}

// ceil(dt / s) for 0 <= dt < 2^31, s < 2^31, rs = (2^32 - 1) / s rounded down: the estimate is at most the quotient and less
// than two below it, since rs > 2^32 / s - 1.
MAASO_HD inline uint32_t walk_rcp(uint32_t s) { return 0xFFFFFFFFu / s; }
MAASO_HD inline uint32_t walk_steps(int32_t dt, uint32_t s, uint32_t rs) {
    const uint32_t d = (uint32_t)dt + s - 1u, q = mul_high(d, rs);
    return q + (d - q * s >= s ? 1u : 0u);
}
MAASO_HD inline uint32_t walk_steps(int64_t dt, uint32_t s, uint32_t rs) {
    const uint64_t d = (uint64_t)dt + (s - 1u);
    return (d >> 32) == 0 ? walk_steps((int32_t)dt, s, rs) : (uint32_t)(d / s);
}

// ceil(dt / s) = (2 (dt + s - 1) m >> 32) >> L with L = ceil(log2 s), m = ceil(2^(31 + L) / s) < 2^32: exact for dt + s - 1 <
// 2^31 (m s - 2^(31 + L) < s <= 2^L; Granlund and Montgomery's division by an invariant).  An entry: {s << 5 | L, m}; s < 2^27.
struct ExactEntry {
    uint32_t step, m;
};
MAASO_HD inline ExactEntry walk_exact_entry(uint32_t s) {
    const uint32_t log2 = bits_of(s - 1u);
    const ExactEntry e = {(s << 5) | log2, (uint32_t)((((uint64_t)1 << (31u + log2)) + (s - 1u)) / s)};
    return e;
}
MAASO_HD inline uint32_t walk_exact_steps(int32_t dt, uint32_t s, uint32_t step, uint32_t m) {
    const uint32_t q = mul_high(2u * ((uint32_t)dt + s - 1u), m);
#ifdef __CUDA_ARCH__
    return __funnelshift_r(q, 0u, step);  // (by the low five bits)
#else
    return q >> (step & 31u);
#endif
}

}  // namespace maaso
