// The walking kernel's bounds on times (walk_kernel.cuh), which the host checks, and what its bodies share.  (Its shared memory and
// what a placement needs of it: route.cuh.)
#pragma once
#include "lane_sim.cuh"

namespace maaso {

// Global memory for one block's running requests: two bytes of it per byte of pool.
__host__ __device__ inline size_t walk_big_scratch(uint32_t pool_bytes) { return (size_t)pool_bytes * 2u; }

// Times are 32-bit offsets from an epoch that each placement moves along (walk_kernel.cuh).  The bounds below
// keep every sum of a round inside 31 bits; a batch whose tables or limits exceed them, checked on the host,
// runs with 64-bit times, and so does, from its start again, a single placement that gets beyond kWalkHorizon.
constexpr int32_t kWalkFar = 0x7FFFFFFF;         // no completion in sight; an arrival beyond the epoch's reach
constexpr int32_t kWalkNowMax = 1 << 27;         // the epoch moves when the dispatcher's clock is this far ahead
constexpr int32_t kWalkHorizon = 0x60000000;     // largest time
constexpr int64_t kWalkStepMax = 1 << 24;        // decode step
constexpr int64_t kWalkPreMax = 1 << 28;         // prefill
constexpr int64_t kWalkLimMax = 1 << 30;         // finite SLO limit

__device__ __forceinline__ void walk_reject_side(const EvalParams& P, uint32_t oc, uint32_t req, uint32_t model) {
    const Dump dump = dump_for(P, oc);
    if (P.rej_by_model) atomicAdd(&P.rej_by_model[(size_t)oc * MAASO_MAX_MODELS + model], 1u);
    if (dump.finish) dump.finish[req] = -1;
    if (dump.first) dump.first[req] = -1;
    if (dump.inst) dump.inst[req] = -1;
}

}  // namespace maaso
