// Layout of the walking kernel's shared memory (eval_walk.cu), used by the validation kernel too, which
// has to know how much of it a placement needs.
#pragma once
#include "lane_sim.cuh"

namespace maaso {

constexpr int kWalkWarps = 16;                    // one block per SM
constexpr int kWalkThreads = 32 * kWalkWarps;
constexpr int kWalkRing = 64;                     // ring entries per warp

// One block: decode-step tables, SLO limits, the completion rings, the pool.
struct WalkLayout {
    uint32_t steps;   // [n_rows][64] u32
    uint32_t lims;    // [n_classes] {TTFT limit, TBT limit (all ones = none), end-to-end limit (64 bits, 2^62 = none)}
    uint32_t ring;    // [warps][kWalkRing] {finish, first token}
    uint32_t ring_b;  // [warps][kWalkRing] {request, instance}
    uint32_t pool;
};
__host__ __device__ inline WalkLayout walk_layout(uint32_t n_rows, uint32_t n_classes) {
    WalkLayout l;
    l.ring = 0;
    l.ring_b = (uint32_t)(kWalkWarps * kWalkRing) * 16u;
    l.lims = l.ring_b + (uint32_t)(kWalkWarps * kWalkRing) * 8u;
    l.steps = l.lims + n_classes * 16u;
    l.pool = (l.steps + n_rows * 256u + 127u) & ~127u;
    return l;
}

// One placement's region: sums (kWalkSums bytes: one set of four 16-byte units per lane, unit-major, then hits by
// class bin), 16 bytes per model, 16 per instance, then per instance its slots: the eight block minima, the stack
// of free slots (a byte each), then blocks of 8 slots with the keys (end index << 6 | slot), the request indices
// and the first-token times.
constexpr uint32_t kWalkLaneSums = 4u * 32u * 16u;
constexpr uint32_t kWalkSums = kWalkLaneSums + 48u;
__host__ __device__ inline uint32_t walk_slot_bytes(uint32_t nblk) { return 32u + ((8u * nblk + 15u) & ~15u) + nblk * 128u; }
__host__ __device__ inline uint32_t walk_region_bytes(uint32_t n_models, uint32_t n_inst, uint32_t slot_bytes) {
    return kWalkSums + 16u * (n_models + n_inst) + slot_bytes;
}

// Times are 32-bit offsets from an epoch that each placement moves along (eval_walk.cu).  The bounds below
// keep every sum of a round inside 31 bits; a batch whose tables or limits exceed them, checked on the host,
// runs on the lane-group kernel, and a single placement that gets beyond kWalkHorizon is handed to the
// one-warp-per-placement kernel, both of which compute in 64 bits.
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
