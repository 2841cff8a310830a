// Layout of the walking kernel's shared memory (walk_kernel.cuh), used by the validation kernel too, which
// has to know how much of it a placement needs.
#pragma once
#include "lane_sim.cuh"

namespace maaso {

// Warps per block, one block per SM: 16 with 128 registers each.  12 with room for 168 serve the engines that fix a request's
// speed better in a batch of at most three placements (or parts of them) per warp, which its longest chains bound (2,000 x
// 17,000 of the paper's shape 9.5 and 9.75 ms, with queues 1,000 x 8,000 2.14 and 2.20; 12,000 x 30,000 under load 5.5 and 4.7).
// With the default engine 12 are 0 to 4 % better where they are better at all (one node, 2,368 x 5,000 1.91 and 1.95 ms, three
// models under load 7,000 x 10,000 1.43 and 1.48) and lose where 16 hold the batch at once or it is lightly loaded (one node
// at 2 requests a second, 2,368 x 4,000 3.55 and 2.32; the paper's shape, 3,000 x 8,000 4.1 and 3.4): 16 always.
constexpr int kWalkWarps = 16, kWalkWarpsFew = 12;
constexpr int kWalkRing = 64;                     // ring entries per warp

constexpr uint32_t kWalkRow = 65u * 8u;           // bytes of a decode-step row
constexpr uint32_t kWalkList = 33u * 32u + 128u;  // list of 32 requests and one behind it, what lanes without an instance read

// One block: the completion rings, SLO limits, decode-step tables, the pool.
struct WalkLayout {
    uint32_t ring;    // [warps][kWalkRing] {finish, first token, request, instance}; 64-bit times: {finish, first token}
    uint32_t ring_b;  // 64-bit times: [warps][kWalkRing] {request, instance}
    uint32_t lims;    // [n_classes] {TTFT limit, TBT limit (all ones = none), end-to-end limit (64 bits, 2^62 = none)}
    uint32_t wide;    // 64-bit times: [n_classes] {TTFT limit (2^62 = none), TBT limit (negative = none)}
    uint32_t steps;   // [n_rows][65] {decode step, 2^32 / step} by running count (walk_dynamic.cuh: exact
                      // reciprocals); a count of 0: a step of 1, an idle clock
    uint32_t list;    // `list`: [warps][kWalkList], requests that need a round, and the dummy region (walk_dynamic.cuh)
    uint32_t pool;
};
__host__ __device__ inline WalkLayout walk_layout(uint32_t n_rows, uint32_t n_classes, bool wide, uint32_t warps, bool list = false) {
    WalkLayout l;
    l.ring = 0;
    l.ring_b = warps * (uint32_t)kWalkRing * 16u;
    l.lims = l.ring_b + (wide ? warps * (uint32_t)kWalkRing * 8u : 0u);
    l.wide = l.lims + n_classes * 16u;
    l.steps = l.wide + (wide ? n_classes * 16u : 0u);
    l.list = (l.steps + n_rows * kWalkRow + 15u) & ~15u;
    l.pool = (l.list + (list ? warps * kWalkList : 0u) + 127u) & ~127u;
    return l;
}

// One placement's region: sums (kWalkSums bytes: one set of four 16-byte units per lane, unit-major, then hits by
// class bin), 16 bytes per model, 16 per instance, with more than 32 instances their resting state (unit-major) and
// a lower bound per model, then per instance its slots: the eight block minima, the stack of free slots (a byte
// each), the keys (end index << 6 | slot, in blocks of 8), then what a running request must remember: {first-token time,
// request index}, 8 bytes (64-bit times: the request indices, then the first-token times).  Keys alone with more than 32
// instances, where the rest is in global memory: shared memory decides how many such placements are resident.  In the
// engines that fix a request's speed at admission: the finish times in falling order, so that the next to free is popped
// off the end.
enum WalkKind : uint32_t { kWalkUsual = 0, kWalkBigKind = 1, kWalkLongKind = 2 };
constexpr uint32_t kWalkLaneSums = 4u * 32u * 16u;
constexpr uint32_t kWalkSums = kWalkLaneSums + 48u;
constexpr uint32_t kWalkBig = 32u;  // more instances than this rest in shared memory
__host__ __device__ inline uint32_t walk_slots_at(uint32_t nblk) { return 32u + ((8u * nblk + 15u) & ~15u); }
// `block`: bytes of 8 slots; kWalkBlock (walk_dynamic.cuh): keys and the rest behind them from a fixed offset on
constexpr uint32_t kWalkKeys = 96u;
constexpr uint32_t kWalkBlock = 96u, kWalkBlockLong = 128u, kWalkBlockKeys = 32u;
__host__ __device__ inline uint32_t walk_slot_bytes(uint32_t b, bool fixed_speed, uint32_t key_bytes, uint32_t block) {
    const uint32_t nblk = (b + 7u) >> 3;
    return fixed_speed ? ((b * key_bytes + 15u) & ~15u) : (block == kWalkBlock ? kWalkKeys : walk_slots_at(nblk)) + nblk * block;
}
__host__ __device__ inline uint32_t walk_rest_bytes(WalkKind kind) { return kind == kWalkUsual ? 0u : (kind == kWalkBigKind ? 48u : 80u); }
__host__ __device__ inline uint32_t walk_region_bytes(uint32_t n_models, uint32_t n_inst, uint32_t slot_bytes, WalkKind kind) {
    return kWalkSums + 16u * (n_models + n_inst) + (kind ? walk_rest_bytes(kind) * n_inst + ((8u * n_models + 15u) & ~15u) : 0u) + slot_bytes;
}
// Placements of more than 32 instances are sorted by the room they need, in steps of kWalkStepBytes; a block's first is
// its largest and decides how many of its warps work side by side.
constexpr uint32_t kWalkStepBytes = 640u;
__host__ __device__ inline uint32_t walk_big_bin(uint32_t need) {
    const uint32_t k = need / kWalkStepBytes;
    return 255u - (k < 255u ? k : 255u);
}
// Global memory for one block's running requests: two bytes of it per byte of pool.
__host__ __device__ inline size_t walk_big_scratch(uint32_t pool_bytes) { return (size_t)pool_bytes * 2u; }

// The most a placement can need: 128 instances of 64 slots, 16 models, 8-byte keys or requests beside 4-byte keys.
constexpr uint32_t kWalkMost = 160u * 1024u;

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
