// Where a placement is scored, and what a call launches for that: buckets, room in shared memory, the choice between the
// kernels.  The host decides what it launches, the validation kernel where a placement goes, and both have to agree, so
// both ask here.  Plain C++ but for the qualifiers: compiles without CUDA.
#pragma once
#include <stdint.h>
#include "../../include/maaso.h"

#ifdef __CUDACC__
#define MAASO_HD __host__ __device__
#else
#define MAASO_HD
#endif

namespace maaso {

// Buckets the validation kernel sorts candidates into.
// 0..5: lane groups of 1,2,4,8,16,32 lanes (one lane per instance)
// 6..8: block layout with 2, 4, 8 warps, one warp per instance, state in registers
// 9:    block layout with 16 warps striding over up to 128 instances, state in shared memory
// 10..18: thread mapping, by how many lanes of a warp work at a time (32, 24, 16, 12, 8, 6, 4, 2, 1:
//        the larger the placements, the fewer fit the warp's pools)
// 19:   one warp per placement with the lane-group code
// 20..30: walking kernel: up to 32 instances by the room a placement needs (one, 2, 4, 8, 16 times a
//        warp's part), more than 32, 64-bit times by the room
constexpr int kNumBuckets = 31;
constexpr int kWalkModes = 5;
constexpr int kWalkBucket0 = 20, kWalkBig0 = kWalkBucket0 + kWalkModes, kWalkLong0 = kWalkBig0 + 1;
constexpr int kWalkBuckets = 2 * kWalkModes + 1;
constexpr int kGenericBlockBucket = 9;
constexpr int kThreadBucket0 = 10;  // buckets 10..18: the thread mapping, by lanes per warp
constexpr int kThreadBuckets = 9;
constexpr int kPack4 = 2, kPack8 = 3;  // in place of the lane groups (Route::pack): up to 4 and up to 8 instances
constexpr int kWideBucket = 19;     // what no other kernel that was launched takes: one warp per placement

// Warps of the walking kernel per block, one block per SM: 16 with 128 registers each.  12 with room for 168 serve the engines
// that fix a request's speed better in a batch of at most three placements (or parts of them) per warp, which its longest chains
// bound (2,000 x 17,000 of the paper's shape 9.5 and 9.75 ms, with queues 1,000 x 8,000 2.14 and 2.20; 12,000 x 30,000 under load
// 5.5 and 4.7).
// With the default engine 12 are 0 to 4 % better where they are better at all (one node, 2,368 x 5,000 1.91 and 1.95 ms, three
// models under load 7,000 x 10,000 1.43 and 1.48) and lose where 16 hold the batch at once or it is lightly loaded (one node
// at 2 requests a second, 2,368 x 4,000 3.55 and 2.32; the paper's shape, 3,000 x 8,000 4.1 and 3.4): 16 always.
constexpr int kWalkWarps = 16, kWalkWarpsFew = 12;
constexpr uint32_t kPackWarps = 14u;              // of the packed kernel (launch_eval_pack)
constexpr int kWalkRing = 64;                     // ring entries per warp
constexpr uint32_t kBlockShared = 227u * 1024u;   // shared memory of a block

// Decode-step rows in shared memory: steps alone, or each with its reciprocal, which spares the rounds a division and takes twice
// the room.  The engines that fix a request's speed never divide by a step: steps alone.  The others carry reciprocals up to so
// many rows; beyond that the room is worth more (more placements fit one warp's part of the pool).  Measured, with and without:
//   up to 32 instances, 32-bit times: 12,000 x 10,000 under load, 100 rows 1.73 and 1.84 ms, 120 1.68 and 1.69, 160 1.76 and 1.70,
//     256 2.36 and 2.01; 4,000 x 8,000 lightly loaded, 120 rows 2.29 and 2.54, 160 3.22 and 2.24; some 20 instances each, 6,000 x
//     8,000, 100 rows 4.02 and 4.04, 120 3.03 and 2.97, 160 2.88 and 2.66
//   more than 32: 2,000 x 5,000, 50 rows 9.29 and 9.39, 60 9.63 and 8.56, 100 7.53 and 6.82 (a few hundred of them, which all run at
//     once either way, 1 to 2 % better with)
//   64-bit times: 5 to 6 % better with, up to 100 rows.  The line there is where the pool still holds every placement.
constexpr uint32_t kWalkRow = 65u * 4u, kWalkRowRcp = 65u * 8u;  // bytes of a row
constexpr uint32_t kWalkRcpRows = 128u, kWalkRcpRowsBig = 52u, kWalkRcpRowsLong = 80u;
constexpr uint32_t kWalkList = 33u * 32u + 128u;  // list of 32 requests and one behind it, what lanes without an instance read

// One block of the walking kernel (walk_kernel.cuh): the completion rings, SLO limits, decode-step tables, the pool.
struct WalkLayout {
    uint32_t ring;    // [warps][kWalkRing] {finish, first token, request, instance}; 64-bit times: {finish, first token}
    uint32_t ring_b;  // 64-bit times: [warps][kWalkRing] {request, instance}
    uint32_t lims;    // [n_classes] {TTFT limit, TBT limit (all ones = none), end-to-end limit (64 bits, 2^62 = none)}
    uint32_t wide;    // 64-bit times: [n_classes] {TTFT limit (2^62 = none), TBT limit (negative = none)}
    uint32_t steps;   // [n_rows][65] decode step by running count, `rcp`: {step, reciprocal}, which is 2^32 / step or (walk_dynamic.cuh)
                      // an exact one; a count of 0: a step of 1, an idle clock
    uint32_t list;    // `list`: [warps][kWalkList], requests that need a round, and the dummy region (walk_dynamic.cuh)
    uint32_t pool;
};
MAASO_HD inline WalkLayout walk_layout(uint32_t n_rows, uint32_t n_classes, bool wide, uint32_t warps, bool rcp, bool list = false) {
    WalkLayout l;
    l.ring = 0;
    l.ring_b = warps * (uint32_t)kWalkRing * 16u;
    l.lims = l.ring_b + (wide ? warps * (uint32_t)kWalkRing * 8u : 0u);
    l.wide = l.lims + n_classes * 16u;
    l.steps = l.wide + (wide ? n_classes * 16u : 0u);
    l.list = (l.steps + n_rows * (rcp ? kWalkRowRcp : kWalkRow) + 15u) & ~15u;
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
MAASO_HD inline uint32_t walk_slots_at(uint32_t nblk) { return 32u + ((8u * nblk + 15u) & ~15u); }
// `block`: bytes of 8 slots; kWalkBlock (walk_dynamic.cuh): keys and the rest behind them from a fixed offset on
constexpr uint32_t kWalkKeys = 96u;
constexpr uint32_t kWalkBlock = 96u, kWalkBlockLong = 128u, kWalkBlockKeys = 32u;
MAASO_HD inline uint32_t walk_slot_bytes(uint32_t b, bool fixed_speed, uint32_t key_bytes, uint32_t block) {
    const uint32_t nblk = (b + 7u) >> 3;
    return fixed_speed ? ((b * key_bytes + 15u) & ~15u) : (block == kWalkBlock ? kWalkKeys : walk_slots_at(nblk)) + nblk * block;
}
MAASO_HD inline uint32_t walk_rest_bytes(WalkKind kind) { return kind == kWalkUsual ? 0u : (kind == kWalkBigKind ? 48u : 80u); }
MAASO_HD inline uint32_t walk_region_bytes(uint32_t n_models, uint32_t n_inst, uint32_t slot_bytes, WalkKind kind) {
    return kWalkSums + 16u * (n_models + n_inst) + (kind ? walk_rest_bytes(kind) * n_inst + ((8u * n_models + 15u) & ~15u) : 0u) + slot_bytes;
}
// Placements of more than 32 instances are sorted by the room they need, in steps of kWalkStepBytes; a block's first is
// its largest and decides how many of its warps work side by side.
constexpr uint32_t kWalkStepBytes = 640u;
MAASO_HD inline uint32_t walk_big_bin(uint32_t need) {
    const uint32_t k = need / kWalkStepBytes;
    return 255u - (k < 255u ? k : 255u);
}

// Packed kernel (eval_pack.cu): a lane's block minima, free slots, keys; 16 bytes so that lanes start in different banks.
constexpr uint32_t kPackLane = 32u + 64u + 256u + 16u;
MAASO_HD inline WalkLayout pack_layout(uint32_t n_rows, uint32_t n_classes) { return walk_layout(n_rows, n_classes, false, kPackWarps, true); }
inline bool pack_fits(uint32_t n_rows, uint32_t n_classes) {
    return pack_layout(n_rows, n_classes).pool + 32u * kPackWarps * kPackLane <= kBlockShared;
}

// What the host has decided for a call.
struct Route {
    uint32_t flags, mapping;
    uint32_t n_rows, n_models, n_classes;
    uint32_t walk_bytes;     // walking kernel: bytes of shared memory one of 16 warps has for a placement, 0 = not used
    uint32_t walk_usual;     // the same for placements of up to 32 instances, with walk_warps warps
    uint32_t walk_warps;
    uint32_t walk_rcp;       // decode-step rows of the walking kernel carry reciprocals: up to 32 instances and 32-bit times,
    uint32_t walk_rcp_big;   // more instances or 64-bit times
    uint32_t walk_parts;     // queues: parts a placement is replayed in, 1 or the number of models
    uint32_t walk_long;      // the whole batch with 64-bit times
    uint32_t walk_all;       // MAASO_MAP_AUTO: the batch goes to the walking kernel whatever its load
    uint32_t pack;           // placements of at most 8 instances that could go to the lane groups share the steps of a warp instead
    uint32_t thread_pool_units;  // thread mapping: 16-byte units one warp has for the cold part of its placements' state, 0 = not used
    uint32_t thread_hot_units;   // and for the hot part (2 units per instance, shared memory)
};

MAASO_HD inline bool route_fixed_speed(uint32_t flags) { return (flags & (MAASO_FLAG_ENGINE_FROZEN | MAASO_FLAG_INSTANCE_QUEUES)) != 0; }
MAASO_HD inline bool route_variant(uint32_t flags) { return route_fixed_speed(flags) || (flags & MAASO_FLAG_TBT_MAXGAP) != 0; }

// The walking and the packed kernel's part of a call that the walking kernel runs: room, and who takes the batch.
// `items`: placements times traces, `insts`: instances times traces; `fits32`: 32-bit times hold the batch's tables and limits.
inline void route_walk(Route& r, uint64_t items, uint64_t insts, uint32_t sm_count, bool fits32) {
    const bool queues = (r.flags & MAASO_FLAG_INSTANCE_QUEUES) != 0;  // always with 64-bit times
    const bool fixed_speed = route_fixed_speed(r.flags);
    r.walk_long = fits32 || queues ? 0u : 1u;
    r.walk_rcp = !fixed_speed && r.n_rows <= kWalkRcpRows ? 1u : 0u;
    r.walk_rcp_big = !fixed_speed && r.n_rows <= (r.walk_long ? kWalkRcpRowsLong : kWalkRcpRowsBig) ? 1u : 0u;
    r.walk_bytes = ((kBlockShared - walk_layout(r.n_rows, r.n_classes, true, kWalkWarps, r.walk_rcp_big != 0).pool) / kWalkWarps) & ~15u;
    // With queues the models of a placement are independent of one another and can be replayed side by side, while the batch is
    // bound by its longest chains: every part scans the whole trace.  A placement has no more parts than instances, and what decides is
    // the number of parts in all, up to twelve a warp, and that of placements, as few models gain less.  Whole and in parts (ms),
    // lightly loaded and (after the semicolon) under load:
    //   two models      4,000 x 6,000 6.9 and 5.7; 3.3 and 3.3    8,000 9.8 and 10.2; 3.7 and 3.8
    //   three           1,000 3.6 and 1.7; 1.9 and 1.5            5,300 7.1 and 5.6; 2.7 and 2.8        16,000 14.8 and 15.4; 6.1 and 7.7
    //   eight           1,330 3.8 and 1.4; 2.6 and 1.1            3,280 4.0 and 3.0; 2.5 and 2.2        5,300 5.2 and 4.6; 3.1 and 3.3
    //     17 instances  1,330 3.9 and 2.2; 2.9 and 2.1            2,660 5.0 and 3.9; 2.8 and 3.4        5,300 8.3 and 7.4; 4.9 and 6.3
    //   sixteen         1,330 2.6 and 1.1; 2.5 and 1.1            3,280 2.9 and 2.4; 2.5 and 2.3        5,300 3.9 and 3.7; 2.7 and 3.6
    //     21 instances  1,330 8.5 and 7.1; 7.6 and 7.1            2,660 10.2 and 9.7; 8.0 and 9.3       5,300 12.8 and 13.2; 10.6 and 13.4
    // (The paper's shape, 2,000 x 17,000: 9.25 and 5.35.)  The warps per block go by the parts (6,000 of them 7.2 ms with 12, 5.3 with 16).
    const uint64_t parts = items * r.n_models < insts ? items * r.n_models : insts;
    r.walk_parts = queues && items <= 3ull * sm_count * kWalkWarpsFew && parts <= 12ull * sm_count * kWalkWarpsFew ? r.n_models : 1u;
    r.walk_warps = fixed_speed && items * r.walk_parts <= 3ull * sm_count * kWalkWarpsFew ? kWalkWarpsFew : kWalkWarps;
    r.walk_usual = ((kBlockShared - walk_layout(r.n_rows, r.n_classes, queues, r.walk_warps, r.walk_rcp != 0, !fixed_speed).pool) / r.walk_warps) & ~15u;
    // Small batches walk whatever their load.  A large one that is not loaded is bound by the instructions of its rounds,
    // which several placements of one warp share in the packed kernel; its steps take the same time however few placements
    // there are, so that the line lies where the walking kernel needs as long.  Measured on 4,000 requests, walking and packed:
    //   one model     at 1 a second 3,000 placements 4.1 and 4.1 ms, 4,096 4.5 and 4.15, 5,000 5.5 and 4.3; at 2 a second 4,096 4.4
    //                 and 4.35, 5,000 4.5 and 4.5, 6,500 6.3 and 4.65; at 4 a second 6,500 4.4 and 4.6, 8,192 5.7 and 4.8
    //   three models  (a third of the lanes of a step at work) at 1 a second 12,288 7.6 and 8.5, 18,432 10.8 and 10.4; at 2 a second
    //                 18,432 8.4 and 10.0, 40,000 16.9 and 17.2; at 4 a second 40,000 11.6 and 15.1 (and it walks by its load: eval_impl)
    // With the optimistic estimate one model at 2 a second 4,096 5.05 and 4.85, three 12,288 7.4 and 8.1, 24,576 13.7 and 12.4.
    // With fixed speeds or queues the alternative is the lane-group kernel, and the lines are early for one model and late for two.
    // Walking (queues: in one piece) and lane groups, 4,000 requests:
    //   fixed speeds    one model at 1 and 2 a second 4,096 7.4 and 9.9, 5.3 and 9.1; 6,144 8.2 and 10.0, 7.1 and 9.4; 8,192 10.6 and
    //                   10.0, 8.4 and 9.3; two at 1 and 3 a second 6,144 6.6 and 7.9, 5.0 and 7.8; 9,000 9.0 and 8.2, 6.4 and 8.0;
    //                   12,288 11.7 and 8.4, 8.2 and 8.4; three at 1 and 4 a second 18,432 11.7 and 15.0, 7.1 and 13.3; 30,000 18.5
    //                   and 20.7, 10.9 and 19.1
    //   queues          one 4,096 7.6 and 9.5, 5.6 and 8.6; 8,192 11.0 and 9.7, 8.9 and 8.7; two 6,144 7.3 and 7.7, 5.9 and 7.6;
    //                   9,000 10.0 and 7.9, 8.4 and 7.9; 12,288 13.1 and 8.2, 10.7 and 8.2; three 9,216 8.7 and 8.7, 6.9 and 8.3;
    //                   18,432 15.8 and 15.0, 12.7 and 14.1
    r.walk_all = items <= (r.n_models == 1 ? 4096u : 6144u * (uint64_t)r.n_models) ? 1u : 0u;
    r.pack = !r.walk_all && !r.walk_long && !route_variant(r.flags) && pack_fits(r.n_rows, r.n_classes) ? 1u : 0u;
}

// Of `grid` blocks, those that replay `big` placements of more than 32 instances, `warps` of them in a block at a time, while the others
// replay `small` smaller ones (each counted once per trace): as many as hold the larger ones at once, and no fewer than their share of
// the work, one of them counted as eight smaller ones (25 warp milliseconds alone and 40 in company, against 4, over 40,000 requests; with
// the default engine, both estimates, and with fixed speeds any weight from 2 to 32 is as good within 2 %, 5 to 1,000 larger ones among 300
// to 30,000).  A smaller placement counts once also where queues have it replayed in parts (Route::walk_parts): its rounds are shared out
// among the parts.  Counted by the parts, 2,500 x 6,000 of which 100 are larger took 7.4 instead of 7.1 ms with two models and 6.8 instead of 6.4
// with three, 5,000 of which 12 are 7.1 instead of 6.8 and 6.6 instead of 6.4.
MAASO_HD inline uint32_t walk_big_share(uint64_t big, uint64_t small, uint32_t warps, uint32_t grid) {
    const uint64_t once = (big + warps - 1u) / warps, share = (8u * big * grid + 8u * big + small - 1u) / (8u * big + small);
    const uint64_t most = grid < big ? grid : big, least = once > share ? once : share;
    return (uint32_t)(most < least ? most : least);
}

// Are the lane groups launched?
MAASO_HD inline bool route_groups(const Route& r) {
    return !r.pack && !r.walk_all && (r.mapping == MAASO_MAP_GROUP || r.mapping == MAASO_MAP_AUTO);
}

// What a placement needs, instance by instance.
struct PlacementSize {
    uint32_t n, slots, slots64;  // walking kernel: shared memory of the slots, with 64-bit times too
    uint32_t units;              // thread mapping: 16-byte units of cold instance state (per instance 2 + key blocks + minima)
    MAASO_HD void add(const Route& r, uint32_t b) {  // (an instance of batch cap `b`; `n` is set before)
        const bool fixed_speed = route_fixed_speed(r.flags);
        const uint32_t key_bytes = fixed_speed && (r.walk_long || (r.flags & MAASO_FLAG_INSTANCE_QUEUES)) ? 8u : 4u;
        slots += walk_slot_bytes(b, fixed_speed, key_bytes, r.walk_long ? kWalkBlockLong : (n > kWalkBig ? kWalkBlockKeys : kWalkBlock));
        slots64 += walk_slot_bytes(b, fixed_speed, fixed_speed ? 8u : 4u, kWalkBlockLong);
        units += 2u + 2u * ((b + 7u) >> 3) + 2u;
    }
};

// Where a valid placement can be scored: its bucket among the lane groups, the block kernels, the packed kernel and the one-warp
// kernel, its bucket among the walking and thread kernels (-1: none), the room it takes in the walking kernel.  One of the two is
// never -1, and every bucket named here is one whose kernel the call launches (route_launches).
struct Home {
    int group, walk;
    uint32_t need;
};
MAASO_HD inline Home route_home(const Route& r, const PlacementSize& s) {
    Home h = {-1, -1, 0u};
    const uint32_t n = s.n;
    if (r.thread_pool_units) {
        // as many lanes per item as placements of this size fit the warp's pools
        const uint32_t cold = n ? r.thread_pool_units / s.units : 32u, hot = n ? r.thread_hot_units / (2u * n) : 32u, fit = cold < hot ? cold : hot;
        const uint32_t lanes[9] = {32, 24, 16, 12, 8, 6, 4, 2, 1};
        for (int i = 0; i < 9 && h.walk < 0; i++)
            if (fit >= lanes[i]) h.walk = kThreadBucket0 + i;
    }
    if (r.walk_bytes) {
        const bool queues = (r.flags & MAASO_FLAG_INSTANCE_QUEUES) != 0, big = n > kWalkBig && !r.walk_long;
        h.need = walk_region_bytes(r.n_models, n, s.slots, r.walk_long || queues ? kWalkLongKind : (big ? kWalkBigKind : kWalkUsual));
        if (big) {
            // (and all of the pool has to hold it if it is handed over)
            const uint32_t later = walk_region_bytes(r.n_models, n, s.slots64, kWalkLongKind);
            if ((h.need > later ? h.need : later) <= r.walk_bytes * (uint32_t)kWalkWarps) h.walk = kWalkBig0;
        } else {
            // one warp's part of the walking kernel's pool, or 2, 4, 8 of them (16 with 64-bit times)
            const uint32_t part = r.walk_long ? r.walk_bytes : r.walk_usual;
            for (uint32_t k = 0; k < (uint32_t)kWalkModes - 1u && h.walk < 0; k++)
                if (h.need <= (part << k)) h.walk = (r.walk_long ? kWalkLong0 : kWalkBucket0) + (int)k;
            if (h.walk < 0 && r.walk_long && h.need <= part * 16u) h.walk = kWalkLong0 + 4;
        }
    }
    if (r.mapping == MAASO_MAP_BLOCK) {
        h.group = n <= 2 ? 6 : (n <= 4 ? 7 : (n <= 8 ? 8 : kGenericBlockBucket));
    } else if (r.pack && n <= 8) {
        h.group = n <= 4 ? kPack4 : kPack8;
    } else if (route_groups(r) && n <= 32) {
        for (h.group = 0; (1u << h.group) < n;) h.group++;
    } else if (h.walk < 0 || (r.mapping != MAASO_MAP_THREAD && !r.walk_bytes)) {
        // More than 32 instances outside the walking and the thread kernel, and whatever their pools cannot hold where the lane
        // groups are not launched.  (One block per placement only when the block mapping is asked for.)
        h.group = kWideBucket;
    }
    return h;
}

// The scoring kernels of a call; `may_leave`: placements may leave the 32-bit horizon in mid-trace.
struct Launches {
    bool groups, pack, walk, big, far, threads, blocks;
    uint32_t wide_from;  // one-warp kernel: the fewest instances of a placement that it takes; 0: it is not launched
};
// `n_inst`: the most instances that a valid placement of the call can have.
inline Launches route_launches(const Route& r, uint64_t n_inst, bool may_leave) {
    Launches l;
    l.groups = route_groups(r);
    l.pack = r.pack != 0;
    l.walk = r.walk_bytes && !r.walk_long;
    l.big = l.walk && n_inst > kWalkBig;
    l.far = r.walk_bytes && (r.walk_long || may_leave || r.pack);
    l.threads = r.thread_pool_units != 0;
    l.blocks = r.mapping == MAASO_MAP_BLOCK;
    // a placement takes the most room with every batch cap at its largest
    l.wide_from = 0;
    for (uint32_t n = 1; n <= (uint32_t)MAASO_MAX_INSTANCES && n <= n_inst && !l.wide_from; n++) {
        PlacementSize s = {n, 0u, 0u, 0u};
        s.add(r, MAASO_WMAX);
        s.slots *= n;
        s.slots64 *= n;
        s.units *= n;
        if (route_home(r, s).group == kWideBucket) l.wide_from = n;
    }
    return l;
}

}  // namespace maaso
