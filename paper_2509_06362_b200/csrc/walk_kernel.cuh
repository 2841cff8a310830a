// Scoring kernel: one warp replays one placement.
//
// What bounds it: the chain of distributor rounds of a placement, each of which depends on the one before, and
// over a large batch the instructions of all rounds.  So a round is kept short, and requests that need none
// do not cost one.  The 32 lanes play two parts:
//   scan    32 requests at a time, one per lane (a coalesced 16-byte load, the next chunk prefetched in
//           registers): which of them could be served at all, by any instance of their model, if nothing had
//           happened since the latest look at it?  Start times only move forward, so what fails is rejected
//           without a round, 32 at a time (about 40 instructions, 16 more per instance of a model if anything
//           gets past the first, instance-blind test).
//   round   lane l is the placement's l-th instance (sorted by model): advance, predict, choose by one
//           reduction, admit.
// Times are 32-bit offsets from an epoch that moves along with the dispatcher's clock (half the instructions of
// 64-bit times).  Instance state is in registers, slot keys and what a running request must remember in shared
// memory: nothing on the chain touches global memory.  Completions go to a small ring and are accounted by all
// lanes together when it fills, so the hash and the sums of the statistics stay off the chain; what they need of
// the request is read from the trace then.
//
// Nothing is counted per rejected request: the request count and the checksum of "all of them rejected"
// are per-class totals of the trace, and a served request takes its own term out again.
//
// What nearly every call runs, the default engine with up to 32 instances and 32-bit times, has a body of its own, written for
// the shortest round (walk_dynamic.cuh).  `Walk` here is the body of all the others.
//
// Measured (B200, whole calls with routing and top-k; lane-group, thread or one-warp kernel before): 143 placements x 500
// requests 0.14 ms (0.56), one node's 10,864 x 10,000 4.2 ms (12.0), 2,000 x 17,000 of the paper's shape 5.9 to 6.4 ms (33.9), with
// queues 5.3 ms (27.8), three models, 100,000 x 100,000 under load 52 ms (135), 2,000 placements of 33 to 128 instances x
// 10,000 6.3 to 7.4 ms (13.8).  Nearly all instructions of a round depend on one another: what the next step
// needs is therefore read from shared memory ahead of the choice, the uncommon outcomes share one branch, and tests of several
// conditions are written without branches (& and | for && and ||).
// What some of the lanes do, an admission or an instance's state out of and into shared memory, all lanes compute, with
// predicated stores and selections: parting the lanes and joining them again took longer than the work (2,000 placements of 33 to 128
// instances x 10,000 8.40 -> 6.75 ms, 500 with fixed speeds 7.54 -> 6.02; masked sub-clusters, 9,000 x 12,000 9.03 -> 7.74; kStraight says
// where not).
// Completions are left in a branch (without it 2 % slower to 2 % faster).
//
// The block's pool of shared memory is split evenly among its warps.  Placements beyond one warp's part run
// first, with half, a quarter, ... of the warps at work and twice, four times, ... the room for each (kWalkModes);
// those of more than 32 instances all need several parts, and a block starts as many warps as its largest allows.
//
// Variants (template arguments of one body, so that each carries nothing of the others):
//   Opt     the distributor predicts with the step time right after admission (optimistic estimate)
//   Eng     0: decode speed follows the running count; 1: fixed at admission (slot keys are finish times, requests
//           are accounted when they are admitted); 2: the same with a queue in front of every instance
//   Wide    64-bit times from time zero: for batches whose tables or limits 32-bit times cannot hold, for queues
//           (which grow to hours where nothing turns requests away), and for placements that leave the 32-bit
//           horizon in mid-trace and are handed over
//   Big     more than 32 instances: lane l takes instances l, l + 32, ... one after the other (those of a model are
//           neighbours, so a round looks at one or two of these strides); their state rests in shared memory
//   Rcp     decode-step rows carry reciprocals (route.cuh: which tables' rows do)
#pragma once
#include <cstring>
#include <type_traits>
#include "steps.cuh"
#include "walk.cuh"

namespace maaso {

constexpr uint32_t kWFull = 0xFFFFFFFFu;
// byte offsets in a placement's sums, after the per-lane ones: hits by class bin, extra distributor rounds
constexpr uint32_t kSByClass = kWalkLaneSums, kSExtra = kWalkLaneSums + 32u;
constexpr int32_t kWPast = -(1 << 30);     // an arrival at least this far before the epoch: beyond every finite limit

extern __shared__ __align__(128) unsigned char walk_smem[];

__device__ __forceinline__ uint4& w4(uint32_t off) { return *reinterpret_cast<uint4*>(walk_smem + off); }
__device__ __forceinline__ uint2& w2(uint32_t off) { return *reinterpret_cast<uint2*>(walk_smem + off); }
__device__ __forceinline__ uint32_t& w1(uint32_t off) { return *reinterpret_cast<uint32_t*>(walk_smem + off); }
__device__ __forceinline__ int64_t& wi(uint32_t off) { return *reinterpret_cast<int64_t*>(walk_smem + off); }
template <class T>
__device__ __forceinline__ T& wt(uint32_t off) { return *reinterpret_cast<T*>(walk_smem + off); }
__device__ __forceinline__ int64_t i64_of(uint32_t lo, uint32_t hi) { return (int64_t)(((uint64_t)hi << 32) | lo); }
__device__ __forceinline__ uint32_t lo32(int64_t v) { return (uint32_t)(uint64_t)v; }
__device__ __forceinline__ uint32_t hi32(int64_t v) { return (uint32_t)((uint64_t)v >> 32); }
__device__ __forceinline__ uint64_t wshfl_xor(uint64_t v, int o) {
    const uint32_t a = __shfl_xor_sync(kWFull, (uint32_t)v, o), b = __shfl_xor_sync(kWFull, (uint32_t)(v >> 32), o);
    return ((uint64_t)b << 32) | a;
}
__device__ __forceinline__ int32_t wshfl(int32_t v, int src) { return __shfl_sync(kWFull, v, src); }
__device__ __forceinline__ int64_t wshfl(int64_t v, int src) {
    return i64_of(__shfl_sync(kWFull, lo32(v), src), __shfl_sync(kWFull, hi32(v), src));
}
__device__ __forceinline__ uint32_t warp_min(uint32_t v) { return __reduce_min_sync(kWFull, v); }
__device__ __forceinline__ uint64_t warp_min(uint64_t v) {  // the smallest high half, the smallest low half that comes with it
    const uint32_t hi = (uint32_t)(v >> 32), mh = __reduce_min_sync(kWFull, hi);
    return ((uint64_t)mh << 32) | __reduce_min_sync(kWFull, hi == mh ? (uint32_t)v : 0xFFFFFFFFu);
}
// Stores of the lanes for which `p` holds, to shared memory by its own addresses, without a branch.
__device__ __forceinline__ void st1_if(bool p, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.u32 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st4_if(bool p, uint32_t a, const uint4& v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %5, 0;\n\t@p st.shared.v4.u32 [%0], {%1, %2, %3, %4};\n\t}"
                 ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void stb_if(bool p, uint32_t a, uint32_t v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.u8 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((uint32_t)p) : "memory");
}
__device__ __forceinline__ void st2_if(bool p, uint32_t a, const uint2& v) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.shared.v2.u32 [%0], {%1, %2};\n\t}" ::"r"(a), "r"(v.x), "r"(v.y), "r"((uint32_t)p) : "memory");
}
// Entry i of the decode-step rows in shared memory (WalkLayout::steps).
__device__ __forceinline__ uint32_t walk_step(const EvalParams& P, uint32_t i) {
    const uint32_t r = i / 65u, w = i - 65u * r;
    return w ? max((uint32_t)P.rows[r * kRowStride + 1u + w], 1u) : 1u;
}

// Accounts the completion ring, one entry per lane and pass, into the lane's own sums in the region `base`:
//   unit 0: sum and maximum of the time to first token; 1: of the end-to-end time; 2: last completion, checksum;
//   3: output tokens, requests served, hits
template <bool Wide>
static __device__ __noinline__ void walk_account(const EvalParams& P, bool dumping, uint32_t oc, uint32_t base, uint32_t ring,
                                                 uint32_t ring_b, uint32_t cnt, int64_t epoch, uint32_t lims, uint32_t wide,
                                                 const uint4* reqs) {
    const uint32_t lane = threadIdx.x & 31u, sums = base + 16u * lane;
    __syncwarp();
    for (uint32_t e = lane; e < cnt; e += 32u) {
        const uint4 ra = w4(ring + e * 16u);
        const uint2 rb = Wide ? w2(ring_b + e * 8u) : make_uint2(ra.z, ra.w);
        const uint4 rec = __ldg(reqs + rb.x);
        const uint4 u0 = w4(sums), u1 = w4(sums + 512u), u2 = w4(sums + 1024u), u3 = w4(sums + 1536u);
        const int64_t fin = Wide ? i64_of(ra.x, ra.y) : epoch + (int32_t)ra.x, first = Wide ? i64_of(ra.z, ra.w) : epoch + (int32_t)ra.y;
        const int64_t arrival = i64_of(rec.x, rec.y);
        const uint32_t S = rec.w & 0xFFFFu, cls = (rec.w >> 16) & 0xFFu;
        const uint4 lim = w4(lims + cls * 16u);
        const int64_t ttft = first - arrival, e2e = fin - arrival;
        bool hit = e2e <= i64_of(lim.z, lim.w);  // (no branches)
        if (Wide) {
            const int64_t l_ttft = wi(wide + cls * 16u), l_tbt = wi(wide + cls * 16u + 8u);
            hit = hit & (ttft <= l_ttft) & ((l_tbt < 0) | (fin - first <= (int64_t)(S - 1u) * l_tbt));
        } else {
            hit = hit & ((lim.x == 0xFFFFFFFFu) | (ttft <= (int64_t)lim.x)) &
                  ((lim.y == 0xFFFFFFFFu) | ((uint64_t)(fin - first) <= (uint64_t)(S - 1u) * lim.y));
        }
        // the request's term as a served one in, its term as a rejected one out
        const uint64_t sum = i64_of(u2.z, u2.w) + served_hash(rb.x, fin, first, rb.y) - rejected_hash(rb.x);
        const int64_t st = i64_of(u0.x, u0.y) + ttft, mt = max(i64_of(u0.z, u0.w), ttft);
        const int64_t se = i64_of(u1.x, u1.y) + e2e, me = max(i64_of(u1.z, u1.w), e2e);
        const int64_t mk = max(i64_of(u2.x, u2.y), fin), tk = i64_of(u3.x, u3.y) + S;
        w4(sums) = make_uint4(lo32(st), hi32(st), lo32(mt), hi32(mt));
        w4(sums + 512u) = make_uint4(lo32(se), hi32(se), lo32(me), hi32(me));
        w4(sums + 1024u) = make_uint4(lo32(mk), hi32(mk), (uint32_t)sum, (uint32_t)(sum >> 32));
        w4(sums + 1536u) = make_uint4(lo32(tk), hi32(tk), u3.z + 1u, u3.w + (hit ? 1u : 0u));
        if (hit) atomicAdd(&w1(base + kSByClass + 4u * min(cls, 7u)), 1u);
        if (dumping) {
            const Dump d = dump_for(P, oc);
            if (d.finish) d.finish[rb.x] = fin;
            if (d.first) d.first[rb.x] = first;
            if (d.inst) d.inst[rb.x] = (int32_t)rb.y;
            if (d.hist) atomicAdd(d.hist + ttft_bin(ttft), 1u);
        }
    }
    __syncwarp();
}

// All live keys of one instance move down by `d`, the counter's value in a key's place (the counter restarts at 0).  Rare.
static __device__ __noinline__ uint32_t walk_rebase(uint32_t area, uint32_t keys, uint32_t nblk, uint32_t d, uint32_t kmin) {
    for (uint32_t b = 0; b <= nblk; b++) {
        const uint32_t p = b ? keys + 32u * (b - 1u) : area;  // the minima, then the keys of each block
        for (uint32_t i = 0; i < 8u; i++) {
            const uint32_t k = w1(p + 4u * i);
            if (k != kKeyEmpty) w1(p + 4u * i) = k - d;
        }
    }
    return kmin != kKeyEmpty ? kmin - d : kmin;
}

// A placement that left the 32-bit horizon is replayed with 64-bit times, once, for every trace of the pass; that
// kernel starts after this one and clears the placement's side outputs first.
static __device__ __noinline__ void walk_hand_over(const EvalParams& P, uint32_t cand, bool fixed_speed) {
    if (atomicExch(&P.code[cand], 0xFFFFFFFEu) == 0xFFFFFFFEu) return;
    const uint32_t lo = P.offsets[cand], n_i = P.offsets[cand + 1] - lo;
    uint32_t slots = 0, mode = 0;
    for (uint32_t i = 0; i < n_i; i++) slots += walk_slot_bytes((P.inst[lo + i] >> 12) & 0xFFu, fixed_speed, fixed_speed ? 8u : 4u, kWalkBlockLong);
    const uint32_t need = walk_region_bytes(P.n_models, n_i, slots, kWalkLongKind);
    while (mode + 1u < (uint32_t)kWalkModes && need > (P.walk_bytes << mode)) mode++;
    // (what 16 parts cannot hold is not in a walking bucket in the first place)
    const uint32_t bucket = (uint32_t)kWalkLong0 + mode, at = atomicAdd(&P.bucket_count[bucket], 1u);
    P.bucket_list[(size_t)bucket * P.n_cand + at] = cand;
}

// One part of a placement's record: adds its sums to what the other parts left there; the last of `parts` completes the record,
// which counts them in its reserved word until then.
static __device__ __noinline__ void walk_add_part(maaso_result* out, uint32_t parts, uint32_t status, uint32_t counted, uint64_t rejected_sum,
                                                  const Stats& st, const uint32_t* h) {
    uint32_t* const w = reinterpret_cast<uint32_t*>(out);
    auto wide = [&](uint32_t at) { return reinterpret_cast<unsigned long long*>(w + at); };
    atomicAdd(w + 2, st.served);
    atomicAdd(w + 3, st.hit);
    for (int i = 0; i < 8; i++)
        if (h[i]) atomicAdd(w + 6 + i, h[i]);
    atomicAdd(wide(14), (unsigned long long)st.sum_ttft);
    atomicMax(wide(16), (unsigned long long)st.max_ttft);
    atomicAdd(wide(18), (unsigned long long)st.sum_e2e);
    atomicMax(wide(20), (unsigned long long)st.max_e2e);
    atomicMax(wide(22), (unsigned long long)st.makespan);
    atomicAdd(wide(24), (unsigned long long)st.tokens);
    atomicAdd(wide(26), (unsigned long long)st.checksum);
    if (status) atomicOr(w + 31, status);
    __threadfence();
    if (atomicAdd(w + 30, 1u) + 1u < parts) return;
    __threadfence();
    auto get = [&](uint32_t at) { return (int64_t)__ldcg(wide(at)); };
    Stats all;
    all.served = __ldcg(w + 2); all.hit = __ldcg(w + 3);
    all.sum_ttft = get(14); all.max_ttft = get(16);
    all.sum_e2e = get(18);  all.max_e2e = get(20);
    all.makespan = get(22); all.tokens = (uint64_t)get(24);
    all.checksum = (uint64_t)get(26) + rejected_sum;
    uint32_t hits[8];
    for (int i = 0; i < 8; i++) hits[i] = __ldcg(w + 6 + i);
    write_result(out, __ldcg(w + 31), counted, counted - all.served, counted, all, hits);
}

// The record of a placement that is through, from its sums in the region `base`; of several parts, see above.
static __device__ __forceinline__ void walk_finish(const EvalParams& P, uint32_t base, uint32_t tr, uint32_t cand, bool use_mask,
                                                   uint32_t cmask, uint32_t status, uint32_t extra, uint32_t parts = 1) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint4 u0 = w4(base + 16u * lane), u1 = w4(base + 16u * lane + 512u), u2 = w4(base + 16u * lane + 1024u), u3 = w4(base + 16u * lane + 1536u);
    Stats st;
    st.sum_ttft = i64_of(u0.x, u0.y); st.max_ttft = i64_of(u0.z, u0.w);
    st.sum_e2e = i64_of(u1.x, u1.y);  st.max_e2e = i64_of(u1.z, u1.w);
    st.makespan = i64_of(u2.x, u2.y); st.checksum = (uint64_t)i64_of(u2.z, u2.w);
    st.tokens = (uint64_t)i64_of(u3.x, u3.y);
    st.served = __reduce_add_sync(kWFull, u3.z);
    st.hit = __reduce_add_sync(kWFull, u3.w);
    // the request count and the checksum of "everything rejected", from the per-class totals
    uint32_t counted_all = 0;
    uint64_t rejected_sum = 0;
    for (uint32_t c = lane; c < P.n_classes; c += 32u)
        if (!use_mask || ((cmask >> c) & 1u)) {
            counted_all += (uint32_t)P.trace_class_tot[tr][2u * c];
            rejected_sum += P.trace_class_tot[tr][2u * c + 1u];
        }
    counted_all = __reduce_add_sync(kWFull, counted_all);
    if (parts == 1u) st.checksum += rejected_sum;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        st.sum_ttft += (int64_t)wshfl_xor((uint64_t)st.sum_ttft, o);
        st.sum_e2e += (int64_t)wshfl_xor((uint64_t)st.sum_e2e, o);
        st.tokens += wshfl_xor(st.tokens, o);
        st.checksum += wshfl_xor(st.checksum, o);
        rejected_sum += wshfl_xor(rejected_sum, o);
        st.max_ttft = max(st.max_ttft, (int64_t)wshfl_xor((uint64_t)st.max_ttft, o));
        st.max_e2e = max(st.max_e2e, (int64_t)wshfl_xor((uint64_t)st.max_e2e, o));
        st.makespan = max(st.makespan, (int64_t)wshfl_xor((uint64_t)st.makespan, o));
    }
    if (lane == 0) {
        uint32_t h[8];
#pragma unroll
        for (int i = 0; i < 8; i++) h[i] = w1(base + kSByClass + 4u * i);
        maaso_result* const out = P.out + (size_t)tr * P.n_cand + cand;
        if (parts == 1u) write_result(out, status, counted_all, counted_all - st.served, (uint64_t)counted_all + extra, st, h);
        else walk_add_part(out, parts, status, counted_all, rejected_sum, st, h);
    }
    __syncwarp();
}

// What one lane knows of its instance.
template <class T>
struct WInst {
    T t;           // clock, a decode-step boundary (may lag `now`)
    T tb;          // last boundary before the next completion if nobody is admitted; "far" while idle.  Fixed speeds: the
                   // earliest finish time
    uint32_t K;    // decode steps done at t since the counter last restarted
    uint32_t kmin; // smallest slot key
    uint32_t w, B;
    uint32_t sw;   // one decode step at the current level (1 while idle)
    uint32_t rsw;  // 2^32 / sw
    uint32_t tag;  // 1 << model (0 for a lane without an instance) | place in the placement as given << 16
    uint32_t area, keys, row;  // byte offsets of its slots, of its first block of keys and of its decode-step row
    uint32_t pre_base, pre_q16, stepB;
    uint32_t pay;  // of what its running requests must remember
};

template <bool Opt, int Eng, bool Wide, bool Big, bool Rcp = (Eng == 0)>
struct Walk {
    using T = typename std::conditional<Wide, int64_t, int32_t>::type;
    using U = typename std::conditional<Wide, uint64_t, uint32_t>::type;
    using Inst = WInst<T>;
    static constexpr bool kFixed = Eng != 0;
    static constexpr bool kAgain = Opt || Eng == 1;  // a wait is followed by a new choice
    static constexpr T kFar = Wide ? (T)((int64_t)1 << 62) : (T)kWalkFar;
    static constexpr U kTier1 = (U)1 << (8 * sizeof(U) - 1);
    static constexpr U kNone = ~(U)0;
    static constexpr uint32_t kKeyBytes = kFixed ? (uint32_t)sizeof(T) : 4u;
    // Fixed speeds and queues, a winner's ring entry and next free slot: without a branch, but for up to 32 instances with 32-bit times, which
    // that makes 1 % slower on average (three models, 12,000 x 6,000 at 400 a second 1.14 and 1.16 ms, the paper's shape up to 2.8 %).
    static constexpr bool kStraight = Wide || Big;
    // Queues: times are below 2^58 (see the admission), so that a key has room for the lane (3 % less than a vote and a search
    // for the winner's bit)
    static constexpr bool kLaneKey = Eng == 2 && Wide && !Big;
    static constexpr bool kAway = Big && !Wide && !kFixed;  // running requests' data in global memory
    static constexpr uint32_t kBlock = Wide ? kWalkBlockLong : (Big ? kWalkBlockKeys : kWalkBlock);
    static constexpr WalkKind kKind = Wide ? kWalkLongKind : (Big ? kWalkBigKind : kWalkUsual);
    static constexpr uint32_t kRest = Wide ? 80u : 48u;
    static constexpr uint32_t kEntry = Rcp ? 8u : 4u, kRow = Rcp ? kWalkRowRcp : kWalkRow;

    // A class's limits; does a first token `since` after the arrival, with `Sm1` more tokens of `step`, meet them?
    struct Limits {
        uint4 a;
        int64_t ttft, tbt;
        __device__ __forceinline__ void load(const WalkLayout& L, uint32_t cls16) {
            a = w4(L.lims + cls16);
            if (Wide) {
                ttft = wi(L.wide + cls16);
                tbt = wi(L.wide + cls16 + 8u);
            }
        }
        __device__ __forceinline__ bool met(U since, uint32_t Sm1, uint32_t step) const {
            const bool end = (int64_t)((uint64_t)Sm1 * step + since) <= i64_of(a.z, a.w);  // (no branches)
            if constexpr (Wide) return (int64_t)since <= ttft && (Sm1 == 0u || tbt < 0 || (int64_t)step <= tbt) && end;
            else return (since <= a.x) & ((Sm1 == 0u) | (step <= a.y)) & end;
        }
    };
    static __device__ __forceinline__ T prefill(uint32_t base, uint32_t q16, uint32_t in_tok) {
        return (T)((U)base + (U)(((uint64_t)q16 * in_tok + 32768u) >> 16));
    }

    // Big: resting state of instance j, unit-major.  `all`: not only what a round changes.  With 32-bit times the
    // last unit is not kept: it is in the instance's entry.
    static __device__ __forceinline__ void put(uint32_t rest, uint32_t n_i, uint32_t j, const Inst& in, bool all) {
        uint4 u[(sizeof(Inst) + 15) / 16];
        memcpy(u, &in, sizeof(Inst));
#pragma unroll
        for (uint32_t k = 0; k < kRest / 16u; k++)
            if (all || k < (Wide ? 3u : 2u)) w4(rest + 16u * (k * n_i + j)) = u[k];
    }
    // What a round changes, of the lanes for which `p` holds.
    static __device__ __forceinline__ void put_if(bool p, uint32_t rest, uint32_t n_i, uint32_t j, const Inst& in) {
        uint4 u[(sizeof(Inst) + 15) / 16];
        memcpy(u, &in, sizeof(Inst));
#pragma unroll
        for (uint32_t k = 0; k < (Wide ? 3u : 2u); k++) st4_if(p, smem_addr(walk_smem) + rest + 16u * (k * n_i + j), u[k]);
    }
    static __device__ __forceinline__ void get(uint32_t rest, uint32_t ents, uint32_t n_i, uint32_t j, Inst& in) {
        uint4 u[(sizeof(Inst) + 15) / 16];
#pragma unroll
        for (uint32_t k = 0; k < kRest / 16u; k++) u[k] = w4(rest + 16u * (k * n_i + j));
        if (!Wide) {
            const uint4 e = w4(ents + 16u * j);
            u[3] = make_uint4(e.y, e.z, e.w, 0u);
        }
        memcpy(&in, u, sizeof(Inst));
        if (!Wide && Opt) in.stepB = w1(in.row + kEntry * in.B);
    }

    // One warp takes the placements of a bucket, one after the other.  `base`: its part of shared memory;
    // `away`: the block's global memory for running requests, two bytes per byte of pool (kAway).
    static __device__ __forceinline__ void bucket(const EvalParams& P, const WalkLayout& L, int bucket, uint32_t base,
                                                  uint32_t static_idx, uint32_t static_total, unsigned char* away) {
        constexpr uint32_t kCap = (uint32_t)kWalkRing;
        const uint32_t smem = smem_addr(walk_smem);
        const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
        const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
        // With a queue in front of every instance the dispatcher never waits, and requests of one model leave no trace on the
        // others': a placement can be replayed in parts, a model each, side by side (EvalParams::walk_parts).
        constexpr bool kParts = Eng == 2 && !Big;
        const uint32_t n_parts = kParts ? P.walk_parts : 1u;
        const uint32_t total = P.bucket_count[bucket] * n_parts * n_traces;
        const uint32_t ring = L.ring + (threadIdx.x >> 5) * kWalkRing * 16u, ring_b = L.ring_b + (threadIdx.x >> 5) * kWalkRing * 8u;
        const bool use_mask = P.class_mask != nullptr && P.n_classes <= 32;
        const uint32_t models = base + kWalkSums, ents = models + 16u * P.n_models, ent = ents + 16u * lane;

        uint32_t idx = static_idx;
        while (idx < total) {
            // ---- the next placement ------------------------------------------------------------------------
            const uint32_t tr = idx % n_traces;
            const uint32_t cand = P.bucket_list[(size_t)bucket * P.n_cand + idx / n_traces / n_parts];
            const uint4* const reqs = P.trace_reqs[tr];
            const uint32_t n_req = P.trace_n[tr];
            uint32_t n_i;
            auto next = [&]() {
                if (lane == 0) idx = static_total + atomicAdd(&P.walk_ctr[bucket - kWalkBucket0], 1u);
                idx = __shfl_sync(kWFull, idx, 0);
            };
            uint4 nxt = make_uint4(0u, 0u, 0u, 0u);  // the lane's request of the next chunk, as loaded
            if (n_req) nxt = __ldg(reqs + min(lane, n_req - 1u));
            Inst in;
            uint32_t rest, lbs;  // Big: resting instances, lower bounds per model; 64-bit times: start times of the entries
            {
                const uint32_t lo = P.offsets[cand];
                n_i = P.offsets[cand + 1] - lo;
                rest = ents + 16u * n_i;
                lbs = rest + kRest * n_i;
                uint32_t area = (Big || Wide) ? lbs + ((8u * P.n_models + 15u) & ~15u) : rest;  // slots of the first instance of a stride
                for (uint32_t i = lane; i < kWalkSums / 16u; i += 32u) w4(base + 16u * i) = make_uint4(0u, 0u, 0u, 0u);
                // instances sorted by model, in their given order within a model (the order in which ties are broken)
                uint32_t before = 0;
                for (uint32_t k = 0; k < P.n_models; k++) {
                    uint32_t n = 0;
                    for (uint32_t s = 0; s < (Big ? n_i : 1u); s += 32u) {
                        const uint32_t j = s + lane, word = j < n_i ? P.inst[lo + j] : 0xFu, m = j < n_i ? word & 0xFu : 0xFFFFFFFFu;
                        const uint32_t b = __ballot_sync(kWFull, m == k);
                        if (m == k) w2(ents + 16u * (before + n + (uint32_t)__popc(b & below))) = make_uint2(word, j);
                        n += (uint32_t)__popc(b);
                    }
                    // per model: smallest prefill base, smallest prediction step, its instances (byte offsets of their entries)
                    if (lane == k) {
                        w4(models + 16u * k) = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, ents + 16u * before, ents + 16u * (before + n));
                        if (Big) wi(lbs + 8u * k) = 0;
                    }
                    before += n;
                }
                __syncwarp();
                for (uint32_t s = 0; s < (Big ? n_i : 1u); s += 32u) {
                    const uint32_t j = s + lane, at = ents + 16u * j;
                    in.t = 0; in.tb = kFar; in.K = 0; in.kmin = kKeyEmpty; in.w = 0; in.B = 1; in.sw = 1; in.rsw = ~0u;
                    in.pre_base = in.pre_q16 = 0; in.stepB = 1; in.tag = 0; in.area = in.keys = in.pay = in.row = L.steps;
                    uint32_t nblk = 0;
                    if (j < n_i) {
                        const uint2 e = w2(at);
                        const uint32_t md = e.x & 0xFu, r = md * P.n_strategies + ((e.x >> 4) & 0xFFu);
                        in.tag = (1u << md) | (e.y << 16);
                        in.B = (e.x >> 12) & 0xFFu;
                        nblk = (in.B + 7u) >> 3;
                        in.row = L.steps + r * kRow;
                        in.pre_base = (uint32_t)P.rows[r * kRowStride];
                        in.pre_q16 = (uint32_t)P.rows[r * kRowStride + 1];
                        in.stepB = w1(in.row + kEntry * in.B);
                        // the smallest step a prediction can use: the step at the batch cap, or (optimistic estimate) at any
                        // level up to it
                        uint32_t ms = in.stepB;
                        if (Opt)
                            for (uint32_t w = 1; w < in.B; w++) ms = min(ms, w1(in.row + kEntry * w));
                        atomicMin(&w1(models + 16u * md), in.pre_base);
                        atomicMin(&w1(models + 16u * md + 4u), ms);
                        // per instance: earliest start, prefill base and slope, smallest prediction step
                        w4(at) = make_uint4(0u, in.pre_base, in.pre_q16, ms);
                    }
                    const uint32_t bytes = nblk ? walk_slot_bytes(in.B, kFixed, kKeyBytes, kBlock) : 0u;
                    uint32_t incl = bytes;
                    for (uint32_t o = 1; o < 32u; o <<= 1) {
                        const uint32_t v = __shfl_up_sync(kWFull, incl, o);
                        if (lane >= o) incl += v;
                    }
                    if (nblk) {
                        in.area = area + incl - bytes;
                        in.keys = kFixed ? in.area : in.area + walk_slots_at(nblk);
                        in.pay = in.keys + 32u * nblk;
                        if (!kFixed) {
                            for (uint32_t i = 0; i < 8u * (nblk + 1u); i++) w1(i < 8u ? in.area + 4u * i : in.keys + 4u * (i - 8u)) = kKeyEmpty;
                            for (uint32_t i = 0; i < in.B; i++) walk_smem[in.area + 32u + i] = (unsigned char)i;
                        }
                    }
                    if (Wide && !Big && j < n_i) wt<T>(rest + 8u * j) = 0;
                    if (Big) {
                        area += __shfl_sync(kWFull, incl, 31);
                        if (j < n_i) put(rest, n_i, j, in, true);
                    }
                }
            }
            uint32_t hasmodel = 0;
            for (uint32_t k = 0; k < P.n_models; k++) {
                const uint2 r = w2(models + 16u * k + 8u);
                hasmodel |= r.x < r.y ? 1u << k : 0u;
            }
            uint32_t parts = 1, mine = 0xFFFFFFFFu;  // parts of the placement; models whose requests are this one's to report
            if constexpr (kParts) {
                if (n_parts > 1u) {
                    const uint32_t k = idx / n_traces % n_parts;
                    const bool first = k == (hasmodel ? (uint32_t)__ffs((int)hasmodel) - 1u : 0u);
                    if (!first && !((hasmodel >> k) & 1u)) {  // (nothing of this model)
                        next();
                        continue;
                    }
                    parts = max(1u, (uint32_t)__popc(hasmodel));
                    mine = (1u << k) | (first ? ~hasmodel : 0u);
                    hasmodel &= 1u << k;
                }
            }
            const uint32_t cmask = use_mask ? P.class_mask[cand] : 0xFFFFFFFFu;
            const bool side = P.rej_by_model != nullptr || (P.dump_row && P.dump_row[cand] >= 0);
            if (Wide && Eng != 2) {
                // a placement handed over has left counts in its side outputs
                const size_t oc = (size_t)tr * P.n_cand + cand;
                if (P.rej_by_model && lane < (uint32_t)MAASO_MAX_MODELS) P.rej_by_model[oc * MAASO_MAX_MODELS + lane] = 0;
                if (P.ttft_hist)
                    for (uint32_t i = lane; i < (uint32_t)MAASO_TTFT_BINS; i += 32u) P.ttft_hist[oc * MAASO_TTFT_BINS + i] = 0;
                __threadfence();
            }
            __syncwarp();

            uint32_t ring_n = 0, status = 0;
            int64_t epoch = 0;
            T now = 0;
            // A time of this lane has left the horizon.  Its next completion may have wrapped then, so from the next round on nothing
            // is asked of the lane, up to the end of the chunk, when the placement is given up: no completion is taken from it (it
            // might have none running), no clock runs past a completion, and no prediction of it is compared (bit 31 of a key
            // says "full").  In the round in which it happens the lane has a free slot and a clock that is right.
            bool bad = false;
            T rel = 0;                     // this lane's request of the chunk: arrival,
            uint32_t c_in = 0, c_meta = 0; // input tokens, output tokens | class | model

            auto flush = [&]() {
                walk_account<Wide>(P, P.dump_row || P.ttft_hist, tr * P.n_cand + cand, base, ring, ring_b, ring_n, epoch, L.lims, L.wide, reqs);
                ring_n = 0;
            };
            auto take_chunk = [&](const uint4& v) {
                const int64_t d = i64_of(v.x, v.y) - epoch;
                if constexpr (Wide) rel = d;
                else rel = d >= (int64_t)kWalkNowMax ? kFar : (d < (int64_t)kWPast ? kWPast : (int32_t)d);
                c_in = v.z;
                c_meta = v.w;
            };
            // Entry of the instance's row: decode step and reciprocal, the latter computed when the level changes if rows have none.
            auto entry = [&](uint32_t at) -> uint2 {
                if constexpr (Rcp) return w2(at);
                else return make_uint2(w1(at), 0u);
            };
            auto is_due = [&](T upto) { return kFixed ? in.tb <= upto : in.tb < upto; };
            // when the instance could start a request
            auto start = [&]() -> T { return kFixed ? (in.w == in.B ? in.tb : now) : (in.w == in.B ? in.tb + (T)in.sw : in.t); };
            // Step `sw` and next completion `left` steps after in.t >= 0; flags what leaves the horizon.
            auto next_end = [&](uint32_t left, bool busy, uint2 step) {
                const uint32_t sw = step.x;
                in.sw = sw;
                in.rsw = Rcp ? step.y : walk_rcp(sw);
                if constexpr (Wide) {
                    in.tb = busy ? in.t + (int64_t)((uint64_t)left * sw) - (int64_t)sw : kFar;
                } else {
                    const uint64_t tc = (uint64_t)left * sw + (uint32_t)in.t;
                    in.tb = busy ? (int32_t)((uint32_t)tc - sw) : kFar;
                    bad = bad | (busy & (tc > (uint64_t)kWalkHorizon));
                }
            };
            auto firsts = [&]() { return in.pay + 32u * ((in.B + 7u) >> 3); };  // 64-bit times: first tokens of the running requests
            // Running requests' first tokens, when the epoch moves by `up`.  (Further back than 32 bits reach: the lane has left
            // the horizon.)
            auto rebase_firsts = [&](T up) {
                if constexpr (!kFixed && !Wide) {
                    for (uint32_t i = 0; i < in.B && in.w > 0; i++) {
                        if (w1(in.keys + 4u * i) == kKeyEmpty) continue;
                        int32_t* const f = kAway ? reinterpret_cast<int32_t*>(away + 2u * (in.keys + 4u * i - L.pool)) : &wt<int32_t>(in.pay + 8u * i);
                        const int64_t v = (int64_t)(kAway ? __ldcg(f) : *f) - up;
                        bad = bad || v < -(int64_t)kWalkFar;
                        if (kAway) __stcg(f, (int32_t)v);
                        else *f = (int32_t)v;
                    }
                }
            };
            // Completions (fixed speeds: slots that free) of the lanes in `due`, one per lane and iteration, until every
            // clock has reached `upto`.
            auto events = [&](bool due, T upto) {
                uint32_t dm = __ballot_sync(kWFull, due);
                while (dm) {
                    if constexpr (kFixed) {
                        if (due) {
                            in.w--;
                            in.tb = in.w > 0 ? wt<T>(in.keys + kKeyBytes * (in.w - 1u)) : kFar;
                            due = in.w > 0 && is_due(upto);
                        }
                    } else {
                        const uint32_t adds = (uint32_t)__popc(dm);
                        if (ring_n + adds > kCap) flush();
                        if (due) {
                            const uint32_t slot = in.kmin & 63u;
                            const uint32_t k8 = in.keys + 4u * slot, kb = in.keys + 4u * (slot & 56u), mb = in.area + ((slot >> 3) << 2);
                            // (the key and its block's minimum go first: what is left is read without them)
                            w1(k8) = kKeyEmpty;
                            w1(mb) = kKeyEmpty;
                            const uint4 k0 = w4(kb), k1 = w4(kb + 16u), m0 = w4(in.area), m1 = w4(in.area + 16u);
                            const uint2 step = entry(in.row + kEntry * in.w - kEntry);
                            uint2 run;  // first token, request; 64-bit times: first token
                            uint32_t rq = 0;
                            if constexpr (kAway) run = __ldcg(reinterpret_cast<const uint2*>(away + 2u * (k8 - L.pool)));
                            else if constexpr (!Wide) run = w2(in.pay + 8u * slot);
                            else run = w2(firsts() + 8u * slot), rq = w1(in.pay + 4u * slot);
                            in.t = in.tb + (T)in.sw;
                            in.K = in.kmin >> 6;
                            in.w--;
                            walk_smem[in.area + 32u + in.w] = (unsigned char)slot;
                            const uint32_t kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                            const uint32_t mv[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                            const uint32_t bmin = min8(kv);
                            const uint32_t e = ring_n + (uint32_t)__popc(dm & below);
                            if constexpr (Wide) {
                                w4(ring + 16u * e) = make_uint4(lo32(in.t), hi32(in.t), run.x, run.y);
                                w2(ring_b + 8u * e) = make_uint2(rq, in.tag >> 16);
                            } else {
                                w4(ring + 16u * e) = make_uint4((uint32_t)in.t, run.x, run.y, in.tag >> 16);
                            }
                            w1(mb) = bmin;
                            in.kmin = min(bmin, min8(mv));
                            const uint32_t left = (in.kmin >> 6) - in.K;
                            const bool busy = in.w > 0;
                            next_end(left, busy, step);
                            due = busy & ((left == 0u) | (in.tb < upto)) & !bad;
                        }
                        ring_n += adds;
                    }
                    dm = __ballot_sync(kWFull, due);
                }
            };
            // Clocks of the lanes in `go` that lag behind `upto` while nothing completes: the next step boundary; an idle
            // instance starts at once.
            auto catch_up = [&](bool go, T upto) {
                if constexpr (Wide) {
                    if (go && in.t < upto) {
                        const uint32_t k = walk_steps((T)(upto - in.t), in.sw, in.rsw);
                        in.t = in.w == 0 ? upto : in.t + (T)((U)k * in.sw);
                        in.K += k;
                    }
                } else {
                    const int32_t dt = go ? max(upto - in.t, 0) : 0;
                    const uint32_t k = walk_steps(dt, in.sw, in.rsw);
                    in.t += (int32_t)(k * in.sw);
                    in.K += k;
                }
            };
            // The next free slot and the step with one request more, read ahead of the choice.
            uint32_t top = 0;
            uint2 more = make_uint2(0u, 0u);
            auto peek = [&]() {
                if (!kFixed) {
                    top = walk_smem[in.area + 32u + in.w];
                    more = entry(in.row + kEntry * in.w + kEntry);
                }
            };
            // One request's times into the ring (`e`: its entry).
            auto record = [&](uint32_t e, T fin, T first, uint32_t req) {
                if constexpr (Wide) {
                    w4(ring + e * 16u) = make_uint4(lo32(fin), hi32(fin), lo32(first), hi32(first));
                    w2(ring_b + e * 8u) = make_uint2(req, in.tag >> 16);
                } else {
                    w4(ring + e * 16u) = make_uint4((uint32_t)fin, (uint32_t)first, req, in.tag >> 16);
                }
            };
            auto record_if = [&](bool p, uint32_t e, T fin, T first, uint32_t req) {
                if constexpr (Wide) {
                    st4_if(p, smem + ring + e * 16u, make_uint4(lo32(fin), hi32(fin), lo32(first), hi32(first)));
                    st2_if(p, smem + ring_b + e * 8u, make_uint2(req, in.tag >> 16));
                } else {
                    st4_if(p, smem + ring + e * 16u, make_uint4((uint32_t)fin, (uint32_t)first, req, in.tag >> 16));
                }
            };
            // "map": prefill at the step boundary (running decodes stall), then occupy a free slot.  With fixed speeds the slot
            // is busy until the finish time, and `queued` takes over the slot that frees first; an instance's finish times
            // are in falling order, the winner's (lane `wl`) are moved by all lanes.  All lanes call it.
            auto admit = [&](bool win, int wl, uint32_t req, uint32_t Sm1, T pre, bool queued) {
                if constexpr (kFixed) {
                    if (ring_n + 1u > kCap) flush();
                    const uint32_t at = __shfl_sync(kWFull, (in.keys << 7) | in.w, wl), a = at >> 7;
                    uint32_t n = at & 127u, level;
                    if (queued) n--;  // the last one goes
                    T v[2], first = now + pre;
#pragma unroll
                    for (uint32_t h = 0; h < 2u; h++) v[h] = 32u * h < n && lane + 32u * h < n ? wt<T>(a + kKeyBytes * (lane + 32u * h)) : kFar;
                    level = n;
                    if (queued) {  // whatever frees together with the slot taken is not busy when the request starts
                        const T tb = wshfl(in.tb, wl);
                        level -= (uint32_t)(__popc(__ballot_sync(kWFull, v[0] == tb)) + __popc(__ballot_sync(kWFull, v[1] == tb)));
                        first = in.tb + pre;
                    }
                    const uint64_t span = (uint64_t)Sm1 * w1(in.row + (win ? kEntry * level : 0u) + kEntry);
                    T fin = first + (T)span;
                    if constexpr (kStraight) {
                        if constexpr (Wide) status = win & (((uint64_t)fin >> 57) != 0) ? (uint32_t)MAASO_CAND_ELOOP : status;  // beyond what the engine takes
                        else bad = bad | (win & ((span > (uint64_t)kWalkHorizon) | (fin > (T)kWalkHorizon)));
                        record_if(win, ring_n, fin, first, req);
                    } else if (win) {
                        bad = bad || span > (uint64_t)kWalkHorizon || fin > (T)kWalkHorizon;
                        record(ring_n, fin, first, req);
                    }
                    ring_n++;
                    fin = wshfl(fin, wl);
                    uint32_t pos = n;
#pragma unroll
                    for (uint32_t h = 0; h < 2u; h++) {
                        pos -= (uint32_t)__popc(__ballot_sync(kWFull, v[h] < fin));
                        if (v[h] < fin) wt<T>(a + kKeyBytes * (lane + 32u * h + 1u)) = v[h];
                    }
                    if (lane == 0) wt<T>(a + kKeyBytes * pos) = fin;
                    __syncwarp();
                    if constexpr (kStraight) {
                        const T next_free = wt<T>(a + kKeyBytes * n);
                        in.w = win ? n + 1u : in.w;
                        in.tb = win ? next_free : in.tb;
                    } else if (win) {
                        in.w = n + 1u;
                        in.tb = wt<T>(a + kKeyBytes * n);
                    }
                } else if (Sm1 == 0u) {  // done at the end of its prefill, never occupies a slot
                    if (ring_n + 1u > kCap) flush();
                    if (win) {
                        in.t += pre;
                        if (in.w > 0) in.tb += pre;
                        if constexpr (!Wide) bad = bad || in.t > (T)kWalkHorizon || (in.w > 0 && in.tb > (T)kWalkHorizon);
                        record(ring_n, in.t, in.t, req);
                    }
                    ring_n++;
                } else if constexpr (!Wide) {
                    // (without a branch: every lane computes what it would leave, the winner takes it)
                    uint32_t nK = in.w > 0 ? in.K : 0u;  // no live end index: the counter restarts
                    if (win && nK + Sm1 > kRelMax) {
                        in.kmin = walk_rebase(in.area, in.keys, (in.B + 7u) >> 3, nK << 6, in.kmin);
                        nK = 0;
                    }
                    const uint32_t nk = ((nK + Sm1) << 6) | top, nmin = min(in.kmin, nk), k8 = in.keys + 4u * top, mb = in.area + ((top >> 1) & 28u);
                    const T nt = in.t + pre;
                    const uint64_t tc = (uint64_t)((nmin >> 6) - nK) * more.x + (uint32_t)nt;
                    st1_if(win, smem + k8, nk);
                    st1_if(win, smem + mb, min(w1(mb), nk));
                    if constexpr (kAway) {
                        if (win) __stcg(reinterpret_cast<uint2*>(away + 2u * (k8 - L.pool)), make_uint2((uint32_t)nt, req));
                    } else {
                        st2_if(win, smem + in.pay + 8u * top, make_uint2((uint32_t)nt, req));
                    }
                    in.t = win ? nt : in.t;
                    in.K = win ? nK : in.K;
                    in.kmin = win ? nmin : in.kmin;
                    in.w = win ? in.w + 1u : in.w;
                    in.sw = win ? more.x : in.sw;
                    in.rsw = win ? (Rcp ? more.y : walk_rcp(more.x)) : in.rsw;
                    in.tb = win ? (T)((uint32_t)tc - more.x) : in.tb;
                    bad = bad | (win & (tc > (uint64_t)kWalkHorizon));
                } else if (win) {  // 64-bit times
                    const uint32_t slot = top;
                    in.t += pre;
                    if (in.w == 0) in.K = 0;  // no live end index: the counter restarts
                    if (in.K + Sm1 > kRelMax) {
                        in.kmin = walk_rebase(in.area, in.keys, (in.B + 7u) >> 3, in.K << 6, in.kmin);
                        in.K = 0;
                    }
                    const uint32_t nk = ((in.K + Sm1) << 6) | slot;
                    w1(in.keys + 4u * slot) = nk;
                    w1(in.pay + 4u * slot) = req;
                    w2(firsts() + 8u * slot) = make_uint2(lo32(in.t), hi32(in.t));
                    atomicMin(&w1(in.area + ((slot >> 3) << 2)), nk);
                    in.kmin = min(in.kmin, nk);
                    in.w++;
                    next_end((in.kmin >> 6) - in.K, true, more);
                }
            };

            for (uint32_t cb = 0; cb < n_req; cb += 32u) {
                take_chunk(nxt);
                nxt = __ldg(reqs + min(cb + 32u + lane, n_req - 1u));
                auto counted = [&]() { return cb + lane < n_req && ((cmask >> ((c_meta >> 16) & 31u)) & 1u) && (!kParts || ((mine >> (c_meta >> 24)) & 1u)); };
                // Which of the chunk's requests from lane `from` on may need the distributor.
                auto test = [&](uint32_t from) -> uint32_t {
                    const uint32_t Sm1 = (c_meta & 0xFFFFu) - 1u, model = c_meta >> 24;
                    const T at = max(now, rel);
                    bool live = lane >= from && counted() && ((hasmodel >> model) & 1u);
                    // (without a branch: every lane has a request, behind the last one the last one once more)
                    const uint4 me = w4(models + 16u * model);
                    Limits lim;
                    lim.load(L, (c_meta >> 12) & 0xFF0u);
                    U since = (U)(at - rel) + me.x;  // earliest first token, since the arrival
                    if (Big && rel != kFar) since = max((T)since, (T)wi(lbs + 8u * model) - rel);
                    live = live & lim.met(since, Sm1, me.y);
                    const uint32_t first = __ballot_sync(kWFull, live);
                    if ((Wide && Big) || first == 0u) return first;
                    // each instance of the model by itself: its start time at the latest look at it, its prefill of this
                    // request, its step (unless they are many)
                    bool ok = !Wide && rel == kFar;
                    uint32_t j = live ? me.z : 0u;
                    const uint32_t j_end = live ? me.w : 0u;
                    if (Big) ok = ok || j_end - j > 8u * 16u;
                    while (__any_sync(kWFull, j < j_end && !ok)) {
                        const uint32_t jj = j < j_end ? j : ents;  // (no branch)
                        const uint4 e = w4(jj);
                        const T t = Wide ? wt<T>(rest + ((jj - ents) >> 1)) : (T)(int32_t)e.x;
                        const U since = (U)(max(at, t) - rel) + (U)prefill(e.y, e.z, c_in);
                        ok = ok | ((j < j_end) & lim.met(since, Sm1, e.w));
                        j += 16u;
                    }
                    return __ballot_sync(kWFull, live && ok);
                };
                uint32_t live = test(0u), done = 0u;  // done: lanes below it have been dealt with (side outputs)
                while (live) {
                    const int src = __ffs((int)live) - 1;
                    const uint32_t req = cb + (uint32_t)src;
                    if (side && lane >= done && lane < (uint32_t)src && counted())
                        walk_reject_side(P, tr * P.n_cand + cand, cb + lane, c_meta >> 24);
                    done = (uint32_t)src + 1u;
                    live &= live - 1u;
                    T arrival = wshfl(rel, src);
                    if constexpr (!Wide) {
                        if (max(now, arrival) >= kWalkNowMax) {  // (or the arrival is out of reach)
                            // move the epoch to the dispatcher's clock (or to the request's arrival, if that is later): what
                            // happens before it is simulated, everything else is measured from there on
                            const uint4 v = __ldg(reqs + req);
                            const int64_t to = max(epoch + now, i64_of(v.x, v.y));
                            const T up = to - epoch >= (int64_t)kFar ? kFar : (T)(to - epoch);
                            // (`up` is cut off only if everything is idle by then)
                            for (uint32_t s = 0; s < (Big ? n_i : 1u); s += 32u) {
                                const bool mine = !Big || s + lane < n_i;
                                if (Big) {
                                    if (mine) get(rest, ents, n_i, s + lane, in);
                                    else in.tag = 0;
                                }
                                events(mine && in.w > 0 && is_due(up) && !bad, up);
                                if (kFixed) {
                                    if (mine && in.w > 0) {
                                        for (uint32_t i = 0; i < in.w; i++) wt<T>(in.keys + kKeyBytes * i) -= up;
                                        in.tb -= up;
                                    }
                                } else if (in.w == 0) {
                                    in.t = in.t > up ? in.t - up : 0;  // an idle instance is where the dispatcher is
                                } else {
                                    catch_up(in.w < in.B, up);
                                    in.t = in.t > up + kWPast ? in.t - up : kWPast;  // a full instance's clock is not looked at
                                    in.tb -= up;
                                    if (mine) rebase_firsts(up);
                                }
                                if (mine && s + lane < n_i) {
                                    const T t = kFixed && in.w < in.B ? 0 : start();
                                    w1(ents + 16u * (s + lane)) = (uint32_t)t;
                                    if (Big) put(rest, n_i, s + lane, in, false);
                                }
                            }
                            if (Big && lane < P.n_models) {
                                const int64_t lb = wi(lbs + 8u * lane) - up;
                                wi(lbs + 8u * lane) = lb < kWPast ? (int64_t)kWPast : lb;
                            }
                            flush();
                            epoch = to;
                            now = 0;
                            take_chunk(__ldg(reqs + min(cb + lane, n_req - 1u)));
                            __syncwarp();
                            arrival = wshfl(rel, src);
                        }
                    }
                    const uint32_t in_tok = __shfl_sync(kWFull, c_in, src), meta = __shfl_sync(kWFull, c_meta, src);
                    const uint32_t Sm1 = (meta & 0xFFFFu) - 1u, model = meta >> 24;
                    Limits lim;
                    lim.load(L, (meta >> 12) & 0xFF0u);
                    now = max(now, arrival);  // pending time: the dispatcher never goes back
                    uint32_t tries = 0;
                    bool again = false, look = false;
                    uint32_t j_lo = 0, j_hi = 32u;  // strides of instances to look at (Big: those of the model)
                    if (Big) {
                        const uint2 r = w2(models + 16u * model + 8u);
                        j_lo = ((r.x - ents) >> 4) & ~31u;
                        j_hi = (r.y - ents) >> 4;
                    }
                    do {
                        tries++;
                        U key = kNone;
                        T t0 = 0, pre = 0, lb = kFar;
                        bool elig = false;
                        uint32_t at = lane;  // the instance behind `key`
                        for (uint32_t s = j_lo; s < j_hi; s += 32u) {
                            if (Big) {
                                get(rest, ents, n_i, min(s + lane, n_i - 1u), in);  // (no branch)
                                in.tag = s + lane < n_i ? in.tag : 0u;
                            }
                            elig = (((in.tag >> model) & 1u) != 0u) & !bad;
                            const T p = prefill(in.pre_base, in.pre_q16, in_tok);
                            // "reduce": what completes before the instance's clock reaches `now`
                            events(elig && is_due(now), now);
                            const bool full = in.w == in.B;
                            if (!kFixed) catch_up(elig && !full, now);
                            if (!Big || Opt) peek();
                            // distributor prediction (Sec. IV-F steps 2-3)
                            const T t = start();
                            uint32_t sB = in.stepB;
                            if (Opt && !full) sB = kFixed ? w1(in.row + kEntry * in.w + kEntry) : more.x;
                            const bool ok = elig && lim.met((U)(t + p - arrival), Sm1, sB);
                            // smallest (tier, predicted first token >= now >= 0), lowest instance among equals
                            const U k = !ok ? kNone : (full ? kTier1 : (U)0) | (kLaneKey ? (U)(t + p) << 5 | lane : (U)(t + p));
                            if (Big) {
                                put_if(elig, rest, n_i, s + lane, in);
                                lb = elig ? min(lb, t + (T)in.pre_base) : lb;
                                if (k < key) { key = k; t0 = t; pre = p; at = s + lane; }
                            } else {
                                key = k; t0 = t; pre = p;
                            }
                            if (Big && !Wide) st1_if(elig, smem + ents + 16u * (s + lane), (uint32_t)t);
                        }
                        const U best = warp_min(key);
                        again = false;
                        int wl;  // the winner's lane
                        if constexpr (kLaneKey) wl = (int)((uint32_t)best & 31u);
                        else wl = __ffs((int)__ballot_sync(kWFull, key == best)) - 1;
                        if (Big && best != kNone) {
                            const uint32_t lowest = __reduce_min_sync(kWFull, key == best ? at : 0xFFFFFFFFu);
                            wl = (int)(lowest & 31u);
                            at = (int)lane == wl ? lowest : min(lane, n_i - 1u);  // (no branch)
                            get(rest, ents, n_i, at, in);
                            peek();
                        }
                        const bool win = (int)lane == wl;
                        bool go = true, queued = false;
                        if (best >= kTier1) {
                            if (Big) {  // rejected, or waits: the model's new bound of any first token
                                const U m = warp_min((U)lb);
                                if (lane == 0) wi(lbs + 8u * model) = (int64_t)(T)m;
                            }
                            if (best == kNone) {  // overflow protection: nobody can meet the deadline
                                if (side && lane == 0) walk_reject_side(P, tr * P.n_cand + cand, req, model);
                                go = false;
                                look = true;
                            } else if (Eng == 2) {
                                queued = true;  // every capable instance is full: queues at the chosen one, the dispatcher goes on
                            } else {
                                // every capable instance is full: wait until the chosen slot frees
                                now = wshfl(t0, wl);
                                if (!kAgain) {
                                    // With the worst-case estimate the next round cannot choose differently: at that time the
                                    // winner has a free slot with the same predicted first token, and no other instance's
                                    // prediction can have become earlier or feasible.  The second round is only counted.
                                    events(win, now);
                                    peek();
                                } else {
                                    again = true;
                                    go = false;
                                    if (tries >= kAttemptCap) { status = MAASO_CAND_ELOOP; again = false; }
                                }
                                if (lane == 0 && (!kAgain || again)) atomicAdd(&w1(base + kSExtra), 1u);
                            }
                        }
                        if (go) {
                            admit(win, wl, req, Sm1, pre, queued);
                            if (Big) {
                                if (!Wide) st1_if(win, smem + ents + 16u * at, (uint32_t)start());
                                put_if(win, rest, n_i, at, in);
                            }
                        }
                        if (!Big && elig) wt<T>(Wide ? rest + 8u * lane : ent) = start();
                        if (kFixed && Wide) status = __reduce_or_sync(kWFull, status);
                    } while (kAgain && again);
                    if ((kAgain || (kFixed && Wide)) && status) break;
                    // The other live requests of the chunk stay live, unless this one was rejected: what the scan went by is out
                    // of date then.  (A wait alone makes few others hopeless: 0 to 0.3 of them on average, and finding out
                    // takes as long as a round.)
                    if (look) {
                        __syncwarp();
                        if (live) live = test((uint32_t)src + 1u);
                    }
                }
                if (side && status == 0u && lane >= done && counted()) walk_reject_side(P, tr * P.n_cand + cand, cb + lane, c_meta >> 24);
                if ((!Wide && __any_sync(kWFull, bad)) || status) break;
            }

            // ---- through the trace: drain, account, write the record ------------------------------------------------
            if (!kFixed && status == 0u) {
                for (uint32_t s = 0; s < (Big ? n_i : 1u); s += 32u) {
                    if (Big) {
                        if (s + lane < n_i) get(rest, ents, n_i, s + lane, in);
                        else in.w = 0;
                    }
                    events(in.w > 0 && !bad, kFar);
                }
            }
            flush();
            next();
            if (!Wide && __any_sync(kWFull, bad)) {
                if (lane == 0) walk_hand_over(P, cand, kFixed);
                continue;
            }
            walk_finish(P, base, tr, cand, use_mask, cmask, status, w1(base + kSExtra), parts);
        }
    }
};

}  // namespace maaso
#include "walk_dynamic.cuh"
namespace maaso {

// Warps of a block that replay placements of more than 32 instances side by side: the room that the list's first, its largest, needs
// decides.
__device__ __forceinline__ uint32_t walk_big_warps(const EvalParams& P, uint32_t warps) {
    const uint32_t cand = P.bucket_list[(size_t)kWalkBig0 * P.n_cand];
    return max(1u, min(warps, P.walk_bytes * kWalkWarps / ((256u - (P.code2[cand] & 0xFFu)) * kWalkStepBytes)));
}

// Blocks that replay the placements of more than 32 instances; the others go to the smaller ones, side by side with them (the kernel
// for those is launched second and starts where this one leaves room).  One kernel after the other, a few hundred of the larger ones
// among 30,000 ran three warps on each SM for 29 of 80 ms; side by side 51 ms (73 -> 51 and 82 -> 51 over two draws).
__device__ __forceinline__ uint32_t walk_big_blocks(const EvalParams& P) {
    const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
    const uint64_t big = (uint64_t)P.bucket_count[kWalkBig0] * n_traces;
    if (P.big_grid == 0u || big == 0u) return 0u;
    uint64_t small = 0;
    for (int mode = 0; mode < kWalkModes; mode++) small += P.bucket_count[kWalkBucket0 + mode];
    return walk_big_share(big, small * n_traces, walk_big_warps(P, (uint32_t)kWalkWarps), P.big_grid);
}

// `Warps`: 16, or 12 for small batches under fixed speeds and queues (route.cuh).  Mode k: the block's warps >> k at work, each with
// 2^k times one warp's part of the pool.  The first placements are dealt out in order, over the SMs first, but not to blocks that
// start late; after that whoever is free takes the next.
template <bool Opt, int Eng, bool Wide, bool Big, int Warps, bool Rcp, bool Apart>
__global__ void __launch_bounds__(32 * Warps, 1) eval_walk_kernel(const __grid_constant__ EvalParams P) {
    constexpr bool kLong = Wide && Eng != 2;  // (queues: 64-bit times in the usual buckets)
    constexpr int kFirst = kLong ? kWalkLong0 : (Big ? kWalkBig0 : kWalkBucket0);
    uint32_t any = 0;
    for (int mode = 0; mode < (Big && !kLong ? 1 : kWalkModes); mode++) any |= P.bucket_count[kFirst + mode];
    if (P.stall_test) any = 0;  // test hook: nothing is scored, every valid candidate keeps its "not scored" mark
    uint32_t blocks = gridDim.x, mine = blockIdx.x;  // blocks that the first placements are dealt out to, this one's number
    if constexpr (Big && !kLong) {
        blocks = min(gridDim.x, any * (P.n_traces > 1 ? P.n_traces : 1u));
        if (P.big_grid) blocks = min(blocks, walk_big_blocks(P));
        if (blockIdx.x >= blocks) return;
        let_next_start();
    } else {
        const uint32_t others = !Big && any ? walk_big_blocks(P) : 0u;
        if (others) {  // some blocks start late: numbers go by who starts first
            if (threadIdx.x == 0) w1(0u) = atomicAdd(&P.work_ctr[15], 1u);  // (where the rings will be)
            __syncthreads();
            mine = w1(0u);
            blocks -= min(blocks, others);
        }
        if (any == 0) {
            wait_for_last();
            return;
        }
    }
    constexpr bool kDynamic = Eng == 0 && !Wide && !Big;
    const WalkLayout L = walk_layout(P.n_rows, P.n_classes, Wide, Warps, Rcp, kDynamic);
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    for (uint32_t i = tid; i < P.n_rows * 65u; i += (32 * Warps)) {
        const uint32_t s = walk_step(P, i);
        if constexpr (!Rcp) w1(L.steps + 4u * i) = kDynamic ? s << 5 : s;
        else if constexpr (kDynamic) {
            const ExactEntry e = walk_exact_entry(s);
            w2(L.steps + 8u * i) = make_uint2(e.step, e.m);
        } else w2(L.steps + 8u * i) = make_uint2(s, walk_rcp(s));
    }
    for (uint32_t c = tid; c < P.n_classes; c += (32 * Warps)) {
        const int64_t a = P.classes[3u * c], b = P.classes[3u * c + 1u], e = P.classes[3u * c + 2u];
        const int64_t none = (int64_t)1 << 62, le = e < 0 ? none : e;
        w4(L.lims + 16u * c) = make_uint4(a < 0 ? 0xFFFFFFFFu : (uint32_t)a, b < 0 ? 0xFFFFFFFFu : (uint32_t)b, lo32(le), hi32(le));
        if (Wide) {
            wi(L.wide + 16u * c) = a < 0 ? none : a;
            wi(L.wide + 16u * c + 8u) = b;
        }
    }
    __syncthreads();
    if constexpr (Big && !kLong) {
        // One list, largest first: the room that the block's first placement needs decides how many warps work, and never more than the
        // block's share of the list: the first blocks to start would take what others have the room for (tables of 100 rows, 500 x
        // 4,000 with and without that bound: fixed speeds 3.90 and 4.14 ms, queues 4.31 and 4.51).
        const uint32_t n = P.bucket_count[kWalkBig0];
        const uint32_t cand = P.bucket_list[(size_t)kWalkBig0 * P.n_cand + blockIdx.x / (P.n_traces > 1 ? P.n_traces : 1u)];
        const uint32_t pool = P.walk_bytes * kWalkWarps, room = (256u - (P.code2[cand] & 0xFFu)) * kWalkStepBytes;
        const uint32_t share = (n * (P.n_traces > 1 ? P.n_traces : 1u) + blocks - 1u) / blocks;
        const uint32_t act = max(1u, min(min((uint32_t)Warps, share), pool / room)), part = (pool / act) & ~127u;
        // (how many that is differs from block to block: the first warps start with what is theirs, the rest with whatever is next)
        uint32_t idx = blockIdx.x;
        if (warp > 0 && warp < act) {
            if ((tid & 31u) == 0) idx = blocks + atomicAdd(&P.walk_ctr[kWalkBig0 - kWalkBucket0], 1u);
            idx = __shfl_sync(kWFull, idx, 0);
        }
        if (warp < act)
            Walk<Opt, Eng, Wide, Big, Rcp>::bucket(P, L, kWalkBig0, L.pool + warp * part, idx, blocks,
                                              reinterpret_cast<unsigned char*>(P.payload) + blockIdx.x * walk_big_scratch(pool));
    } else {
        for (int mode = kWalkModes - 1; mode >= 0; mode--) {
            if (P.bucket_count[kFirst + mode] == 0) continue;  // the same for the whole block
            const uint32_t act = (uint32_t)Warps >> mode, part = (kLong ? P.walk_bytes : P.walk_usual) << mode;
            using Body = typename std::conditional<kDynamic, WalkDynamic<Opt, Rcp, Apart>, Walk<Opt, Eng, Wide, Big, Rcp>>::type;
            if (warp < act) {
                uint32_t idx = warp * blocks + mine;
                if (mine >= blocks) {
                    if ((tid & 31u) == 0) idx = act * blocks + atomicAdd(&P.walk_ctr[kFirst + mode - kWalkBucket0], 1u);
                    idx = __shfl_sync(kWFull, idx, 0);
                }
                Body::bucket(P, L, kFirst + mode, L.pool + warp * part, idx, act * blocks, nullptr);
            }
            if (mode) __syncthreads();
        }
        wait_for_last();
    }
}

template <bool Opt, int Eng, bool Wide, bool Big, bool Rcp, int Warps = kWalkWarps, bool Apart = false>
static cudaError_t launch_walk(const EvalParams& P, int grid, bool overlap, cudaStream_t stream) {
    auto kernel = eval_walk_kernel<Opt, Eng, Wide, Big, Warps, Rcp, Apart>;
    const size_t smem = walk_layout(P.n_rows, P.n_classes, Wide, Warps, Rcp, Eng == 0 && !Wide && !Big).pool + (Big || (Wide && Eng != 2) ? P.walk_bytes * kWalkWarps : P.walk_usual * Warps);
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    // `overlap`: its blocks may start before the kernel ahead of it has ended
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t config = {};
    config.gridDim = dim3((unsigned)grid);
    config.blockDim = dim3(32u * Warps);
    config.dynamicSmemBytes = smem;
    config.stream = stream;
    config.attrs = &attr;
    config.numAttrs = overlap ? 1u : 0u;
    return cudaLaunchKernelEx(&config, kernel, P);
}

}  // namespace maaso
