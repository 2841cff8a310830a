// Scoring kernel of the default engine: one warp replays one placement of at most 32 instances.
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
// Measured (B200; lane-group or thread kernel before): 143 placements x 500 requests 0.26 ms (0.44), 10,864 x
// 10,000 8.6 ms (12.2), 2,000 x 17,000 of the paper's shape 15.0 ms (33.8), 100,000 x 100,000 under load 122 ms
// (132), 64 x 20,000 8.6 ms (18.9).  A round with one completion takes 290 warp instructions and, alone on its
// scheduler, 1,360 cycles.
//
// The block's pool of shared memory is split evenly among its warps.  Placements beyond one warp's part run
// first, with half, a quarter, ... of the warps at work and twice, four times, ... the room for each (kWalkModes).
#include "walk.cuh"

namespace maaso {

constexpr uint32_t kWFull = 0xFFFFFFFFu;
// byte offsets in a placement's sums, after the per-lane ones: hits by class bin, extra distributor rounds
constexpr uint32_t kSByClass = kWalkLaneSums, kSExtra = kWalkLaneSums + 32u;
constexpr int32_t kWFar = 0x7FFFFFFF;      // an arrival beyond the epoch's reach; an idle instance's next boundary
constexpr int32_t kWPast = -(1 << 30);     // an arrival at least this far before the epoch: beyond every finite limit

extern __shared__ __align__(128) unsigned char walk_smem[];

__device__ __forceinline__ uint4& w4(uint32_t off) { return *reinterpret_cast<uint4*>(walk_smem + off); }
__device__ __forceinline__ uint2& w2(uint32_t off) { return *reinterpret_cast<uint2*>(walk_smem + off); }
__device__ __forceinline__ uint32_t& w1(uint32_t off) { return *reinterpret_cast<uint32_t*>(walk_smem + off); }
__device__ __forceinline__ int64_t& wi(uint32_t off) { return *reinterpret_cast<int64_t*>(walk_smem + off); }
__device__ __forceinline__ int64_t i64_of(uint32_t lo, uint32_t hi) { return (int64_t)(((uint64_t)hi << 32) | lo); }
__device__ __forceinline__ uint32_t lo32(int64_t v) { return (uint32_t)(uint64_t)v; }
__device__ __forceinline__ uint32_t hi32(int64_t v) { return (uint32_t)((uint64_t)v >> 32); }
__device__ __forceinline__ uint64_t wshfl_xor(uint64_t v, int o) {
    const uint32_t a = __shfl_xor_sync(kWFull, (uint32_t)v, o), b = __shfl_xor_sync(kWFull, (uint32_t)(v >> 32), o);
    return ((uint64_t)b << 32) | a;
}

// Accounts the completion ring, one entry per lane and pass, into the lane's own sums in the region `base`:
//   unit 0: sum and maximum of the time to first token; 1: of the end-to-end time; 2: last completion, checksum;
//   3: output tokens, requests served, hits
static __device__ __noinline__ void walk_account(const EvalParams& P, bool dumping, uint32_t oc, uint32_t base, uint32_t ring,
                                                 uint32_t ring_b, uint32_t cnt, uint32_t lims, const uint4* reqs) {
    const uint32_t lane = threadIdx.x & 31u, sums = base + 16u * lane;
    __syncwarp();
    for (uint32_t e = lane; e < cnt; e += 32u) {
        const uint2 rb = w2(ring_b + e * 8u);
        const uint4 rec = __ldg(reqs + rb.x);
        const uint4 ra = w4(ring + e * 16u);
        uint4 u0 = w4(sums), u1 = w4(sums + 512u), u2 = w4(sums + 1024u), u3 = w4(sums + 1536u);
        const int64_t fin = i64_of(ra.x, ra.y), first = i64_of(ra.z, ra.w), arrival = i64_of(rec.x, rec.y);
        const uint32_t S = rec.w & 0xFFFFu, cls = (rec.w >> 16) & 0xFFu;
        const uint4 lim = w4(lims + cls * 16u);
        const int64_t ttft = first - arrival, e2e = fin - arrival;
        const bool hit = (lim.x == 0xFFFFFFFFu || ttft <= (int64_t)lim.x) && e2e <= i64_of(lim.z, lim.w) &&
                         (lim.y == 0xFFFFFFFFu || (uint64_t)(fin - first) <= (uint64_t)(S - 1u) * lim.y);
        // the request's term as a served one in, its term as a rejected one out
        const uint64_t sum = i64_of(u2.z, u2.w) + served_hash(rb.x, fin, first, rb.y) - rejected_hash(rb.x);
        const int64_t st = i64_of(u0.x, u0.y) + ttft, mt = max(i64_of(u0.z, u0.w), ttft);
        const int64_t se = i64_of(u1.x, u1.y) + e2e, me = max(i64_of(u1.z, u1.w), e2e);
        const int64_t mk = max(i64_of(u2.x, u2.y), fin), tk = i64_of(u3.x, u3.y) + S;
        w4(sums) = make_uint4(lo32(st), hi32(st), lo32(mt), hi32(mt));
        w4(sums + 512u) = make_uint4(lo32(se), hi32(se), lo32(me), hi32(me));
        w4(sums + 1024u) = make_uint4(lo32(mk), hi32(mk), (uint32_t)sum, (uint32_t)(sum >> 32));
        w4(sums + 1536u) = make_uint4(lo32(tk), hi32(tk), u3.z + 1u, u3.w + (hit ? 1u : 0u));
        if (hit) atomicAdd(&w1(base + kSByClass + 4u * (cls < 7u ? cls : 7u)), 1u);
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

// Keys of block b of an instance with nblk blocks.
__device__ __forceinline__ uint32_t walk_block(uint32_t area, uint32_t nblk, uint32_t b) {
    return area + 32u + ((8u * nblk + 15u) & ~15u) + 128u * b;
}

// All live end indices of one instance move down by the counter value K (which restarts at 0).  Rare.
static __device__ __noinline__ uint32_t walk_rebase(uint32_t area, uint32_t nblk, uint32_t K, uint32_t kmin) {
    const uint32_t d = K << 6;
    for (uint32_t b = 0; b <= nblk; b++) {
        const uint32_t p = b ? walk_block(area, nblk, b - 1u) : area;  // the minima, then the keys of each block
        for (uint32_t i = 0; i < 8u; i++) {
            const uint32_t k = w1(p + 4u * i);
            if (k != kKeyEmpty) w1(p + 4u * i) = k - d;
        }
    }
    return kmin != kKeyEmpty ? kmin - d : kmin;
}

// A placement that left the 32-bit horizon goes to the one-warp-per-placement kernel, once, for every trace of
// the pass; that kernel starts after this one and clears the placement's side outputs first.
static __device__ __noinline__ void walk_hand_over(const EvalParams& P, uint32_t cand) {
    if (atomicExch(&P.code[cand], 0xFFFFFFFFu) == 0xFFFFFFFFu) return;
    const uint32_t at = atomicAdd(&P.bucket_count[kWideBucket], 1u);
    P.bucket_list[(size_t)kWideBucket * P.n_cand + at] = cand;
}

// What one lane knows of its instance.
struct WInst {
    int32_t T;     // clock, a decode-step boundary (may lag `now`)
    int32_t tb;    // last boundary before the next completion if nobody is admitted; kWFar while idle
    uint32_t K;    // decode steps done at T since the counter last restarted
    uint32_t kmin; // smallest slot key
    uint32_t w, B;
    uint32_t sw;   // one decode step at the current level (valid while w > 0)
    float rsw;     // 1 / sw
    uint32_t pre_base, pre_q16, stepB;
    uint32_t tag;  // 1 << model (0 for a lane without an instance) | place in the placement as given << 16
    uint32_t area, keys, row;  // byte offsets of its slots, of its first block of keys and of its decode-step row
};

// ceil(dt / s) for 1 <= dt < 2^31 and a quotient below 2^16, rs = 1 / s to a few units in the last place: the
// float estimate is within one of the true quotient and is fixed up exactly.
__device__ __forceinline__ uint32_t walk_steps(uint32_t dt, uint32_t s, float rs) {
    const uint32_t q = (uint32_t)(__uint2float_rz(dt) * rs);
    const int32_t r = (int32_t)(dt - q * s);
    return q + (r > 0 ? 1u : 0u) + (r > (int32_t)s ? 1u : 0u) - (r <= -(int32_t)s ? 1u : 0u);
}


// One warp takes the placements of a bucket, one after the other.  `base`: its part of shared memory.
template <bool OPT>
__device__ __forceinline__ void walk_bucket(const EvalParams& P, const WalkLayout& L, int bucket, uint32_t base,
                                            uint32_t static_idx, uint32_t static_total) {
    constexpr uint32_t kCap = (uint32_t)kWalkRing;
    const uint32_t lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
    const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
    const uint32_t total = P.bucket_count[bucket] * n_traces;
    const uint32_t ring = L.ring + (threadIdx.x >> 5) * kWalkRing * 16u, ring_b = L.ring_b + (threadIdx.x >> 5) * kWalkRing * 8u;
    const bool use_mask = P.class_mask != nullptr && P.n_classes <= 32;
    const uint32_t models = base + kWalkSums, ents = models + 16u * P.n_models, ent = ents + 16u * lane;

    uint32_t idx = static_idx;
    while (idx < total) {
        // ---- the next placement ----------------------------------------------------------------------------
        const uint32_t tr = idx % n_traces;
        const uint32_t cand = P.bucket_list[(size_t)bucket * P.n_cand + idx / n_traces];
        const uint4* const reqs = P.trace_reqs[tr];
        const uint32_t n_req = P.trace_n[tr];
        uint32_t n_i;
        uint4 nxt = make_uint4(0u, 0u, 0u, 0u);  // the lane's request of the next chunk, as loaded
        if (n_req) nxt = __ldg(reqs + min(lane, n_req - 1u));
        WInst in;
        in.T = 0; in.tb = kWFar; in.K = 0; in.kmin = kKeyEmpty; in.w = 0; in.B = 1; in.sw = 1; in.rsw = 1.0f;
        in.pre_base = in.pre_q16 = 0; in.stepB = 1; in.tag = 0; in.area = in.keys = in.row = L.steps;
        {
            const uint32_t lo = P.offsets[cand];
            n_i = P.offsets[cand + 1] - lo;
            for (uint32_t i = lane; i < kWalkSums / 16u; i += 32u) w4(base + 16u * i) = make_uint4(0u, 0u, 0u, 0u);
            // instances sorted by model, in their given order within a model (the order in which ties are broken)
            const uint32_t word = lane < n_i ? P.inst[lo + lane] : 0u, m = lane < n_i ? word & 0xFu : 0xFFFFFFFFu;
            uint32_t before = 0, at = 0;
            for (uint32_t k = 0; k < P.n_models; k++) {
                const uint32_t b = __ballot_sync(kWFull, m == k), n = (uint32_t)__popc(b);
                if (m == k) at = before + (uint32_t)__popc(b & below);
                // per model: smallest prefill base, smallest prediction step, its instances (byte offsets of their entries)
                if (lane == k) w4(models + 16u * k) = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, ents + 16u * before, ents + 16u * (before + n));
                before += n;
            }
            if (lane < n_i) w2(ents + 16u * at) = make_uint2(word, lane);
            __syncwarp();
            uint32_t nblk = 0;
            if (lane < n_i) {
                const uint2 e = w2(ent);
                const uint32_t md = e.x & 0xFu, r = md * P.n_strategies + ((e.x >> 4) & 0xFFu);
                in.tag = (1u << md) | (e.y << 16);
                in.B = (e.x >> 12) & 0xFFu;
                nblk = (in.B + 7u) >> 3;
                in.row = L.steps + r * 256u;
                in.pre_base = (uint32_t)P.rows[r * kRowStride];
                in.pre_q16 = (uint32_t)P.rows[r * kRowStride + 1];
                // the smallest step a prediction can use: the step at the batch cap, or (optimistic estimate) at any
                // level up to it
                in.stepB = w1(in.row + 4u * in.B - 4u);
                uint32_t ms = in.stepB;
                if (OPT)
                    for (uint32_t w = 0; w + 1u < in.B; w++) ms = min(ms, w1(in.row + 4u * w));
                atomicMin(&w1(models + 16u * md), in.pre_base);
                atomicMin(&w1(models + 16u * md + 4u), ms);
                // per instance: earliest start, prefill base and slope, smallest prediction step
                w4(ent) = make_uint4(0u, in.pre_base, in.pre_q16, ms);
            }
            const uint32_t bytes = nblk ? walk_slot_bytes(nblk) : 0u;
            uint32_t incl = bytes;
            for (uint32_t o = 1; o < 32u; o <<= 1) {
                const uint32_t v = __shfl_up_sync(kWFull, incl, o);
                if (lane >= o) incl += v;
            }
            if (nblk) {
                in.area = ents + 16u * n_i + incl - bytes;
                in.keys = walk_block(in.area, nblk, 0u);
                for (uint32_t b = 0; b <= nblk; b++) {
                    const uint32_t p = b ? in.keys + 128u * (b - 1u) : in.area;
                    w4(p) = make_uint4(kKeyEmpty, kKeyEmpty, kKeyEmpty, kKeyEmpty);
                    w4(p + 16u) = make_uint4(kKeyEmpty, kKeyEmpty, kKeyEmpty, kKeyEmpty);
                }
                for (uint32_t i = 0; i < in.B; i++) walk_smem[in.area + 32u + i] = (unsigned char)i;
            }
        }
        const uint32_t hasmodel = __reduce_or_sync(kWFull, in.tag & 0xFFFFu);
        const uint32_t cmask = use_mask ? P.class_mask[cand] : 0xFFFFFFFFu;
        const bool side = P.rej_by_model != nullptr || (P.dump_row && P.dump_row[cand] >= 0);
        __syncwarp();

        uint32_t ring_n = 0, status = 0;
        int64_t epoch = 0;
        int32_t now = 0;
        bool bad = false;              // a time of this lane has left the horizon
        int32_t rel = 0;               // this lane's request of the chunk: arrival,
        uint32_t c_in = 0, c_meta = 0; // input tokens, output tokens | class | model

        auto flush = [&]() {
            walk_account(P, P.dump_row || P.ttft_hist, tr * P.n_cand + cand, base, ring, ring_b, ring_n, L.lims, reqs);
            ring_n = 0;
        };
        auto take_chunk = [&](const uint4& v) {
            const int64_t d = i64_of(v.x, v.y) - epoch;
            rel = d >= (int64_t)kWalkNowMax ? kWFar : (d < (int64_t)kWPast ? kWPast : (int32_t)d);
            c_in = v.z;
            c_meta = v.w;
        };
        // Level, step and next completion after an admission or a retirement at in.T >= 0; flags what leaves the horizon.
        auto next_end = [&](uint32_t left) {
            in.sw = w1(in.row + 4u * in.w - 4u);
            in.rsw = rcp_approx((float)in.sw);
            const uint64_t tc = (uint64_t)left * in.sw + (uint32_t)in.T;
            bad = bad || tc > (uint64_t)kWalkHorizon;
            in.tb = (int32_t)((uint32_t)tc - in.sw);
        };
        // Completions of the lanes in `due`, one per lane and iteration, until every clock has reached `upto`.
        auto events = [&](bool due, int32_t upto) {
            uint32_t dm = __ballot_sync(kWFull, due);
            while (dm) {
                const uint32_t adds = (uint32_t)__popc(dm);
                if (ring_n + adds > kCap) flush();
                if (due) {
                    const uint32_t slot = in.kmin & 63u;
                    const uint32_t kb = in.keys + ((slot >> 3) << 7), k8 = kb + 4u * (slot & 7u);
                    const uint4 k0 = w4(kb), k1 = w4(kb + 16u), m0 = w4(in.area), m1 = w4(in.area + 16u);
                    const uint2 ft = w2(k8 + 64u + 4u * (slot & 7u));
                    const uint32_t rq = w1(k8 + 32u);
                    in.T = in.tb + (int32_t)in.sw;
                    in.K = in.kmin >> 6;
                    in.w--;
                    walk_smem[in.area + 32u + in.w] = (unsigned char)slot;
                    // the smallest of the other keys: keys are unique, so the retired one wraps to all ones
                    const uint32_t km = in.kmin + 1u;
                    const uint32_t kv[8] = {k0.x - km, k0.y - km, k0.z - km, k0.w - km, k1.x - km, k1.y - km, k1.z - km, k1.w - km};
                    const uint32_t mv[8] = {m0.x - km, m0.y - km, m0.z - km, m0.w - km, m1.x - km, m1.y - km, m1.z - km, m1.w - km};
                    const uint32_t bmin = min8(kv);
                    const uint32_t e = ring_n + (uint32_t)__popc(dm & below);
                    const int64_t fin = epoch + in.T;
                    w4(ring + 16u * e) = make_uint4(lo32(fin), hi32(fin), ft.x, ft.y);
                    w2(ring_b + 8u * e) = make_uint2(rq, in.tag >> 16);
                    w1(k8) = kKeyEmpty;
                    w1(in.area + ((slot >> 3) << 2)) = bmin + km;
                    in.kmin = min(bmin, min8(mv)) + km;
                    // (an instance that is now idle reads the word before its row, and its next boundary is far)
                    const uint32_t left = (in.kmin >> 6) - in.K;
                    const bool busy = in.w > 0;
                    in.sw = w1(in.row + 4u * in.w - 4u);
                    in.rsw = rcp_approx((float)in.sw);
                    const uint64_t tc = (uint64_t)left * in.sw + (uint32_t)in.T;
                    in.tb = busy ? (int32_t)((uint32_t)tc - in.sw) : kWFar;
                    bad = bad || (busy && tc > (uint64_t)kWalkHorizon);
                    due = busy && (left == 0u || in.tb < upto) && !bad;
                }
                ring_n += adds;
                dm = __ballot_sync(kWFull, due);
            }
        };

        for (uint32_t cb = 0; cb < n_req; cb += 32u) {
            take_chunk(nxt);
            nxt = __ldg(reqs + min(cb + 32u + lane, n_req - 1u));
            // Which of the chunk's requests from lane `from` on may need the distributor.
            auto test = [&](uint32_t from) -> uint32_t {
                const uint32_t Sm1 = (c_meta & 0xFFFFu) - 1u, cls = (c_meta >> 16) & 0xFFu, model = c_meta >> 24;
                const int32_t at = max(now, rel);
                bool live = lane >= from && cb + lane < n_req && ((cmask >> (cls & 31u)) & 1u) && ((hasmodel >> model) & 1u);
                uint4 me = make_uint4(0u, 0u, 0u, 0u), lim = me;
                if (live) {
                    me = w4(models + 16u * model);
                    lim = w4(L.lims + ((c_meta >> 12) & 0xFF0u));
                    const uint32_t since = (uint32_t)(at - rel) + me.x;  // earliest first token, since the arrival
                    live = since <= lim.x && (Sm1 == 0u || me.y <= lim.y) &&
                           (int64_t)((uint64_t)Sm1 * me.y + since) <= i64_of(lim.z, lim.w);
                }
                uint32_t fit = __ballot_sync(kWFull, live);
                if (fit == 0u) return 0u;
                // each instance of the model by itself: its start time at the latest look at it, its prefill of this
                // request, its step
                bool ok = rel == kWFar;
                uint32_t j = live ? me.z : 0u;
                const uint32_t j_end = live ? me.w : 0u;
                while (__any_sync(kWFull, j < j_end)) {
                    if (j < j_end) {
                        const uint4 e = w4(j);
                        const uint32_t since = (uint32_t)(max(at, (int32_t)e.x) - rel) + e.y +
                                               (uint32_t)(((uint64_t)e.z * c_in + 32768u) >> 16);
                        ok = ok || (since <= lim.x && (Sm1 == 0u || e.w <= lim.y) &&
                                    (int64_t)((uint64_t)Sm1 * e.w + since) <= i64_of(lim.z, lim.w));
                        j = ok ? j_end : j + 16u;
                    }
                }
                return __ballot_sync(kWFull, live && ok);
            };
            uint32_t live = test(0u), done = 0u;  // done: lanes below it have been dealt with (side outputs)
            while (live) {
                const int src = __ffs((int)live) - 1;
                const uint32_t req = cb + (uint32_t)src;
                if (side && lane >= done && lane < (uint32_t)src && ((cmask >> ((c_meta >> 16) & 31u)) & 1u))
                    walk_reject_side(P, tr * P.n_cand + cand, cb + lane, c_meta >> 24);
                done = (uint32_t)src + 1u;
                live &= live - 1u;
                int32_t arrival = __shfl_sync(kWFull, rel, src);
                if (arrival == kWFar || now >= kWalkNowMax) {
                    // move the epoch to the dispatcher's clock (or to the request's arrival, if that is later): what
                    // happens before it is simulated, everything else is measured from there on
                    const uint4 v = __ldg(reqs + req);
                    const int64_t to = max(epoch + now, i64_of(v.x, v.y));
                    const int32_t up = to - epoch >= (int64_t)kWFar ? kWFar : (int32_t)(to - epoch);
                    events(in.tb < up, up);
                    if (in.w == 0) {
                        in.T = in.T > up ? in.T - up : 0;  // an idle instance is where the dispatcher is
                    } else {
                        if (in.w < in.B && in.T < up) {
                            const uint32_t k = walk_steps((uint32_t)(up - in.T), in.sw, in.rsw);
                            in.T += (int32_t)(k * in.sw);
                            in.K += k;
                        }
                        in.T = in.T > up + kWPast ? in.T - up : kWPast;  // the clock of a full instance is not looked at
                        in.tb -= up;
                    }
                    if (lane < n_i) w1(ent) = (uint32_t)(in.w == in.B ? in.tb + (int32_t)in.sw : in.T);
                    epoch = to;
                    now = 0;
                    take_chunk(__ldg(reqs + min(cb + lane, n_req - 1u)));
                    __syncwarp();
                    arrival = __shfl_sync(kWFull, rel, src);
                }
                const uint32_t in_tok = __shfl_sync(kWFull, c_in, src), meta = __shfl_sync(kWFull, c_meta, src);
                const uint32_t Sm1 = (meta & 0xFFFFu) - 1u;
                const bool elig = (in.tag >> (meta >> 24)) & 1u;
                const uint4 lim = w4(L.lims + ((meta >> 12) & 0xFF0u));
                const int32_t pre = (int32_t)(in.pre_base + (uint32_t)(((uint64_t)in.pre_q16 * in_tok + 32768u) >> 16));
                now = max(now, arrival);  // pending time: the dispatcher never goes back
                uint32_t tries = 0;
                bool again = false;
                do {
                    tries++;
                    // "reduce": what completes before the instance's clock reaches `now`
                    events(elig && in.tb < now, now);
                    const bool full = in.w == in.B;
                    if (elig && !full && in.T < now) {
                        if (in.w == 0) {
                            in.T = now;  // an idle instance starts at once
                        } else {
                            const uint32_t k = walk_steps((uint32_t)(now - in.T), in.sw, in.rsw);
                            in.T += (int32_t)(k * in.sw);
                            in.K += k;
                        }
                    }
                    // distributor prediction (Sec. IV-F steps 2-3)
                    const int32_t t0 = full ? in.tb + (int32_t)in.sw : in.T;
                    uint32_t sB = in.stepB;
                    if (OPT && !full) sB = w1(in.row + 4u * in.w);
                    const uint32_t since = (uint32_t)(t0 + pre - arrival);
                    const bool ok = elig && since <= lim.x && (Sm1 == 0u || sB <= lim.y) &&
                                    (int64_t)((uint64_t)Sm1 * sB + since) <= i64_of(lim.z, lim.w);
                    // the choice: smallest (tier, predicted first token >= now >= 0), lowest instance among equals
                    const uint32_t key = ok ? (full ? 0x80000000u : 0u) | (uint32_t)(t0 + pre) : 0xFFFFFFFFu;
                    const uint32_t best = __reduce_min_sync(kWFull, key);
                    again = false;
                    bool win = false;
                    if (best != 0xFFFFFFFFu) {
                        const int winner = __ffs((int)__ballot_sync(kWFull, key == best)) - 1;
                        win = (int)lane == winner;
                        if (best >> 31) {
                            // every capable instance is full: wait until the chosen slot frees
                            now = __shfl_sync(kWFull, t0, winner);
                            if (!OPT) {
                                // With the worst-case estimate the next round cannot choose differently: at that time
                                // the winner has a free slot with the same predicted first token, and no other
                                // instance's prediction can have become earlier or feasible.  The second round is
                                // only counted.
                                tries++;
                                events(win, now);
                            } else {
                                again = true;
                                win = false;
                                if (tries >= kAttemptCap) { status = MAASO_CAND_ELOOP; again = false; }
                            }
                        }
                        if (Sm1 == 0u && !again && status == 0u) {  // done at the end of its prefill, never occupies a slot
                            if (ring_n + 1u > kCap) flush();
                            if (win) {
                                in.T += pre;
                                if (in.w > 0) in.tb += pre;
                                bad = bad || in.T > kWalkHorizon || (in.w > 0 && in.tb > kWalkHorizon);
                                const int64_t fin = epoch + in.T;
                                w4(ring + ring_n * 16u) = make_uint4(lo32(fin), hi32(fin), lo32(fin), hi32(fin));
                                w2(ring_b + ring_n * 8u) = make_uint2(req, in.tag >> 16);
                            }
                            ring_n++;
                            win = false;
                        }
                    } else if (side && lane == 0) {
                        walk_reject_side(P, tr * P.n_cand + cand, req, meta >> 24);  // overflow protection: nobody can meet the deadline
                    }
                    if (win) {
                        // "map": prefill at the step boundary (running decodes stall), then occupy a free slot
                        const uint32_t slot = walk_smem[in.area + 32u + in.w];
                        in.T += pre;
                        if (in.w == 0) in.K = 0;  // no live end index: the counter restarts
                        if (in.K + Sm1 > kRelMax) {
                            in.kmin = walk_rebase(in.area, (in.B + 7u) >> 3, in.K, in.kmin);
                            in.K = 0;
                        }
                        const uint32_t nk = ((in.K + Sm1) << 6) | slot;
                        const uint32_t k8 = in.keys + ((slot >> 3) << 7) + 4u * (slot & 7u);
                        const int64_t first = epoch + in.T;
                        w1(k8) = nk;
                        w1(k8 + 32u) = req;
                        w2(k8 + 64u + 4u * (slot & 7u)) = make_uint2(lo32(first), hi32(first));
                        atomicMin(&w1(in.area + ((slot >> 3) << 2)), nk);
                        in.kmin = min(in.kmin, nk);
                        in.w++;
                        next_end((in.kmin >> 6) - in.K);
                    }
                    if (elig) w1(ent) = (uint32_t)(in.w == in.B ? in.tb + (int32_t)in.sw : in.T);
                    // after a plain admission the other live requests of the chunk stay live; a rejection or a wait has
                    // changed what the scan goes by
                    if ((best >> 31) && !again) {
                        __syncwarp();
                        if (live) live = test((uint32_t)src + 1u);
                    }
                } while (OPT && again);
                if (tries > 1u && lane == 0) w1(base + kSExtra) += tries - 1u;
                if (OPT && status) break;
            }
            if (side && status == 0u && lane >= done && cb + lane < n_req && ((cmask >> ((c_meta >> 16) & 31u)) & 1u))
                walk_reject_side(P, tr * P.n_cand + cand, cb + lane, c_meta >> 24);
            if (__any_sync(kWFull, bad) || (OPT && status)) break;
        }

        // ---- through the trace: drain, account, write the record ------------------------------------------------
        if (status == 0u) events(in.w > 0 && !bad, kWFar);
        flush();
        if (lane == 0) idx = static_total + atomicAdd(&P.walk_ctr[bucket - kWalkBucket0], 1u);
        idx = __shfl_sync(kWFull, idx, 0);
        if (__any_sync(kWFull, bad)) {
            if (lane == 0) walk_hand_over(P, cand);
            continue;
        }
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
        for (uint32_t c = lane; c < P.n_classes; c += 32u)
            if (!use_mask || ((cmask >> c) & 1u)) {
                counted_all += (uint32_t)P.trace_class_tot[tr][2u * c];
                st.checksum += P.trace_class_tot[tr][2u * c + 1u];
            }
        counted_all = __reduce_add_sync(kWFull, counted_all);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            st.sum_ttft += (int64_t)wshfl_xor((uint64_t)st.sum_ttft, o);
            st.sum_e2e += (int64_t)wshfl_xor((uint64_t)st.sum_e2e, o);
            st.tokens += wshfl_xor(st.tokens, o);
            st.checksum += wshfl_xor(st.checksum, o);
            st.max_ttft = max(st.max_ttft, (int64_t)wshfl_xor((uint64_t)st.max_ttft, o));
            st.max_e2e = max(st.max_e2e, (int64_t)wshfl_xor((uint64_t)st.max_e2e, o));
            st.makespan = max(st.makespan, (int64_t)wshfl_xor((uint64_t)st.makespan, o));
        }
        if (lane == 0) {
            uint32_t h[8];
#pragma unroll
            for (int i = 0; i < 8; i++) h[i] = w1(base + kSByClass + 4u * i);
            write_result(P.out + tr * P.n_cand + cand, status, counted_all, counted_all - st.served,
                         (uint64_t)counted_all + w1(base + kSExtra), st, h);
        }
        __syncwarp();
    }
}

template <bool OPT>
__global__ void __launch_bounds__(kWalkThreads, 1) eval_walk_kernel(const __grid_constant__ EvalParams P) {
    if (P.stall_test) return;  // test hook: nothing is scored, every valid candidate keeps its "not scored" mark
    const WalkLayout L = walk_layout(P.n_rows, P.n_classes);
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    for (uint32_t i = tid; i < P.n_rows * 64u; i += kWalkThreads)
        w1(L.steps + 4u * i) = (uint32_t)P.rows[(i >> 6) * kRowStride + 2 + (i & 63u)];
    for (uint32_t c = tid; c < P.n_classes; c += kWalkThreads) {
        const int64_t a = P.classes[3u * c], b = P.classes[3u * c + 1u], e = P.classes[3u * c + 2u];
        const int64_t le = e < 0 ? (int64_t)1 << 62 : e;
        w4(L.lims + 16u * c) = make_uint4(a < 0 ? 0xFFFFFFFFu : (uint32_t)a, b < 0 ? 0xFFFFFFFFu : (uint32_t)b, lo32(le), hi32(le));
    }
    __syncthreads();
    // mode k: the block's warps >> k at work, each with 2^k times one warp's part of the pool.  The first placements
    // are dealt out in order, over the SMs first; after that whoever is free takes the next.
    for (int mode = kWalkModes - 1; mode >= 0; mode--) {
        const int bucket = kWalkBucket0 + mode;
        if (P.bucket_count[bucket] == 0) continue;  // the same for the whole block
        const uint32_t act = (uint32_t)kWalkWarps >> mode;
        if (warp < act)
            walk_bucket<OPT>(P, L, bucket, L.pool + warp * (P.walk_bytes << mode), warp * gridDim.x + blockIdx.x, act * gridDim.x);
        if (mode) __syncthreads();
    }
}

cudaError_t launch_eval_walk(const EvalParams& P, int sm_count, cudaStream_t stream) {
    auto kernel = (P.flags & MAASO_FLAG_PRED_OPTIMISTIC) ? eval_walk_kernel<true> : eval_walk_kernel<false>;
    const size_t smem = walk_layout(P.n_rows, P.n_classes).pool + P.walk_bytes * kWalkWarps;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<sm_count, kWalkThreads, smem, stream>>>(P);
    return cudaGetLastError();
}

}  // namespace maaso
