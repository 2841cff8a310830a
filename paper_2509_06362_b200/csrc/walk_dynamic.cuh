// Walking kernel's body for the engine whose decode speed follows the running count, placements of at most 32 instances,
// 32-bit times: what nearly every call runs.  Same scan and same round as Walk (walk_kernel.cuh), written for the shortest chain.
//
// What bounds it: the chain of rounds of the longest placements, each instruction waited for in turn (5 to 6 cycles for an
// addition, 13 more where a comparison is waited for, 18 for a warp-wide minimum, 30 for shared memory or a shuffle, 36 for
// finding a lowest bit, 20 to 40 for a vote and its branch: clock() around chains of each), and over a large batch the ALU
// pipe, which takes a warp instruction every second cycle.  So
//   - the scan leaves a list of the requests that need a round, with what a round needs of them, in shared memory, and a round
//     reads the next entry ahead: no bit search, no shuffles, no limits to look up;
//   - everything an admission needs is there before the choice: next free slot, its block's minimum, the step with one
//     request more;
//   - the choice's key names the lane: one minimum and one comparison;
//   - the usual path shares no value with the uncommon ones (what merged with them cost 30 instructions a round);
//   - a wait is one operation on the winner's slots: the request takes over the slot that frees;
//   - a step count is a high product and a shift (exact reciprocals), without a correction (large tables, whose rows have none: a
//     division);
//   - chunks that need no round are skipped in a loop of their own, and under load, where the clock is far ahead and only requests
//     with much time can still be served, the trace's list of those is scanned instead (one in five requests: three models,
//     30,000 x 30,000 under load 9.15 -> 5.93 ms, 1,000 x 60,000 2.43 -> 1.64, one node's 10,864 x 10,000 4.62 -> 4.47; lightly
//     loaded 0 to 1 % better);
//   - shared memory is addressed directly (5 % against references into the block's array);
//   - lower bounds for the scan are written when a list is through, not on every round.
// Measured against the body that it replaced here (that of Walk): warp instructions of a round that admits 189 -> 135, with a
// completion before 286 -> 214, with a wait 304 -> 171; 2,000 x 17,000 of the paper's shape 8.9 -> 6.4 ms, one node's 10,864 x
// 10,000 6.4 -> 4.63, three models under load 12,000 x 30,000 4.51 -> 4.25, masked sub-clusters 9,000 x 12,000 18.3 -> 15.9.
// Dropped: completions without a branch (a lone warp 1 % faster, in company up to 4 % slower: thirteen selections); the accounting of
// completions inlined (+7 %); two requests of different models in one round (most rounds of a loaded placement wait, which makes
// the second one's look stale: +2 to 15 %); levels by address and block minima by atomics (as fast).
#pragma once

namespace maaso {

// A load that stays where it is written, ahead of what it is for (the compiler moves a plain one down to its use).
__device__ __forceinline__ uint4 load_ahead(const uint4* p) {
    uint4 v;
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

// Shared memory by its own 32-bit addresses (the layout's offsets with the base of the block's part added).
__device__ __forceinline__ uint4 ld4(uint32_t a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ uint2 ld2(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t ld1(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ uint32_t ldb(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void st4(uint32_t a, const uint4& v) {
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ void st2(uint32_t a, const uint2& v) {
    asm volatile("st.shared.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(v.x), "r"(v.y) : "memory");
}
__device__ __forceinline__ void st1(uint32_t a, uint32_t v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void stb(uint32_t a, uint32_t v) { asm volatile("st.shared.u8 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void min_shared(uint32_t a, uint32_t v) { asm volatile("red.shared.min.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }

// `Rcp`: the decode-step rows carry reciprocals.  `Apart`: patient requests are also looked at by themselves (EvalParams::trace_patient).
template <bool Opt, bool Rcp, bool Apart>
struct WalkDynamic {
    static constexpr uint32_t kEntry = Rcp ? 8u : 4u;
    using Limits = typename Walk<Opt, 0, false, false>::Limits;
    static constexpr int32_t kFar = kWalkFar;
    // A key: tier << 31 | (predicted first token - now, at most kOffMax) << 5 | lane.  From kOffMax on (a minute ahead) the
    // offsets are compared in full.
    static constexpr uint32_t kTier1 = 1u << 31, kNone = ~0u, kOffMax = (1u << 26) - 2u, kFast = kOffMax << 5;
    static constexpr uint32_t kRoom = 32u;         // the ring is accounted when it has as many entries: one iteration adds up to 32

    static __device__ __forceinline__ void bucket(const EvalParams& P, const WalkLayout& L0, int bucket, uint32_t base0,
                                                  uint32_t static_idx, uint32_t static_total, unsigned char*) {
        const uint32_t smem = smem_addr(walk_smem), base = base0 + smem;
        WalkLayout L = L0;
        L.ring += smem; L.lims += smem; L.steps += smem; L.list += smem;
        const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, below = (1u << lane) - 1u;
        const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
        const uint32_t total = P.bucket_count[bucket] * n_traces;
        const uint32_t ring = L.ring + warp * kWalkRing * 16u, list = L.list + warp * kWalkList, dummy = list + 33u * 32u;
        const bool use_mask = P.class_mask != nullptr && P.n_classes <= 32;
        const uint32_t models = base + kWalkSums, ents = models + 16u * P.n_models;

        uint32_t idx = static_idx;
        while (idx < total) {
            // ---- the next placement ------------------------------------------------------------------------
            const uint32_t tr = idx % n_traces;
            const uint32_t cand = P.bucket_list[(size_t)bucket * P.n_cand + idx / n_traces];
            const uint4* const reqs = P.trace_reqs[tr];
            const uint32_t n_req = P.trace_n[tr];
            uint4 nxt = make_uint4(0u, 0u, 0u, 0u);  // the lane's request of the next chunk, as loaded
            if (n_req) nxt = __ldg(reqs + min(lane, n_req - 1u));
            const uint32_t lo = P.offsets[cand], n_i = P.offsets[cand + 1] - lo;
            // this lane's instance (see WInst)
            int32_t t = 0, tc = kFar;  // clock, next completion
            uint32_t K = 0, kmin = kKeyEmpty, w = 0, B = 1, bit = 0, place = 0, area = dummy, pay = dummy, row = L.steps, pre_base = 0, pre_q16 = 0, stepB = 1, low_step = 1;
            uint32_t ent = dummy + 96u;
            {
                for (uint32_t i = lane; i < kWalkSums / 16u; i += 32u) st4(base + 16u * i, make_uint4(0u, 0u, 0u, 0u));
                // instances sorted by model, in their given order within a model (the order in which ties are broken)
                const uint32_t word = lane < n_i ? P.inst[lo + lane] : 0xFu, m = lane < n_i ? word & 0xFu : 0xFFFFFFFFu;
                uint32_t before = 0;
                for (uint32_t k = 0; k < P.n_models; k++) {
                    const uint32_t b = __ballot_sync(kWFull, m == k), n = (uint32_t)__popc(b);
                    if (m == k) st2(ents + 16u * (before + (uint32_t)__popc(b & below)), make_uint2(word, lane));
                    // per model: smallest prefill base, smallest prediction step, its instances (byte offsets of their entries)
                    if (lane == k) st4(models + 16u * k, make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, ents + 16u * before, ents + 16u * (before + n)));
                    before += n;
                }
                __syncwarp();
                uint32_t bytes = 0;
                if (lane < n_i) {
                    ent = ents + 16u * lane;
                    const uint2 e = ld2(ent);
                    const uint32_t md = e.x & 0xFu, r = md * P.n_strategies + ((e.x >> 4) & 0xFFu);
                    bit = 1u << md;  // of its model; 0 from when it has left the horizon on: nothing is asked of it any more (see Walk)
                    place = e.y;
                    B = (e.x >> 12) & 0xFFu;
                    row = L.steps + r * (Rcp ? kWalkRowRcp : kWalkRow);
                    pre_base = (uint32_t)P.rows[r * kRowStride];
                    pre_q16 = (uint32_t)P.rows[r * kRowStride + 1];
                    stepB = ld1(row + kEntry * B) >> 5;
                    // the smallest step a prediction can use: the step at the batch cap, or (optimistic estimate) at any
                    // level up to it
                    low_step = stepB;
                    if (Opt)
                        for (uint32_t l = 1; l < B; l++) low_step = min(low_step, ld1(row + kEntry * l) >> 5);
                    min_shared(models + 16u * md, pre_base);
                    min_shared(models + 16u * md + 4u, low_step);
                    // per instance: earliest start, prefill base and slope, smallest prediction step
                    st4(ent, make_uint4(0u, pre_base, pre_q16, low_step));
                    bytes = walk_slot_bytes(B, false, 4u, kWalkBlock);
                }
                uint32_t incl = bytes;
                for (uint32_t o = 1; o < 32u; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(kWFull, incl, o);
                    if (lane >= o) incl += v;
                }
                if (bytes) {
                    area = ents + 16u * n_i + incl - bytes;
                    pay = area + kWalkKeys + 4u * ((B + 7u) & ~7u);
                    for (uint32_t i = 0; i < 8u; i++) st1(area + 4u * i, kKeyEmpty);
                    for (uint32_t i = area + kWalkKeys; i < pay; i += 4u) st1(i, kKeyEmpty);
                    for (uint32_t i = 0; i < B; i++) stb(area + 32u + i, i);
                }
            }
            uint32_t hasmodel = 0;
            for (uint32_t k = 0; k < P.n_models; k++) {
                const uint2 r = ld2(models + 16u * k + 8u);
                hasmodel |= r.x < r.y ? 1u << k : 0u;
            }
            const uint32_t cmask = use_mask ? P.class_mask[cand] : 0xFFFFFFFFu;
            const bool side = P.rej_by_model != nullptr || (P.dump_row && P.dump_row[cand] >= 0);
            __syncwarp();

            uint32_t step = 32u, rcp = 0x80000000u, sw = 1u;  // entry of the current level (0: an idle clock), its step
            // the next free slot, its block's smallest key, the entry of one request more
            uint32_t top = 0, top_min = 0;
            uint2 more = make_uint2(0u, 0u);
            uint32_t ring_n = 0, status = 0, extra = 0;  // extra: distributor rounds beyond one per request
            int64_t epoch = 0;
            int32_t now = 0;
            int32_t rel = 0;                // this lane's request of the chunk: arrival,
            uint32_t c_in = 0, c_meta = 0;  // input tokens, output tokens | class | model

            auto flush = [&]() {
                walk_account<false>(P, P.dump_row || P.ttft_hist, tr * P.n_cand + cand, base0, ring - smem, 0u, ring_n, epoch, L0.lims, 0u, reqs);
                ring_n = 0;
            };
            auto take_chunk = [&](const uint4& v) {
                const int64_t d = i64_of(v.x, v.y) - epoch;
                rel = d >= (int64_t)kWalkNowMax ? kFar : (d < (int64_t)kWPast ? kWPast : (int32_t)d);
                c_in = v.z;
                c_meta = v.w;
            };
            auto entry = [&](uint32_t at) -> uint2 {
                if constexpr (Rcp) return ld2(at);
                else return make_uint2(ld1(at), 0u);
            };
            auto peek = [&]() {
                more = entry(row + kEntry * w + kEntry);
                top = ldb(area + 32u + w);  // (a full instance's is not looked at)
                top_min = ld1(area + ((top >> 1) & 28u));
            };
            peek();
            // The next completion, counted from the clock; false: it leaves the horizon.
            auto next_end = [&](bool busy) -> bool {
                const uint64_t ahead = (uint64_t)((kmin >> 6) - K) * sw;
                const uint32_t end = (uint32_t)ahead + (uint32_t)t;
                tc = busy ? (int32_t)end : kFar;
                const bool in = !busy | (((uint32_t)(ahead >> 32) == 0u) & (max((uint32_t)ahead, end) <= (uint32_t)kWalkHorizon));
                if (!in) bit = 0;
                return in;
            };
            // One completion in each of the lanes in `due` (their set: `dm`); then whether another one is due.  `stay`: at the time
            // `now`, while the clock is already beyond it (see the wait).
            auto retire = [&](bool due, uint32_t dm, int32_t upto, bool stay) -> bool {
                if (due) {
                    const uint32_t s = kmin & 63u, keys = area + kWalkKeys, kb = keys + 4u * (s & 56u), mb = area + ((s >> 1) & 28u);
                    // (the key and its block's minimum go first: what is left is read without them)
                    st1(keys + 4u * s, kKeyEmpty);
                    st1(mb, kKeyEmpty);
                    const uint4 k0 = ld4(kb), k1 = ld4(kb + 16u), m0 = ld4(area), m1 = ld4(area + 16u);
                    const uint2 cur = entry(row + kEntry * w - kEntry), run = ld2(pay + 8u * s);
                    const uint32_t kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                    const uint32_t mv[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                    if (!stay) {
                        t = tc;
                        K = kmin >> 6;
                    }
                    w--;
                    stb(area + 32u + w, s);
                    st4(ring + 16u * (ring_n + (uint32_t)__popc(dm & below)), make_uint4((uint32_t)(stay ? now : tc), run.x, run.y, place));
                    top = s;
                    more = make_uint2(step, rcp);
                    step = cur.x;
                    rcp = cur.y;
                    sw = step >> 5;
                    top_min = min8(kv);
                    st1(mb, top_min);
                    kmin = min(top_min, min8(mv));
                    const bool busy = w > 0u, in = next_end(busy);
                    due = busy & in & (((kmin >> 6) == K) | (!stay & (tc < upto + (int32_t)sw)));
                }
                return due;
            };
            // Completions of the lanes in `due` until every clock has reached `upto`.  (`w` of a lane that is due is not 0.)
            auto events = [&](bool due, int32_t upto) {
                uint32_t dm = __ballot_sync(kWFull, due);
                while (dm) {
                    if (ring_n >= kRoom) flush();
                    due = retire(due, dm, upto, false);
                    ring_n += (uint32_t)__popc(dm);
                    dm = __ballot_sync(kWFull, due);
                }
            };
            // Decode steps until `dt` later; 2 (dt + step - 1) < 2^32.
            auto steps_of = [&](int32_t dt) -> uint32_t {
                if constexpr (Rcp) return walk_exact_steps(dt, sw, step, rcp);
                else return ((uint32_t)dt + sw - 1u) / sw;
            };
            auto start = [&]() -> int32_t { return w == B ? tc : t; };
            // What is rare, out of the rounds' way.  Moves the epoch for request `src` of the chunk at `cb` of `arr`, to the dispatcher's
            // clock (or to the request's arrival, if that is later): what happens before it is simulated, everything else is
            // measured from there on.
            auto move_epoch = [&](const uint4* arr, uint32_t n_arr, uint32_t cb, uint32_t src, bool patient, int32_t& mark) {
                const uint4 v = __ldg(arr + cb + src);
                const int64_t to = max(epoch + now, i64_of(v.x, v.y));
                const int32_t up = to - epoch >= (int64_t)kFar ? kFar : (int32_t)(to - epoch);  // (cut off only if all is idle by then)
                events(w > 0 && bit && tc - (int32_t)sw < up, min(up, kFar - (int32_t)kWalkStepMax));
                if (w == 0) {
                    t = t > up ? t - up : 0;  // an idle instance is where the dispatcher is
                } else {
                    if (w < B && t < up) {
                        const uint32_t k = steps_of(up - t);
                        t += (int32_t)(k * sw);
                        K += k;
                    }
                    t = t > up + kWPast ? t - up : kWPast;  // a full instance's clock is not looked at
                    tc -= up;
                    // running requests' first tokens (further back than 32 bits reach: the lane has left the horizon)
                    for (uint32_t i = 0; i < B; i++) {
                        if (ld1(area + kWalkKeys + 4u * i) == kKeyEmpty) continue;
                        const int64_t f = (int64_t)(int32_t)ld1(pay + 8u * i) - up;
                        if (f < -(int64_t)kFar) bit = 0;
                        st1(pay + 8u * i, (uint32_t)(int32_t)f);
                    }
                }
                st1(ent, (uint32_t)start());
                flush();
                epoch = to;
                now = 0;
                if (Apart && !patient) mark = 0;
                take_chunk(__ldg(arr + min(cb + lane, n_arr - 1u)));
                __syncwarp();
            };

            // The chunk: 32 requests from `cb` on of the trace or, where the dispatcher's clock is so far ahead that all others are too
            // late (or none of them counts), of its patient ones alone (EvalParams::trace_patient).
            const uint32_t n_pat = Apart ? P.trace_n_patient[tr] : 0u;
            const uint4* const pats = Apart ? P.trace_patient[tr] : nullptr;
            const uint32_t* const pat_idx = reinterpret_cast<const uint32_t*>(pats + n_pat);
            const bool only_pat = Apart && n_pat && use_mask && (cmask & P.impatient) == 0u;
            const uint4* arr = reqs;
            uint32_t cb = 0, n_arr = n_req, first_lane = 0;
            int32_t mark = 0;  // while the list is read: where the trace goes on; else the dispatcher's clock before which it is not turned to again
            bool apart = false;
            auto counted = [&]() { return cb + lane < n_arr && ((cmask >> ((c_meta >> 16) & 31u)) & 1u); };
            auto turn_to = [&](bool patient, uint32_t at) {
                apart = patient;
                arr = patient ? pats : reqs;
                n_arr = patient ? n_pat : n_req;
                cb = at & (patient ? ~0u : ~31u);
                first_lane = patient ? 0u : at & 31u;
                nxt = __ldg(arr + min(cb + lane, n_arr - 1u));
            };
            // Goes on behind the last patient request that has been looked at.  The list's next 32 reach so far that they and what is between
            // them are worth the turn once the clock is the others' patience beyond the last of them; behind its end it never is.  (Turning after
            // every chunk in vain, 30,000 requests, 10,000 placements: all patient ones in the first tenth 8.0 instead of 7.5 ms, one in 1,000 after
            // that 7.9 instead of 7.3.)
            auto leave = [&]() {
                const int32_t reach = cb < n_pat ? __reduce_max_sync(kWFull, rel) : kFar;
                const uint32_t to = max((uint32_t)mark, cb ? __ldg(pat_idx + min(cb, n_pat) - 1u) + 1u : 0u);
                mark = reach >= kWalkNowMax ? kFar : reach + P.patience;
                turn_to(false, to);
            };
            // Which of the chunk's requests from lane `from` on may need the distributor.
            auto test = [&](uint32_t from) -> uint32_t {
                const uint32_t Sm1 = (c_meta & 0xFFFFu) - 1u, model = c_meta >> 24;
                const int32_t at = max(now, rel);
                bool live = (lane >= from) & counted() & ((hasmodel >> model) & 1u);
                // (without a branch: every lane has a request, behind the last one the last one once more)
                const uint4 me = ld4(models + 16u * model);
                Limits lim;
                lim.a = ld4(L.lims + ((c_meta >> 12) & 0xFF0u));
                live = live & lim.met((uint32_t)(at - rel) + me.x, Sm1, me.y);  // earliest first token, since the arrival
                const uint32_t first = __ballot_sync(kWFull, live);
                if (Opt || first == 0u) return first;
                // each instance of the model by itself: its start time at the latest look at it, its prefill of this
                // request, its step; two at a time, as what one waits for is a chain of loads and products (30,000 x 30,000 under load
                // 9.42 -> 9.15 ms, one node's first 148 1 % less)
                bool ok = rel == kFar;
                uint32_t j = live ? me.z : 0u;
                const uint32_t j_end = live ? me.w : 0u;
                do {
                    const bool one = j < j_end, two = j + 16u < j_end;
                    const uint4 e = ld4(one ? j : ents), f = ld4(two ? j + 16u : ents);  // (no branch)
                    const uint32_t since = (uint32_t)(max(at, (int32_t)e.x) - rel) + (uint32_t)Walk<Opt, 0, false, false>::prefill(e.y, e.z, c_in);
                    const uint32_t since2 = (uint32_t)(max(at, (int32_t)f.x) - rel) + (uint32_t)Walk<Opt, 0, false, false>::prefill(f.y, f.z, c_in);
                    ok = ok | (one & lim.met(since, Sm1, e.w)) | (two & lim.met(since2, Sm1, f.w));
                    j += 32u;
                } while (__any_sync(kWFull, j < j_end && !ok));
                return __ballot_sync(kWFull, live && ok);
            };
            auto report = [&](uint32_t served, uint32_t end) {
                if (lane < end && counted() && !((served >> lane) & 1u)) walk_reject_side(P, tr * P.n_cand + cand, cb + lane, c_meta >> 24);
            };

            if (only_pat) turn_to(true, 0u);
            for (;; cb += 32u) {
                uint32_t live = 0;
                for (; cb < n_arr; cb += 32u) {  // (a loop of its own: under load most chunks need no round)
                    take_chunk(nxt);
                    nxt = load_ahead(arr + min(cb + 32u + lane, n_arr - 1u));
                    if (Apart && apart && !only_pat && __any_sync(kWFull, (cb + lane < n_pat) & (rel >= now - P.patience))) break;
                    live = test(Apart ? first_lane : 0u);
                    if (live) break;
                    if (Apart) {
                        if (!apart && n_pat && first_lane == 0u && now >= mark && !__any_sync(kWFull, rel >= now - P.trace_lead[tr])) {
                            mark = (int32_t)(cb + 32u);
                            turn_to(true, __ldg(pat_idx + n_pat + cb / 32u));
                            cb -= 32u;
                        }
                        first_lane = 0;
                    } else if (side) {
                        report(0u, 32u);
                    }
                }
                if (live == 0u) {
                    if (!(Apart && apart) || only_pat) break;
                    leave();
                    cb -= 32u;
                    continue;
                }
                const uint32_t req_of = Apart && apart ? __ldg(pat_idx + min(cb + lane, n_pat - 1u)) : cb + lane;  // the lane's request
                if (Apart) first_lane = 0;
                bool gone = false;  // (its rounds are over)
                uint32_t from = 0, served = 0, end = 32u;  // `end`: where a failed placement stops
                do {
                    // The list of requests that need a round, up to one that is out of the epoch's reach; what the keys need room
                    // for (an end index is at most 2^16 beyond one before it), a placement that left the horizon: one vote for all that is
                    // rare (under load 1.6 % less).
                    const bool mine = ((live >> lane) & 1u) != 0u, beyond = mine & (max(now, rel) >= kWalkNowMax), high = (w > 0) & (K > kRelMax - (40u << 16));
                    uint32_t far = 0;
                    if (__any_sync(kWFull, beyond | high | (bit == 0u && lane < n_i))) {
                        if (__any_sync(kWFull, bit == 0u && lane < n_i)) {
                            gone = true;
                            break;
                        }
                        far = __ballot_sync(kWFull, beyond);
                        if (__any_sync(kWFull, high) && w > 0) {
                            const uint32_t d = K << 6;
                            for (uint32_t at = area; at < pay; at += at == area + 28u ? 68u : 4u) {  // block minima, keys
                                const uint32_t k = ld1(at);
                                if (k != kKeyEmpty) st1(at, k - d);
                            }
                            if (kmin != kKeyEmpty) kmin -= d;
                            peek();
                            K = 0;
                        }
                        if (far) live &= (far & (0u - far)) - 1u;
                    }
                    uint32_t n = (uint32_t)__popc(live);
                    if (((live >> lane) & 1u) != 0u) {
                        // {arrival, input tokens, model bit | lane << 16, keys below this take the usual path; `Apart`: request}
                        // {bound of the first token after the arrival, of the step, of the end + 1, output tokens - 1 | the factor of the step in
                        // the bound of the end << 16 (the same, 0 without a limit)}
                        const uint32_t out = c_meta & 0xFFFFu, at = list + 32u * (uint32_t)__popc(live & below);
                        const uint4 l = ld4(L.lims + ((c_meta >> 12) & 0xFF0u));
                        const bool endless = (l.w >> 30) != 0u;
                        st4(at, make_uint4((uint32_t)rel, c_in, (1u << (c_meta >> 24)) | (lane << 16), Apart ? req_of : (out == 1u ? 0u : kFast)));
                        st4(at + 16u, make_uint4(min(l.x, 0xFFFFFFFEu) + 1u, out == 1u ? 0xFFFFFFFFu : l.y, endless ? 0xFFFFFFFFu : l.z + 1u, (out - 1u) | (endless ? 0u : (out - 1u) << 16)));
                    }
                    __syncwarp();
                    bool move = far != 0u;
                    from = move ? (uint32_t)__ffs((int)far) - 1u : 32u;  // where the next pass over the chunk starts
                    uint32_t i = 0;
                    uint4 q = ld4(list);  // the request of this round
                    uint32_t tries = 0, rejected = 0;
                    while (i < n) {
                        const uint4 lim = ld4(list + 32u * i + 16u), qn = ld4(list + 32u * i + 32u);
                        const int32_t arrival = (int32_t)q.x;
                        // (keys below `usual` take the usual path; one token: none)
                        const uint32_t req = Apart ? q.w : cb + (q.z >> 16), usual = Apart ? (lim.w ? kFast : 0u) : q.w;
                        now = max(now, arrival);  // pending time: the dispatcher never goes back
                        const bool elig = (bit & q.z) != 0u;
                        const int32_t pre = (int32_t)(pre_base + (uint32_t)(((uint64_t)pre_q16 * q.y + 32768u) >> 16));
                        const uint32_t Sm1 = lim.w & 0xFFFFu;
                        // the bound that the class and the prediction's step put on the first token after the arrival
                        auto bound = [&](uint32_t sB) -> uint32_t {
                            const int64_t left = (int64_t)lim.z - (int64_t)((uint64_t)(lim.w >> 16) * sB);
                            return min(lim.x, lo32(left) & ~(uint32_t)((int32_t)hi32(left) >> 31));
                        };
                        uint32_t could = ~0u;
                        // Could any instance serve it if nothing happened since the latest look at them?  With the optimistic estimate waits
                        // follow one another and leave little of a list: asked ahead of each round instead of in the scan (three
                        // models, 12,000 x 30,000: 10.6 -> 8.2 ms; with the worst-case estimate 4.25 -> 4.38, a chain 5 to 8 % longer).
                        if (Opt)
                            could = __ballot_sync(kWFull, elig & (low_step <= lim.y) & ((uint32_t)(max(now, start()) + pre - arrival) < bound(low_step)));
                        // "reduce": what completes before the instance's clock reaches `now`
                        bool due = elig & (tc < now + (int32_t)sw);
                        uint32_t dm = __ballot_sync(kWFull, due);
                        if (Opt && could == 0u) {
                            rejected |= 1u << (q.z >> 16);
                            i++;
                            q = qn;
                            tries = 0;
                            continue;
                        }
                        while (dm) {
                            due = retire(due, dm, now, false);
                            ring_n += (uint32_t)__popc(dm);
                            dm = __ballot_sync(kWFull, due);
                            if (ring_n >= kRoom) flush();
                        }
                        const bool full = w == B;
                        {
                            const uint32_t k = steps_of(elig & !full ? max(now - t, 0) : 0);
                            t += (int32_t)(k * sw);
                            K += k;
                        }
                        // distributor prediction (Sec. IV-F steps 2-3)
                        const uint32_t sB = Opt && !full ? more.x >> 5 : stepB, most = bound(sB);
                        const int32_t t0 = full ? tc : t, first = t0 + pre;
                        const bool ok = elig & (sB <= lim.y) & ((uint32_t)(first - arrival) < most);
                        // smallest (tier, predicted first token >= now), lowest instance among equals
                        const uint32_t key = ok ? (min((uint32_t)(first - now), kOffMax) << 5) + (full ? lane + kTier1 : lane) : kNone;
                        const uint32_t best = __reduce_min_sync(kWFull, key);
                        // "map": prefill at the step boundary (running decodes stall), then occupy a free slot.  Every lane computes what it
                        // would leave and one takes it: without a branch that only one lane takes 3 to 6 % less (computed ahead of the
                        // choice, while it is under way, 1 to 3 % less alone but 3 % more under load, where most rounds wait).
                        auto admit = [&](bool win) {
                            const uint32_t nK = w > 0u ? K : 0u, nk = ((nK + Sm1) << 6) | top, nmin = min(kmin, nk), n_sw = more.x >> 5;
                            const uint64_t ahead = (uint64_t)((nmin >> 6) - nK) * n_sw;
                            const uint32_t n_end = (uint32_t)ahead + (uint32_t)first;
                            const bool n_in = ((uint32_t)(ahead >> 32) == 0u) & (max((uint32_t)ahead, n_end) <= (uint32_t)kWalkHorizon);
                            st1_if(win, area + kWalkKeys + 4u * top, nk);
                            st2_if(win, pay + 8u * top, make_uint2((uint32_t)first, req));
                            st1_if(win, area + ((top >> 1) & 28u), min(top_min, nk));
                            t = win ? first : t;
                            K = win ? nK : K;
                            kmin = win ? nmin : kmin;
                            w = win ? w + 1u : w;
                            step = win ? more.x : step;
                            rcp = win ? more.y : rcp;
                            sw = win ? n_sw : sw;
                            tc = win ? (int32_t)n_end : tc;
                            bit = win & !n_in ? 0u : bit;
                        };
                        if (best < usual) {
                            admit(key == best);
                            peek();
                        } else if (best == kNone) {
                            // overflow protection: nobody can meet the deadline.  What the scan went by is out of date: once more
                            rejected |= 1u << (q.z >> 16);
                            if (!Opt) {
                                from = (q.z >> 16) + 1u;
                                move = false;
                                break;
                            }
                        } else {
                            const bool waits = best >= kTier1;
                            uint32_t wl = best & 31u;  // the winner's lane
                            if (((best >> 5) & 0x3FFFFFFu) == kOffMax) {  // more than a minute ahead: compared in full
                                const uint32_t k = ok & (full == waits) ? (uint32_t)first : kNone, b = __reduce_min_sync(kWFull, k);
                                wl = (uint32_t)__ffs((int)__ballot_sync(kWFull, k == b)) - 1u;
                            }
                            const bool win = lane == wl;
                            if (waits) {
                                // every capable instance is full: wait until the chosen slot frees
                                now = __shfl_sync(kWFull, t0, (int)wl);
                                extra++;
                                if (Opt || usual == 0u) {  // a new choice
                                    if (Opt && ++tries >= kAttemptCap) {
                                        status = MAASO_CAND_ELOOP;
                                        from = end = q.z >> 16;
                                        break;
                                    }
                                    if (now >= kWalkNowMax) {  // (for the same request)
                                        from = q.z >> 16;
                                        move = true;
                                        break;
                                    }
                                    continue;
                                }
                                // With the worst-case estimate the next round cannot choose differently: at that time the winner has
                                // a free slot with the same predicted first token, and no other instance's prediction can have become
                                // earlier or feasible.  So it is only counted, and the request takes the slot over.
                                bool twin;
                                {  // (without a branch, as above, 1 to 2 % less; the other lanes look at their first slot)
                                    const uint32_t s = win ? kmin & 63u : 0u, keys = area + kWalkKeys, kb = keys + 4u * (s & 56u), mb = area + ((s >> 1) & 28u);
                                    st1_if(win, keys + 4u * s, kKeyEmpty);
                                    st1_if(win, mb, kKeyEmpty);
                                    const uint4 k0 = ld4(kb), k1 = ld4(kb + 16u), m0 = ld4(area), m1 = ld4(area + 16u);
                                    const uint2 run = ld2(pay + 8u * s);
                                    const uint32_t kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                                    const uint32_t mv[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                                    const uint32_t bmin = min8(kv), others = min(bmin, min8(mv));
                                    const uint32_t nK = kmin >> 6, nk = ((nK + Sm1) << 6) | s, nmin = min(others, nk);
                                    st4_if(win, ring + 16u * ring_n, make_uint4((uint32_t)t0, run.x, run.y, place));
                                    st1_if(win, keys + 4u * s, nk);
                                    st2_if(win, pay + 8u * s, make_uint2((uint32_t)first, req));
                                    st1_if(win, mb, min(bmin, nk));
                                    const uint64_t ahead = (uint64_t)((nmin >> 6) - nK) * sw;
                                    const uint32_t n_end = (uint32_t)ahead + (uint32_t)first;
                                    const bool n_in = ((uint32_t)(ahead >> 32) == 0u) & (max((uint32_t)ahead, n_end) <= (uint32_t)kWalkHorizon);
                                    K = win ? nK : K;
                                    t = win ? first : t;
                                    kmin = win ? nmin : kmin;
                                    tc = win ? (int32_t)n_end : tc;
                                    bit = win & !n_in ? 0u : bit;
                                    twin = win & ((others >> 6) == nK);
                                }
                                if (++ring_n >= kRoom) flush();
                                uint32_t tm = __ballot_sync(kWFull, twin | (now >= kWalkNowMax));
                                if (tm) {
                                    // others that complete at the very boundary the request waited for
                                    while ((tm = __ballot_sync(kWFull, twin)) != 0u) {
                                        twin = retire(twin, tm, 0, true);
                                        if (++ring_n >= kRoom) flush();
                                    }
                                    peek();
                                    if (now >= kWalkNowMax && i + 1u < n) {
                                        n = i + 1u;
                                        from = qn.z >> 16;
                                        move = true;
                                    }
                                }
                            } else if (usual == 0u) {  // one token: done at the end of its prefill, never occupies a slot
                                if (win) {
                                    t = first;
                                    if (w > 0) tc += pre;
                                    if (t > (int32_t)kWalkHorizon || (w > 0 && (uint32_t)tc > (uint32_t)kWalkHorizon)) bit = 0;
                                    st4(ring + 16u * ring_n, make_uint4((uint32_t)t, (uint32_t)t, req, place));
                                }
                                if (++ring_n >= kRoom) flush();
                            } else {  // (as above)
                                admit(win);
                                peek();
                            }
                        }
                        i++;
                        q = qn;
                        tries = 0;
                    }
                    if (!Opt) st1(ent, (uint32_t)start());  // for the scan
                    // (what is in the list was admitted, up to where the list was left, unless it was rejected)
                    served |= live & (from < 32u ? (1u << from) - 1u : ~0u) & ~rejected;
                    __syncwarp();
                    if (status) break;
                    if (move) move_epoch(arr, n_arr, cb, from, apart, mark);
                    else if (from >= 32u) break;
                    live = test(from);
                } while (live);
                if (!Apart && side) report(served, end);
                if (gone | (status != 0u)) break;
            }

            // ---- through the trace: drain, account, write the record ------------------------------------------------
            if (status == 0u) events(w > 0 && bit, kFar - (int32_t)kWalkStepMax);
            flush();
            if (lane == 0) idx = static_total + atomicAdd(&P.walk_ctr[bucket - kWalkBucket0], 1u);
            idx = __shfl_sync(kWFull, idx, 0);
            if (__any_sync(kWFull, lane < n_i && bit == 0u)) {
                if (lane == 0) walk_hand_over(P, cand, false);
                continue;
            }
            walk_finish(P, base0, tr, cand, use_mask, cmask, status, extra);
        }
    }
};

}  // namespace maaso
