// Scoring kernel for many lightly loaded placements of at most 8 instances: the placements of a warp share its steps.
//
// What bounds it: instruction issue and the chain of steps together.  Where most requests are served, nearly every request
// needs a distributor round in every placement, and a round of the walking kernel leaves all but a few lanes idle.  Here a
// group of 4 or 8 lanes replays one placement, lane = instance, and the groups of a warp take the same request of the same
// trace at the same time: one step of about 400 warp instructions is 4 or 8 rounds.  The request and its limits are the
// same in all lanes, the choice is a butterfly inside the group, completions of all groups are worked off together.  Under
// load the walking kernel is the better one: it skips what is turned away, and a step here waits for every group.
//
// The rest is the walking kernel's: 32-bit times from an epoch (here the same for the warp, moved to a request's
// arrival), keys in shared memory, a ring of completions (one part per group) accounted by the group's lanes.  A running
// request's first token and index (8 bytes per slot) and the sums are in global memory: what is left in shared memory is
// the same for every placement.  A completion copies them into its ring entry in the background (cp.async): waited for, that
// load stopped all groups of the warp and took a quarter of the time (1.7 of 7.2 cycles between two instructions of a warp).
// A slot has two entries in turn, so that a new occupant does not write what is still being copied.
//
// Measured (B200; with the load waited for, 64-bit lane groups, walking kernel in place of this one): 9,000 placements of one
// node x 5,000 requests at 2 a second 6.1 ms (8.0, 13.3, 14.2), 10,864 x 2,500 x 16 arrival rates 29.5 (32.9), with the optimistic
// estimate 31.9 (34.6); at 8 a second half of the 9,000 are loaded and they walk (5.3 ms, and less since).  Groups of 2 lanes for
// placements of one and two instances were slower (12.3 against 9.4 and 142 against 132 ms): 16 placements step through more
// completions one after the other than 8 do.  Dropped: what the next completion has to be accounted with kept in registers, loaded
// when its key becomes the smallest (+30 % and more: the register's next load waits for the last); this kernel in the manner of
// walk_dynamic.cuh (+4 to +33 %: it spills at 128 registers); the next request read by all lanes at once (-2 %, optimistic +4 %).
#include "walk_kernel.cuh"

namespace maaso {

// A lane's running requests, two entries per slot in turn: {first token from the epoch, request}; then sums (64 bytes), hits by
// class bin (32).
constexpr uint32_t kPackPay = 128u * 8u, kPackScratch = kPackPay + 128u;
constexpr uint32_t kPackRelMax = (1u << 25) - 2u;  // largest end index of a key: end index << 7 | entry in turn << 6 | slot

size_t pack_scratch(int grid) { return (size_t)grid * 32u * kPackWarps * kPackScratch; }

// Accounts a group's ring, one entry per lane and pass (lane `li` of `G`; `mine`: the lane's sums).  An entry: first token from the
// epoch, request, finish time from the epoch, instance.
static __device__ __noinline__ void pack_account(const EvalParams& P, bool dumping, uint32_t oc, unsigned char* mine, uint32_t* bins,
                                                 uint32_t ring, int64_t epoch, uint32_t li, uint32_t G, uint32_t cnt, uint32_t lims,
                                                 const uint4* reqs) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (li < cnt) {
        uint4* const sums = reinterpret_cast<uint4*>(mine);
        const uint4 u0 = __ldcg(sums), u1 = __ldcg(sums + 1), u2 = __ldcg(sums + 2), u3 = __ldcg(sums + 3);
        int64_t st = i64_of(u0.x, u0.y), mt = i64_of(u0.z, u0.w), se = i64_of(u1.x, u1.y), me = i64_of(u1.z, u1.w);
        int64_t mk = i64_of(u2.x, u2.y), tk = i64_of(u3.x, u3.y);
        uint64_t sum = (uint64_t)i64_of(u2.z, u2.w);
        uint32_t served = u3.z, hits = u3.w;
        for (uint32_t e = li; e < cnt; e += G) {
            const uint4 ra = w4(ring + e * 16u);
            const uint2 rb = make_uint2(ra.y, ra.w);
            const uint4 rec = __ldg(reqs + rb.x);
            const int64_t fin = epoch + (int32_t)ra.z, first = epoch + (int32_t)ra.x, arrival = i64_of(rec.x, rec.y);
            const uint32_t S = rec.w & 0xFFFFu, cls = (rec.w >> 16) & 0xFFu;
            const uint4 lim = w4(lims + cls * 16u);
            const int64_t ttft = first - arrival, e2e = fin - arrival;
            const bool hit = (e2e <= i64_of(lim.z, lim.w)) & ((lim.x == 0xFFFFFFFFu) | (ttft <= (int64_t)lim.x)) &
                             ((lim.y == 0xFFFFFFFFu) | ((uint64_t)(fin - first) <= (uint64_t)(S - 1u) * lim.y));
            // the request's term as a served one in, its term as a rejected one out
            sum += served_hash(rb.x, fin, first, rb.y) - rejected_hash(rb.x);
            st += ttft;
            mt = max(mt, ttft);
            se += e2e;
            me = max(me, e2e);
            mk = max(mk, fin);
            tk += S;
            served++;
            hits += hit ? 1u : 0u;
            if (hit) atomicAdd(bins + (cls < 7u ? cls : 7u), 1u);
            if (dumping) {
                const Dump d = dump_for(P, oc);
                if (d.finish) d.finish[rb.x] = fin;
                if (d.first) d.first[rb.x] = first;
                if (d.inst) d.inst[rb.x] = (int32_t)rb.y;
                if (d.hist) atomicAdd(d.hist + ttft_bin(ttft), 1u);
            }
        }
        __stcg(sums, make_uint4(lo32(st), hi32(st), lo32(mt), hi32(mt)));
        __stcg(sums + 1, make_uint4(lo32(se), hi32(se), lo32(me), hi32(me)));
        __stcg(sums + 2, make_uint4(lo32(mk), hi32(mk), (uint32_t)sum, (uint32_t)(sum >> 32)));
        __stcg(sums + 3, make_uint4(lo32(tk), hi32(tk), served, hits));
    }
    __syncwarp();
}

// Copies what a running request must remember into its ring entry, in the background.
__device__ __forceinline__ void copy_run(uint32_t entry, const uint2* run) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(entry + smem_addr(walk_smem)), "l"(run) : "memory");
}

// Work items of a batch: of groups of eight lanes, of all.
__device__ __forceinline__ uint32_t pack_items8(const EvalParams& P) { return (P.bucket_count[kPack8] + 3u) / 4u; }
__device__ __forceinline__ uint32_t pack_total(const EvalParams& P) {
    return (pack_items8(P) + (P.bucket_count[kPack4] + 7u) / 8u) * (P.n_traces > 1 ? P.n_traces : 1u);
}

// One warp takes work items, one after the other: 32 / G placements of the bucket whose groups have G lanes, the largest
// placements first.  (One numbering for both buckets: starting on each from the same warps would have some replay an item
// of each in a row where there is one item for each warp.)
// `Straight`: completions and admissions without a branch; every lane computes what it would leave, those concerned take it.  Where the
// longest items decide, that is better (one node's 10,864 x 5,000 with 12 warps 6.28 -> 6.03 ms), over many waves of items the
// instructions count (16 rates x 10,864 x 10,000 121.2 and 122.1 ms, worst-case estimate 112.5 and 113.2).
template <bool Opt, bool Straight>
static __device__ __forceinline__ void pack_items(const EvalParams& P, const WalkLayout& L, uint32_t idx, uint32_t static_total) {
    using W = Walk<Opt, 0, false, false>;
    using Limits = typename W::Limits;
    constexpr int32_t kFar = kWalkFar;
    constexpr uint32_t kTier1 = 1u << 31, kNone = ~0u;
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, below = (1u << lane) - 1u;
    const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
    const uint32_t n8 = pack_items8(P), total = pack_total(P);
    const uint32_t area = L.pool + threadIdx.x * kPackLane, keys = area + 96u, smem = smem_addr(walk_smem);
    unsigned char* const scratch = reinterpret_cast<unsigned char*>(P.payload) + ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * kPackScratch;
    uint2* const pay = reinterpret_cast<uint2*>(scratch);
    const bool use_mask = P.class_mask != nullptr && P.n_classes <= 32;

    while (idx < total) {
        // ---- the next placements ------------------------------------------------------------------------------
        const uint32_t tr = idx % n_traces, item = idx / n_traces;
        const bool eight = item < n8;
        const uint32_t G = eight ? 8u : 4u, g = lane / G, li = lane & (G - 1u), gmask = ((1u << G) - 1u) << (lane - li);
        const uint32_t bucket = eight ? kPack8 : kPack4, count = P.bucket_count[bucket];
        const uint32_t at = (eight ? item : item - n8) * (32u / G) + g;
        const bool valid = at < count;
        const uint32_t cap = 2u * G;  // a group's part of the ring
        const uint32_t ring = L.ring + (warp * kWalkRing + g * cap) * 16u;
        const uint32_t cand = P.bucket_list[(size_t)bucket * P.n_cand + (valid ? at : count - 1u)], oc = tr * P.n_cand + cand;
        const uint4* const reqs = P.trace_reqs[tr];
        const uint32_t n_req = P.trace_n[tr];
        uint4 nxt = make_uint4(0u, 0u, 0u, 0u);
        if (n_req) nxt = __ldg(reqs + min(lane, n_req - 1u));
        WInst<int32_t> in;
        in.t = 0; in.tb = kFar; in.K = 0; in.kmin = kKeyEmpty; in.w = 0; in.B = 1; in.sw = 1; in.rsw = ~0u;
        in.pre_base = in.pre_q16 = 0; in.stepB = 1; in.tag = 0; in.row = L.steps;
        {
            const uint32_t lo = P.offsets[cand], n_i = P.offsets[cand + 1] - lo;
            if (valid && li < n_i) {
                const uint32_t word = P.inst[lo + li], md = word & 0xFu, r = md * P.n_strategies + ((word >> 4) & 0xFFu);
                in.tag = 1u << md;
                in.B = (word >> 12) & 0xFFu;
                in.row = L.steps + r * kWalkRowRcp;
                in.pre_base = (uint32_t)P.rows[r * kRowStride];
                in.pre_q16 = (uint32_t)P.rows[r * kRowStride + 1];
                in.stepB = w1(in.row + 8u * in.B);
            }
        }
        for (uint32_t i = 0; i < 8u + ((in.B + 7u) & ~7u); i++) w1(i < 8u ? area + 4u * i : keys + 4u * (i - 8u)) = kKeyEmpty;
        for (uint32_t i = 0; i < in.B; i++) walk_smem[area + 32u + i] = (unsigned char)i;
#pragma unroll
        for (uint32_t i = 0; i < 6u; i++) __stcg(reinterpret_cast<uint4*>(scratch + kPackPay) + i, make_uint4(0u, 0u, 0u, 0u));
        __threadfence();
        __syncwarp();
        const uint32_t cmask = use_mask ? P.class_mask[cand] : 0xFFFFFFFFu;
        const bool side = valid && (P.rej_by_model != nullptr || (P.dump_row && P.dump_row[cand] >= 0));
        uint32_t ring_n = 0, status = 0, extra = 0;
        int64_t epoch = 0;
        int32_t now = 0, rel = 0;
        uint32_t c_in = 0, c_meta = 0;
        bool bad = false;  // a time of this lane has left the horizon: nothing is asked of it any more (see the walking kernel)

        auto bins = [&]() { return reinterpret_cast<uint32_t*>(scratch - li * kPackScratch + kPackPay + 64u); };
        auto flush = [&]() {
            pack_account(P, P.dump_row || P.ttft_hist, oc, scratch + kPackPay, bins(), ring, epoch, li, G, ring_n, L.lims, reqs);
            ring_n = 0;
        };
        auto take_chunk = [&](const uint4& v) {
            const int64_t d = i64_of(v.x, v.y) - epoch;
            rel = d >= (int64_t)kWalkNowMax ? kFar : (d < (int64_t)kWPast ? kWPast : (int32_t)d);
            c_in = v.z;
            c_meta = v.w;
        };
        auto next_end = [&](uint32_t left, bool busy, uint2 step) {
            const uint32_t sw = step.x;
            in.sw = sw;
            in.rsw = step.y;
            const uint64_t tc = (uint64_t)left * sw + (uint32_t)in.t;
            in.tb = busy ? (int32_t)((uint32_t)tc - sw) : kFar;
            bad = bad | (busy & (tc > (uint64_t)kWalkHorizon));
        };
        // Completions of the lanes in `due` before `upto`, one per lane and iteration.
        auto events = [&](bool due, int32_t upto) {
            uint32_t dm = __ballot_sync(kWFull, due);
            while (dm) {
                const uint32_t adds = (uint32_t)__popc(dm & gmask);
                if (__any_sync(kWFull, ring_n + adds > cap)) flush();
                if constexpr (Straight) {
                    // (the other lanes look at their first slot)
                    const uint32_t run = due ? in.kmin & 127u : 0u, slot = run & 63u, kb = keys + ((slot >> 3) << 5), mb = area + ((slot >> 3) << 2);
                    const uint32_t e = ring + 16u * (ring_n + (uint32_t)__popc(dm & gmask & below));
                    if (due) copy_run(e, pay + run);
                    st1_if(due, smem + keys + (slot << 2), kKeyEmpty);
                    st1_if(due, smem + mb, kKeyEmpty);
                    const uint4 k0 = w4(kb), k1 = w4(kb + 16u), m0 = w4(area), m1 = w4(area + 16u);
                    const uint2 step = w2(in.row + 8u * in.w - 8u);
                    const int32_t nt = in.tb + (int32_t)in.sw;
                    const uint32_t nK = in.kmin >> 7, nw = in.w - 1u;
                    stb_if(due, smem + area + 32u + nw, run ^ 64u);
                    st2_if(due, smem + e + 8u, make_uint2((uint32_t)nt, li));
                    const uint32_t kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                    const uint32_t mv[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                    const uint32_t bmin = min8(kv), nmin = min(bmin, min8(mv)), left = (nmin >> 7) - nK;
                    st1_if(due, smem + mb, bmin);
                    const bool busy = nw > 0u;
                    const uint64_t tc = (uint64_t)left * step.x + (uint32_t)nt;
                    const int32_t ntb = busy ? (int32_t)((uint32_t)tc - step.x) : kFar;
                    in.t = due ? nt : in.t;
                    in.K = due ? nK : in.K;
                    in.w = due ? nw : in.w;
                    in.kmin = due ? nmin : in.kmin;
                    in.tb = due ? ntb : in.tb;
                    in.sw = due ? step.x : in.sw;
                    in.rsw = due ? step.y : in.rsw;
                    bad = bad | (due & busy & (tc > (uint64_t)kWalkHorizon));
                    due = due & busy & ((left == 0u) | (ntb < upto)) & !bad;
                } else if (due) {
                    const uint32_t slot = in.kmin & 63u, run = in.kmin & 127u, kb = keys + ((slot >> 3) << 5);
                    const uint32_t e = ring + 16u * (ring_n + (uint32_t)__popc(dm & gmask & below));
                    copy_run(e, pay + run);
                    w1(keys + (slot << 2)) = kKeyEmpty;
                    w1(area + ((slot >> 3) << 2)) = kKeyEmpty;
                    const uint4 k0 = w4(kb), k1 = w4(kb + 16u), m0 = w4(area), m1 = w4(area + 16u);
                    const uint2 step = w2(in.row + 8u * in.w - 8u);
                    in.t = in.tb + (int32_t)in.sw;
                    in.K = in.kmin >> 7;
                    in.w--;
                    walk_smem[area + 32u + in.w] = (unsigned char)(run ^ 64u);
                    w2(e + 8u) = make_uint2((uint32_t)in.t, li);
                    const uint32_t kv[8] = {k0.x, k0.y, k0.z, k0.w, k1.x, k1.y, k1.z, k1.w};
                    const uint32_t mv[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
                    const uint32_t bmin = min8(kv);
                    w1(area + ((slot >> 3) << 2)) = bmin;
                    in.kmin = min(bmin, min8(mv));
                    const uint32_t left = (in.kmin >> 7) - in.K;
                    const bool busy = in.w > 0;
                    next_end(left, busy, step);
                    due = busy & ((left == 0u) | (in.tb < upto)) & !bad;
                }
                ring_n += adds;
                dm = __ballot_sync(kWFull, due);
            }
        };
        // A clock that lags behind `upto` while nothing completes: the next step boundary; an idle instance starts at once.
        auto catch_up = [&](bool go, int32_t upto) {
            const int32_t dt = go ? max(upto - in.t, 0) : 0;
            const uint32_t k = walk_steps(dt, in.sw, in.rsw);
            in.t += (int32_t)(k * in.sw);
            in.K += k;
        };

        for (uint32_t cb = 0; cb < n_req; cb += 32u) {
            take_chunk(nxt);
            nxt = __ldg(reqs + min(cb + 32u + lane, n_req - 1u));
            const uint32_t n_chunk = min(32u, n_req - cb);
            // what the keys need room for: an end index is at most 2^16 beyond one before it (else one request at a time)
            if (Straight && __any_sync(kWFull, (in.w > 0) & (in.K > kPackRelMax - (40u << 16))) && in.w > 0) {
                in.kmin = walk_rebase(area, keys, (in.B + 7u) >> 3, in.K << 7, in.kmin);
                in.K = 0;
            }
            for (uint32_t i = 0; i < n_chunk; i++) {
                int32_t arrival = __shfl_sync(kWFull, rel, (int)i);
                const uint32_t in_tok = __shfl_sync(kWFull, c_in, (int)i), meta = __shfl_sync(kWFull, c_meta, (int)i);
                if (arrival == kFar) {
                    // move the epoch to this arrival: what happens before it is simulated, the rest is measured from there on
                    const uint4 v = __ldg(reqs + cb + i);
                    const int64_t to = i64_of(v.x, v.y);
                    const int32_t up = to - epoch >= (int64_t)kFar ? kFar : (int32_t)(to - epoch);
                    events(in.w > 0 && in.tb < up && !bad, up);
                    if (in.w == 0) {
                        in.t = in.t > up ? in.t - up : 0;
                    } else {
                        catch_up(in.w < in.B, up);
                        in.t = in.t > up + kWPast ? in.t - up : kWPast;  // a full instance's clock is not looked at
                        in.tb -= up;
                        // running requests' first tokens (further back than 32 bits reach: the lane has left the horizon)
                        for (uint32_t s = 0; s < in.B; s++) {
                            const uint32_t k = w1(keys + 4u * s);
                            if (k == kKeyEmpty) continue;
                            int32_t* const f = reinterpret_cast<int32_t*>(pay + (k & 127u));
                            const int64_t v = (int64_t)*f - up;
                            bad = bad || v < -(int64_t)kFar;
                            *f = (int32_t)v;
                        }
                    }
                    now = max(now - up, 0);
                    flush();
                    epoch = to;
                    take_chunk(__ldg(reqs + min(cb + lane, n_req - 1u)));
                    arrival = 0;
                }
                const uint32_t Sm1 = (meta & 0xFFFFu) - 1u, model = meta >> 24;
                const bool counted = (cmask >> ((meta >> 16) & 31u)) & 1u;
                Limits lim;
                lim.load(L, (meta >> 12) & 0xFF0u);
                now = max(now, arrival);  // pending time: the dispatcher never goes back
                const int32_t pre = W::prefill(in.pre_base, in.pre_q16, in_tok);
                bool act = counted;  // this group still has to place the request
                asm volatile("cp.async.commit_group;" ::: "memory");  // what earlier steps copy (see the admission)
                for (uint32_t tries = 1;; tries++) {
                    const bool elig = act & (((in.tag >> model) & 1u) != 0u) & !bad;
                    events(elig & (in.tb < now), now);
                    const bool full = in.w == in.B;
                    catch_up(elig & !full, now);
                    uint32_t top = walk_smem[area + 32u + in.w];
                    uint2 more = w2(in.row + 8u * in.w + 8u);
                    // distributor prediction (Sec. IV-F steps 2-3)
                    const int32_t t = full ? in.tb + (int32_t)in.sw : in.t;
                    const bool ok = elig & lim.met((uint32_t)(t + pre - arrival), Sm1, Opt && !full ? more.x : in.stepB);
                    // smallest (tier, predicted first token), lowest instance among equals
                    const uint32_t key = ok ? (full ? kTier1 : 0u) | (uint32_t)(t + pre) : kNone;
                    uint32_t best = min(key, __shfl_xor_sync(kWFull, key, 1));
                    best = min(best, __shfl_xor_sync(kWFull, best, 2));
                    if (G > 4u) best = min(best, __shfl_xor_sync(kWFull, best, 4));
                    const uint32_t equal = __ballot_sync(kWFull, key == best) & gmask;
                    const bool chosen = (key == best) & ((equal & below) == 0u);  // (the winner, without a search for its bit)
                    bool win = chosen & (best < kTier1);
                    const bool slow = act & (best >= kTier1);
                    bool again = false;
                    if (__any_sync(kWFull, slow)) {
                        const bool waits = slow && best != kNone;
                        // overflow protection: nobody can meet the deadline
                        if (side && slow && !waits && li == 0u && status == 0u) walk_reject_side(P, oc, cb + i, model);
                        // every capable instance is full: wait until the chosen slot frees
                        const int32_t frees = __shfl_sync(kWFull, t, __ffs((int)equal) - 1);
                        if (waits) now = frees;
                        if (!Opt) {
                            // the second round cannot choose differently (see the walking kernel): it is only counted
                            const bool mine = waits & chosen;
                            events(mine, now);
                            win = win || mine;
                            top = walk_smem[area + 32u + in.w];
                            more = w2(in.row + 8u * in.w + 8u);
                        } else {
                            again = waits;
                            if (waits && tries >= kAttemptCap) { status = MAASO_CAND_ELOOP; again = false; }
                        }
                        if (waits && (!Opt || again)) extra++;
                    }
                    // prefill at the step boundary (running decodes stall), then occupy a free slot
                    if (Sm1 == 0u) {  // done at the end of its prefill, never occupies a slot
                        const uint32_t adds = __ballot_sync(kWFull, win) & gmask ? 1u : 0u;
                        if (__any_sync(kWFull, ring_n + adds > cap)) flush();
                        if (win) {
                            in.t += pre;
                            if (in.w > 0) in.tb += pre;
                            bad = bad || in.t > kWalkHorizon || (in.w > 0 && in.tb > kWalkHorizon);
                            w4(ring + ring_n * 16u) = make_uint4((uint32_t)in.t, cb + i, (uint32_t)in.t, li);
                        }
                        ring_n += adds;
                    } else {
                        // The entry taken now is the slot's last but one: copies of earlier steps have to be through, this step's not.
                        asm volatile("cp.async.wait_group 0;" ::: "memory");
                        if constexpr (Straight) {
                            const uint32_t nK = in.w > 0 ? in.K : 0u, nk = ((nK + Sm1) << 7) | top, nmin = min(in.kmin, nk);  // (no live end index: the counter restarts)
                            const int32_t nt = in.t + pre;
                            const uint64_t tc = (uint64_t)((nmin >> 7) - nK) * more.x + (uint32_t)nt;
                            st1_if(win, smem + keys + 4u * (top & 63u), nk);
                            if (win) pay[top] = make_uint2((uint32_t)nt, cb + i);
                            const uint32_t mb = smem + area + ((top >> 1) & 28u);
                            st1_if(win, mb, min(ld1(mb), nk));
                            in.t = win ? nt : in.t;
                            in.K = win ? nK : in.K;
                            in.kmin = win ? nmin : in.kmin;
                            in.w = win ? in.w + 1u : in.w;
                            in.sw = win ? more.x : in.sw;
                            in.rsw = win ? more.y : in.rsw;
                            in.tb = win ? (int32_t)((uint32_t)tc - more.x) : in.tb;
                            bad = bad | (win & (tc > (uint64_t)kWalkHorizon));
                        } else if (win) {
                            in.t += pre;
                            if (in.w == 0) in.K = 0;  // no live end index: the counter restarts
                            if (in.K + Sm1 > kPackRelMax) {
                                in.kmin = walk_rebase(area, keys, (in.B + 7u) >> 3, in.K << 7, in.kmin);
                                in.K = 0;
                            }
                            const uint32_t nk = ((in.K + Sm1) << 7) | top;
                            w1(keys + 4u * (top & 63u)) = nk;
                            pay[top] = make_uint2((uint32_t)in.t, cb + i);
                            const uint32_t mb = area + ((top >> 1) & 28u);
                            w1(mb) = min(w1(mb), nk);
                            in.kmin = min(in.kmin, nk);
                            in.w++;
                            next_end((in.kmin >> 7) - in.K, true, more);
                        }
                    }
                    if (!Opt) break;
                    act = again;
                    if (!__any_sync(kWFull, again)) break;
                }
            }
            // a group that has left the horizon, or ran out of rounds, is out
            const uint32_t out = __ballot_sync(kWFull, bad || status);
            if (out & gmask) {
                in.tag = 0; in.w = 0; in.tb = kFar; in.kmin = kKeyEmpty; in.t = 0; in.sw = 1; in.rsw = ~0u; now = 0;
            }
        }

        // ---- through the trace: drain, account, write the records -----------------------------------------------------
        events(in.w > 0 && !bad, kFar);
        flush();
        if (lane == 0) idx = static_total + atomicAdd(&P.work_ctr[0], 1u);
        idx = __shfl_sync(kWFull, idx, 0);
        const bool away = (__ballot_sync(kWFull, bad) & gmask) != 0u;
        __threadfence();
        __syncwarp();
        const uint4* const sums = reinterpret_cast<const uint4*>(scratch + kPackPay);
        const uint4 u0 = __ldcg(sums), u1 = __ldcg(sums + 1), u2 = __ldcg(sums + 2), u3 = __ldcg(sums + 3);
        Stats st;
        st.sum_ttft = i64_of(u0.x, u0.y); st.max_ttft = i64_of(u0.z, u0.w);
        st.sum_e2e = i64_of(u1.x, u1.y);  st.max_e2e = i64_of(u1.z, u1.w);
        st.makespan = i64_of(u2.x, u2.y); st.checksum = (uint64_t)i64_of(u2.z, u2.w);
        st.tokens = (uint64_t)i64_of(u3.x, u3.y);
        st.served = u3.z;
        st.hit = u3.w;
        // the request count and the checksum of "everything rejected", from the per-class totals
        uint32_t counted_all = 0;
        for (uint32_t c = li; c < P.n_classes; c += G)
            if (!use_mask || ((cmask >> c) & 1u)) {
                counted_all += (uint32_t)P.trace_class_tot[tr][2u * c];
                st.checksum += P.trace_class_tot[tr][2u * c + 1u];
            }
        for (uint32_t o = 1; o < G; o <<= 1) {
            st.sum_ttft += (int64_t)wshfl_xor((uint64_t)st.sum_ttft, (int)o);
            st.sum_e2e += (int64_t)wshfl_xor((uint64_t)st.sum_e2e, (int)o);
            st.tokens += wshfl_xor(st.tokens, (int)o);
            st.checksum += wshfl_xor(st.checksum, (int)o);
            st.max_ttft = max(st.max_ttft, (int64_t)wshfl_xor((uint64_t)st.max_ttft, (int)o));
            st.max_e2e = max(st.max_e2e, (int64_t)wshfl_xor((uint64_t)st.max_e2e, (int)o));
            st.makespan = max(st.makespan, (int64_t)wshfl_xor((uint64_t)st.makespan, (int)o));
            st.served += __shfl_xor_sync(kWFull, st.served, (int)o);
            st.hit += __shfl_xor_sync(kWFull, st.hit, (int)o);
            counted_all += __shfl_xor_sync(kWFull, counted_all, (int)o);
        }
        if (valid && li == 0u) {
            if (away) {
                walk_hand_over(P, cand, false);
            } else {
                uint32_t h[8];
#pragma unroll
                for (int i = 0; i < 8; i++) h[i] = __ldcg(bins() + i);
                write_result(P.out + oc, status, counted_all, counted_all - st.served, (uint64_t)counted_all + extra, st, h);
            }
        }
        __syncwarp();
    }
}

// Do 12 warps per SM serve so many items better than 14 (of `grid` SMs)?  See launch_eval_pack.
constexpr uint32_t kPackFewWaves = 2u, kPackFewAgain = 16u;
__device__ __forceinline__ bool pack_few(uint32_t items, uint32_t grid) {
    const uint32_t wave = kWalkWarpsFew * grid;
    return items <= wave || (items > kPackFewAgain * grid && items <= kPackFewWaves * wave);
}

// `Warps`: 14 with 128 registers each, or 12 with room for 168.  `one_of_two`: both are launched, and the number of items decides which
// of them replays the batch (launch_eval_pack).
template <bool Opt, int Warps>
__global__ void __launch_bounds__(32 * Warps, 1) eval_pack_kernel(const __grid_constant__ EvalParams P, bool one_of_two) {
    if (P.stall_test) return;  // test hook: nothing is scored, every valid candidate keeps its "not scored" mark
    const uint32_t items = pack_total(P);
    if (items == 0) return;
    if (one_of_two && pack_few(items, gridDim.x) != (Warps == kWalkWarpsFew)) return;
    let_next_start();
    const WalkLayout L = pack_layout(P.n_rows, P.n_classes);
    const uint32_t tid = threadIdx.x, warp = tid >> 5;
    for (uint32_t i = tid; i < P.n_rows * 65u; i += 32u * Warps) {
        const uint32_t s = walk_step(P, i);
        w2(L.steps + 8u * i) = make_uint2(s, walk_rcp(s));
    }
    for (uint32_t c = tid; c < P.n_classes; c += 32u * Warps) {
        const int64_t a = P.classes[3u * c], b = P.classes[3u * c + 1u], e = P.classes[3u * c + 2u], le = e < 0 ? (int64_t)1 << 62 : e;
        w4(L.lims + 16u * c) = make_uint4(a < 0 ? 0xFFFFFFFFu : (uint32_t)a, b < 0 ? 0xFFFFFFFFu : (uint32_t)b, lo32(le), hi32(le));
    }
    __syncthreads();
    pack_items<Opt, Warps == kWalkWarpsFew>(P, L, warp * gridDim.x + blockIdx.x, gridDim.x * Warps);
}

template <int Warps>
static cudaError_t launch_pack(const EvalParams& P, int grid, bool one_of_two, cudaStream_t stream, int* launches) {
    const size_t smem = pack_layout(P.n_rows, P.n_classes).pool + 32u * Warps * kPackLane;
    auto kernel = (P.flags & MAASO_FLAG_PRED_OPTIMISTIC) ? eval_pack_kernel<true, Warps> : eval_pack_kernel<false, Warps>;
    cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, 32 * Warps, smem, stream>>>(P, one_of_two);
    ++*launches;
    return cudaGetLastError();
}
// A batch whose items 12 warps per SM hold at once is bound by its longest items, which take 154 to 158 registers there and spill
// nothing (14 warps: 88 to 100 bytes).  14 and not 16 for the rest: their shared memory fits a partition that leaves 60 KB of L1
// instead of 28 (16 rates, 10,864 x 2,500: 29.5 and 31.7 ms, optimistic estimate 32.0 and 33.5).  With more items 12 take a second
// wave that 14 do not need, or hardly; from 16 items per SM on both take two, which 12 run faster; the third wave again is better shared
// by 14, and beyond it neither is better throughout (0.92 to 1.14 of the time).  One model on one node, 2,500 requests at 1 a second, 12
// and 14 warps: 1,497 items (10,000 placements; 12 warps on each of 148 SMs hold 1,776) 2.94 and 3.25 ms, 1,646 3.00 and 3.23, 1,797
// 3.95 and 3.37, 1,945 4.65 and 3.48, 2,094 4.78 and 4.35, 2,318 4.83 and 5.17, 2,540 4.88 and 5.49, 3,243 5.61 and 5.75, 3,510 5.71 and
// 6.16, 3,731 7.18 and 6.34, 4,026 7.52 and 6.60; the optimistic estimate and two traces within 2 % of these ratios; two models, 12,800 x
// 3,000 (one wave) 3.50 and 3.88, 16,000 (in the second) 5.07 and 4.60, 24,000 6.24 and 6.73.
// An item is four to eight placements, and how many items a batch has is known on the device alone: where the placements leave it
// open, both kernels are launched and one of them returns at once.  (14 first: the shorter batches' tail is what the walking
// kernel, which is launched next, starts beside.)
cudaError_t launch_eval_pack(const EvalParams& P, int grid, cudaStream_t stream, int* launches) {
    const uint64_t placements = (uint64_t)P.n_cand * (P.n_traces > 1 ? P.n_traces : 1u), wave = (uint64_t)kWalkWarpsFew * (uint64_t)grid;
    if (placements > 8 * kPackFewWaves * wave) return launch_pack<kPackWarps>(P, grid, false, stream, launches);
    const bool both = placements > 4 * wave;
    const cudaError_t e = both ? launch_pack<kPackWarps>(P, grid, true, stream, launches) : cudaSuccess;
    return e != cudaSuccess ? e : launch_pack<kWalkWarpsFew>(P, grid, both, stream, launches);
}

}  // namespace maaso
