// Candidate decode + validation (constraints (c) and (d) of Sec. IV-C, table ranges) and
// sorting of valid candidates into launch buckets; helpers for the per-request dump buffers.
#include "walk.cuh"

namespace maaso {

// Where a valid candidate can be scored.  `code` = its bucket among the lane-group / block buckets (0..9, or the
// one-warp bucket) and its cost bin, `code2` = its bucket among the thread-mapping and walking buckets and the bin;
// 0xFFFFFFFF = it has no such place.  A candidate with both is placed by the batch-wide choice plan_kernel makes
// (MAASO_MAP_AUTO).
constexpr uint32_t kNowhere = 0xFFFFFFFFu;
__device__ __forceinline__ int t_row(int b) { return b < kWalkBucket0 ? b - kThreadBucket0 : kThreadBuckets + b - kWalkBucket0; }

struct Place {
    uint32_t status, code, code2;
    bool loaded;  // the trace asks for more than the placement can decode
};

// Validation (constraints (c) and (d) of Sec. IV-C, table ranges) and routing of candidate c; writes the record of an
// invalid one and marks a valid one "not scored" (ETIMEOUT): the scoring kernel overwrites the record when it
// finishes the candidate, so a kernel that gave up leaves no record undefined.
__device__ __forceinline__ Place place_candidate(const EvalParams& P, uint32_t c) {
    const uint32_t lo = P.offsets[c], hi = P.offsets[c + 1];
    uint32_t status = 0, n = 0, sum_b = 0;
    PlacementSize size = {0u, 0u, 0u, 0u};
    uint64_t supply = 0; // decode tokens per second the placement can produce with every slot busy
    if (hi < lo || hi > P.n_inst) {
        status = MAASO_CAND_EBADINST;  // malformed CSR row
    } else {
        n = hi - lo;
        if (n > MAASO_MAX_INSTANCES) {
            status = MAASO_CAND_ETOOMANY;
        } else {
            size.n = n;
            uint64_t devsum = 0;
            for (uint32_t i = 0; i < n; i++) {
                const uint32_t word = P.inst[lo + i];
                const uint32_t m = word & 0xFu, s = (word >> 4) & 0xFFu, b = (word >> 12) & 0xFFu;
                if ((word >> 20) != 0 || m >= P.n_models || s >= P.n_strategies || b < 1 || b > MAASO_WMAX) {
                    status |= MAASO_CAND_EBADINST;
                    continue;
                }
                sum_b += b;
                size.add(P, b);
                supply += b * 1000000u / (uint32_t)P.rows[(m * P.n_strategies + s) * kRowStride + 1 + b];
                devsum += (uint64_t)P.devices[s];
                if (P.devices[s] < P.min_devices[m]) status |= MAASO_CAND_EMEMFIT;
            }
            if (devsum > P.budget) status |= MAASO_CAND_EBUDGET;
        }
    }
    Home home = {-1, -1, 0u};
    if (!status) home = route_home(P, size);
    if (P.dump_row) P.dump_row[c] = -1;
    const uint32_t n_traces = P.n_traces > 1 ? P.n_traces : 1u;
    for (uint32_t t = 0; t < n_traces; t++) {
        const size_t oc = (size_t)t * P.n_cand + c;  // the candidate's record in trace t's block
        if (P.rej_by_model)
            for (int m = 0; m < MAASO_MAX_MODELS; m++) P.rej_by_model[oc * MAASO_MAX_MODELS + m] = 0;
        uint4* o = reinterpret_cast<uint4*>(P.out + oc);
        o[0] = make_uint4(status ? status : MAASO_CAND_ETIMEOUT, 0, 0, 0);
        for (int i = 1; i < 8; i++) o[i] = make_uint4(0, 0, 0, 0);
    }
    // Cost estimate: the total batch cap (how many requests the placement can have in flight;
    // it tracks the number of served requests and so the number of simulation events).
    const uint32_t bin = (kCostBins - 1) - min((uint32_t)(kCostBins - 1), sum_b / 8u);
    Place r;
    r.status = status;
    r.code = home.group >= 0 ? (((uint32_t)home.group << 8) | bin) : kNowhere;
    r.code2 = home.walk >= 0 ? (((uint32_t)home.walk << 8) | (home.walk == kWalkBig0 ? walk_big_bin(home.need) : bin)) : kNowhere;
    r.loaded = (uint64_t)P.demand_tok_s >= 2ull * supply;
    return r;
}

__global__ void prep_kernel(const EvalParams P) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P.n_cand) return;
    const Place r = place_candidate(P, c);
    P.code[c] = r.code;
    P.code2[c] = r.code2;
    const uint32_t bin = (r.code != kNowhere ? r.code : r.code2) & 0xFFu;
    const int bg = (int)(r.code >> 8), bt = (int)(r.code2 >> 8);
    if (r.code != kNowhere && r.code2 != kNowhere) {
        atomicAdd(&P.hist[(bg == kWideBucket ? kHistBothW : kHistBothG + bg) * kCostBins + bin], 1u);
        atomicAdd(&P.hist[(kHistBothT + t_row(bt)) * kCostBins + bin], 1u);
        // loaded beyond what it can decode: most of its requests will be turned away, which the
        // walking and the thread kernel do for next to nothing
        atomicAdd(&P.bucket_count[kCtrBoth], 1u);
        if (r.loaded) atomicAdd(&P.bucket_count[kCtrLoaded], 1u);
    } else if (r.code != kNowhere) {
        atomicAdd(&P.hist[(bg == kWideBucket ? kHistWide : kHistOnlyG + bg) * kCostBins + bin], 1u);
    } else if (r.code2 != kNowhere) {
        atomicAdd(&P.hist[(kHistOnlyT + t_row(bt)) * kCostBins + bin], 1u);
    }
}

// Exclusive prefix sums of 256 counts by one warp (lane l holds counts 8l .. 8l+7); returns the total.
__device__ __forceinline__ uint32_t warp_scan_256(uint32_t (&v)[8]) {
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t sum = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const uint32_t x = v[i];
        v[i] = sum;
        sum += x;
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= (uint32_t)o) incl += x;
    }
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] += incl - sum;
    return __shfl_sync(0xFFFFFFFFu, incl, 31);
}

// One block, one warp per bucket, eight cost bins per lane: (0) the batch-wide choice for the candidates that can go
// either way (MAASO_MAP_AUTO): the walking kernel if the batch is small, or if most of them are loaded beyond their decode
// capacity, else the packed kernel or the lane groups (the thread kernel in the walking kernel's place, and from
// P.thread_min_cand loaded ones on, only where MAASO_THREAD_MIN_CAND allows it: 0 otherwise); (1) if the resident lane-group grid has warps to spare, promote
// the most expensive candidates of the narrower lane-group buckets to a warp of their own (bucket 5) so that their
// event handling is not serialised with other candidates' in the same warp; (2) turn the per-bin histograms into
// write cursors (bins in decreasing cost order).
__global__ void __launch_bounds__(1024) plan_kernel(const EvalParams P) {
    __shared__ uint32_t tot[6], s_cut;
    const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31u;
    const uint32_t n_both = P.bucket_count[kCtrBoth], n_loaded = P.bucket_count[kCtrLoaded];
    const bool use_threads = P.walk_all || (n_loaded >= P.thread_min_cand && 2u * n_loaded >= n_both);
    auto counts = [&](int b, uint32_t (&v)[8]) {  // final counts of bucket b in this lane's bins
        const uint32_t only = b == kWideBucket ? kHistWide : (b < kThreadBucket0 ? kHistOnlyG + b : kHistOnlyT + t_row(b));
        const uint32_t both = b == kWideBucket ? kHistBothW : (b < kThreadBucket0 ? kHistBothG + b : kHistBothT + t_row(b));
        const bool take = (b == kWideBucket || b < kThreadBucket0) ? !use_threads : use_threads;
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = P.hist[only * kCostBins + 8u * lane + i] + (take ? P.hist[both * kCostBins + 8u * lane + i] : 0u);
    };
    if (threadIdx.x == 0) s_cut = 0;
    uint32_t v[8];
    if (P.group_warps) {
        if (warp <= 5) {
            counts((int)warp, v);
            const uint32_t t = warp_scan_256(v);
            if (lane == 0) tot[warp] = t;
        }
        __syncthreads();
        if (warp == 0) {
            // warps the lane-group buckets need; every work item exists once per trace, and a promoted candidate takes a
            // warp in each of them
            uint32_t need = 0, narrow[8] = {0, 0, 0, 0, 0, 0, 0, 0}, add[8];
            for (int b = 0; b <= 5; b++) need += (tot[b] + (32u >> b) - 1) / (32u >> b);
            const uint32_t n_tr = P.n_traces > 1 ? P.n_traces : 1u;
            const uint64_t need_all = (uint64_t)need * n_tr;
            const uint32_t spare = P.group_warps > need_all ? (uint32_t)((P.group_warps - need_all) / n_tr * P.promote_pct / 100) : 0;
            for (int b = 0; b < 5; b++) {
                counts(b, add);
#pragma unroll
                for (int i = 0; i < 8; i++) narrow[i] += add[i];
            }
            uint32_t before[8], n = 0;
#pragma unroll
            for (int i = 0; i < 8; i++) before[i] = narrow[i];
            warp_scan_256(before);
#pragma unroll
            for (int i = 0; i < 8; i++) n += before[i] + narrow[i] <= spare ? 1u : 0u;  // prefix sums are monotone
            n = __reduce_add_sync(0xFFFFFFFFu, n);
            if (lane == 0) s_cut = n;
        }
    }
    __syncthreads();
    const uint32_t cut = s_cut;  // bins below `cut` are promoted
    for (int b = (int)warp; b < kNumBuckets; b += 32) {
        counts(b, v);
        if (b <= 5 && cut) {
            uint32_t add[8];
            for (int x = 0; x < 5; x++) {
                if (b == 5) counts(x, add);
#pragma unroll
                for (int i = 0; i < 8; i++)
                    if (8u * lane + i < cut) v[i] = b == 5 ? v[i] + add[i] : 0u;
            }
        }
        const uint32_t total = warp_scan_256(v);
#pragma unroll
        for (int i = 0; i < 8; i++) P.hist[(kHistCursor + b) * kCostBins + 8u * lane + i] = v[i];
        if (lane == 0) P.bucket_count[b] = total;
    }
    if (threadIdx.x == 0) {
        P.bucket_count[kCtrCut] = cut;
        P.bucket_count[kCtrUseThreads] = use_threads ? 1u : 0u;
    }
}

__global__ void scatter_kernel(const EvalParams P) {
    const uint32_t c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= P.n_cand) return;
    const uint32_t cg = P.code[c], ct = P.code2[c];
    if (cg == kNowhere && ct == kNowhere) return;
    const uint32_t code = (cg != kNowhere && ct != kNowhere) ? (P.bucket_count[kCtrUseThreads] ? ct : cg) : (cg != kNowhere ? cg : ct);
    uint32_t b = code >> 8;
    const uint32_t bin = code & 0xFFu;
    if (b < 5 && bin < P.bucket_count[kCtrCut]) b = 5;
    const uint32_t pos = atomicAdd(&P.hist[(kHistCursor + b) * kCostBins + bin], 1u);
    P.bucket_list[(size_t)b * P.n_cand + pos] = c;
}

// All of the above in one launch, for a batch of at most kPrepOne candidates that the walking kernel takes whatever
// its load: one block, histograms in shared memory, nothing to be cleared beforehand.  Three launches and a clear
// are 20 us of a small call's 300.
__global__ void __launch_bounds__(kPrepOne) prep_one_kernel(const EvalParams P) {
    extern __shared__ uint32_t one_hist[];  // [kNumBuckets][kCostBins]
    const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
    for (uint32_t i = tid; i < (uint32_t)(kNumBuckets * kCostBins); i += kPrepOne) one_hist[i] = 0;
    for (uint32_t i = tid; i < 128u; i += kPrepOne) P.bucket_count[i] = 0;  // bucket counts and work counters
    __syncthreads();
    uint32_t code = kNowhere;
    if (tid < P.n_cand) {
        const Place r = place_candidate(P, tid);
        code = r.code2 != kNowhere ? r.code2 : r.code;
        P.code[tid] = code;
        P.code2[tid] = code;
    }
    if (code != kNowhere) atomicAdd(&one_hist[code], 1u);  // bucket << 8 | bin is its place in the histograms
    __syncthreads();
    for (uint32_t b = warp; b < (uint32_t)kNumBuckets; b += kPrepOne / 32) {
        uint32_t v[8];
#pragma unroll
        for (int i = 0; i < 8; i++) v[i] = one_hist[b * kCostBins + 8u * lane + i];
        const uint32_t total = warp_scan_256(v);
#pragma unroll
        for (int i = 0; i < 8; i++) one_hist[b * kCostBins + 8u * lane + i] = v[i];
        if (lane == 0) P.bucket_count[b] = total;
    }
    __syncthreads();
    if (code != kNowhere) {
        const uint32_t pos = atomicAdd(&one_hist[code], 1u);
        P.bucket_list[(size_t)(code >> 8) * P.n_cand + pos] = tid;
    }
}

__global__ void dump_map_kernel(const EvalParams P, const uint32_t* dump_idx) {
    const uint32_t d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= P.dump_n) return;
    const uint32_t c = dump_idx[d];
    if (c < P.n_cand) P.dump_row[c] = (int32_t)d;
}

__global__ void dump_fill_kernel(int64_t* finish, int64_t* first, int32_t* inst, size_t n) {
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        if (finish) finish[i] = -2;
        if (first) first[i] = -2;
        if (inst) inst[i] = -2;
    }
}

// A class whose requests may get their first token and their end more than `patience` us after their arrival.
__device__ __forceinline__ bool is_patient(const int64_t* classes, uint32_t cls, int64_t patience) {
    const int64_t ttft = classes[cls * 3 + 0], e2e = classes[cls * 3 + 2];
    return (ttft < 0 || ttft > patience) && (e2e < 0 || e2e > patience);
}

// The checksum term of a rejected request depends on the request alone: computed once per trace, with the
// prepared record.
// Prepared trace records for the lane-group kernel (layout: common.cuh), and how many of a tile's requests are patient ones
// (kScanTile threads).
__global__ void cook_trace_kernel(const uint4* reqs, const int64_t* classes, uint4* out, uint64_t* rej_hash, uint32_t n, PatientList list) {
    const uint32_t r = blockIdx.x * blockDim.x + threadIdx.x;
    bool patient = false;
    if (r < n) {
        const Request q = decode_request(reqs[r]);
        const int64_t l_ttft = classes[q.cls * 3 + 0], l_tbt = classes[q.cls * 3 + 1], l_e2e = classes[q.cls * 3 + 2];
        const int64_t dl_ttft = l_ttft < 0 ? INT64_MAX : q.arrival + l_ttft;
        const int64_t dl_e2e = l_e2e < 0 ? INT64_MAX : q.arrival + l_e2e;
        const uint32_t tbt32 = (l_tbt < 0 || l_tbt > 0xFFFFFFFFll) ? 0xFFFFFFFFu : (uint32_t)l_tbt;
        const uint64_t h = rejected_hash(r);
        rej_hash[r] = h;
        auto lo = [](uint64_t v) { return (uint32_t)v; };
        auto hi = [](uint64_t v) { return (uint32_t)(v >> 32); };
        uint4* o = out + (size_t)r * kCookedWords;
        o[0] = make_uint4(lo((uint64_t)q.arrival), hi((uint64_t)q.arrival), lo((uint64_t)dl_ttft), hi((uint64_t)dl_ttft));
        o[1] = make_uint4(lo((uint64_t)dl_e2e), hi((uint64_t)dl_e2e), q.in_tokens, tbt32);
        o[2] = make_uint4(lo(h), hi(h), (q.S - 1u) | (q.cls << 16) | (q.model << 24), 0u);
        patient = is_patient(classes, q.cls, list.patience);
    }
    if (list.counts) {
        const int k = __syncthreads_count(patient);
        if (threadIdx.x == 0) list.counts[blockIdx.x] = (uint32_t)k;
    }
}

// Scan tiles of the thread mapping.  Tile t (kScanTile requests) is a header followed by one
// 16-byte record per request.
//   record: {arrival - the tile's base arrival (all ones: does not fit 32 bits, look at the full record),
//            TTFT limit, end-to-end limit (each clamped to 32 bits; all ones = none, or too large to
//            matter here), model | cls << 8 | (output tokens - 1) << 16}.  Once the dispatcher's clock has
//            passed arrival + limit, no instance can serve the request in time.
//   header units 0..3: eight int64, entry k (classes 7 and up share entry 7) = the largest arrival +
//            min(TTFT, end-to-end limit) over the tile's requests of that class: INT64_MAX if one of
//            them has no limit, INT64_MIN if the tile has none, so "clock beyond the entries of the
//            classes I count" means the whole tile is late;
//   unit 4: base arrival (int64) = arrival of the tile's first request;
//   units 5..20: per class slot a 256-bit map of the tile's requests of that class;
//   units 21..36: the same per model (models 7 and up share slot 7).
// And the tile's part of the list of patient requests: here and not on the host or in a kernel of its own, as loading a trace is bound
// by the host's pass over the requests and by the number of copies and launches (with all three 0.037, 0.069 and 0.387 ms for 500, 10,000
// and 100,000 requests, this way 0.032, 0.061 and 0.343, without a list 0.030, 0.061 and 0.342).
__global__ void scan_trace_kernel(const uint4* reqs, const int64_t* classes, uint4* scan, uint32_t n, PatientList list) {
    const uint32_t tile = blockIdx.x, t = threadIdx.x;  // kScanTile threads
    __shared__ int64_t thr[8];
    if (t < 8) thr[t] = INT64_MIN;
    __syncthreads();
    const uint32_t r = tile * kScanTile + t;
    uint4* const base = scan + (size_t)tile * (kScanTile + kScanHdrUnits);
    const int64_t base_arrival = decode_request(reqs[tile * kScanTile]).arrival;
    uint32_t cslot = 0xFFu, mslot = 0xFFu;
    uint4 raw = make_uint4(0u, 0u, 0u, 0u);
    bool patient = false;
    if (r < n) {
        raw = reqs[r];
        const Request q = decode_request(raw);
        patient = is_patient(classes, q.cls, list.patience);
        const int64_t l_ttft = classes[q.cls * 3 + 0], l_e2e = classes[q.cls * 3 + 2];
        const uint32_t t32 = (l_ttft < 0 || l_ttft >= 0xFFFFFFFFll) ? 0xFFFFFFFFu : (uint32_t)l_ttft;
        const uint32_t e32 = (l_e2e < 0 || l_e2e >= 0xFFFFFFFFll) ? 0xFFFFFFFFu : (uint32_t)l_e2e;
        const int64_t rel = q.arrival - base_arrival;
        const uint32_t rel32 = rel >= 0xFFFFFFFFll ? 0xFFFFFFFFu : (uint32_t)rel;
        base[kScanHdrUnits + t] = make_uint4(rel32, t32, e32, q.model | (q.cls << 8) | ((q.S - 1u) << 16));
        const uint32_t lim32 = min(t32, e32);
        const int64_t v = lim32 == 0xFFFFFFFFu ? INT64_MAX : q.arrival + (int64_t)lim32;
        cslot = q.cls < 7 ? q.cls : 7;
        mslot = q.model < 7 ? q.model : 7;
        atomicMax(reinterpret_cast<long long*>(&thr[cslot]), (long long)v);
    }
    uint32_t* const words = reinterpret_cast<uint32_t*>(base);
    for (uint32_t k = 0; k < 8; k++) {
        const uint32_t cb = __ballot_sync(0xFFFFFFFFu, cslot == k), mb = __ballot_sync(0xFFFFFFFFu, mslot == k);
        if ((t & 31u) == 0) {
            words[(kScanHdrClassBits + 2 * k) * 4 + (t >> 5)] = cb;
            words[(kScanHdrModelBits + 2 * k) * 4 + (t >> 5)] = mb;
        }
    }
    __syncthreads();
    if (t < 4) {
        const uint64_t a = (uint64_t)thr[2 * t], b = (uint64_t)thr[2 * t + 1];
        base[t] = make_uint4((uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32));
    }
    if (t == 4) base[kScanHdrBase] = make_uint4((uint32_t)base_arrival, (uint32_t)((uint64_t)base_arrival >> 32), 0u, 0u);
    if (t >= 5 && t < 8) base[kScanHdrUnits - 3 + (t - 5)] = make_uint4(0u, 0u, 0u, 0u);  // padding units 37..39
    if (list.counts) {
        __shared__ uint32_t before[kScanTile / 32], own[kScanTile / 32];
        uint32_t at = 0;  // patient requests ahead of this one: those of earlier tiles, of earlier warps, of earlier lanes
        for (uint32_t i = t; i < tile; i += kScanTile) at += list.counts[i];
        at = __reduce_add_sync(0xFFFFFFFFu, at);
        const uint32_t set = __ballot_sync(0xFFFFFFFFu, patient), lane = t & 31u;
        if (lane == 0) before[t >> 5] = at, own[t >> 5] = (uint32_t)__popc(set);
        __syncthreads();
        at = 0;
        for (uint32_t v = 0; v < kScanTile / 32; v++) at += before[v] + (v < t >> 5 ? own[v] : 0u);
        if (lane == 0 && r < n) list.ahead[r / 32u] = at;
        if (patient) {
            at += (uint32_t)__popc(set & ((1u << lane) - 1u));
            list.reqs[at] = raw;
            list.idx[at] = r;
        }
    }
}
size_t scan_trace_units(uint32_t n) {
    const size_t tiles = ((size_t)n + kScanTile - 1) / kScanTile;
    return (tiles ? tiles : 1) * (kScanTile + kScanHdrUnits);
}
uint32_t scan_trace_tiles(uint32_t n) { return (uint32_t)(((uint64_t)n + kScanTile - 1) / kScanTile); }
// Everything that is prepared of a trace, on the legacy stream.
cudaError_t launch_cook_trace(const uint4* reqs, const int64_t* classes, uint4* cooked, uint64_t* rej_hash, uint4* scan, const PatientList& list, uint32_t n) {
    if (n == 0) return cudaSuccess;
    cook_trace_kernel<<<scan_trace_tiles(n), kScanTile>>>(reqs, classes, cooked, rej_hash, n, list);
    scan_trace_kernel<<<scan_trace_tiles(n), kScanTile>>>(reqs, classes, scan, n, list);
    return cudaGetLastError();
}

cudaError_t launch_prep(const EvalParams& P, const uint32_t* dump_idx, cudaStream_t stream, int* launches) {
    if (P.dump_n) {
        const size_t n = (size_t)P.dump_n * P.n_req;
        if (n) {
            dump_fill_kernel<<<(unsigned)min((size_t)4096, (n + 255) / 256), 256, 0, stream>>>(
                P.dump_finish, P.dump_first, P.dump_inst, n);
            (*launches)++;
        }
    }
    if (P.n_cand <= (uint32_t)kPrepOne && P.walk_all) {
        prep_one_kernel<<<1, kPrepOne, kNumBuckets * kCostBins * 4, stream>>>(P);
        (*launches)++;
    } else {
        prep_kernel<<<(P.n_cand + 255) / 256, 256, 0, stream>>>(P);
        plan_kernel<<<1, 1024, 0, stream>>>(P);
        scatter_kernel<<<(P.n_cand + 255) / 256, 256, 0, stream>>>(P);
        (*launches) += 3;
    }
    if (P.dump_n) {
        dump_map_kernel<<<(P.dump_n + 255) / 256, 256, 0, stream>>>(P, dump_idx);
        (*launches)++;
    }
    return cudaGetLastError();
}

}  // namespace maaso
