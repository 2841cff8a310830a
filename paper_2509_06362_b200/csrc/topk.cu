// Grid-level top-k over result records.  Every pass reduces chunks of records to their k best; passes repeat
// until one chunk is left, whose k best, in order, are the answer.
//
// What bounds it: one read of the 64 bytes per record that decide (two of the record's four sectors) for a large
// n, and launches and block-wide barriers for a small one.  So a block does not sort its chunk: it maps the
// ranking to one 64-bit word per record that never contradicts the exact order, narrows the chunk down to
// little more than k survivors with histograms of 11 bits of that word at a time (starting at the highest bit
// in which the chunk's words differ, so one or two rounds do), and only the survivors are ranked exactly, each
// by counting who is before it.  A chunk is 8,192 records (16,384 if that makes it the only one): 123 blocks
// for 10^6 records, and their 64 best each are one more chunk.  Measured, k = 64 (sorting every chunk in shared
// memory before): 300 records 19 us with its launch (79), 10,000 23 (194), 10^6 52 (435); k = 1024 of 10^6 569 (682).
#include "common.cuh"

namespace maaso {

constexpr int kChunk = 8192;       // records per block
constexpr int kChunkOne = 16384;   // and if one block can take them all
constexpr int kTopkThreads = 1024;
constexpr int kDigits = 2048;      // 11 bits
constexpr uint32_t kSurvivors = MAASO_MAX_TOPK + MAASO_MAX_TOPK / 4 + 128;

struct Entry {
    uint64_t sum_ttft;
    uint32_t n_hit;
    uint32_t n_served;
    uint32_t idx;    // candidate index; 0xFFFFFFFF = padding
    uint32_t valid;  // 1 = scored candidate
};
static_assert(sizeof(Entry) == 24, "entry layout");

// true if a ranks strictly before b: scored first, more hits, lower mean first-token latency
// (exact: sum_a * n_b < sum_b * n_a in 128 bits; nothing served ranks after something served),
// lower index.
__device__ __forceinline__ bool ranks_before(const Entry& a, const Entry& b) {
    if (a.valid != b.valid) return a.valid > b.valid;
    if (a.valid) {
        if (a.n_hit != b.n_hit) return a.n_hit > b.n_hit;
        const bool sa = a.n_served > 0, sb = b.n_served > 0;
        if (sa != sb) return sa;
        if (sa) {
            const uint64_t l_lo = a.sum_ttft * (uint64_t)b.n_served;
            const uint64_t l_hi = __umul64hi(a.sum_ttft, (uint64_t)b.n_served);
            const uint64_t r_lo = b.sum_ttft * (uint64_t)a.n_served;
            const uint64_t r_hi = __umul64hi(b.sum_ttft, (uint64_t)a.n_served);
            if (l_hi != r_hi) return l_hi < r_hi;
            if (l_lo != r_lo) return l_lo < r_lo;
        }
    }
    return a.idx < b.idx;
}

// Order 1 ranks by a score: the entry carries the bit pattern of the score mapped so that
// unsigned order = descending score (as sum_ttft with n_served = 1, n_hit = 0), NaN = not valid.
__device__ __forceinline__ uint64_t descending_key(double s) {
    const uint64_t b = (uint64_t)__double_as_longlong(s);
    const uint64_t ascending = (b >> 63) ? ~b : (b | (1ull << 63));
    return ~ascending;
}

// The ranking as one word, larger = better, equal words = look closer: a ranks before b => word(a) >= word(b).
// Scores: the mapped bit pattern without its lowest bit, below a bit that says valid.  Records: valid, hits,
// something served, and the whole microseconds of the mean first-token time, 30 bits, clamped (the floor of the
// exact quotient, so a lower mean never gets the smaller word).  1 = not valid, 0 = padding.
__device__ __forceinline__ uint64_t rank_word(const Entry& v, bool by_score) {
    if (!v.valid) return v.idx == 0xFFFFFFFFu ? 0 : 1;
    if (by_score) return (1ull << 63) | (~v.sum_ttft >> 1);
    uint64_t r = (1ull << 63) | ((uint64_t)v.n_hit << 31);
    if (v.n_served) {
        const uint64_t m = (v.sum_ttft >> 32) ? v.sum_ttft / v.n_served : (uint64_t)((uint32_t)v.sum_ttft / v.n_served);
        const uint32_t c = m > 0x3FFFFFFFull ? 0x3FFFFFFFu : (uint32_t)m;
        r |= (1ull << 30) | (0x3FFFFFFFu - c);
    }
    return r;
}

// What tells records of equal words apart, level by level: the rest of the score, or the whole microseconds of a
// clamped mean; 64 bits of the mean's fraction, high half first (two different quotients with 32-bit divisors
// differ by more than 2^-64); the index.  Never 0 (out) nor all ones (in).
__device__ __forceinline__ uint64_t tie_word(const Entry& v, bool by_score, int level) {
    if (level == 3) return 1ull + (uint64_t)(0xFFFFFFFFu - v.idx);
    if (!v.valid || (!by_score && !v.n_served)) return 1ull;
    if (by_score) return 1ull + (level == 0 ? (~v.sum_ttft & 1ull) : 0ull);
    const uint64_t whole = v.sum_ttft / v.n_served;
    if (level == 0) return 1ull + (~whole >> 1);
    const uint64_t r0 = (v.sum_ttft - whole * v.n_served) << 32, q0 = r0 / v.n_served;
    if (level == 1) return 1ull + (((~whole & 1ull) << 32) | (0xFFFFFFFFull - q0));
    return 1ull + (0xFFFFFFFFull - ((r0 - q0 * v.n_served) << 32) / v.n_served);
}

__device__ __forceinline__ Entry load_entry(const maaso_result* src_res, const Entry* src_ent, const double* scores, uint64_t g, uint64_t n) {
    Entry v;
    v.sum_ttft = 0; v.n_hit = 0; v.n_served = 0; v.idx = 0xFFFFFFFFu; v.valid = 0;
    if (g < n) {
        if (src_ent) {
            v = src_ent[g];
        } else if (scores) {
            const double sc = scores[g];
            v.idx = (uint32_t)g;
            v.valid = sc == sc ? 1u : 0u;
            v.n_served = 1;
            v.sum_ttft = descending_key(sc);
        } else {
            const uint4 a = __ldg(reinterpret_cast<const uint4*>(src_res + g));      // status, counted, served, hit
            const uint4 d = __ldg(reinterpret_cast<const uint4*>(src_res + g) + 3);  // .., .., sum_ttft lo, hi
            v.idx = (uint32_t)g;
            v.valid = a.x == 0 ? 1u : 0u;
            v.n_served = a.z;
            v.n_hit = a.w;
            v.sum_ttft = ((uint64_t)d.w << 32) | d.z;
        }
    }
    return v;
}

// src_ent == null: first pass, entries are built from records (or scores) [0, n).  Otherwise entries
// come from src_ent[0, n).  Block b reduces its chunk to its k best and writes them to dst_ent[b*k ..] (padding
// behind them) or, in the final pass, candidate indices / records to out_idx / out_res.
__global__ void __launch_bounds__(kTopkThreads)
topk_pass_kernel(const maaso_result* src_res, const Entry* src_ent, uint64_t n, uint32_t chunk, uint32_t k,
                 Entry* dst_ent, int final_pass, const maaso_result* all_res, uint32_t* out_idx,
                 maaso_result* out_res, const double* scores) {
    extern __shared__ __align__(16) unsigned char topk_smem[];
    Entry* const surv = reinterpret_cast<Entry*>(topk_smem);                                  // [kSurvivors]
    uint64_t* const swd = reinterpret_cast<uint64_t*>(topk_smem + kSurvivors * sizeof(Entry));  // [kSurvivors] their words
    uint32_t* const hist = reinterpret_cast<uint32_t*>(swd + kSurvivors);                     // [kDigits]
    uint64_t* const word = reinterpret_cast<uint64_t*>(hist + kDigits);                       // [chunk]
    __shared__ unsigned long long s_ones, s_zeros;
    __shared__ uint32_t s_part[32], s_bin, s_above, s_in, s_cnt, s_valid;
    __shared__ uint32_t sel[MAASO_MAX_TOPK];
    const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5;
    const uint64_t base = (uint64_t)blockIdx.x * chunk;
    const uint32_t have = n > base ? (uint32_t)min((uint64_t)chunk, n - base) : 0u;
    const bool by_score = scores != nullptr;
    const uint32_t cap = min(kSurvivors, k + k / 4u + 128u);
    for (uint32_t i = tid; i < have; i += kTopkThreads) word[i] = rank_word(load_entry(src_res, src_ent, scores, base + i, n), by_score);
    uint64_t lo = 1;  // the survivors: word >= lo
    for (int level = 0;; level++) {
        // the bits in which the words differ, of the valid records if there are enough of them
        if (tid == 0) { s_ones = 0; s_zeros = 0; s_cnt = 0; s_valid = 0; }
        __syncthreads();
        uint64_t ones = 0, zeros = 0;
        uint32_t n_any = 0, n_valid = 0;
        for (uint32_t i = tid; i < have; i += kTopkThreads) {
            const uint64_t w = word[i];
            if (w) n_any++;
            if (w > 1) { ones |= w; zeros |= ~w; n_valid++; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            ones |= __shfl_xor_sync(0xFFFFFFFFu, ones, o);
            zeros |= __shfl_xor_sync(0xFFFFFFFFu, zeros, o);
        }
        n_any = __reduce_add_sync(0xFFFFFFFFu, n_any);
        n_valid = __reduce_add_sync(0xFFFFFFFFu, n_valid);
        if (lane == 0 && n_any) {
            atomicAdd(&s_cnt, n_any);
            atomicAdd(&s_valid, n_valid);
            atomicOr(&s_ones, (unsigned long long)ones);
            atomicOr(&s_zeros, (unsigned long long)zeros);
        }
        __syncthreads();
        if (s_cnt <= cap) break;  // nothing to narrow
        uint64_t common = s_ones & ~s_zeros, diff = s_ones & s_zeros;
        if (s_valid < k) { common = 0; diff = ~0ull; }
        int shift = diff ? max(0, 53 - __clzll((long long)diff)) : 0;
        uint64_t prefix = shift + 11 >= 64 ? 0ull : common & (~0ull << (shift + 11));
        uint32_t above = 0, m = 0;
        for (;;) {
            for (uint32_t i = tid; i < kDigits; i += kTopkThreads) hist[i] = 0;
            __syncthreads();
            const uint64_t pmask = shift + 11 >= 64 ? 0ull : ~0ull << (shift + 11);
            for (uint32_t i = tid; i < have; i += kTopkThreads) {
                const uint64_t w = word[i];
                if (w && (w & pmask) == prefix) atomicAdd(&hist[(uint32_t)(w >> shift) & (kDigits - 1)], 1u);
            }
            __syncthreads();
            // thread t owns digits 2047 - 2t and 2046 - 2t: counts from the top
            const uint32_t d1 = kDigits - 1 - 2u * tid, c1 = hist[d1], c0 = hist[d1 - 1u];
            uint32_t incl = c1 + c0;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
                if (lane >= (uint32_t)o) incl += v;
            }
            if (lane == 31u) s_part[warp] = incl;
            __syncthreads();
            if (warp == 0) {
                uint32_t p = s_part[lane];
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, p, o);
                    if (lane >= (uint32_t)o) p += v;
                }
                s_part[lane] = p;
            }
            __syncthreads();
            const uint32_t before = above + incl - c1 - c0 + (warp ? s_part[warp - 1u] : 0u);
            if (before < k && before + c1 + c0 >= k) {  // the k-th best is in one of this thread's digits
                const bool first = before + c1 >= k;
                s_bin = first ? d1 : d1 - 1u;
                s_above = first ? before : before + c1;
                s_in = first ? c1 : c0;
            }
            __syncthreads();
            above = s_above;
            m = above + s_in;
            prefix |= (uint64_t)s_bin << shift;
            if (m <= cap || shift == 0) break;
            shift = max(0, shift - 11);
            prefix &= ~0ull << (shift + 11);
        }
        lo = prefix;
        if (m <= cap) break;
        // more equal words at the threshold than there is room for: what is above it is in, what is below is out, and
        // the rest is told apart by the next word (the last of them is different for every record)
        __syncthreads();
        for (uint32_t i = tid; i < have; i += kTopkThreads) {
            const uint64_t w = word[i];
            word[i] = w > lo ? ~0ull : (w == lo ? tie_word(load_entry(src_res, src_ent, scores, base + i, n), by_score, level) : 0ull);
        }
        lo = 1;
        __syncthreads();
    }
    // the survivors
    __syncthreads();
    if (tid == 0) s_cnt = 0;
    __syncthreads();
    for (uint32_t i = tid; i < have; i += kTopkThreads)
        if (word[i] >= lo) {
            const uint32_t at = atomicAdd(&s_cnt, 1u);
            const Entry v = load_entry(src_res, src_ent, scores, base + i, n);
            surv[at] = v;
            swd[at] = rank_word(v, by_score);
        }
    __syncthreads();
    const uint32_t m = s_cnt;
    // exact ranks: how many survivors are before this one (the word decides, equal words are compared in full)
    // 2^lg threads share one survivor, eight at most (of 143 records 11.4 -> 9 us; the best 200 of 200,000 52 -> 45 us).  Shifts, as divisions
    // by a number that the survivors decide cost 1 to 2 us (the best 31 of 200,000 by score 22.6, this way 20.2).
    const uint32_t lg = m <= (uint32_t)kTopkThreads / 8 ? 3u : m <= (uint32_t)kTopkThreads / 4 ? 2u : m <= (uint32_t)kTopkThreads / 2 ? 1u : 0u;
    const uint32_t per = 1u << lg;
    for (uint32_t i0 = 0; i0 < m; i0 += (uint32_t)kTopkThreads >> lg) {
        const uint32_t i = i0 + (tid >> lg);
        uint32_t r = 0;
        if (i < m) {
            const uint64_t w = swd[i];
            const Entry v = surv[i];
            for (uint32_t j = tid & (per - 1u); j < m; j += per) {
                const uint64_t x = swd[j];
                if (x > w || (x == w && j != i && ranks_before(surv[j], v))) r++;
            }
        }
        for (uint32_t o = 1; o < per; o <<= 1) r += __shfl_xor_sync(0xFFFFFFFFu, r, (int)o);
        if (i < m && (tid & (per - 1u)) == 0 && r < k) {
            if (!final_pass) {
                dst_ent[(uint64_t)blockIdx.x * k + r] = surv[i];
            } else {
                out_idx[r] = surv[i].idx;
                sel[r] = surv[i].idx;
            }
        }
    }
    const uint32_t pad = min(m, k);
    for (uint32_t i = pad + tid; i < k; i += kTopkThreads) {
        if (!final_pass) {
            Entry v;
            v.sum_ttft = 0; v.n_hit = 0; v.n_served = 0; v.idx = 0xFFFFFFFFu; v.valid = 0;
            dst_ent[(uint64_t)blockIdx.x * k + i] = v;
        } else {
            out_idx[i] = 0xFFFFFFFFu;
            sel[i] = 0xFFFFFFFFu;
        }
    }
    if (final_pass && out_res) {
        __syncthreads();
        for (uint32_t i = tid; i < 8u * k; i += kTopkThreads) {
            const uint32_t idx = sel[i >> 3];
            reinterpret_cast<uint4*>(out_res)[i] = idx != 0xFFFFFFFFu ? reinterpret_cast<const uint4*>(all_res + idx)[i & 7u]
                                                                      : make_uint4(0u, 0u, 0u, 0u);
        }
    }
}

static size_t topk_smem_bytes(uint32_t chunk) { return kSurvivors * (sizeof(Entry) + 8) + kDigits * 4 + (size_t)chunk * 8; }

size_t topk_scratch_bytes(uint64_t n_cand, uint32_t k) {
    const uint64_t blocks = (n_cand + kChunk - 1) / kChunk;
    return (size_t)(blocks * k * sizeof(Entry)) * 2 + 64;
}

// scratch: at least topk_scratch_bytes(n_cand, k), 16-byte aligned.
cudaError_t launch_topk(const maaso_result* results, uint64_t n_cand, uint32_t k, void* scratch,
                        uint32_t* out_idx, maaso_result* out_res, cudaStream_t stream, int* launches,
                        const double* scores) {
    cudaError_t err = cudaFuncSetAttribute(topk_pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)topk_smem_bytes(kChunkOne));
    if (err != cudaSuccess) return err;
    const uint64_t blocks0 = (n_cand + kChunk - 1) / kChunk;
    Entry* buf[2];
    buf[0] = reinterpret_cast<Entry*>(scratch);
    buf[1] = buf[0] + blocks0 * k;
    const Entry* src_ent = nullptr;
    uint64_t n = n_cand;
    int which = 0;
    for (;;) {
        const bool final_pass = n <= (uint64_t)kChunkOne;
        const uint32_t chunk = final_pass ? (uint32_t)kChunkOne : (uint32_t)kChunk;
        const uint64_t blocks = final_pass ? 1 : (n + kChunk - 1) / kChunk;
        topk_pass_kernel<<<(unsigned)blocks, kTopkThreads, topk_smem_bytes(final_pass ? (uint32_t)(n < 64 ? 64 : (n + 63) / 64 * 64) : chunk), stream>>>(
            results, src_ent, n, chunk, k, buf[which], final_pass ? 1 : 0, results, out_idx, out_res, scores);
        (*launches)++;
        if (final_pass) break;
        src_ent = buf[which];
        n = blocks * k;
        which ^= 1;
    }
    return cudaGetLastError();
}

// ---- top-k for callers that cannot allocate ---------------------------------------------------
// The partial lists of the passes live in a fixed array inside the library image instead of
// memory obtained at run time.  Every pass writes each entry the next pass reads, so nothing
// in the array has to be cleared between calls.
constexpr uint64_t kNoAllocMaxCand = MAASO_NOALLOC_MAX_CAND;
constexpr uint32_t kNoAllocMaxK = MAASO_NOALLOC_MAX_K;
constexpr size_t kNoAllocBytes =
    ((((kNoAllocMaxCand + kChunk - 1) / kChunk) * kNoAllocMaxK * sizeof(Entry) * 2 + 64) + 255) / 256 * 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// The device address of the array on the current device: its name is only a host-side handle and
// must not be handed to a kernel.  Looked up on every call (no allocation, no stream work), so no
// cached pointer can go stale when a context is re-created, and host threads share nothing.
static cudaError_t noalloc_scratch(void** out) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    *out = p;
    return cudaSuccess;
}

}  // namespace maaso

extern "C" MAASO_API int maaso_topk_noalloc(const maaso_result* results, uint64_t n_cand, uint32_t k,
                                            uint32_t order, uint32_t* out_idx, maaso_result* out_res,
                                            void* cuda_stream) {
    using namespace maaso;
    if (k == 0) return MAASO_OK;
    if (!out_idx || (!results && n_cand) || order != 0) return MAASO_EINVAL;
    if (n_cand > kNoAllocMaxCand || k > kNoAllocMaxK) return MAASO_ETOOBIG;  // beyond the fixed scratch
    void* scratch = nullptr;
    if (noalloc_scratch(&scratch) != cudaSuccess) {
        cudaGetLastError();
        return MAASO_ECUDA;
    }
    int launches = 0;
    const cudaError_t e = launch_topk(results, n_cand, k, scratch, out_idx, out_res, (cudaStream_t)cuda_stream,
                                      &launches, nullptr);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return MAASO_ECUDA;
    }
    return MAASO_OK;
}
