// Composite serving score of Sec. IV-D from the integer result records, in IEEE double with
// explicitly rounded operations (no fused multiply-add), so that it reproduces a plain
// sequential evaluation bit for bit.
#include "common.cuh"

namespace maaso {

__global__ void score_kernel(const maaso_result* res, uint64_t n, maaso_score_params p, double* out) {
    const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 a = reinterpret_cast<const uint4*>(res + i)[0];  // status, counted, served, hit
    const uint4 d = reinterpret_cast<const uint4*>(res + i)[3];  // .., .., sum_ttft
    const uint4 m = reinterpret_cast<const uint4*>(res + i)[5];  // max_e2e, makespan
    const uint4 t = reinterpret_cast<const uint4*>(res + i)[6];  // tokens, checksum
    if (a.x != 0) { out[i] = -1.0; return; }
    const uint32_t n_counted = a.y, n_served = a.z, n_hit = a.w;
    const int64_t sum_ttft = (int64_t)(((uint64_t)d.w << 32) | d.z);
    const int64_t makespan = (int64_t)(((uint64_t)m.w << 32) | m.z);
    const uint64_t tokens = ((uint64_t)t.y << 32) | t.x;
    double phis = 0.0, phit = 0.0, phil = 0.0;
    if (n_counted > 0) phis = __ddiv_rn((double)n_hit, (double)n_counted);           // Phi_S^n: SLO satisfaction ratio
    if (n_served > 0 && makespan > 0) {
        const double thr = __ddiv_rn((double)tokens, __dmul_rn((double)makespan, 1e-6));  // tokens per second
        phit = __ddiv_rn(thr < p.gamma_t ? thr : p.gamma_t, p.gamma_t);                   // Phi_T^n
    }
    if (n_served > 0) {
        const double lat = __dmul_rn(__ddiv_rn((double)sum_ttft, (double)n_served), 1e-6);  // mean time to first token, s
        double room = __dadd_rn(p.gamma_l, -lat);
        if (room < 0.0) room = 0.0;
        phil = __ddiv_rn(room, p.gamma_l);                                                // Phi_L^n
    }
    const double x = __dmul_rn(p.alpha, phis);
    const double y = __dmul_rn(p.beta, phit);
    const double z = __dmul_rn(__dadd_rn(1.0, -p.beta), phil);
    out[i] = __dadd_rn(__dadd_rn(x, y), z);
}

cudaError_t launch_score(const maaso_result* res, uint64_t n, const maaso_score_params& p, double* out,
                         cudaStream_t stream) {
    if (n) score_kernel<<<(unsigned)((n + 255) / 256), 256, 0, stream>>>(res, n, p, out);
    return cudaGetLastError();
}

// Upper edge (microseconds) of a histogram bin of ttft_bin; the last bin is open.
__device__ __forceinline__ int64_t ttft_bin_upper(uint32_t b) {
    if (b == 0) return 1023;
    if (b >= (uint32_t)(MAASO_TTFT_BINS - 1)) return INT64_MAX;
    const uint32_t e = 10u + (b - 1u) / 2u, h = (b - 1u) & 1u;
    return ((int64_t)1 << e) + (int64_t)(h + 1u) * ((int64_t)1 << (e - 1)) - 1;
}

struct PermilleList {
    uint32_t v[16];
};

// Eight lanes per candidate: lane l holds bins 8l .. 8l+7 (two 16-byte loads; a warp reads four histograms), and a scan over
// the lanes gives the cumulative counts.  They go to shared memory, where lane j searches for the bin that rank j falls into, six
// steps for all ranks at once.  Bound by the read of the histograms and the instructions around it: 10^6 histograms, three
// ranks, 67 us (every lane counting its bins below every target 75, every lane working out every target with 16 lanes a
// histogram 218, one thread per histogram 496).  Histograms are words, so they may start at any word: beside a 16-byte
// boundary they are read word by word (`Words`).  `U`: 32 bits where all counts of the warp's histograms are small.
template <class U>
__device__ __forceinline__ void percentiles_of(const U (&c)[8], U below, U* all, uint32_t l, const PermilleList& pm, uint32_t n_p, int64_t* o, bool write) {
    if constexpr (sizeof(U) == 4) {
        uint4* const v = reinterpret_cast<uint4*>(all + 8u * l);
        v[0] = make_uint4(below + c[0], below + c[1], below + c[2], below + c[3]);
        v[1] = make_uint4(below + c[4], below + c[5], below + c[6], below + c[7]);
    } else {
#pragma unroll
        for (int i = 0; i < 8; i++) all[8u * l + i] = below + c[i];
    }
    __syncwarp();
    const U total = all[MAASO_TTFT_BINS - 1];
    for (uint32_t j = l; j < n_p; j += 8u) {
        const uint32_t p = pm.v[j];
        // the rank's target count: ceil(p total / 1000), at least 1
        U target = sizeof(U) == 4 && total <= 4000000u ? (U)((p * (uint32_t)total + 999u) / 1000u) : (U)(((uint64_t)p * total + 999u) / 1000u);
        if (target < 1) target = 1;
        uint32_t bin = 0;  // how many bins end below it
#pragma unroll
        for (uint32_t step = MAASO_TTFT_BINS / 2u; step > 0u; step >>= 1)
            if (all[bin + step - 1u] < target) bin += step;
        if (write) o[j] = total ? ttft_bin_upper(bin) : -1;
    }
}

template <bool Words>
__global__ void __launch_bounds__(256) ttft_percentile_kernel(const uint32_t* hist, uint64_t n, const __grid_constant__ PermilleList pm, uint32_t n_p, int64_t* out) {
    const uint64_t c = ((uint64_t)blockIdx.x * 256u + threadIdx.x) >> 3;
    const uint32_t l = threadIdx.x & 7u;
    uint4 a = make_uint4(0u, 0u, 0u, 0u), b = a;
    if (c < n) {
        const uint32_t* h = hist + c * MAASO_TTFT_BINS + 8u * l;
        if (Words) {
            a = make_uint4(__ldg(h), __ldg(h + 1), __ldg(h + 2), __ldg(h + 3));
            b = make_uint4(__ldg(h + 4), __ldg(h + 5), __ldg(h + 6), __ldg(h + 7));
        } else {
            a = __ldg(reinterpret_cast<const uint4*>(h));
            b = __ldg(reinterpret_cast<const uint4*>(h) + 1);
        }
    }
    const bool small = (a.x | a.y | a.z | a.w | b.x | b.y | b.z | b.w) < (1u << 25);  // 64 of them stay below 2^31
    int64_t* const o = out + c * n_p;
    __shared__ __align__(16) unsigned long long s_all[32 * (MAASO_TTFT_BINS + 2)];  // cumulative counts, a histogram per 8 threads
    unsigned long long* const mine = s_all + (threadIdx.x >> 3) * (MAASO_TTFT_BINS + 2);
    if (__all_sync(0xFFFFFFFFu, small)) {
        uint32_t s[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 1; i < 8; i++) s[i] += s[i - 1];
        uint32_t incl = s[7];
#pragma unroll
        for (int k = 1; k < 8; k <<= 1) {
            const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, k, 8);
            if (l >= (uint32_t)k) incl += v;
        }
        percentiles_of(s, incl - s[7], reinterpret_cast<uint32_t*>(mine), l, pm, n_p, o, c < n);
    } else {
        unsigned long long s[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 1; i < 8; i++) s[i] += s[i - 1];
        unsigned long long incl = s[7];
#pragma unroll
        for (int k = 1; k < 8; k <<= 1) {
            const unsigned long long v = __shfl_up_sync(0xFFFFFFFFu, incl, k, 8);
            if (l >= (uint32_t)k) incl += v;
        }
        percentiles_of(s, incl - s[7], mine, l, pm, n_p, o, c < n);
    }
}

cudaError_t launch_ttft_percentiles(const uint32_t* hist, uint64_t n, const uint32_t* permille, uint32_t n_p,
                                    int64_t* out, cudaStream_t stream) {
    PermilleList pm;
    for (uint32_t j = 0; j < 16; j++) pm.v[j] = j < n_p ? permille[j] : 0;
    if (n) {
        auto kernel = reinterpret_cast<uintptr_t>(hist) % 16u ? ttft_percentile_kernel<true> : ttft_percentile_kernel<false>;
        kernel<<<(unsigned)((n + 31) / 32), 256, 0, stream>>>(hist, n, pm, n_p, out);
    }
    return cudaGetLastError();
}

}  // namespace maaso
