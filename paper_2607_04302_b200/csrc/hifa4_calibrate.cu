// Smooth-QK calibration (Eq. "sqk", "Calibration-Static Deployment") and the applicability gate ("Adaptive Applicability
// Gate"), without leaving the device:
//   scan      per (sample, KV head, channel) the largest magnitude of Q and of K; for the gate also the exact histogram
//             of |K| and the two global maxima - one pass over the activations
//   finalize  gate decision (if asked for) and the factors s, 1/s
// |x| of a 16-bit float is a 15-bit pattern whose integer order is the order of the values, so a 32768-bin histogram of
// the patterns is the exact distribution of |K| and the nearest-rank percentile is read off its running sum.
//
// Bound: the bytes of the activations.  32 samples x 1024 tokens x 32 / 8 heads x 128 channels (336 MB): 52 us at the
// measured copy rate.  As five kernels - a maximum of K and one of Q with 8 atomics per thread and 256 tokens, a separate
// histogram pass over K, a one-CTA gate, the factors - it took 33 + 104 + 22 + 24 + 6 us; now clear 2.5, scan 58, factors
// 7 us under ncu, and the whole call 68 instead of 195 us.
#include "hifa4_internal.h"
#include "hifa4_device.cuh"

namespace hifa4 {

constexpr int HIST_BINS = 32768;
constexpr int SCAN_THREADS = 1024, SCAN_GROUP = 512;      // two groups of 16 warps per CTA, one CTA per SM
constexpr int SCAN_UNROLL = 8;                            // 16-byte loads in flight per thread

struct ScanJob {
    const uint4 *q, *k;
    long long q_rows, k_rows;         // S * H * Ncal
    int Hq, Hkv, Ncal, C;             // C = d / 8 vectors per row
    uint32_t *qmax, *kmax;            // [S,Hkv,d], cleared
    uint32_t *hist, *gmax;            // gate: [HIST_BINS] and {max|K|, max|Q|}, cleared; else null
    HeadMap qmap;
};

// One group of 512 threads takes rows r0..r1-1 of x [S, H, Ncal, d]: maxima in registers (thread t always holds vector
// t % C of a row) while the rows belong to one (sample, KV head), then one reduction through shared memory and d atomics.
template <typename T, bool HIST>
__device__ __forceinline__ void scan_rows(const uint4* __restrict__ x, long long r0, long long r1, const HeadMap* map, int H,
                                          int Hkv, int Ncal, int C, int tid, int bar, uint4* red, uint32_t* __restrict__ ws,
                                          uint32_t* hist_s, uint32_t* __restrict__ gmax)
{
    uint4 acc = make_uint4(0, 0, 0, 0);
    auto take = [&](uint4 v) {
        v.x &= 0x7FFF7FFFu; v.y &= 0x7FFF7FFFu; v.z &= 0x7FFF7FFFu; v.w &= 0x7FFF7FFFu;
        acc.x = max16<T>(acc.x, v.x); acc.y = max16<T>(acc.y, v.y);
        acc.z = max16<T>(acc.z, v.z); acc.w = max16<T>(acc.w, v.w);
        if (HIST) {
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                atomicAdd(&hist_s[w[i] & 0xFFFFu], 1u);
                atomicAdd(&hist_s[w[i] >> 16], 1u);
            }
        }
    };
    auto key_of = [&](long long sh) { return (sh / H) * Hkv + (map ? (int)map->kv_of[sh % H] : (int)(sh % H)); };
    long long r = r0;
    while (r < r1) {
        long long sh = r / Ncal;                          // sample * H + head
        const long long key = key_of(sh);
        long long end = (++sh) * Ncal;
        while (end < r1 && key_of(sh) == key) end = (++sh) * Ncal;     // heads of one KV head follow one another
        end = min(end, r1);
        const uint4* p = x + r * C;
        const long long n = (end - r) * C;
        long long i = tid;
        for (; i + (SCAN_UNROLL - 1) * SCAN_GROUP < n; i += SCAN_UNROLL * SCAN_GROUP) {
            uint4 v[SCAN_UNROLL];
#pragma unroll
            for (int u = 0; u < SCAN_UNROLL; ++u) v[u] = __ldcs(p + i + u * SCAN_GROUP);
#pragma unroll
            for (int u = 0; u < SCAN_UNROLL; ++u) take(v[u]);
        }
        for (; i < n; i += SCAN_GROUP) take(__ldcs(p + i));
        red[tid] = acc;
        acc = make_uint4(0, 0, 0, 0);
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(SCAN_GROUP) : "memory");
        const int words = 4 * C;                          // 32-bit words per row of the table: 32, 64 or 128
        if (tid < words) {
            const uint32_t* rw = reinterpret_cast<const uint32_t*>(red) + tid;
            uint32_t m = 0;
            for (int row = 0; row < SCAN_GROUP / C; ++row) m = max16<T>(m, rw[row * words]);
            float lo, hi;
            Pair16<T>::unpack(m, lo, hi);
            uint32_t* o = ws + key * (8 * C) + 2 * tid;   // non-negative floats order like their bit patterns
            atomicMax(o, __float_as_uint(lo));
            atomicMax(o + 1, __float_as_uint(hi));
            if (gmax) {
                const uint32_t top = __reduce_max_sync(0xffffffffu, __float_as_uint(fmaxf(lo, hi)));
                if ((tid & 31) == 0) atomicMax(gmax, top);
            }
        }
        asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(SCAN_GROUP) : "memory");
        r = end;
    }
}

// CTA i takes the i-th share of Q's rows and of K's.  Threads 512.. take the K share (and its histogram, 128 KB of
// counters in shared memory) and then help with the end of the Q share, threads 0..511 its beginning: the histogram's
// shared-memory atomics, 22 us on their own at the size above, run under the other group's loads.
template <typename T, bool HIST>
__global__ void __launch_bounds__(SCAN_THREADS, 1)
calibrate_scan_kernel(const __grid_constant__ ScanJob job)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    extern __shared__ uint32_t hist_s[];
    __shared__ uint4 red[2][SCAN_GROUP];
    const int tid = threadIdx.x;
    if (HIST) {
        for (int i = tid; i < HIST_BINS / 4; i += SCAN_THREADS) reinterpret_cast<uint4*>(hist_s)[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");    // the counters and maxima have been cleared
    const long long nb = gridDim.x, b = blockIdx.x;
    const long long q0 = job.q_rows * b / nb, q1 = job.q_rows * (b + 1) / nb;
    const long long k0 = job.k_rows * b / nb, k1 = job.k_rows * (b + 1) / nb;
    const long long k_cost = (k1 - k0) * (HIST ? 2 : 1);  // a K row with its histogram counts as two
    const long long spare = (q1 - q0) - k_cost;
    const long long qm = q1 - (spare > 0 ? spare / 2 : 0);
    if (tid < SCAN_GROUP) {
        scan_rows<T, false>(job.q, q0, qm, &job.qmap, job.Hq, job.Hkv, job.Ncal, job.C, tid, 1, red[0], job.qmax, nullptr,
                            HIST ? job.gmax + 1 : nullptr);
    } else {
        scan_rows<T, HIST>(job.k, k0, k1, nullptr, job.Hkv, job.Hkv, job.Ncal, job.C, tid - SCAN_GROUP, 2, red[1], job.kmax, hist_s,
                           HIST ? job.gmax : nullptr);
        scan_rows<T, false>(job.q, qm, q1, &job.qmap, job.Hq, job.Hkv, job.Ncal, job.C, tid - SCAN_GROUP, 2, red[1], job.qmax, nullptr,
                            HIST ? job.gmax + 1 : nullptr);
    }
    if (HIST) {
        __syncthreads();
        for (int i = tid; i < HIST_BINS; i += SCAN_THREADS)
            if (hist_s[i]) atomicAdd(&job.hist[i], hist_s[i]);
    }
}

__global__ void __launch_bounds__(256)
clear_kernel(uint32_t* __restrict__ a, long long na, uint32_t* __restrict__ b, int nb)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const long long step = (long long)gridDim.x * 256, i0 = (long long)blockIdx.x * 256 + threadIdx.x;
    for (long long i = i0; i < na; i += step) a[i] = 0;
    for (long long i = i0; i < nb; i += step) b[i] = 0;
}

// Nearest-rank 99th percentile of S non-negative values: the (S / 100 + 1)-th largest, found from the top, one pass over the
// values per distinct one (their bit patterns order like integers).  Counting the values below each candidate instead took
// S^2 loads: 38 samples, 40 / 8 heads, 256 channels 300 us, now under 10.
__device__ __forceinline__ double percentile99(const float* __restrict__ v, int S, long long stride)
{
    const long long rank = (long long)ceil(0.99 * (double)S) < 1 ? 1 : (long long)ceil(0.99 * (double)S);
    long long left = S - rank + 1;
    uint32_t top = 0, limit = 0xFFFFFFFFu;
    while (left > 0) {
        long long count = 0;
        top = 0;
#pragma unroll 8
        for (int m = 0; m < S; ++m) {
            const uint32_t u = __float_as_uint(v[m * stride]);
            if (u < limit) {
                count = u > top ? 1 : count + (u == top);
                top = max(top, u);
            }
        }
        if (count == 0) break;
        left -= count;
        limit = top;
    }
    return (double)__uint_as_float(top);
}

constexpr int FIN_THREADS = 256;

// Pattern of rank `rank` (from 1) in the histogram; the whole CTA takes part and gets the result.
__device__ __forceinline__ uint32_t hist_select(const uint32_t* __restrict__ hist, unsigned long long rank)
{
    __shared__ unsigned long long s_warp[FIN_THREADS / 32];
    __shared__ uint32_t s_found;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int PER_WARP = HIST_BINS / (FIN_THREADS / 32);          // bins of a warp, 64 at a time (2 per lane)
    const uint2* hw = reinterpret_cast<const uint2*>(hist + warp * PER_WARP);
    unsigned long long sum = 0;
#pragma unroll 16
    for (int i = 0; i < PER_WARP / 64; ++i) {
        const uint2 h = hw[i * 32 + lane];
        sum += (unsigned long long)h.x + h.y;
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) s_warp[warp] = sum;
    if (tid == 0) s_found = 0;
    __syncthreads();
    unsigned long long before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    if (before < rank && rank <= before + sum) {                      // the rank falls in this warp's bins
        for (int i = 0; i < PER_WARP / 64; ++i) {
            const uint2 h = hw[i * 32 + lane];
            unsigned long long c = (unsigned long long)h.x + h.y;     // inclusive scan over the lanes
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long up = __shfl_up_sync(0xffffffffu, c, o);
                if (lane >= o) c += up;
            }
            const unsigned long long all = __shfl_sync(0xffffffffu, c, 31), mine = before + c - h.x - h.y;
            if (rank <= before + all) {
                if (mine < rank && rank <= before + c)
                    s_found = (uint32_t)(warp * PER_WARP + i * 64 + 2 * lane + (rank > mine + h.x ? 1 : 0));
                break;
            }
            before += all;
        }
    }
    __syncthreads();
    return s_found;
}

// s = Kagg^alpha / Qagg^(1-alpha); 1 where degenerate.  The per-sample maxima are combined over the S samples by
// root-mean-square (aggregator 0, the paper's choice), mean (1) or nearest-rank 99th percentile (2).
// hist non-null: the gate chooses alpha and bypass (every CTA reads the histogram for itself, 128 KB from L2); gmax:
// {max|K|, max|Q|}; stats[0..3] = rho_K, T_K/Q, branch (0 bypass, 1 strong, 2 mild), alpha.
template <typename T>
__global__ void __launch_bounds__(FIN_THREADS)
smooth_finalize_kernel(const float* __restrict__ kmax, const float* __restrict__ qmax, int S, int n, double alpha, int bypass,
                       int aggregator, const uint32_t* __restrict__ hist, const uint32_t* __restrict__ gmax,
                       unsigned long long rank, float* __restrict__ stats, float* __restrict__ s, float* __restrict__ inv_s)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (hist) {
        const double p99 = (double)In16<T>::to_f((uint16_t)hist_select(hist, rank));
        const float mk = __uint_as_float(gmax[0]), mq = __uint_as_float(gmax[1]);
        const double rho = p99 > 0.0 ? (double)mk / p99 : 0.0;
        const double t = mq > 0.f ? (double)mk / (double)mq : 0.0;
        const int branch = (rho >= 6.0 && t >= 2.0) ? (t > 3.0 ? 1 : 2) : 0;
        alpha = branch == 1 ? 0.5 : branch == 2 ? 0.25 : 0.0;
        bypass = branch == 0;
        if (stats && blockIdx.x == 0 && threadIdx.x == 0) {
            stats[0] = (float)rho;
            stats[1] = (float)t;
            stats[2] = (float)branch;
            stats[3] = (float)alpha;
        }
    }
    const int i = blockIdx.x * FIN_THREADS + threadIdx.x;
    if (i >= n) return;
    double sv = 1.0;
    if (!bypass) {
        double kagg, qagg;
        if (aggregator == 2) {
            kagg = percentile99(kmax + i, S, n);
            qagg = percentile99(qmax + i, S, n);
        } else {
            double ks = 0, qs = 0;
#pragma unroll 8
            for (int m = 0; m < S; ++m) {
                const double a = kmax[(long long)m * n + i], b = qmax[(long long)m * n + i];
                ks += aggregator == 1 ? a : a * a;
                qs += aggregator == 1 ? b : b * b;
            }
            kagg = aggregator == 1 ? ks / S : sqrt(ks / S);
            qagg = aggregator == 1 ? qs / S : sqrt(qs / S);
        }
        if (kagg > 0 && qagg > 0) sv = pow(kagg, alpha) / pow(qagg, 1.0 - alpha);
    }
    const float sf = (float)sv;
    s[i] = sf;
    inv_s[i] = __frcp_rn(sf);
}

// ------------------------------------------------------------------------------- launchers
template <typename T, bool HIST>
static cudaError_t launch_scan(const ScanJob& job, cudaStream_t st)
{
    const size_t smem = HIST ? HIST_BINS * sizeof(uint32_t) : 0;
    auto kern = calibrate_scan_kernel<T, HIST>;
    static SmemOptIn opt_in;
    if (smem && !opt_in.ensure(kern, (int)smem)) return cudaErrorInvalidValue;
    int dev = 0, sms = 148;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const long long want = ((job.q_rows + job.k_rows) * job.C + 4 * SCAN_THREADS - 1) / (4 * SCAN_THREADS);
    return launch_dependent(kern, (unsigned)(want < sms ? want : sms), SCAN_THREADS, smem, st, job);
}

cudaError_t launch_calibrate(int dtype, const void* q_cal, const void* k_cal, const HeadMap& qmap, int S, int Hq, int Hkv,
                             int Ncal, int d, double alpha, bool bypass, int aggregator, float* absmax_ws, void* gate_ws,
                             float* d_stats, float* s, float* inv_s, cudaStream_t st)
{
    const long long n = (long long)S * Hkv * d;
    float *kmax = absmax_ws, *qmax = absmax_ws + n;
    uint32_t* hist = reinterpret_cast<uint32_t*>(gate_ws);
    uint32_t* gmax = hist ? hist + HIST_BINS : nullptr;
    cudaError_t e;
    if (hist) {
        if ((e = launch_dependent(clear_kernel, 64, 256, 0, st, reinterpret_cast<uint32_t*>(absmax_ws), 2 * n, hist, HIST_BINS + 2)) != cudaSuccess)
            return e;
    } else if ((e = cudaMemsetAsync(absmax_ws, 0, 2 * n * sizeof(float), st)) != cudaSuccess) {
        return e;
    }
    if (!bypass) {
        ScanJob job{};
        job.q = (const uint4*)q_cal; job.k = (const uint4*)k_cal;
        job.q_rows = (long long)S * Hq * Ncal; job.k_rows = (long long)S * Hkv * Ncal;
        job.Hq = Hq; job.Hkv = Hkv; job.Ncal = Ncal; job.C = d / 8;
        job.qmax = (uint32_t*)qmax; job.kmax = (uint32_t*)kmax;
        job.hist = hist; job.gmax = gmax;
        job.qmap = qmap;
        if (dtype == HIFA4_F16) e = hist ? launch_scan<__half, true>(job, st) : launch_scan<__half, false>(job, st);
        else e = hist ? launch_scan<__nv_bfloat16, true>(job, st) : launch_scan<__nv_bfloat16, false>(job, st);
        if (e != cudaSuccess) return e;
    }
    unsigned long long rank = (unsigned long long)ceil(0.99 * (double)((long long)S * Hkv * Ncal * d));   // nearest-rank percentile
    if (rank < 1) rank = 1;
    const int nf = Hkv * d;
    const unsigned blocks = (unsigned)((nf + FIN_THREADS - 1) / FIN_THREADS);
    auto fin = dtype == HIFA4_F16 ? smooth_finalize_kernel<__half> : smooth_finalize_kernel<__nv_bfloat16>;
    return launch_dependent(fin, blocks, FIN_THREADS, 0, st, (const float*)kmax, (const float*)qmax, S, nf, alpha, bypass ? 1 : 0, aggregator,
                            (const uint32_t*)hist, (const uint32_t*)gmax, rank, d_stats, s, inv_s);
}

}  // namespace hifa4
