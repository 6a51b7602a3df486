// Smooth-QK scaling fused with HIF4 quantization (Algorithm 1 lines 1 and 3).  Q, K and V are quantized by one
// launch: 128-bit coalesced loads, a team of four lanes per 64-element group, shuffle reductions,
// packed f32x2 arithmetic.
#include <type_traits>

#include "hifa4_internal.h"
#include "hifa4_device.cuh"
#include "hifa4_ptx.cuh"

namespace hifa4 {

using namespace ptx;

// A team of four lanes owns a 64-element group; lane j owns its level-2 units j and j + 4 (8 elements each), so that the
// team's 16-byte loads and image stores cover 64 contiguous bytes each.
// The kernel is bound by instruction issue, the ALU pipe (logic, permutes, shifts, 16-bit maxima, conversions; half rate)
// first, before it is bound by memory; hence four lanes instead of eight (what a lane does once per group was a third of
// the instructions), maxima, shift selection and metadata on packed 16-bit patterns, and multiplications where they
// replace logic: 17 executed warp instructions per element of a lane instead of 25.  Q, K and V of 32 / 8 heads, d = 128,
// bf16: N = 8192 49.7 -> 41.5 us (230 MB, 5.5 TB/s), N = 4096 27.4 -> 24.7 us; persistent CTAs that load the next piece
// under the current one were slower (64 us: fewer independent chains per scheduler), and so were one share per thread
// (48 us) and three or five CTAs per SM.
struct Group {                        // constants of a 64-element group whose maximum magnitude is A
    uint32_t s_bits;                  // the scale S = smallest E6M2 value with 7 S >= A (clamped to the code range)
    uint64_t inv44, s44;              // {4/S, 4/S}, {S/4, S/4}
    uint32_t c0_bits;                 // bits(-magic * S/4)
};
// Biased quotient y = RZ(x * RN(4/S)) + magic * 2^k, magic = 1.5 * 2^23 + 8: rounds to the nearest multiple of 2^k, ties to
// even (see e6m2_inv4 on the ties); the low bits of y are m + 8 >= 1, m the signed code; fma(y, S/4, -magic * 2^k * S/4) =
// m * 2^k * S/4 without rounding (magic * (4 + M) has at most 24 significant bits).
constexpr uint32_t Q_MAGIC_BITS = 0x4B400008u;
__device__ __forceinline__ Group group_of(float A)
{
    Group g;
    // S = A / 7 rounded up to two mantissa bits.  1/7 is rounded down, so A = 7 S gives at most S; any other A with at most
    // 11 significant bits exceeds 7 S by 2^-11 of itself or more, which the two roundings cannot hide.
    const uint32_t t = (__float_as_uint(__fmul_rn(A, __uint_as_float(0x3E124924u))) + 0x1FFFFFu) & 0xFFE00000u;
    g.s_bits = min(max(t, 0x27800000u), 0x47600000u);              // codes 0 and 255
    const float s4 = __uint_as_float(g.s_bits - (2u << 23));
    float r;                                                       // 4/S correctly rounded: S has three significant bits, so the
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s4));         // residual is exact and one step decides the rounding
    r = fmaf(fmaf(-s4, r, 1.f), r, r);
    g.inv44 = pack2(r, r);
    g.s44 = pack2(s4, s4);
    g.c0_bits = __float_as_uint(__fmul_rn(-12582920.f, s4));
    return g;
}

// Shifts of the two subgroups of a unit from their maxima At (packed), k_t * 2^7 in the two halves:
// k_t = max(need_t, need_other - 1), need = number of 1.75 S, 3.5 S exceeded (the pair rule of the level-2 bit).
template <typename T> __device__ __forceinline__ uint32_t unit_shifts(uint32_t At, float S);
// BF16 patterns: x_t = max(bits(At_t) - bits(1.75 S) - 1 + 2^7, 0) = need_t * 2^7 + fraction; 1.75 S is a BF16 value, and
// -bits(1.75 S) - 1 + 2^7 is the complement of bits(0.875 S).
template <> __device__ __forceinline__ uint32_t unit_shifts<__nv_bfloat16>(uint32_t At, float S)
{
    const uint32_t b = __float_as_uint(0.875f * S);
    const uint32_t x = __viaddmax_s16x2(At, ~__byte_perm(b, b, 0x3232), 0u);
    return __viaddmax_s16x2(__byte_perm(x, x, 0x1032), 0xFF80FF80u, x) & 0x01800180u;
}
// FP16 subnormals have no binades, so FP16 maxima are widened first.
template <> __device__ __forceinline__ uint32_t unit_shifts<__half>(uint32_t At, float S)
{
    float a0, a1;
    Pair16<__half>::unpack(At, a0, a1);
    const int b = (int)__float_as_uint(0.875f * S) + 1;
    const int x0 = max((int)__float_as_uint(a0) - b, 0), x1 = max((int)__float_as_uint(a1) - b, 0);
    const int k0 = max(x0, x1 - (1 << 23)) >> 23, k1 = max(x1, x0 - (1 << 23)) >> 23;
    return (uint32_t)(k0 << 7 | k1 << 23);
}

// xw: the 16 values as packed pairs (words 0-3 unit j, 4-7 unit j + 4), already smoothed and rounded to T.  Returns the
// BF16 image in xw; CODES: also the packed nibbles of the two units and the group's metadata word (same on every lane).
// False: the group's maximum lies above 7 S of the largest scale (in FP16: it is an infinity, a smoothed product may round to
// one; 7 S is not an FP16 value), or the group holds a NaN, whose bit pattern would run into its neighbours' nibbles.  What was
// formed is then void and quantize16_general has to do it.
template <typename T, bool CODES>
__device__ __forceinline__ bool quantize16(uint32_t (&xw)[8], int j, uint32_t (&nib)[2], uint32_t& meta_word)
{
    uint32_t At[2];                                               // {subgroup 0, subgroup 1} of each unit; a NaN wins
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        const uint32_t m0 = max16_nan<T>(abs16<T>(xw[4 * u]), abs16<T>(xw[4 * u + 1]));
        const uint32_t m1 = max16_nan<T>(abs16<T>(xw[4 * u + 2]), abs16<T>(xw[4 * u + 3]));
        At[u] = max16_nan<T>(__byte_perm(m0, m1, 0x5410), __byte_perm(m0, m1, 0x7632));
    }
    uint32_t A2 = max16_nan<T>(At[0], At[1]);
    A2 = max16_nan<T>(A2, __byte_perm(A2, A2, 0x1032));
    A2 = max16_nan<T>(A2, __shfl_xor_sync(0xffffffffu, A2, 1));
    A2 = max16_nan<T>(A2, __shfl_xor_sync(0xffffffffu, A2, 2));
    float A, Ah;
    Pair16<T>::unpack(A2, Ah, A);
    const Group g = group_of(A);                                  // A = 0 gives code 0 and an all-zero group
    uint32_t ks[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        ks[u] = unit_shifts<T>(At[u], __uint_as_float(g.s_bits));
        const uint32_t ks0 = ks[u] << 16, ks1 = ks[u] & 0xFFFF0000u;          // k << 23
        const uint64_t mm = pack2(__uint_as_float(Q_MAGIC_BITS + ks0), __uint_as_float(Q_MAGIC_BITS + ks1));
        const uint64_t cc = pack2(__uint_as_float(g.c0_bits + ks0), __uint_as_float(g.c0_bits + ks1));
        // element i of subgroup 0 is paired with element i of subgroup 1: one pair of constants serves four operations
        float x[8], v[8], y[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) Pair16<T>::unpack(xw[4 * u + i], x[2 * i], x[2 * i + 1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint64_t yy = add2(mul2_rz(pack2(x[i], x[4 + i]), g.inv44), mm);
            unpack2(fma2(yy, g.s44, cc), v[i], v[4 + i]);
            unpack2(yy, y[i], y[4 + i]);
        }
        // at most 6 significant bits: the upper halves of the FP32 patterns are the BF16 values
#pragma unroll
        for (int i = 0; i < 4; ++i) xw[4 * u + i] = __byte_perm(__float_as_uint(v[2 * i]), __float_as_uint(v[2 * i + 1]), 0x7632);
        if (CODES) {
            // nibbles m + 8 of a subgroup add up in the low 16 bits (magic * 16^i is zero there except for its 8), then all
            // eight are turned from offset to sign-magnitude form: negative where bit 3 is clear, |m| = 8 - (m + 8)
            uint32_t h[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                h[t] = __float_as_uint(y[4 * t + 3]) * 16u + __float_as_uint(y[4 * t + 2]);
                h[t] = h[t] * 16u + __float_as_uint(y[4 * t + 1]);
                h[t] = h[t] * 16u + __float_as_uint(y[4 * t]);
            }
            const uint32_t b = __byte_perm(h[0], h[1], 0x5410);
            const uint32_t neg = ~b & 0x88888888u, one = neg >> 3;
            nib[u] = (((b & 0x77777777u) ^ (one * 7u)) + one) | neg;
        }
    }
    if (CODES) {
        // level-2 bit of a unit: both subgroups shifted; level-3 bit: k = 2, or k = 1 without the level-2 bit.  Both units
        // at once: k of (unit, subgroup) at bits 0, 16 (unit j) and 8, 24 (unit j + 4)
        const uint32_t w = (ks[0] >> 7) | (ks[1] << 1);
        const uint32_t nz = w | (w >> 1), aa = nz & (nz >> 16) & 0x00000101u;
        const uint32_t l3 = ((w >> 1) | (w & ~(aa * 0x00010001u))) & 0x01010101u;
        uint32_t part = ((aa | (aa >> 4)) & 0x11u) << (8 + j);
        part |= ((l3 | (l3 >> 15)) & 0x0303u) << (16 + 2 * j);
        part |= __shfl_xor_sync(0xffffffffu, part, 1);
        part |= __shfl_xor_sync(0xffffffffu, part, 2);
        meta_word = part | ((g.s_bits >> 21) - 316u);             // + scale code 4 (exponent - 79) + mantissa
    }
    return A <= 401408.f;
}

// The same for any values: widened, and clamped where the maximum exceeds 7 S.  A warp that has a group for it runs it over
// all its shares, after the usual form, in a function of its own (see requantize).
template <typename T, bool CODES>
__device__ __forceinline__ void quantize16_general(uint32_t (&xw)[8], int j, uint32_t (&nib)[2], uint32_t& meta_word)
{
    float a[4], A = 0.f;                                          // maxima of the lane's subgroups and of the group; a NaN loses
#pragma unroll
    for (int t = 0; t < 4; ++t) {
        float x[4];
        Pair16<T>::unpack(xw[2 * t], x[0], x[1]);
        Pair16<T>::unpack(xw[2 * t + 1], x[2], x[3]);
        a[t] = fmaxf(max3(fabsf(x[0]), fabsf(x[1]), fabsf(x[2])), fabsf(x[3]));
        A = fmaxf(A, a[t]);
    }
    A = fmaxf(A, __shfl_xor_sync(0xffffffffu, A, 1));
    A = fmaxf(A, __shfl_xor_sync(0xffffffffu, A, 2));
    const Hif4Group g = hif4_group(A);
    uint32_t part = 0;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
        float x[8], y[8];
#pragma unroll
        for (int i = 0; i < 4; ++i) Pair16<T>::unpack(xw[4 * u + i], x[2 * i], x[2 * i + 1]);
        if (A > g.top) {
#pragma unroll
            for (int i = 0; i < 8; ++i) x[i] = x[i] > g.top ? g.top : x[i] < -g.top ? -g.top : x[i];     // a NaN stays one
            a[2 * u] = fminf(a[2 * u], g.top);
            a[2 * u + 1] = fminf(a[2 * u + 1], g.top);
        }
        uint32_t w[4];
        int l2, k0, k1;
        hif4_unit(x, a[2 * u], a[2 * u + 1], g, w, y, l2, k0, k1);
#pragma unroll
        for (int i = 0; i < 4; ++i) xw[4 * u + i] = w[i];
        if (CODES) {
            nib[u] = hif4_unit_nibbles(y);
            part |= hif4_unit_meta(j + 4 * u, l2, k0, k1);
        }
    }
    if (CODES) {
        part |= __shfl_xor_sync(0xffffffffu, part, 1);
        part |= __shfl_xor_sync(0xffffffffu, part, 2);
        meta_word = part | (uint32_t)g.code;
    }
}

struct QuantJob {                     // one launch quantizes Q, K and V (any of them may be absent)
    const uint16_t *q, *k, *v;        // [B,Hq,N,d], [B,Hkv,N,d], [B,Hkv,N,d]
    const float *s, *inv_s;           // [Hkv,d] Smooth-QK factors for Q and K, or null
    uint8_t *q_codes, *k_codes, *v_codes;
    uint32_t *q_meta, *k_meta, *v_meta;
    uint16_t *q_img, *k_img, *v_img;
    float *q_mu, *k_sum;              // Q-Mean auxiliary outputs or null
    int Hq, Hkv, N, d;
    unsigned q_blocks, k_blocks;      // CTAs [0, q_blocks) take Q, the next k_blocks K, the rest V
    unsigned row_blocks_per_head;     // N * d / 16 / (256 * UPT)
    unsigned v_tiles;                 // 64 x 64 tiles of V, two per CTA
    HeadMap qmap;
};

constexpr int QUANT_THREADS = 256;
// Lane shares (16 elements) per thread, template parameter UPT: 2 where a head holds a multiple of 512 of them (64 bytes of
// loads in flight per thread), else 1.

// Q and K: groups along d.  One head is N*d/16 lane shares; a CTA takes 256 * UPT consecutive ones, thread t the shares t,
// t + 256 (all loads are issued before any arithmetic).  The shares of a thread have their channels, hence their Smooth-QK
// factors, in common.  Returns whether the usual form did for all of them.
template <typename T, int UPT, bool CODES, bool QM, bool GENERAL>
__device__ __forceinline__ bool quantize_rows_cta(const uint16_t* __restrict__ x, const float* __restrict__ scale,
                                                  int kv_row, long long head, unsigned blk_in_head, int N, int d,
                                                  uint8_t* __restrict__ codes, uint32_t* __restrict__ meta,
                                                  uint16_t* __restrict__ img, float* __restrict__ mu_out,
                                                  float* __restrict__ ksum_out)
{
    const int spr = d >> 4;                                                   // lane shares per row
    const int j = threadIdx.x & 3;
    const unsigned s0 = blk_in_head * (QUANT_THREADS * UPT) + threadIdx.x;    // share inside the head
    const long long g0 = head * (long long)N * (d >> 6) + (s0 >> 2);          // 64-element group
    const uint4* src = reinterpret_cast<const uint4*>(x) + g0 * 8 + j;
    uint4 raw[UPT][2];
#pragma unroll
    for (int r = 0; r < UPT; ++r) {
        raw[r][0] = __ldg(src + r * (QUANT_THREADS * 2));
        raw[r][1] = __ldg(src + r * (QUANT_THREADS * 2) + 4);
    }
    const int c0 = (int)((s0 >> 2) & (unsigned)((d >> 6) - 1)) * 64 + j * 8;  // first channel; the other unit is 32 further
    float4 sv[4];
    if (scale) {
        const float4* sp = reinterpret_cast<const float4*>(scale + (long long)kv_row * d + c0);
        sv[0] = __ldg(sp); sv[1] = __ldg(sp + 1); sv[2] = __ldg(sp + 8); sv[3] = __ldg(sp + 9);
    }
    bool done = true;
#pragma unroll
    for (int r = 0; r < UPT; ++r) {
        const long long grp = g0 + r * (QUANT_THREADS / 4);
        uint32_t xw[8] = {raw[r][0].x, raw[r][0].y, raw[r][0].z, raw[r][0].w, raw[r][1].x, raw[r][1].y, raw[r][1].z, raw[r][1].w};
        if (scale) {                                       // FP32 product, rounded once to the activation dtype
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float lo, hi, a, b;
                Pair16<T>::unpack(xw[i], lo, hi);
                const float4 f = sv[i >> 1];
                unpack2(mul2(pack2(lo, hi), (i & 1) ? pack2(f.z, f.w) : pack2(f.x, f.y)), a, b);
                xw[i] = Pair16<T>::round_pack(a, b);
            }
        }
        if (QM) {
            // Q-Mean auxiliary (Algorithm 1 lines 2 and 6).  A row of d channels sits in d/16 consecutive,
            // aligned lanes; the sum runs in double, where it is exact for any row whose values span fewer
            // than ~40 binades, so its order does not matter.
            const long long row = head * N + (s0 + r * QUANT_THREADS) / (unsigned)spr;
            const bool first = ((threadIdx.x & (unsigned)(spr - 1)) == 0);
            double sum = 0.0;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                float lo, hi;
                Pair16<T>::unpack(xw[i], lo, hi);
                sum += (double)lo + (double)hi;
            }
            for (int off = 1; off < spr; off <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
            if (mu_out) {                                  // q_z = round_in(q~ - mu), mu = FP16(mean)
                const float mu = __half2float(__double2half(sum / (double)d));
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    float lo, hi;
                    Pair16<T>::unpack(xw[i], lo, hi);
                    xw[i] = Pair16<T>::round_pack(In16<T>::round_d((double)lo - (double)mu), In16<T>::round_d((double)hi - (double)mu));
                }
                if (first) mu_out[row] = mu;
            } else if (first) {
                ksum_out[row] = __half2float(__double2half(sum));
            }
        }
        uint32_t nib[2], mw;
        if constexpr (GENERAL) quantize16_general<T, CODES>(xw, j, nib, mw);
        else done &= quantize16<T, CODES>(xw, j, nib, mw);
        uint4* dst = reinterpret_cast<uint4*>(img) + grp * 8 + j;
        dst[0] = make_uint4(xw[0], xw[1], xw[2], xw[3]);
        dst[4] = make_uint4(xw[4], xw[5], xw[6], xw[7]);
        if (CODES) {
            uint32_t* cw = reinterpret_cast<uint32_t*>(codes) + grp * 8 + j;
            cw[0] = nib[0];
            cw[4] = nib[1];
            if (j == 0) meta[grp] = mw;
        }
    }
    return done;
}

// V: groups of 64 tokens per channel; outputs are stored transposed ([.., d, N]).  Half a CTA (128 threads) transposes a
// 64-token x 64-channel tile through shared memory.  The tile is kept as 64 rows of 8 16-byte chunks, chunk c of row r
// stored at position c ^ f(r) with f(r) = 2 (r / 8) mod 8 + r / 32, so that both the row-wise 16-byte stores and the
// column-wise 4-byte reads (a thread reads two adjacent channels of 8 consecutive tokens, a warp 8 channel pairs x 4
// lanes) are free of bank conflicts.  The general form reads its values from global memory instead.
template <typename T, bool CODES, bool GENERAL>
__device__ __forceinline__ bool quantize_tokens_half(uint4* tile, bool valid, const uint16_t* __restrict__ x, long long bh, int tok0,
                                                     int ch0, int N, int d, uint8_t* __restrict__ codes,
                                                     uint32_t* __restrict__ meta, uint16_t* __restrict__ img)
{
    const int tid = threadIdx.x & 127;
    const uint16_t* src = x + (bh * N + tok0) * (long long)d + ch0;
    auto swz = [](int r) { return ((r >> 3) * 2 & 7) + (r >> 5); };
    if constexpr (!GENERAL) {
        if (valid) {
            uint4 v[4];
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int idx = tid + it * 128;
                v[it] = __ldg(reinterpret_cast<const uint4*>(src + (long long)(idx >> 3) * d) + (idx & 7));
            }
#pragma unroll
            for (int it = 0; it < 4; ++it) {
                const int idx = tid + it * 128, r = idx >> 3;
                tile[r * 8 + ((idx & 7) ^ swz(r))] = v[it];
            }
        }
        __syncthreads();
    }
    if (!valid) return true;
    const int cp = tid >> 2, j = tid & 3;                          // channel pair, lane of the team
    const uint32_t* tw = reinterpret_cast<const uint32_t*>(tile);
    uint32_t wa[8], wb[8];                                         // channels 2 cp and 2 cp + 1, token pairs
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = 8 * (j + 4 * u) + 2 * i;
            uint32_t t0, t1;
            if constexpr (GENERAL) {
                t0 = __ldg(reinterpret_cast<const uint32_t*>(src + (long long)r * d) + cp);
                t1 = __ldg(reinterpret_cast<const uint32_t*>(src + (long long)(r + 1) * d) + cp);
            } else {
                const int pos = (((cp >> 2) ^ swz(r)) << 2) | (cp & 3);
                t0 = tw[r * 32 + pos];
                t1 = tw[(r + 1) * 32 + pos];
            }
            wa[4 * u + i] = __byte_perm(t0, t1, 0x5410);
            wb[4 * u + i] = __byte_perm(t0, t1, 0x7632);
        }
    bool done = true;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        uint32_t (&xw)[8] = c ? wb : wa;
        uint32_t nib[2], mw;
        if constexpr (GENERAL) quantize16_general<T, CODES>(xw, j, nib, mw);
        else done &= quantize16<T, CODES>(xw, j, nib, mw);
        const long long orow = bh * d + ch0 + 2 * cp + c;             // row of the transposed outputs
        uint4* dst = reinterpret_cast<uint4*>(img + orow * (long long)N + tok0) + j;
        dst[0] = make_uint4(xw[0], xw[1], xw[2], xw[3]);
        dst[4] = make_uint4(xw[4], xw[5], xw[6], xw[7]);
        if (CODES) {
            uint32_t* cw = reinterpret_cast<uint32_t*>(codes + orow * (N / 2) + tok0 / 2) + j;
            cw[0] = nib[0];
            cw[4] = nib[1];
            if (j == 0) meta[orow * (N / 64) + tok0 / 64] = mw;
        }
    }
    return done;
}

template <typename T, int UPT, bool CODES, bool QM, bool GENERAL>
__device__ __forceinline__ bool quantize_cta(const QuantJob& job, uint4* tiles)
{
    unsigned blk = blockIdx.x;
    if (blk < job.q_blocks + job.k_blocks) {
        const bool is_q = blk < job.q_blocks;
        if (!is_q) blk -= job.q_blocks;
        const unsigned head = blk / job.row_blocks_per_head;             // b * H + h
        const unsigned in_head = blk - head * job.row_blocks_per_head;
        if (is_q)
            return quantize_rows_cta<T, UPT, CODES, QM, GENERAL>(job.q, job.s, job.qmap.kv_of[head % (unsigned)job.Hq], head, in_head, job.N,
                                 job.d, job.q_codes, job.q_meta, job.q_img, job.q_mu, nullptr);
        return quantize_rows_cta<T, UPT, CODES, QM, GENERAL>(job.k, job.inv_s, (int)(head % (unsigned)job.Hkv), head, in_head, job.N, job.d,
                                 job.k_codes, job.k_meta, job.k_img, nullptr, job.k_sum);
    }
    blk -= job.q_blocks + job.k_blocks;
    const unsigned half = threadIdx.x >> 7, t = 2 * blk + half;
    const unsigned tok_blocks = job.N / 64, ch_blocks = job.d / 64;
    const unsigned tb = t % tok_blocks, rest = t / tok_blocks;
    const unsigned cb = rest % ch_blocks, bh = rest / ch_blocks;
    return quantize_tokens_half<T, CODES, GENERAL>(tiles + half * (64 * 8), t < job.v_tiles, job.v, bh, tb * 64, cb * 64, job.N, job.d,
                                                   job.v_codes, job.v_meta, job.v_img);
}

// Out of line, and from the inputs in global memory on, so that nothing of the usual path lives across it: a branch to the general
// form inside quantize16, even one that is never taken, costs 1 to 6 % (the shares of a thread no longer interleave), and an
// inlined second pass 2 to 8 % (spills at the 64 registers of four CTAs per SM).
template <typename T, int UPT, bool CODES, bool QM>
__device__ __noinline__ void requantize(const QuantJob& job)
{
    quantize_cta<T, UPT, CODES, QM, true>(job, nullptr);
}

template <typename T, int UPT, bool CODES, bool QM>
__global__ void __launch_bounds__(QUANT_THREADS, 4)
quantize_qkv_kernel(const __grid_constant__ QuantJob job)
{
    // a dependent grid launched with programmatic stream serialization (the attention kernel) may start
    // becoming resident as this grid's CTAs retire; it waits for this grid's completion before it reads.  This grid does the
    // same behind its predecessor (back-to-back calls: 44.2 -> 42.8 us at N = 8192, 30.6 -> 28.9 us for a whole d = 64 prefill)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __shared__ uint4 tiles[2 * 64 * 8];
    const bool done = quantize_cta<T, UPT, CODES, QM, false>(job, tiles);
    if (!__all_sync(0xffffffffu, done)) requantize<T, UPT, CODES, QM>(job);
}

// ------------------------------------------------------------------------------- launchers
cudaError_t launch_quantize_qkv(int dtype, const hifa4_shape& sh, const HeadMap& qmap, const void* q,
                                const void* k, const void* v, const float* s, const float* inv_s,
                                const hifa4_qkv& out, bool with_codes, cudaStream_t st)
{
    QuantJob job{};
    job.q = (const uint16_t*)q; job.k = (const uint16_t*)k; job.v = (const uint16_t*)v;
    job.s = s; job.inv_s = inv_s;
    job.q_codes = out.q_codes; job.k_codes = out.k_codes; job.v_codes = out.v_codes;
    job.q_meta = out.q_meta; job.k_meta = out.k_meta; job.v_meta = out.v_meta;
    job.q_img = (uint16_t*)out.q_mma; job.k_img = (uint16_t*)out.k_mma; job.v_img = (uint16_t*)out.v_mma;
    job.q_mu = out.q_mu; job.k_sum = out.k_sum;
    job.Hq = sh.Hq; job.Hkv = sh.Hkv; job.N = sh.N; job.d = sh.d;
    const long long head_shares = (long long)sh.N * sh.d / 16;
    const int upt = head_shares % (QUANT_THREADS * 2) == 0 ? 2 : 1;
    job.row_blocks_per_head = (unsigned)(head_shares / (QUANT_THREADS * upt));
    job.q_blocks = q ? (unsigned)sh.B * sh.Hq * job.row_blocks_per_head : 0u;
    job.k_blocks = k ? (unsigned)sh.B * sh.Hkv * job.row_blocks_per_head : 0u;
    job.v_tiles = v ? (unsigned)sh.B * sh.Hkv * (sh.N / 64) * (sh.d / 64) : 0u;
    const unsigned v_blocks = (job.v_tiles + 1) / 2;
    job.qmap = qmap;
    const unsigned long long total = (unsigned long long)job.q_blocks + job.k_blocks + v_blocks;
    if (total == 0) return cudaSuccess;
    if (total > 0x7FFFFFFFull) return cudaErrorInvalidConfiguration;
    const bool qm = out.q_mu != nullptr;
    auto pick = [&](auto t) {
        using T = decltype(t);
        auto by_upt = [&](auto codes, auto q_mean) {
            constexpr bool C = decltype(codes)::value, M = decltype(q_mean)::value;
            return upt == 2 ? quantize_qkv_kernel<T, 2, C, M> : quantize_qkv_kernel<T, 1, C, M>;
        };
        using Yes = std::true_type;
        using No = std::false_type;
        return with_codes ? (qm ? by_upt(Yes(), Yes()) : by_upt(Yes(), No())) : (qm ? by_upt(No(), Yes()) : by_upt(No(), No()));
    };
    auto kern = dtype == HIFA4_F16 ? pick(__half()) : pick(__nv_bfloat16());
    return launch_dependent(kern, (unsigned)total, QUANT_THREADS, 0, st, job);
}

}  // namespace hifa4
