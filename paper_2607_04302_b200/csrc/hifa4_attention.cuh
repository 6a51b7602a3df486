// Declarations shared by the attention kernels: launch arguments, the in-register HIF4 quantizer
// of P and the host-side TMA descriptor helper.
#pragma once
#include <cuda.h>
#include <type_traits>

#include "hifa4_internal.h"
#include "hifa4_device.cuh"
#include "hifa4_ptx.cuh"

namespace hifa4 {

using namespace ptx;

struct DebugReq {
    int n_blocks;
    int blocks[HIFA4_MAX_DEBUG_BLOCKS * 3];
    uint8_t* p_codes;
    float* p_step;
    float* l_out;
    float* m_out;
};

struct AttnArgs {
    int B, Hq, Hkv, N;
    int causal, out_dtype;
    int group_heads;              // CTA order: groups of this many (batch, query head) pairs, one group after the other
    int unit_heads, group_units;  // two-block kernel: query heads per unit (G, or 1 under a custom head map), units per group
    float c0, c1;                 // sigma, sigma * log2(e)
    uint64_t c1c1;                // {c1, c1}, the operand of packed instructions as it stands
    int normalizer;               // 1: l accumulates the unquantized P (mismatched), not P-hat
    unsigned long long* hist;     // mass-error histogram [n_bins + 2] or null
    int n_bins;
    double hist_lo, hist_inv_w;   // bin = floor((eps - lo) * inv_w)
    int p_f32;                    // keep P in FP32 before quantization (variant; default FP16)
    int qmean;                    // add mu_i * k_sum_j to the raw scores (Algorithm 1 line 6)
    const float* q_mu;            // [B,Hq,N]
    const float* k_sum;           // [B,Hkv,N]
    // kind::f8f6f4 experiment (Q K^T on E4M3 images of element x micro-exponent, one accumulator per 64-channel group)
    const void *q_f8, *k_f8;      // [B,H,N,d] bytes, else null
    const float *q_gs, *k_gs;     // [B,H,N,d/64] group scales S/4
    const void* q_raw;            // raw-Q launch (Q is quantized inside the kernel): the 16-bit Q [B,Hq,N,d], else null
    const float* q_scale;         // raw-Q launch: Smooth-QK factors of Q [Hkv,d] or null
    int in_dtype;                 // raw-Q launch: HIFA4_F16 or HIFA4_BF16
    void* out;
    int* d_status;
    HeadMap map;
    DebugReq dbg;
};

template <int D, int BC>
struct Cfg {
    static constexpr int BR = 128;
    static constexpr int KSUB = D / 64;                    // 64-channel sub-tiles of Q and K
    static constexpr int PSUB = BC / 64;                   // 64-key chunks of P and V^T
    static constexpr int Q_SUB_BYTES = BR * 128;
    static constexpr int K_SUB_BYTES = BC * 128;
    static constexpr int V_CHUNK_BYTES = (D + 16) * 128;   // D rows of V^T + 16 rows of ones
    static constexpr int P_SUB_BYTES = BR * 128;
    static constexpr int Q_OFF = 0;
    static constexpr int K_OFF = Q_OFF + KSUB * Q_SUB_BYTES;
    static constexpr int V_OFF = K_OFF + KSUB * K_SUB_BYTES;
    static constexpr int P_OFF = V_OFF + PSUB * V_CHUNK_BYTES;
    static constexpr int BAR_OFF = P_OFF + PSUB * P_SUB_BYTES;
    static constexpr int SMEM_BYTES = BAR_OFF + 64 + 1024;  // + alignment slack
    static constexpr int O_COLS = D + 16;
    static constexpr int S_COL = (D == 64) ? 128 : (D == 128 ? 256 : 384);
    static constexpr int TMEM_COLS = (D == 64) ? 256 : 512;
    static_assert(S_COL + BC <= TMEM_COLS, "tensor memory budget");
};

__device__ __forceinline__ float f16_round(float x) { return __half2float(__float2half_rn(x)); }

// Quantize NU*8 consecutive softmax weights of one 64-key HIF4 group (already rounded to FP16,
// held as floats, all >= 0) and return the BF16 image of P-hat as NU*4 packed words (element 2i
// in the low half of word i).  A is the maximum of the whole group (the caller combines partial
// maxima when a group is split over threads) and At[t] the maxima of this thread's 4-key
// subgroups.  Optionally dumps nibbles and subgroup steps.
//
// Arithmetic (all exact): the element code is m = RNE(p / step).  q = RZ(p * (1/step)) lands
// exactly on j + 1/2 for every tie (see e6m2_inv4), y = q + 1.5 * 2^23 rounds q to the nearest
// integer with ties to even, and fma(y, step, -1.5 * 2^23 * step) = m * step without rounding.
// The shift of a 4-key subgroup with maximum At is read off the float bit patterns:
// n - 1 = max((bits(At) - bits(1.75 S) - 1) >> 23, -1); the pair rule "level-2 bit = 1 iff
// max(need) = 2 or min(need) >= 1" is a = (n0 + n1 + 2) >> 2 and the shifts are max(n, a).
template <int NU>
__device__ __forceinline__ void quantize_p_units(const float (&p)[NU * 8], const float (&At)[NU * 2], float A,
                                                 uint32_t (&w)[NU * 4], uint8_t* dump_codes, float* dump_step,
                                                 float* sum_out = nullptr)
{
    if (sum_out) *sum_out = 0.f;
    if (A == 0.f) {
#pragma unroll
        for (int i = 0; i < NU * 4; ++i) w[i] = 0u;
        if (dump_codes) {
#pragma unroll
            for (int i = 0; i < NU / 2; ++i) reinterpret_cast<uint4*>(dump_codes)[i] = make_uint4(0, 0, 0, 0);
        }
        if (dump_step) {
#pragma unroll
            for (int i = 0; i < NU / 2; ++i) reinterpret_cast<float4*>(dump_step)[i] = make_float4(0, 0, 0, 0);
        }
        return;
    }
    const int code = e6m2_code_for_max(A);
    const float S = e6m2_value(code);
    const uint32_t inv4_bits = __float_as_uint(e6m2_inv4(code));
    const uint32_t s4_bits = __float_as_uint(S) - (2u << 23);              // S / 4
    const int t1 = (int)__float_as_uint(1.75f * S) + 1;
    const float MAGIC = 12582912.f;                                        // 1.5 * 2^23
#pragma unroll
    for (int u = 0; u < NU; ++u) {                   // one level-2 unit = 8 keys
        const int n0 = max(((int)__float_as_uint(At[2 * u]) - t1) >> 23, -1);       // need - 1
        const int n1 = max(((int)__float_as_uint(At[2 * u + 1]) - t1) >> 23, -1);
        const int a = (n0 + n1 + 4) >> 2;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int k = max((h ? n1 : n0) + 1, a);
            const float inv_step = __uint_as_float(inv4_bits - ((uint32_t)k << 23));
            const float step = __uint_as_float(s4_bits + ((uint32_t)k << 23));
            const float negc = -MAGIC * step;
            float v[4];
            uint32_t packed = 0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float y = __fadd_rn(__fmul_rz(p[8 * u + 4 * h + i], inv_step), MAGIC);
                v[i] = fmaf(y, step, negc);
                if (sum_out) *sum_out += v[i];            // exact: every term is a multiple of S/4, the sum < 2^11 of them
                if (dump_codes) packed |= (__float_as_uint(y) & 15u) << (8 * i);
            }
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[4 * u + 2 * h]) : "f"(v[1]), "f"(v[0]));
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(w[4 * u + 2 * h + 1]) : "f"(v[3]), "f"(v[2]));
            if (dump_step) dump_step[2 * u + h] = step;
            if (dump_codes) reinterpret_cast<uint32_t*>(dump_codes)[2 * u + h] = packed;
        }
    }
}

// Fused form of Algorithm 1 lines 9-10 for NU*8 consecutive keys of one 64-key group: takes the raw
// score accumulators (masked ones already -inf), forms P = exp2(acc * c1 - mL) rounded to FP16 and
// quantizes it unit by unit, so that the exponentials (MUFU pipe) and the quantizer arithmetic
// (ALU/FMA pipes) of a warp interleave.  A is the group maximum of P, which the caller gets from
// the group maximum of the accumulators through the same instruction sequence
// (p_of_score): that is exact because fma, ex2.approx (checked exhaustively over [-40, 0]) and
// the FP16 rounding are all monotone non-decreasing.
template <bool PF32 = false>
__device__ __forceinline__ float p_of_score(float acc, float c1, float mL)
{
    const float e = ex2_approx(fmaf(acc, c1, -mL));
    return PF32 ? e : f16_round(e);                    // PF32: the variant that keeps P in FP32
}

// Arithmetic of the fused form.  P is FP16, so the quantizer runs on packed FP16 pairs from the conversion on and
// hands over a packed BF16 image: no widening back to FP32, no repacking.  The softmax warps are bound by instruction
// issue and by the power the SM draws, and two factors with one product and one FMA per pair are the fewest instructions found: one
// reciprocal split into two constants (a product and an FMA per pair, then an addition; shift constants by five operations instead of
// three) takes 152 instead of 142 us at 32 / 8 heads, d = 128, causal, N = 4096, and 539 instead of 504 at N = 8192 (B200, back to
// back, two-block kernel before its waits by vote).  In units of S/2:
//   q = RN(p * c1)                  c1 * c2 = 2/S up to 7e-5, two FP16 factors per mantissa of S, c2 = 2, 1.40, 0.74, 0.74 (one FP16
//   y = fma(q, c2, 2^(9+k))         constant errs by 2^-12, which is not enough).  The factors are chosen so that the rounding of q lands on
//                                   the side of a rounding tie on which p lies, and for p on the tie on the side of the even
//                                   multiple: the FMA rounds p * 2/S to the nearest multiple of the subgroup's step, ties to
//                                   even, exactly.  The low bits of y are the element code m
//   v = fma_bf16(y, c, -n)          the bit pattern of y read as BF16 is 2^E (1 + m/128) with E known from k, so one BF16 FMA
//                                   with c = step * 128 * 2^-E, n = step * 128 gives m * step exactly
// (P exceeds 1 where the running maximum, an FP16 value, was rounded down: up to e^8 for scaled scores of 16384 to 32768.)
// Groups whose maximum is below 2^-12 move a factor 2^12 from c1 to c2: c1 stays finite.  The shift k of a 4-key subgroup
// is read off the bit pattern of its largest q: need = number of thresholds 1.75 S, 3.5 S that p exceeds, then
// k_t = max(need_t, need_other - 1) (that is the pair rule: the level-2 bit is set iff max(need) = 2 or min(need) >= 1,
// and a subgroup that needs no shift of its own still gets one when its partner needs two), which is the need of
// max(q_t, q_other / 2); the two subgroups of a unit share packed 16-bit integer operations, whose sum carries k straight
// into the exponent of the magic constant.  tests/test_p_quantizer_factors.py checks the scheme on every finite FP16 P
// under every scale a group maximum can select and every shift.
// The FP32-P variant keeps the FP32 form of the same scheme: q = RZ(p * (4/S)) (exactly on ties, see e6m2_inv4),
// y = q + 1.5 * 2^(23+k), v = fma(y, S/4, -magic*S/4), two elements per f32x2 operation.
template <bool PF32> struct PQuantConst;        // per (row, 64-key group, tile) constants of the fused quantizer
template <> struct PQuantConst<true> {
    uint64_t c1c1, nml, inv44, s44;
    uint32_t c0_bits, s4_bits;
    int tadd;
};
template <> struct PQuantConst<false> {
    uint64_t c1c1, nml;
    uint32_t f1, f2, tadd, n;                    // packed pairs of equal halves: c1, c2, threshold, -step * 128 at k = 0
    uint32_t s4_bits;                            // P-hat dump only
};

// Constants from the group maximum A of P.  A = 0 (every key masked) needs no branch: the scale stays finite, every p
// is 0 and every product below is an exact zero.
template <bool PF32>
__device__ __forceinline__ PQuantConst<PF32> p_quant_const(uint64_t c1c1, float mL, float A)
{
    PQuantConst<PF32> k;
    k.c1c1 = c1c1;
    k.nml = pack2(-mL, -mL);
    if constexpr (PF32) {
        const int code = e6m2_code_for_max(A);
        const float S = e6m2_value(code);
        const float inv4 = e6m2_inv4(code);
        const float S4 = __uint_as_float(__float_as_uint(S) - (2u << 23)); // S / 4
        k.tadd = (1 << 23) - ((int)__float_as_uint(1.75f * S) + 1);
        k.c0_bits = __float_as_uint(-12582912.f * S4);                     // -1.5 * 2^23 * S/4
        k.s4_bits = __float_as_uint(S4);
        k.inv44 = pack2(inv4, inv4);
        k.s44 = pack2(S4, S4);
    } else {
        // t: the upper bits of S, the smallest E6M2 value with 7 S >= A, as a float (exponent, two mantissa bits).  The constant
        // is below 1/7 by less than 2^-25: the product never exceeds S where A = 7 S, and A has 11 significant bits
        const uint32_t t = (__float_as_uint(fmaxf(A, 0x1p-24f) * __uint_as_float(0x3E124924u)) + 0x1FFFFFu) >> 21;
        const uint32_t sel = 0x1010u + 0x2222u * (t & 3u);                 // both halves = entry M of a table of four
        const uint32_t top = A < 0x1p-12f ? 0x30003000u : 0u;              // 2^12
        k.f1 = __byte_perm(0x3C923C00u, 0x3E303F38u, sel) + (127u - (t >> 2)) * 0x04000400u - top;
        k.f2 = __byte_perm(0x3D9A4000u, 0x39E939E9u, sel) + top;
        k.tadd = __byte_perm(0x22FF24FFu, 0x1F421F42u, sel) + top;         // 1023 - bits(RN(1.75 S c1)) + bits(512)
        k.n = t * 0x00200020u + 0x76807680u;                               // 0x8000 | bits(step * 128), - bits(512) >> 3
        k.s4_bits = (t << 21) - (2u << 23);
    }
    return k;
}

// P = exp2(acc * c1 - mL) for the 8 keys of unit u: FP16 pairs in natural order, or FP32 values (PF32).
template <int NU>
__device__ __forceinline__ void exp_unit(const float (&acc)[NU * 8], int u, const PQuantConst<false>& k, uint32_t (&p)[4])
{
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float t0, t1;
        unpack2(fma2(pack2(acc[8 * u + 2 * i], acc[8 * u + 2 * i + 1]), k.c1c1, k.nml), t0, t1);
        asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(p[i]) : "f"(ex2_approx(t1)), "f"(ex2_approx(t0)));
    }
}
template <int NU>
__device__ __forceinline__ void exp_unit(const float (&acc)[NU * 8], int u, const PQuantConst<true>& k, float (&p)[8])
{
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
        float t0, t1;
        unpack2(fma2(pack2(acc[8 * u + i], acc[8 * u + i + 1]), k.c1c1, k.nml), t0, t1);
        p[i] = ex2_approx(t0);
        p[i + 1] = ex2_approx(t1);
    }
}

// One level-2 unit: P -> P-hat image words w[0..3]; codes / ks0, ks1: the element codes and k << 23 for the dump.
__device__ __forceinline__ void quantize_unit(const uint32_t (&p)[4], const PQuantConst<false>& k, uint32_t (&w)[4],
                                              uint32_t (&codes)[2], int& ks0, int& ks1)
{
    uint32_t q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = h2_mul(p[i], k.f1);
    const uint32_t a = h2_max(q[0], q[1]), b = h2_max(q[2], q[3]);
    const uint32_t At = h2_max(__byte_perm(a, b, 0x5410), __byte_perm(a, b, 0x7632));     // {subgroup 0, subgroup 1}
    const uint32_t Bt = __viaddmax_s16x2(__byte_perm(At, At, 0x1032), 0xFC00FC00u, At);   // max(A_t, A_other / 2)
    const uint32_t x = __viaddmax_s16x2(Bt, k.tadd, 0x60006000u);                          // bits(512 * 2^k) + fraction
    const uint32_t magic = x & 0xFC00FC00u;                                                // 512 * 2^k
    const uint32_t n = k.n + (magic >> 3);                                                 // -step * 128 (+ k << 7)
    const uint32_t c = n - magic - 0x40804080u;                                            // step * 128 * 2^-E, E = 65 + 8 k
    const uint32_t magic0 = dup_lo(magic), magic1 = dup_hi(magic);
    uint32_t y[4];
    y[0] = h2_fma(q[0], k.f2, magic0);
    y[1] = h2_fma(q[1], k.f2, magic0);
    y[2] = h2_fma(q[2], k.f2, magic1);
    y[3] = h2_fma(q[3], k.f2, magic1);
    w[0] = bf2_fma(y[0], dup_lo(c), dup_lo(n));
    w[1] = bf2_fma(y[1], dup_lo(c), dup_lo(n));
    w[2] = bf2_fma(y[2], dup_hi(c), dup_hi(n));
    w[3] = bf2_fma(y[3], dup_hi(c), dup_hi(n));
    codes[0] = __byte_perm(y[0], y[1], 0x6420) & 0x0F0F0F0Fu;
    codes[1] = __byte_perm(y[2], y[3], 0x6420) & 0x0F0F0F0Fu;
    ks0 = (int)(((magic - 0x60006000u) & 0xFFFFu) << 13);
    ks1 = (int)(((magic - 0x60006000u) >> 16) << 13);
}
// The packed operations pair key i of subgroup 0 with key i of subgroup 1, so that one pair of per-subgroup constants
// (magic, c) serves four packed operations.  On bit patterns, with x_t = max(bits(At_t) + tadd, 0) = need_t * 2^23 +
// fraction: k_t * 2^23 = max(x_t, x_other - 2^23) with the fraction masked off.
__device__ __forceinline__ void quantize_unit(const float (&p)[8], const PQuantConst<true>& k, uint32_t (&w)[4],
                                              uint32_t (&codes)[2], int& ks0, int& ks1)
{
    const int MAGIC_BITS = 0x4B400000;                                    // 1.5 * 2^23
    const float At0 = fmaxf(max3(p[0], p[1], p[2]), p[3]);
    const float At1 = fmaxf(max3(p[4], p[5], p[6]), p[7]);
    const int x0 = max((int)__float_as_uint(At0) + k.tadd, 0);
    const int x1 = max((int)__float_as_uint(At1) + k.tadd, 0);
    ks0 = max(x0, x1 - (1 << 23)) & (int)0xFF800000;
    ks1 = max(x1, x0 - (1 << 23)) & (int)0xFF800000;
    const uint64_t mm = pack2(__int_as_float(MAGIC_BITS + ks0), __int_as_float(MAGIC_BITS + ks1));
    const uint64_t cc = pack2(__int_as_float((int)k.c0_bits + ks0), __int_as_float((int)k.c0_bits + ks1));
    float v[8], c[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint64_t y = add2(mul2_rz(pack2(p[i], p[4 + i]), k.inv44), mm);
        unpack2(fma2(y, k.s44, cc), v[i], v[4 + i]);
        unpack2(y, c[i], c[4 + i]);
    }
    // BF16 image: every value has at most 8 significant bits, so the upper halves of the FP32 patterns
    // are the BF16 values (a byte permute instead of a conversion)
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __byte_perm(__float_as_uint(v[2 * i]), __float_as_uint(v[2 * i + 1]), 0x7632);
#pragma unroll
    for (int h = 0; h < 2; ++h)
        codes[h] = (__float_as_uint(c[4 * h]) & 15u) | ((__float_as_uint(c[4 * h + 1]) & 15u) << 8) |
                   ((__float_as_uint(c[4 * h + 2]) & 15u) << 16) | ((__float_as_uint(c[4 * h + 3]) & 15u) << 24);
}

// Units U0..U1-1 of a thread's NU units: acc -> P -> P-hat image words w[4u..4u+3].
// The exponentials of unit u+1 are issued before unit u is quantized, so that the MUFU latency of
// one unit hides behind the ALU/FMA work of the previous one.
template <int NU, int U0, int U1, bool DBG, bool PF32 = false>
__device__ __forceinline__ void exp_quantize_units(const float (&acc)[NU * 8], const PQuantConst<PF32>& k, bool zero_group,
                                                   uint32_t (&w)[NU * 4], uint8_t* dump_codes, float* dump_step)
{
    using P8 = std::conditional_t<PF32, float[8], uint32_t[4]>;
    P8 pn;
    exp_unit<NU>(acc, U0, k, pn);
#pragma unroll
    for (int u = U0; u < U1; ++u) {
        P8 p;
#pragma unroll
        for (int i = 0; i < (PF32 ? 8 : 4); ++i) p[i] = pn[i];
        if (u + 1 < U1) exp_unit<NU>(acc, u + 1, k, pn);
        uint32_t wu[4], codes[2];
        int ks0, ks1;
        quantize_unit(p, k, wu, codes, ks0, ks1);
#pragma unroll
        for (int i = 0; i < 4; ++i) w[4 * u + i] = wu[i];
        if (DBG) {
            if (dump_step) {
                dump_step[2 * u] = zero_group ? 0.f : __int_as_float((int)k.s4_bits + ks0);
                dump_step[2 * u + 1] = zero_group ? 0.f : __int_as_float((int)k.s4_bits + ks1);
            }
            if (dump_codes) {
                reinterpret_cast<uint32_t*>(dump_codes)[2 * u] = codes[0];
                reinterpret_cast<uint32_t*>(dump_codes)[2 * u + 1] = codes[1];
            }
        }
    }
}

// Maximum of 64 values in 31 three-input maxima and one of two: seven chains of nine, then their results and the last value.
__device__ __forceinline__ float max64(const float (&p)[64])
{
    float t[8];
#pragma unroll
    for (int c = 0; c < 7; ++c) {
        t[c] = max3(p[9 * c], p[9 * c + 1], p[9 * c + 2]);
        t[c] = max3(t[c], p[9 * c + 3], p[9 * c + 4]);
        t[c] = max3(t[c], p[9 * c + 5], p[9 * c + 6]);
        t[c] = max3(t[c], p[9 * c + 7], p[9 * c + 8]);
    }
    t[7] = p[63];
    const float mx = max3(max3(t[0], t[1], t[2]), t[3], t[4]);
    return fmaxf(max3(mx, t[5], t[6]), t[7]);
}

// Rescale of a row's history: the D channels and the normaliser column of [O | l] at tensor-memory address t_o times
// rsc, 64 columns per round trip (the other columns of the ones block are never read).  The caller waits for the stores.
// Unrolled only for d = 256 (one CTA per SM, registers to spare: 540 -> 518 us at N = 8192, 16 heads); at the 96 registers of
// the d = 128 kernels ptxas would overlap two round trips and spill (80 to 120 bytes of reloads per tile: 34.9 against
// 32.9 us for 8 heads, B = 2, N = 2048).
template <int D>
__device__ __forceinline__ void rescale_columns(uint32_t t_o, float rsc)
{
    const uint64_t rr = pack2(rsc, rsc);
    auto scale32 = [&](uint32_t (&r)[32]) {
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
            float x0, x1;
            unpack2(mul2(pack2(__uint_as_float(r[i]), __uint_as_float(r[i + 1])), rr), x0, x1);
            r[i] = __float_as_uint(x0);
            r[i + 1] = __float_as_uint(x1);
        }
    };
    uint32_t rl[1];
    tmem_ld1(t_o + D, rl);
#pragma unroll (D > 128 ? D / 64 : 1)
    for (int cc = 0; cc < D / 64; ++cc) {
        uint32_t r0[32], r1[32];
        tmem_ld32(t_o + cc * 64, r0);
        tmem_ld32(t_o + cc * 64 + 32, r1);
        tmem_wait_ld();
        scale32(r0);
        tmem_st32(t_o + cc * 64, r0);
        scale32(r1);
        tmem_st32(t_o + cc * 64 + 32, r1);
    }
    rl[0] = __float_as_uint(__uint_as_float(rl[0]) * rsc);
    tmem_st1(t_o + D, rl);
}

// A warp stores 64 bytes of each of its 32 rows (lane = row, 16 words each): through a swizzled 2 KB tile of shared
// memory, so that a store instruction covers whole 64-byte pieces of 8 rows.  Rows at or past `rows` are not written.
__device__ __forceinline__ void store_rows64(uint32_t stage, const uint32_t (&w)[16], uint8_t* dst, size_t row_bytes,
                                             int rows, int lane)
{
#pragma unroll
    for (int c = 0; c < 4; ++c)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                     ::"r"(stage + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4)), "r"(w[4 * c]), "r"(w[4 * c + 1]), "r"(w[4 * c + 2]),
                       "r"(w[4 * c + 3]) : "memory");
    __syncwarp();
    const int c = lane & 3;
#pragma unroll
    for (int it = 0; it < 4; ++it) {
        const int r = it * 8 + (lane >> 2);
        uint4 v;
        asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(stage + r * 64 + ((c ^ ((r >> 1) & 3)) << 4)));
        if (r < rows) *reinterpret_cast<uint4*>(dst + (size_t)r * row_bytes + c * 16) = v;
    }
    __syncwarp();
}

// Whole 64-key group held by one thread; the image goes to row `row` of a 128-byte-swizzled
// shared-memory tile (the layout a K-major tcgen05 operand descriptor with SWIZZLE_128B reads).
__device__ __forceinline__ void quantize_p64(const float (&p)[64], uint32_t p_sub_base, int row,
                                             uint8_t* dump_codes, float* dump_step, float* sum_out = nullptr)
{
    float At[16];
#pragma unroll
    for (int t = 0; t < 16; ++t) At[t] = fmaxf(max3(p[4 * t], p[4 * t + 1], p[4 * t + 2]), p[4 * t + 3]);
    float A4[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) A4[t] = fmaxf(max3(At[4 * t], At[4 * t + 1], At[4 * t + 2]), At[4 * t + 3]);
    const float A = fmaxf(max3(A4[0], A4[1], A4[2]), A4[3]);
    uint32_t w[32];
    quantize_p_units<8>(p, At, A, w, dump_codes, dump_step, sum_out);
    const uint32_t row_base = p_sub_base + (row >> 3) * 1024 + (row & 7) * 128;
    const int sw = row & 7;
#pragma unroll
    for (int u = 0; u < 8; ++u)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                     ::"r"(row_base + ((u ^ sw) << 4)), "r"(w[4 * u]), "r"(w[4 * u + 1]), "r"(w[4 * u + 2]), "r"(w[4 * u + 3]) : "memory");
}

// BF16 tensor [heads][rows][cols] (cols contiguous), box [1][box_rows][64 cols], 128-byte swizzle,
// out-of-range elements read as zero.  Returns false if the driver entry point is unavailable or
// the encode fails.
bool make_bf16_map(CUtensorMap* m, void* base, uint64_t heads, uint64_t rows, uint64_t cols, uint32_t box_rows);

// Warp-specialised kernel for d = 128, Bc = 128 (hifa4_attention_ws.cu).
int launch_attention_ws(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st);

// Warp-specialised kernels for Bc = 64, d = 64, 128 or 256 (hifa4_attention_ws64.cu).
int launch_attention_ws64(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st);
// The same with two query blocks per CTA that share the K / V tiles, d = 128 (hifa4_attention_pair.cu).
int launch_attention_pair(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, int Bc, cudaStream_t st);
// The same on pairs of SMs, d = 256 (hifa4_attention_cta2.cu).
bool attention_cta2_pays(const hifa4_shape& sh, const hifa4_attn_params& prm, int unit_heads);
int launch_attention_cta2(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st);
// Self-test instantiations (d = 128, Bc = 64): one bounded wait is made to run out (see hifa4_selftest_wait_timeout).
int launch_attention_pair_selftest(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st);
int launch_attention_ws64_selftest(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st);

}  // namespace hifa4
