// Warp-specialised HiFA4 attention forward for Bc = 64 or 128, d = 128 (Algorithm 1 lines 4-13) with two 128-row query blocks per
// CTA that share the K and V^T tiles.
//
// The two blocks ("halves") belong to query heads of one KV head, so every K and V^T tile is loaded once for 256
// query rows instead of once for 128: with one block per CTA and two CTAs per SM the tiles cross L2 -> SM at 9 TB/s,
// and leaving those loads out altogether made long launches of that kernel 13-16 % shorter (the clocks of long launches follow
// the power they draw).  Against the 64-key kernel (sustained, us; two-block against 64-key): 32 / 32 heads, causal, N = 4096 157 against
// 168, N = 8192 whole calls 580 against 606; not causal N = 8192, 2048 blocks 1016 against 1064.  It executes 10.3 instructions per 32
// scores; of its 132 us at N = 4096 (32 / 8 heads, BF16 output) the quantizer of P with two factors, which all attention kernels
// share, saved 10 and the waits by vote with the P V issuer's look-ahead, which only this kernel has, another 10.
// hifa4_dispatch.h says when it is taken.  d = 64 stays with the 64-key kernel (350 against 380 us, 12 / 4 heads, B = 2, N = 8192,
// both with an earlier quantizer: its tiles are half as large and its softmax share twice).  Apart from the
// shared tiles the halves run independently of one another, each as the 64-key kernel (hifa4_attention_ws64.cu) runs a
// CTA.  Warps:
//   0-15   softmax / quantize: warps 8h..8h+3 own the even key tiles of half h, warps 8h+4..8h+7 the odd ones, one
//          thread per query row and tile
//   16     one thread: work list, TMA loads of the K and V^T tiles (three-stage rings)
//   17, 18 one thread each: TMA load of the half's Q, issuer of its S = Q K^T
//   19     one thread: issuer of [O | l] += P-hat [V | 1] of both halves, whichever is ready
// (five warps per scheduler partition, 20 in all, leave 96 registers per thread; six would leave 80)
// One CTA per SM, persistent: the grid has one CTA per pair of blocks, and a running CTA takes over the next pending
// one with cluster launch control (heaviest first, in grid order) while its last tiles are in flight, so that loads,
// the first S and the set-up of the next pair run under the epilogue of the current one.  Tiles are numbered through
// all pairs of a CTA (t per half, c for the tiles loaded); barrier phases follow those numbers.
// Tensor memory, per half: [O | l] d+16 columns, S 64, P-hat 32 (2 x 240 of 512 columns at d = 128).  Output goes
// through 2 KB of shared memory per warp, so that stores cover whole 64-byte row pieces.
// Template flags: Q-Mean (key sums staged in eight slots by the loader, as in the 64-key kernel); B128: 128-key tiles, each a
// pair of 64-key ones whose owners exchange their maxima (one more hand-off per tile, one rescale less).  Against the
// 128-key kernel (hifa4_attention_ws.cu): 32 / 8 heads, causal, whole calls with an earlier quantizer, N = 4096 191 against 213 us, N =
// 8192 637 against 722; causal, N = 1024, 576 blocks 37.0 against 42.5.
// Every wait is bounded (see hifa4_attention_ws.cu for the failure protocol).
#include "hifa4_attention.cuh"
#include "hifa4_dispatch.h"

namespace hifa4 {

struct PairCfg {
    static constexpr int D = 128, BC = 64, STAGES = 3;
    static constexpr int NSW = 16, W_LD = 16, W_QK = 17, W_PV = 19, THREADS = 20 * 32;
    static constexpr int NU = BC / 8, QSUB = D / 64;
    static constexpr int Q_HALF = QSUB * 16384;
    static constexpr int K_SUB = BC * 128, K_STAGE = QSUB * K_SUB;
    static constexpr int V_STAGE = (D + 16) * 128;          // D rows of V^T + 16 rows of ones, 64 keys wide
    static constexpr int K_OFF = 2 * Q_HALF;
    static constexpr int V_OFF = K_OFF + STAGES * K_STAGE;
    static constexpr int STG_OFF = V_OFF + STAGES * V_STAGE;   // output staging, 2 KB per softmax warp
    static constexpr int MX_OFF = STG_OFF + NSW * 2048;     // running maxima handed from tile t to t+1: [half][t % 2][128] floats;
                                                            // 128-key tiles: maxima of the halves of a tile, [half][t % 4][128]
    static constexpr int KSUM_OFF = MX_OFF + 2 * 4 * 512;   // Q-Mean: channel sums of a tile's 64 keys, slot = tile % 8
    static constexpr int MISC_OFF = KSUM_OFF + 8 * 256;
    static constexpr int SMEM_BYTES = MISC_OFF + 1024 + 1024;
    static constexpr int O_COLS = D + 16;
    static constexpr int S_COL = O_COLS, P_COL = S_COL + 64, H_COLS = O_COLS + 96, TMEM_COLS = 512;
    static_assert(2 * H_COLS <= TMEM_COLS && SMEM_BYTES <= 227 * 1024, "tensor memory or shared memory budget");
    static_assert(MX_OFF % 1024 == 0 && MISC_OFF % 16 == 0, "addresses below are formed with xor");
};

namespace pairk {
// Per half (HALF barriers each, half 1 after half 0): QF Q landed, QD last S of the pair complete (Q may be replaced), SFR
// S buffer free (4 arrivals), SF[t % 2] S complete, PGO P-hat stored and history rescaled (4), PV[t % 2] P V complete,
// MR[t % 2] (128-key tiles: t % 4) maxima published (4), OE output columns read (8).  Ring (index = stage): KF / VF tile landed, KE / VE
// tile read by both halves.  WF / WE[pair % 2]: work record written / read by all (20); CL: answer of the launch control;
// KSF[tile % 8]; AB, per half: its softmax warps have come to a pair without a block for it (8, Q-Mean only).  SF, PV and MR
// come in twos because each group of softmax warps sees every second tile only: a parity wait must not be two phases behind.
enum { QF = 0, QD = 1, SFR = 2, PGO = 3, SF = 4, PV = 6, MR = 8, OE = 12, HALF = 16,
       KF = 32, KE = 35, VF = 38, VE = 41, WF = 44, WE = 46, CL = 48, KSF = 49, AB = 57, N_BARS = 59 };
constexpr uint32_t WAIT_POLLS = 1u << 18;            // a poll may keep the thread suspended for up to about 4 us
struct Work {                         // one pair of query blocks
    int n_max;                        // key tiles to load; 0: no more work
    int bh_kv;
    int n[2];                         // key tiles of the halves (0: no block)
    int q0[2], bh_q[2];
};
}  // namespace pairk

static __device__ __forceinline__ uint64_t fma2_here(uint64_t a, uint64_t b, uint64_t c)      // stays between the loads around it
{
    uint64_t r;
    asm volatile("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
static __device__ __forceinline__ int ld_flag(uint32_t addr)
{
    int v;
    asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
static __device__ __forceinline__ void st_flag(uint32_t addr, int v)
{
    asm volatile("st.volatile.shared.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
static __device__ __forceinline__ bool wait_pair(uint32_t bar, uint32_t parity, uint32_t abort_flag)
{
#pragma unroll 1
    for (uint32_t i = 0; i < pairk::WAIT_POLLS; ++i) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 63u && ld_flag(abort_flag)) return false;
    }
    return false;
}
// The same for a whole warp.  The verdict is a vote: the warp stays together where a wait fails, and the compiler knows it, keeps
// the loop state in uniform registers and no reconvergence state; a waiting warp issues one instruction per poll instead of a
// loop's worth.
static __device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, uint32_t abort_flag)
{
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
#pragma unroll 1
    for (uint32_t i = 0; i < pairk::WAIT_POLLS / 4; ++i) {
        if (__all_sync(0xffffffffu, mbar_try_wait4(bar, parity))) return true;
        if ((i & 15u) == 15u && __any_sync(0xffffffffu, ld_flag(abort_flag))) return false;
    }
    return false;
}
// The same where the warps wait longest, for P V and, with 128-key tiles, for the other half's maxima: each thread polls in the
// plain loop and the vote comes once at the end (32 / 8 heads, N = 4096, causal, 134.4 against 135.3 us).
static __device__ __forceinline__ bool wait_long(uint32_t bar, uint32_t parity, uint32_t abort_flag)
{
    return __all_sync(0xffffffffu, wait_pair(bar, parity, abort_flag));
}
static __device__ __forceinline__ int uni(int v) { return __shfl_sync(0xffffffffu, v, 0); }      // the same in all lanes, and the compiler knows
static __device__ __forceinline__ void arrive0(uint32_t bar, int lane)      // one arrival from lane 0 of a converged warp
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.eq.s32 p, %1, 0;\n\t"
                 "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
                 ::"r"(bar), "r"(lane) : "memory");
}
// Ask for the next pending CTA of this grid; the 16-byte answer lands at `dst` and completes on `bar`.
static __device__ __forceinline__ void launch_control_ask(uint32_t dst, uint32_t bar)
{
    fence_proxy_async_smem();
    mbar_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(dst), "r"(bar) : "memory");
}
static __device__ __forceinline__ int launch_control_answer(uint32_t src)   // blockIdx.x of the CTA taken over, or -1
{
    uint32_t got, x;
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b128 a;\n\t"
                 "ld.shared.b128 a, [%2];\n\t"
                 "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, a;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t"
                 "mov.u32 %1, 0;\n\t"
                 "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %1, a;\n\t}"
                 : "=r"(got), "=r"(x) : "r"(src) : "memory");
    return got ? (int)x : -1;
}

// SELFTEST: as in the 64-key kernel, the instantiation whose wait for P V runs out.  The softmax warps withhold the arrivals that
// release P V; a CTA takes one pair only and two tiles of it at most, and the issuer first waits, with the full limit, until their
// loads have landed, their S = Q K^T are complete and the launch control has answered: when its 2^6 polls begin, nothing is in
// flight.  The softmax warps then leave through the abort exits of wait_warp and wait_long, the issuers of S through theirs.
template <bool QM, bool B128, bool SELFTEST = false>
__global__ void __launch_bounds__(PairCfg::THREADS, 1)
attention_fwd_pair_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                          const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ AttnArgs args)
{
    using namespace pairk;
    using C = PairCfg;
    constexpr int D = C::D, BC = C::BC, STAGES = C::STAGES, NU = C::NU, O_COLS = C::O_COLS;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t k_s = smem_base + C::K_OFF, v_s = smem_base + C::V_OFF, bars = smem_base + C::MISC_OFF;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + C::MISC_OFF + 8 * N_BARS);
    const uint32_t abort_flag = bars + 8 * N_BARS + 8;
    constexpr int CL_OFF = C::MISC_OFF + 512;                 // answer of the launch control (16-byte aligned)
    volatile Work* work = reinterpret_cast<volatile Work*>(smem_gen + C::MISC_OFF + 544);    // [2]

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int N = args.N;

    if (warp == C::W_LD && lane == 0) {
        // A CTA that starts after another one reported a failure does nothing: one thread reads the status word and
        // publishes the verdict, so that all roles agree on it.
        int status_now = args.d_status ? *reinterpret_cast<volatile int*>(args.d_status) : 0;
        tma_prefetch_desc(&tmap_q); tma_prefetch_desc(&tmap_k); tma_prefetch_desc(&tmap_v);
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(bar(KF + s), 1); mbar_init(bar(KE + s), 2);
            mbar_init(bar(VF + s), 1); mbar_init(bar(VE + s), 2);
        }
        for (int h = 0; h < 2; ++h) {
            const int b = h * HALF;
            mbar_init(bar(b + QF), 1); mbar_init(bar(b + QD), 1); mbar_init(bar(b + SFR), 4); mbar_init(bar(b + PGO), 4);
            for (int s = 0; s < 2; ++s) {
                mbar_init(bar(b + SF + s), 1); mbar_init(bar(b + PV + s), 1);
            }
            for (int s = 0; s < 4; ++s) mbar_init(bar(b + MR + s), 4);
            mbar_init(bar(b + OE), 8);
            mbar_init(bar(WF + h), 1); mbar_init(bar(WE + h), 20); mbar_init(bar(AB + h), 8);
        }
        mbar_init(bar(CL), 1);
        for (int s = 0; s < 8; ++s) mbar_init(bar(KSF + s), 1);
        fence_barrier_init();
        // nothing the preceding kernel of the stream wrote is touched before this point (programmatic launch)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (status_now != 0) status_now = *reinterpret_cast<volatile int*>(args.d_status);
        st_flag(abort_flag, status_now != 0 ? 2 : 0);
    }
    if (warp == C::W_LD) { __syncwarp(); tmem_alloc(smem_u32((const void*)tmem_slot), C::TMEM_COLS); tmem_relinquish(); }
    for (int i = tid; i < STAGES * 128; i += C::THREADS) {        // ones rows under every V^T stage
        const int st = i / 128, off = (i % 128) * 16;
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};"
                     ::"r"(v_s + st * C::V_STAGE + D * 128 + off), "r"(0x3F803F80u) : "memory");
    }
    fence_proxy_async_smem();
    tc_fence_before();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    const bool dead = ld_flag(abort_flag) != 0;

    auto fail = [&](int site) {
        st_flag(abort_flag, 1);
        if (args.d_status) atomicCAS(args.d_status, 0, HIFA4_ERR_TIMEOUT + 16 * site);
    };

    if (dead) {
        // fall through to the common exit
    } else if (warp == C::W_LD) {
        // ------------------------------------------------------------------ work list, K and V^T loads
        if (elect_one()) {
            // Order of the pairs: units (KV heads with their G query heads; single query heads under a custom head map) in
            // groups whose K / V images fit in L2 together; inside a group the position in the unit's list of blocks is
            // outermost, and that list runs from the last query block (the heaviest under a causal mask) to the first, all
            // heads of the unit for each block.
            const int G = args.unit_heads, n_qt = (N + 127) / 128, Hu = args.Hq / G;
            const int blocks = n_qt * G, pairs = (blocks + 1) >> 1, gu = args.group_units;
            int stk = 0, stv = 0, c = 0;                      // ring stages, tile count
            uint32_t phk = 1, phv = 1;                        // parity that the "empty" waits use: the first round passes
            int idx = (int)blockIdx.x;
            for (int it = 0;; ++it) {
                if (it >= 2 && !wait_pair(bar(WE + (it & 1)), (uint32_t)((it >> 1) - 1) & 1u, abort_flag)) { fail(16); break; }
                volatile Work& w = work[it & 1];
                int n_max = 0, bh_kv = 0;
                if (idx >= 0) {
                    const int grp_i = idx / (pairs * gu), in_grp = idx - grp_i * (pairs * gu);
                    const int p = in_grp / gu, unit = grp_i * gu + (in_grp - p * gu);
                    const int b = unit / Hu, h0 = (unit - b * Hu) * G;
                    bh_kv = b * args.Hkv + args.map.kv_of[h0];
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf) {
                        const int r = 2 * p + hf, qi = r / G, q0 = (n_qt - 1 - qi) * 128;
                        const int last_key = args.causal ? min(q0 + 127, N - 1) : N - 1;
                        int n = r >= blocks ? 0 : B128 ? 2 * (last_key / 128 + 1) : last_key / BC + 1;
                        if (SELFTEST) n = min(n, 2);
                        w.n[hf] = n;
                        w.q0[hf] = q0;
                        w.bh_q[hf] = b * args.Hq + h0 + (r - qi * G);
                        n_max = max(n_max, n);
                    }
                }
                w.n_max = n_max;
                w.bh_kv = bh_kv;
                mbar_arrive(bar(WF + (it & 1)));
                if (idx < 0) break;
                // K and V^T stages become free at different times (S runs a tile or two ahead of P V, and a half may lag the
                // other): the two rings are refilled independently of one another
                int jk = 0, jv = 0;
                uint32_t idle = 0;
                bool ok = true;
                while (jv < n_max) {
                    if (++idle > 4 * WAIT_POLLS || ((idle & 63u) == 63u && ld_flag(abort_flag))) {
                        if (idle > 4 * WAIT_POLLS) fail(1);
                        ok = false;
                        break;
                    }
                    if (jk < n_max && mbar_test_wait(bar(KE + stk), phk)) {
                        idle = 0;
                        mbar_expect_tx(bar(KF + stk), C::K_STAGE);
#pragma unroll
                        for (int s = 0; s < C::QSUB; ++s)
                            tma_load_3d(k_s + stk * C::K_STAGE + s * C::K_SUB, &tmap_k, bar(KF + stk), 64 * s, jk * BC, bh_kv);
                        if (QM) {
                            // slot c % 8 held the sums of tile c-8: this load follows S(c-3) of both halves, hence their pull
                            // of S(c-4) by the warps that read the slot during tile c-8 or by warps that waited for them since;
                            // a half without a block frees the pair's tiles only after its warps have come to that pair
                            // (tests/test_pair_keysum_order.py).  (B128: a tile may lie past the last key; its scores are masked
                            // whatever is added to them)
                            const int key = B128 ? min(jk * BC, N - BC) : jk * BC;
                            mbar_expect_tx(bar(KSF + (c & 7)), 256);
                            bulk_load(smem_base + C::KSUM_OFF + (c & 7) * 256, args.k_sum + (size_t)bh_kv * N + key, 256, bar(KSF + (c & 7)));
                            ++c;
                        }
                        if (jk == max(n_max - 3, 0)) launch_control_ask(smem_base + CL_OFF, bar(CL));
                        ++jk;
                        if (++stk == STAGES) { stk = 0; phk ^= 1u; }
                    }
                    if (jv < jk && mbar_test_wait(bar(VE + stv), phv)) {
                        idle = 0;
                        mbar_expect_tx(bar(VF + stv), D * 128);
                        tma_load_3d(v_s + stv * C::V_STAGE, &tmap_v, bar(VF + stv), jv * BC, 0, bh_kv);
                        ++jv;
                        if (++stv == STAGES) { stv = 0; phv ^= 1u; }
                    }
                }
                if (!ok) break;
                if (!wait_pair(bar(CL), (uint32_t)it & 1u, abort_flag)) { fail(17); break; }
                if (SELFTEST) break;
                idx = launch_control_answer(smem_base + CL_OFF);
            }
        }
    } else if (warp < C::NSW) {
        // ------------------------------------------------------------------ softmax / quantize
        const int hf = warp >> 3, grp = (warp >> 2) & 1, quarter = warp & 3;
        const int r_loc = quarter * 32 + lane;                    // row inside the block = TMEM lane
        const uint32_t t_o = tmem + ((uint32_t)(quarter * 32) << 16) + hf * C::H_COLS;   // [O | l], then S, then P-hat
        const float LOG2E = 1.4426950408889634f;
        const uint32_t mx_own = smem_base + C::MX_OFF + hf * 2048 + grp * 512 + r_loc * 4;
        const uint32_t b_h = bar(hf * HALF), b_own = b_h + 8 * grp, b_oth = b_own ^ 8;   // (b_h is a multiple of 16)
        int t0 = 0;                                               // tiles of this half before the current pair
        int c0 = 0;                                               // tiles loaded before the current pair
        bool ok = true;
        for (int it = 0; ok; ++it) {
            if (!wait_warp(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(18); break; }
            volatile Work& w = work[it & 1];
            const int n_max = uni(w.n_max);
            if (n_max == 0) break;
            const int n_tiles = uni(w.n[hf]), q0 = uni(w.q0[hf]);
            if (QM && n_tiles == 0) arrive0(bar(AB + hf), lane);
            const int row = q0 + r_loc;
            float m_run = -INFINITY;
            const float mu_row = (QM && n_tiles > 0 && row < N) ? args.q_mu[(size_t)w.bh_q[hf] * N + row] : 0.f;

            for (int jt = (t0 ^ grp) & 1; jt < n_tiles; jt += 2) {
                const int t = t0 + jt, j0 = jt * BC;               // t % 2 == grp
                const uint32_t ph = (uint32_t)(t >> 1) & 1u, ph_prev = (uint32_t)((t - 1) >> 1) & 1u;
                if (!wait_warp(b_own + 8 * SF, ph, abort_flag)) { fail(8); ok = false; break; }
                tc_fence_after();
                float p[BC];
                {
                    uint32_t r[BC];
                    tmem_ld32(t_o + C::S_COL, reinterpret_cast<uint32_t(&)[32]>(r[0]));
                    tmem_ld32(t_o + C::S_COL + 32, reinterpret_cast<uint32_t(&)[32]>(r[32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < BC; ++i) p[i] = __uint_as_float(r[i]);
                }
                tc_fence_before();                                 // S(t) is in registers: S(t+1) may overwrite it
                __syncwarp();
                arrive0(b_h + 8 * SFR, lane);

                if (QM) {                                          // Q-Mean correction (line 6): + mu_i * sum_c k~_jc
                    const int c = c0 + jt;
                    if (!wait_warp(bar(KSF + (c & 7)), (uint32_t)(c >> 3) & 1u, abort_flag)) { fail(15); ok = false; break; }
                    const uint32_t ks_s = smem_base + C::KSUM_OFF + (c & 7) * 256;
                    const uint64_t mu2 = pack2(mu_row, mu_row);
#pragma unroll
                    for (int i = 0; i < BC; i += 8) {
                        float4 ka, kb;
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(ka.x), "=f"(ka.y), "=f"(ka.z), "=f"(ka.w) : "r"(ks_s + 4 * i));
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(kb.x), "=f"(kb.y), "=f"(kb.z), "=f"(kb.w) : "r"(ks_s + 4 * i + 16));
                        unpack2(fma2_here(mu2, pack2(ka.x, ka.y), pack2(p[i], p[i + 1])), p[i], p[i + 1]);
                        unpack2(fma2_here(mu2, pack2(ka.z, ka.w), pack2(p[i + 2], p[i + 3])), p[i + 2], p[i + 3]);
                        unpack2(fma2_here(mu2, pack2(kb.x, kb.y), pack2(p[i + 4], p[i + 5])), p[i + 4], p[i + 5]);
                        unpack2(fma2_here(mu2, pack2(kb.z, kb.w), pack2(p[i + 6], p[i + 7])), p[i + 6], p[i + 7]);
                    }
                }
                if ((args.causal && (j0 + BC - 1 > q0)) || (j0 + BC > N)) {   // masked scores become -inf: exp gives exact zeros
                    const int key_lim = args.causal ? min(row, N - 1) : N - 1;
#pragma unroll
                    for (int i = 0; i < BC; ++i) p[i] = (j0 + i > key_lim) ? -INFINITY : p[i];
                }
                // (no instruction: unties the scores from the two blocks of 32 registers that the loads fill; without it ptxas spills 48
                // bytes in the plain form, with it none there, and with Q-Mean or 128-key tiles still 8 to 12)
#pragma unroll
                for (int i = 0; i < BC; ++i) asm volatile("" : "+f"(p[i]));
                const float mx = max64(p);                         // row maximum = maximum of the tile's single 64-key group
                float oth = -INFINITY;
                if constexpr (B128) {
                    // 128-key tile = tiles t and t ^ 1: both groups take the maximum over both halves and keep the running
                    // maximum for themselves; its second half finds the history rescaled.  Four slots and barriers: those
                    // of tile t serve tile t+4, after P V(t+1), hence after the other group has read them.
                    const float own = f16_round(mx * args.c0);
                    const uint32_t sl = (uint32_t)(t & 2) * 512u, b_mr = b_h + 8 * MR + 8 * (t & 2);
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(mx_own + sl), "f"(own) : "memory");
                    __syncwarp();
                    arrive0(b_mr + 8 * grp, lane);
                    if (!wait_long(b_mr + 8 * (grp ^ 1), (uint32_t)(t >> 2) & 1u, abort_flag)) { fail(12); ok = false; break; }
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(oth) : "r"((mx_own ^ 512u) + sl) : "memory");
                } else if (jt > 0) {                               // running maximum after the previous tile, from its owner
                    if (!wait_warp(b_oth + 8 * MR, ph_prev, abort_flag)) { fail(12); ok = false; break; }
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(m_run) : "r"(mx_own ^ 512u) : "memory");
                }
                // running maximum and rescale factor (lines 7-8), both FP16 values.  No branch: r = 1 exactly
                // when the maximum did not move; at jt = 0 (m = -inf) r = 0 is never applied.
                const float m_new = fmaxf(B128 ? fmaxf(m_run, oth) : m_run, f16_round(mx * args.c0));
                if (!B128) {
                    asm volatile("st.shared.f32 [%0], %1;" ::"r"(mx_own), "f"(m_new) : "memory");   // for the owner of the next tile
                    __syncwarp();
                    arrive0(b_own + 8 * MR, lane);
                }
                const float rsc = B128 && (t & 1) ? 1.f : f16_round(ex2_approx((m_run - m_new) * LOG2E));
                m_run = m_new;
                const float mL = m_run * LOG2E;
                const float A = p_of_score<false>(mx, args.c1, mL); // = max of P over the group (monotone map)

                // P = exp(S - m) in FP16 (line 9), P-hat = HIF4(P) (line 10)
                uint32_t pw[NU * 4];
                const auto qc = p_quant_const<false>(args.c1c1, mL, A);
                exp_quantize_units<NU, 0, NU, false, false>(p, qc, false, pw, nullptr, nullptr);
                // the P-hat columns and [O | l] are free once P V of the previous tile has completed
                if (jt > 0) {
                    if (!wait_long(b_oth + 8 * PV, ph_prev, abort_flag)) { fail(10); ok = false; break; }
                    tc_fence_after();
                }
                tmem_st32(t_o + C::P_COL, pw);
                if (jt > 0 && __any_sync(0xffffffffu, rsc != 1.f)) rescale_columns<D>(t_o, rsc);   // line 8
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                if (!SELFTEST) arrive0(b_h + 8 * PGO, lane);
            }
            if (!ok) break;
            t0 += n_tiles;
            c0 += n_max;

            // finalize: out = O / l with l rounded to FP16 (line 13); group grp writes channels (d/2) grp ..
            if (n_tiles > 0) {
                if (!wait_warp(b_h + 8 * PV + 8 * ((t0 - 1) & 1), (uint32_t)((t0 - 1) >> 1) & 1u, abort_flag)) { fail(11); ok = false; break; }
                tc_fence_after();
                constexpr int NC = D / 2 / 32;                     // 32-column chunks of this thread's channel half
                uint32_t lr[1];
                tmem_ld1(t_o + D, lr);
                tmem_wait_ld();
                const float l16 = f16_round(__uint_as_float(lr[0]));
                // O / l as the correctly rounded quotient from the correctly rounded reciprocal: q0 = O * y,
                // q = fma(fma(-q0, l, O), y, q0) (Markstein's correction step; no value here is near the ends of
                // the FP32 range: l >= 2^-24 is an FP16 value and |O| <= l * max|V|)
                const float rl = __frcp_rn(l16);
                const size_t orow = (size_t)w.bh_q[hf] * N + q0 + quarter * 32;      // first row of this warp
                const int rows = N - q0 - quarter * 32;            // rows of the warp inside the sequence (may exceed 32)
                const uint32_t stage = smem_base + C::STG_OFF + (uint32_t)warp * 2048u;
#pragma unroll 1
                for (int cc = 0; cc < NC; ++cc) {
                    uint32_t r[32];
                    tmem_ld32(t_o + grp * (D / 2) + cc * 32, r);
                    tmem_wait_ld();
                    if (cc == NC - 1) {                            // the next pair's P V may overwrite [O | l]
                        tc_fence_before();
                        __syncwarp();
                        arrive0(b_h + 8 * OE, lane);
                    }
                    float o[32];
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const float a = __uint_as_float(r[i]);
                        const float x0 = a * rl;
                        o[i] = fmaf(fmaf(-x0, l16, a), rl, x0);
                    }
                    const int col = grp * (D / 2) + cc * 32;
                    if (args.out_dtype == HIFA4_F32) {
#pragma unroll
                        for (int pc = 0; pc < 2; ++pc) {
                            uint32_t wd[16];
#pragma unroll
                            for (int i = 0; i < 16; ++i) wd[i] = __float_as_uint(o[16 * pc + i]);
                            store_rows64(stage, wd, reinterpret_cast<uint8_t*>(args.out) + (orow * D + col + 16 * pc) * 4, D * 4, rows, lane);
                        }
                    } else {
                        uint32_t wd[16];
#pragma unroll
                        for (int i = 0; i < 16; ++i)
                            wd[i] = args.out_dtype == HIFA4_F16 ? Pair16<__half>::round_pack(o[2 * i], o[2 * i + 1])
                                                                : Pair16<__nv_bfloat16>::round_pack(o[2 * i], o[2 * i + 1]);
                        store_rows64(stage, wd, reinterpret_cast<uint8_t*>(args.out) + (orow * D + col) * 2, D * 2, rows, lane);
                    }
                }
            }
            __syncwarp();
            arrive0(bar(WE + (it & 1)), lane);
        }
    } else if (warp < C::W_PV) {
        // ------------------------------------------------------------------ Q loads, issuer of S = Q K^T (one half)
        if (elect_one()) {
            const int hf = warp - C::W_QK;
            constexpr uint32_t idesc_s = umma_idesc_bf16(128, BC);
            const uint32_t q_s = smem_base + hf * C::Q_HALF, b_h = bar(hf * HALF);
            const uint32_t q_lo = umma_desc_lo(q_s), k_lo = umma_desc_lo(k_s), d_s = tmem + hf * C::H_COLS + C::S_COL;
            int t = 0, st = 0, nq = 0, nab = 0;               // tile, ring stage, Q loads so far, pairs without a block
            uint32_t ph = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                if (!wait_pair(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(19); break; }
                volatile Work& w = work[it & 1];
                const int n_max = w.n_max, n_tiles = w.n[hf], q0 = w.q0[hf], bh_q = w.bh_q[hf];
                if (n_max == 0) break;
                mbar_arrive(bar(WE + (it & 1)));
                if (n_tiles > 0) {
                    if (nq > 0 && !wait_pair(b_h + 8 * QD, (uint32_t)(nq - 1) & 1u, abort_flag)) { fail(5); break; }
                    mbar_expect_tx(b_h + 8 * QF, C::Q_HALF);
#pragma unroll
                    for (int s = 0; s < C::QSUB; ++s) tma_load_3d(q_s + s * 16384, &tmap_q, b_h + 8 * QF, 64 * s, q0, bh_q);
                    if (!wait_pair(b_h + 8 * QF, (uint32_t)nq & 1u, abort_flag)) { fail(3); break; }
                    ++nq;
                } else if (QM) {                              // key-sum slots: the warps may still be at the pair before
                    if (!wait_pair(bar(AB + hf), (uint32_t)nab & 1u, abort_flag)) { fail(20); break; }
                    ++nab;
                }
                for (int jt = 0; jt < n_max; ++jt) {          // S(t): K tile landed, S(t-1) in registers
                    if (!wait_pair(bar(KF + st), ph, abort_flag)) { fail(4); ok = false; break; }
                    if (jt < n_tiles) {
                        if (t > 0 && !wait_pair(b_h + 8 * SFR, (uint32_t)(t - 1) & 1u, abort_flag)) { fail(6); ok = false; break; }
                        tc_fence_after();
                        const uint32_t b0 = k_lo + st * (C::K_STAGE >> 4);
#pragma unroll
                        for (int kk = 0; kk < D / 16; ++kk)   // 16 channels per step
                            umma_bf16_ss_lo(d_s, q_lo + (kk >> 2) * (16384 >> 4) + (kk & 3) * 2,
                                            b0 + (kk >> 2) * (C::K_SUB >> 4) + (kk & 3) * 2, idesc_s, kk ? 1u : 0u);
                        umma_commit(b_h + 8 * SF + 8 * (t & 1));
                        umma_commit(bar(KE + st));
                        if (jt + 1 == n_tiles) umma_commit(b_h + 8 * QD);
                        ++t;
                    } else {
                        mbar_arrive(bar(KE + st));            // the other half's tile only
                    }
                    if (++st == STAGES) { st = 0; ph ^= 1u; }
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ issuer of [O | l] += P-hat [V | 1], both halves
        if (elect_one()) {
            // The time between "P-hat stored and history rescaled" and the issue of P V is part of the chain that sets the
            // tile period (20 ns of sleep between polls cost 2.5 %): everything else that a tile waits for (its V^T stage, the
            // output of the block before) is seen to ahead, and an armed half costs one poll per round (N = 4096, causal,
            // 134.1 -> 132.1 us; B = 4, N = 2048, non-causal, 254 -> 250)
            constexpr uint32_t idesc_o = umma_idesc_bf16(128, O_COLS);
            const uint32_t v_lo = umma_desc_lo(v_s);
            int it[2] = {0, 0}, jt[2] = {0, 0}, n_max[2] = {0, 0}, n_tiles[2] = {0, 0}, st[2] = {0, 0};
            uint32_t ph[2] = {0, 0}, t[2] = {0, 0}, no[2] = {0, 0};      // parities of the ring round, the tile and the block count
            bool first[2] = {true, true}, done[2] = {false, false}, armed[2] = {false, false};
            constexpr uint32_t POLLS = SELFTEST ? 1u << 6 : 4 * WAIT_POLLS;
            uint32_t idle = 0;
            if constexpr (SELFTEST) {
                bool quiet = wait_pair(bar(WF), 0, abort_flag) && wait_pair(bar(CL), 0, abort_flag);
                for (int j = 0; quiet && j < work[0].n_max; ++j) quiet = wait_pair(bar(VF + j), 0, abort_flag);
                for (int hf = 0; hf < 2; ++hf)
                    for (int j = 0; quiet && j < work[0].n[hf]; ++j) quiet = wait_pair(bar(hf * HALF + SF + j), 0, abort_flag);
                if (!quiet) fail(2);
            }
            while (!(done[0] && done[1])) {
                if (++idle > POLLS || ((idle & 63u) == 63u && ld_flag(abort_flag))) { if (idle > POLLS) fail(7); break; }
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    if (armed[hf]) {
                        if (!mbar_test_wait(bar(hf * HALF + PGO), t[hf])) continue;
                        idle = 0;
                        tc_fence_after();
                        const uint32_t b0 = v_lo + st[hf] * (C::V_STAGE >> 4);
                        const uint32_t acc0 = jt[hf] > 0 ? 1u : 0u;
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)          // 16 keys per step; channels and ones block
                            umma_bf16_ts_lo(tmem + hf * C::H_COLS, tmem + hf * C::H_COLS + C::P_COL + kk * 8, b0 + kk * 2, idesc_o, kk ? 1u : acc0);
                        umma_commit(bar(hf * HALF + PV + (int)t[hf]));
                        umma_commit(bar(VE + st[hf]));
                        armed[hf] = false;
                        t[hf] ^= 1u;
                        if (jt[hf] + 1 == n_tiles[hf]) { no[hf] ^= 1u; first[hf] = false; }
                        ++jt[hf];
                        if (++st[hf] == STAGES) { st[hf] = 0; ph[hf] ^= 1u; }
                    }
                    if (armed[hf] || done[hf]) continue;
                    if (jt[hf] == n_max[hf]) {                  // next pair
                        if (!mbar_test_wait(bar(WF + (it[hf] & 1)), (uint32_t)(it[hf] >> 1) & 1u)) continue;
                        volatile Work& w = work[it[hf] & 1];
                        n_max[hf] = w.n_max;
                        n_tiles[hf] = w.n[hf];
                        jt[hf] = 0;
                        if (n_max[hf] == 0) { done[hf] = true; continue; }
                        mbar_arrive(bar(WE + (it[hf] & 1)));
                        ++it[hf];
                        idle = 0;
                    }
                    if (!mbar_test_wait(bar(VF + st[hf]), ph[hf])) continue;                              // V^T tile landed
                    if (jt[hf] < n_tiles[hf]) {
                        // the first P V of a block overwrites the output columns of the block before
                        armed[hf] = jt[hf] > 0 || first[hf] || mbar_test_wait(bar(hf * HALF + OE), no[hf] ^ 1u);
                    } else {
                        idle = 0;
                        mbar_arrive(bar(VE + st[hf]));          // the other half's tile only
                        ++jt[hf];
                        if (++st[hf] == STAGES) { st[hf] = 0; ph[hf] ^= 1u; }
                    }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == C::W_LD) {
        __syncwarp();
        if (ld_flag(abort_flag) == 1) let_copies_land();
        tmem_dealloc(tmem, C::TMEM_COLS);
    }
}

template <bool QM, bool B128, bool SELFTEST = false>
static int launch_pair(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st)
{
    using C = PairCfg;
    CUtensorMap mq, mk, mv;
    if (!make_bf16_map(&mq, qkv.q_mma, (uint64_t)sh.B * sh.Hq, sh.N, C::D, 128)) return HIFA4_ERR_CUDA;
    if (!make_bf16_map(&mk, qkv.k_mma, (uint64_t)sh.B * sh.Hkv, sh.N, C::D, C::BC)) return HIFA4_ERR_CUDA;
    if (!make_bf16_map(&mv, qkv.v_mma, (uint64_t)sh.B * sh.Hkv, C::D, sh.N, C::D)) return HIFA4_ERR_CUDA;
    auto kern = attention_fwd_pair_kernel<QM, B128, SELFTEST>;
    static SmemOptIn opt_in;
    if (!opt_in.ensure(kern, C::SMEM_BYTES)) return HIFA4_ERR_CUDA;
    const int blocks = (sh.N + 127) / 128 * args.unit_heads;
    const unsigned grid = (unsigned)(((blocks + 1) / 2) * (sh.Hq / args.unit_heads) * sh.B);
    return launch_dependent(kern, grid, C::THREADS, C::SMEM_BYTES, st, mq, mk, mv, args) == cudaSuccess ? HIFA4_OK : HIFA4_ERR_CUDA;
}

bool attention_pair_pays(const hifa4_shape& sh, const hifa4_attn_params& prm)
{
    if (sh.d != 128 || (prm.Bc != 64 && prm.Bc != 128) || prm.normalizer || prm.p_dtype == HIFA4_F32) return false;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return false;
    const int G = heads_per_unit(sh);
    const long long unit_blocks = (long long)((sh.N + 127) / 128) * G, units = (long long)(sh.Hq / G) * sh.B;
    return two_blocks_faster(prm.Bc, sh.N, prm.causal != 0, prm.qmean != 0, unit_blocks * units, (unit_blocks + 1) / 2 * units, sms);
}

int launch_attention_pair_selftest(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st)
{
    return launch_pair<false, false, true>(sh, qkv, args, st);
}

int launch_attention_pair(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, int Bc, cudaStream_t st)
{
    if (sh.d != 128) return HIFA4_ERR_UNSUPPORTED;
    if (Bc == 128) return args.qmean ? launch_pair<true, true>(sh, qkv, args, st) : launch_pair<false, true>(sh, qkv, args, st);
    return args.qmean ? launch_pair<true, false>(sh, qkv, args, st) : launch_pair<false, false>(sh, qkv, args, st);
}

}  // namespace hifa4
