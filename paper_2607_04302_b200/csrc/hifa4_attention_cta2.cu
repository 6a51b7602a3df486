// Warp-specialised HiFA4 attention forward for d = 256, Bc = 64 (Algorithm 1 lines 4-13) on pairs of SMs.
//
// A cluster of two CTAs takes two 128-row query blocks of one KV head, one per CTA, and runs both GEMMs as
// tcgen05.mma.cta_group::2 with M = 256: each CTA holds half of every K and V^T tile and its tensor core reads the other
// half from its partner, so a tile crosses L2 -> SM once for 256 query rows and half of it sits in each shared memory.
// That leaves room for S of a whole step of two tiles (N = 128, the full rate of the tensor cores) and for two P-hat
// buffers, for which d = 256 has no tensor memory with one CTA per tile (there Q takes 128 columns).  16 / 8 heads, causal,
// N = 8192: 440 us against 487 in the 64-key kernel, 475 against 545 under the power cap (N = 4096, B = 2, non-causal: 448
// against 498, 475 against 525).
// Warps of a CTA:
//   0-7    softmax / quantize: warps 0-3 own the even key tiles, warps 4-7 the odd ones, one thread per row and tile
//   8-11   history, one thread per row: rescale of [O | l], output
//   12     one thread: TMA loads of the CTA's Q block and of its half of the K and V^T tiles; in CTA 0 also the work list
//   13     CTA 0 only, one thread: issuer of S = Q K^T
//   14, 15 CTA 0 only, one thread each: issuers of [O | l] += P-hat [V | 1], a part each
// What bounds it: the chain P V(t) - rescale - P V(t+1), since at 256 rows some row's maximum moves in nearly every tile.
// With the rescale in the softmax warps, which own alternate tiles but finish both tiles of a step together, the chain held
// them up: 562 us.  P V is therefore issued in two parts, channels 0..127 and channels 128..255 with the ones block, each
// with its own barriers, so that one part is rescaled while the other is multiplied; and S is issued in four pieces of 64
// channels, at most two of them in flight, with P V in between (all of S at once: 496 us; pieces of 32 channels, two in
// flight, leave the tensor cores idle between them: 700 us; three of 64: no difference).  A single issuer that polls for
// both kinds of work spends 800 clk per part of P V in its loop, next to warps that fill the issue slots: 460 us.
// (d = 128 in this form, with three groups of softmax warps, stays behind two independent blocks per SM, which hide one
// another's chain: 2.5 against 2.0 ms at N = 16384, 32 / 8 heads, causal.)
// N of a cta_group::2 MMA is a multiple of 32 and CTA r supplies the r-th half of its B rows: CTA 0 holds the K rows of a
// step's first tile, the V^T rows of channels 0..63, 128..191 and 16 rows of ones, CTA 1 the K rows of the second tile, the
// V^T rows of 64..127, 192..255 and 16 rows of ones.  Tensor memory (columns): channels 0..127, 128..191, ones 16, channels
// 192..255, ones 16 (0..287), S 128, P-hat 2 x 32.
// Persistent through cluster launch control as hifa4_attention_pair.cu, whose order of pairs it shares; a shorter or absent
// second block runs along under its mask, and so does a step's second tile past the last key.  Tiles are numbered through
// all pairs of a cluster (t, even at a pair's first tile); barrier phases follow those numbers.  Barriers that both CTAs
// arrive on live in CTA 0.
// Template flag: Q-Mean.  Every wait is bounded (see hifa4_attention_ws.cu for the failure protocol).
#include "hifa4_attention.cuh"

namespace hifa4 {

struct Cta2Cfg {
    static constexpr int D = 256, BC = 64, QSUB = D / 64;
    static constexpr int K_STAGES = 2, V_STAGES = 4;
    static constexpr int NSW = 8, W_HIST = 8, W_LD = 12, W_QK = 13, W_PV = 14, THREADS = 512;
    static constexpr int NU = BC / 8;
    static constexpr int Q_BYTES = QSUB * 16384;            // sub-tiles of 64 channels x 128 rows
    static constexpr int K_SUB = 64 * 128, K_STAGE = QSUB * K_SUB;     // this CTA's 64 of a step's 128 keys
    static constexpr int V_ROWS = D / 4;                    // this CTA's channels of either part of P V
    static constexpr int V_HI = V_ROWS * 128, V_ONES = 2 * V_HI, V_STAGE = V_ONES + 16 * 128;    // second part, ones inside a stage
    static constexpr int K_OFF = Q_BYTES, V_OFF = K_OFF + K_STAGES * K_STAGE;
    static constexpr int STG_OFF = V_OFF + V_STAGES * V_STAGE;         // output staging, 2 KB per history warp
    static constexpr int MX_OFF = STG_OFF + 4 * 2048;       // running maxima handed from tile t to t+1: [t % 2][128] floats
    static constexpr int RS_OFF = MX_OFF + 1024;            // rescale factors for the history warps: [t % 4][128] floats
    static constexpr int KSUM_OFF = RS_OFF + 2048;          // Q-Mean: channel sums of a step's 128 keys, slot = step % 4
    static constexpr int MISC_OFF = KSUM_OFF + 4 * 512;
    static constexpr int SMEM_BYTES = MISC_OFF + 1024 + 1024;
    static constexpr int HI_COL = D / 2, L_COL = D / 2 + V_ROWS, S_COL = D + 32, P_COL = S_COL + 128, TMEM_COLS = 512;
    static_assert(P_COL + 64 <= TMEM_COLS && SMEM_BYTES <= 227 * 1024, "tensor memory or shared memory budget");
    static_assert(K_OFF % 1024 == 0 && V_STAGE % 1024 == 0 && MX_OFF % 1024 == 0 && MISC_OFF % 16 == 0,
                  "swizzle atoms, addresses formed with xor, bulk copies");
};

namespace cta2 {
// In CTA 0, for both: QF Q blocks landed, KF / VF halves landed, SFR S of a step pulled (16 arrivals), GL / GH[t % 2] P-hat
// stored and first / second part of the history rescaled or, at a pair's first tile, output (16), WE[pair % 2] work record
// read (28), CL answer of the launch control, SC[piece % 2] piece of S complete.  In each CTA: QD last S of the pair
// complete, KE stage free, SF S of a step complete, PL / PH[t % 2] first / second part of P V complete, PV[t % 4] both, and
// the V^T stage free (2), MR[t % 4] maxima and rescale factors published (4 arrivals; the softmax warps may be two tiles
// ahead of the history warps), WF[pair % 2] work record written, KSF[step % 4] Q-Mean key sums landed.
enum { PL = 0, PH = 2, PV = 4, MR = 8, GL = 12, GH = 14, WF = 16, WE = 18, SF = 20, SFR = 21, QF = 22, QD = 23, CL = 24,
       KF = 25, KE = 27, VF = 29, KSF = 33, SC = 37, N_BARS = 39 };
constexpr uint32_t WAIT_POLLS = 1u << 18;            // a poll may keep the thread suspended for up to about 4 us
struct Work {
    int n_max;                        // steps of two key tiles; 0: no more work
    int bh_kv;
    int q0[2], bh_q[2];
    int store[2];                     // 0: the second block is a stand-in, nothing is written
};

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t at_rank(uint32_t addr, uint32_t rank)   // the same shared-memory address in CTA `rank`
{
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_remote(uint32_t addr, int v)
{
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void arrive_remote(uint32_t addr)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// The same from lane 0 of a converged warp, where no memory but tensor memory is handed over (ordered by the tcgen05 fences):
// without cluster scope, whose release waits ~1100 clk for the warp's earlier memory operations.
__device__ __forceinline__ void arrive_remote0(uint32_t addr, int lane)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.eq.s32 p, %1, 0;\n\t"
                 "@p mbarrier.arrive.shared::cluster.b64 _, [%0];\n\t}"
                 ::"r"(addr), "r"(lane) : "memory");
}
__device__ __forceinline__ void arrive_local0(uint32_t addr, int lane)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.eq.s32 p, %1, 0;\n\t"
                 "@p mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}"
                 ::"r"(addr), "r"(lane) : "memory");
}
__device__ __forceinline__ bool poll_cluster(uint32_t bar, uint32_t parity)  // for data written by the other CTA's threads
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
__device__ __forceinline__ int flag(uint32_t addr)
{
    int v;
    asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity, uint32_t abort_flag)
{
#pragma unroll 1
    for (uint32_t i = 0; i < WAIT_POLLS; ++i) {
        if (CLUSTER ? poll_cluster(bar, parity) : mbar_try_wait(bar, parity)) return true;
        if ((i & 63u) == 63u && flag(abort_flag)) return false;
    }
    return false;
}
// TMA load into this CTA's shared memory whose bytes count on a barrier of either CTA of the pair (no multicast).
__device__ __forceinline__ void load_3d(uint32_t dst, const void* tmap, uint32_t bar, int c0, int c1, int c2)
{
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
                 "[%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void mma_ss(uint32_t d, uint32_t a_lo, uint32_t b_lo, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 ad, bd;\n\t"
                 "setp.ne.b32 p, %5, 0;\n\t"
                 "mov.b64 ad, {%1, %3};\n\t"
                 "mov.b64 bd, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], ad, bd, %4, p;\n\t}"
                 ::"r"(d), "r"(a_lo), "r"(b_lo), "r"(UMMA_DESC_HI_SW128), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a_tmem, uint32_t b_lo, uint32_t idesc, uint32_t accumulate)
{
    asm volatile("{\n\t.reg .pred p;\n\t.reg .b64 bd;\n\t"
                 "setp.ne.b32 p, %5, 0;\n\t"
                 "mov.b64 bd, {%2, %3};\n\t"
                 "tcgen05.mma.cta_group::2.kind::f16 [%0], [%1], bd, %4, p;\n\t}"
                 ::"r"(d), "r"(a_tmem), "r"(b_lo), "r"(UMMA_DESC_HI_SW128), "r"(idesc), "r"(accumulate) : "memory");
}
// Arrive on this barrier of both CTAs once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3) : "memory");
}
__device__ __forceinline__ void commit_local(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void launch_control_ask(uint32_t dst, uint32_t bar)
{
    fence_proxy_async_smem();
    mbar_expect_tx(bar, 16);
    asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
                 ::"r"(dst), "r"(bar) : "memory");
}
__device__ __forceinline__ int launch_control_answer(uint32_t src)          // blockIdx.x of the first CTA taken over, or -1
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
// NC columns of [O | l] at tensor-memory address t times r; the caller waits for the stores.
template <int NC>
__device__ __forceinline__ void scale_columns(uint32_t t, float r)
{
    const uint64_t rr = pack2(r, r);
#pragma unroll
    for (int c = 0; c < NC; c += 64) {
        constexpr int H = NC < 64 ? 1 : 2;
        uint32_t a[H][32];
#pragma unroll
        for (int h = 0; h < H; ++h) tmem_ld32(t + c + 32 * h, a[h]);
        tmem_wait_ld();
#pragma unroll
        for (int h = 0; h < H; ++h) {
#pragma unroll
            for (int i = 0; i < 32; i += 2) {
                float x0, x1;
                unpack2(mul2(pack2(__uint_as_float(a[h][i]), __uint_as_float(a[h][i + 1])), rr), x0, x1);
                a[h][i] = __float_as_uint(x0);
                a[h][i + 1] = __float_as_uint(x1);
            }
            tmem_st32(t + c + 32 * h, a[h]);
        }
    }
}
}  // namespace cta2

template <bool QM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(Cta2Cfg::THREADS, 1)
attention_fwd_cta2_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                          const __grid_constant__ CUtensorMap tmap_v, const __grid_constant__ AttnArgs args)
{
    using namespace cta2;
    using C = Cta2Cfg;
    constexpr int D = C::D, BC = C::BC, NU = C::NU;

    extern __shared__ uint8_t smem_raw[];
    const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;       // the same in both CTAs
    uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
    const uint32_t k_s = smem_base + C::K_OFF, v_s = smem_base + C::V_OFF, bars = smem_base + C::MISC_OFF;
    auto bar = [&](int i) { return bars + 8u * (uint32_t)i; };
    volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(smem_gen + C::MISC_OFF + 8 * N_BARS);
    const uint32_t abort_flag = bars + 8 * N_BARS + 8;
    constexpr int CL_OFF = C::MISC_OFF + 512, WORK_OFF = C::MISC_OFF + 544;
    volatile Work* work = reinterpret_cast<volatile Work*>(smem_gen + WORK_OFF);     // [2]

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int N = args.N;
    const uint32_t rank = cluster_rank();

    if (warp == C::W_LD && lane == 0) {
        // CTA 0 reads the status word for both: a cluster that starts after another one reported a failure does nothing
        int status_now = rank == 0 && args.d_status ? *reinterpret_cast<volatile int*>(args.d_status) : 0;
        tma_prefetch_desc(&tmap_q); tma_prefetch_desc(&tmap_k); tma_prefetch_desc(&tmap_v);
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar(PL + s), 1); mbar_init(bar(PH + s), 1); mbar_init(bar(GL + s), 16); mbar_init(bar(GH + s), 16);
            mbar_init(bar(WF + s), 1); mbar_init(bar(WE + s), 2 * C::NSW + 12); mbar_init(bar(SC + s), 1);
            mbar_init(bar(KF + s), 1); mbar_init(bar(KE + s), 1);
        }
        for (int s = 0; s < 4; ++s) {
            mbar_init(bar(MR + s), 4); mbar_init(bar(VF + s), 1); mbar_init(bar(PV + s), 2); mbar_init(bar(KSF + s), 1);
        }
        mbar_init(bar(SF), 1); mbar_init(bar(SFR), 16);
        mbar_init(bar(QF), 1); mbar_init(bar(QD), 1); mbar_init(bar(CL), 1);
        fence_barrier_init();
        // nothing the preceding kernel of the stream wrote is touched before this point (programmatic launch)
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (rank == 0) {
            if (status_now != 0) status_now = *reinterpret_cast<volatile int*>(args.d_status);
        }
        st_remote(at_rank(abort_flag, rank), 0);
        if (rank == 0 && status_now != 0) st_remote(at_rank(abort_flag, 0), 2);
        *reinterpret_cast<volatile int*>(smem_gen + C::MISC_OFF + 8 * N_BARS + 12) = rank == 0 ? (status_now != 0) : 0;
    }
    if (warp == C::W_LD) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32((const void*)tmem_slot)), "r"(C::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    }
    for (int i = tid; i < C::V_STAGES * 128; i += C::THREADS) {        // ones rows under every V^T stage
        const int st = i / 128, off = (i % 128) * 16;
        asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};"
                     ::"r"(v_s + st * C::V_STAGE + C::V_ONES + off), "r"(0x3F803F80u) : "memory");
    }
    fence_proxy_async_smem();
    tc_fence_before();
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    cluster_sync();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    int verdict;                                              // CTA 0's, the same for both
    asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(verdict) : "r"(at_rank(bars + 8 * N_BARS + 12, 0)) : "memory");
    const bool dead = verdict != 0;

    auto fail = [&](int site) {
        st_remote(at_rank(abort_flag, 0), 1);
        st_remote(at_rank(abort_flag, 1), 1);
        if (args.d_status) atomicCAS(args.d_status, 0, HIFA4_ERR_TIMEOUT + 16 * site);
    };

    if (dead) {
        // fall through to the common exit
    } else if (warp == C::W_LD) {
        // ------------------------------------------------------------------ work list (CTA 0), loads
        if (elect_one()) {
            // order of the pairs: as in hifa4_attention_pair.cu
            const int G = args.unit_heads, n_qt = (N + 127) / 128, Hu = args.Hq / G;
            const int blocks = n_qt * G, pairs = (blocks + 1) >> 1, gu = args.group_units;
            const uint32_t qf = at_rank(bar(QF), 0);
            int stk = 0, stv = 0, c = 0;                      // ring stages, step count (Q-Mean)
            uint32_t phk = 1, phv = 1;                        // parity that the "empty" waits use: the first round passes
            int idx = (int)blockIdx.x >> 1;
            for (int it = 0;; ++it) {
                volatile Work& w = work[it & 1];
                int n_max = 0, bh_kv = 0, q0 = 0, bh_q = 0;
                if (rank == 0) {
                    if (it >= 2 && !wait<true>(bar(WE + (it & 1)), (uint32_t)((it >> 1) - 1) & 1u, abort_flag)) { fail(16); break; }
                    int rec[8] = {0, 0, 0, 0, 0, 0, 0, 0};
                    if (idx >= 0) {
                        const int grp_i = idx / (pairs * gu), in_grp = idx - grp_i * (pairs * gu);
                        const int p = in_grp / gu, unit = grp_i * gu + (in_grp - p * gu);
                        const int b = unit / Hu, h0 = (unit - b * Hu) * G;
                        rec[1] = b * args.Hkv + args.map.kv_of[h0];
#pragma unroll
                        for (int hf = 0; hf < 2; ++hf) {
                            const int r = 2 * p + hf < blocks ? 2 * p + hf : 2 * p, qi = r / G, q0 = (n_qt - 1 - qi) * 128;
                            const int last_key = args.causal ? min(q0 + 127, N - 1) : N - 1;
                            rec[0] = max(rec[0], last_key / (2 * BC) + 1);
                            rec[2 + hf] = q0;
                            rec[4 + hf] = b * args.Hq + h0 + (r - qi * G);
                            rec[6 + hf] = 2 * p + hf < blocks;
                        }
                    }
                    n_max = rec[0]; bh_kv = rec[1]; q0 = rec[2]; bh_q = rec[4];
#pragma unroll
                    for (uint32_t rk = 0; rk < 2; ++rk) {
                        const uint32_t dst = at_rank(smem_base + WORK_OFF + (it & 1) * (uint32_t)sizeof(Work), rk);
#pragma unroll
                        for (int i = 0; i < 8; ++i) st_remote(dst + 4 * i, rec[i]);
                        arrive_remote(at_rank(bar(WF + (it & 1)), rk));
                    }
                } else {
                    if (!wait<true>(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(21); break; }
                    n_max = w.n_max; bh_kv = w.bh_kv; q0 = w.q0[1]; bh_q = w.bh_q[1];
                }
                if (n_max == 0) break;
                if (rank == 1) arrive_remote(at_rank(bar(WE + (it & 1)), 0));
                int jk = 0, jv = 0;
                bool q_done = false, ok = true;
                uint32_t idle = 0;
                while (jv < 2 * n_max || !q_done) {
                    if (++idle > 4 * WAIT_POLLS || ((idle & 63u) == 63u && flag(abort_flag))) {
                        if (idle > 4 * WAIT_POLLS) fail(1);
                        ok = false;
                        break;
                    }
                    if (jk < n_max && mbar_try_wait(bar(KE + stk), phk)) {
                        idle = 0;
                        if (rank == 0) mbar_expect_tx(bar(KF + stk), 2 * C::K_STAGE);
                        const uint32_t kf = at_rank(bar(KF + stk), 0);
#pragma unroll
                        for (int s = 0; s < C::QSUB; ++s)
                            load_3d(k_s + stk * C::K_STAGE + s * C::K_SUB, &tmap_k, kf, 64 * s, jk * 2 * BC + 64 * (int)rank, bh_kv);
                        if (QM) {
                            // slot c % 4 held the sums of step c-4: this load follows S(c-2), hence the pull of S(c-3) by the
                            // warps that read the slot during step c-4.  (N may end inside a step.)
                            const uint32_t bytes = min(2 * BC, N - jk * 2 * BC) * 4u;
                            mbar_expect_tx(bar(KSF + (c & 3)), bytes);
                            bulk_load(smem_base + C::KSUM_OFF + (c & 3) * 512, args.k_sum + (size_t)bh_kv * N + jk * 2 * BC, bytes, bar(KSF + (c & 3)));
                            ++c;
                        }
                        if (rank == 0 && jk == max(n_max - 2, 0)) launch_control_ask(smem_base + CL_OFF, bar(CL));
                        ++jk;
                        if (++stk == C::K_STAGES) { stk = 0; phk ^= 1u; }
                    }
                    if (!q_done && (it == 0 || mbar_try_wait(bar(QD), (uint32_t)(it - 1) & 1u))) {
                        idle = 0;
                        q_done = true;
                        if (rank == 0) mbar_expect_tx(bar(QF), 2 * C::Q_BYTES);
#pragma unroll
                        for (int s = 0; s < C::QSUB; ++s) load_3d(smem_base + s * 16384, &tmap_q, qf, 64 * s, q0, bh_q);
                    }
                    if (jv < 2 * jk && mbar_try_wait(bar(PV + stv), phv)) {
                        idle = 0;
                        if (rank == 0) mbar_expect_tx(bar(VF + stv), 4 * C::V_HI);
                        const uint32_t vf = at_rank(bar(VF + stv), 0);
                        load_3d(v_s + stv * C::V_STAGE, &tmap_v, vf, jv * BC, C::V_ROWS * (int)rank, bh_kv);
                        load_3d(v_s + stv * C::V_STAGE + C::V_HI, &tmap_v, vf, jv * BC, D / 2 + C::V_ROWS * (int)rank, bh_kv);
                        ++jv;
                        if (++stv == C::V_STAGES) { stv = 0; phv ^= 1u; }
                    }
                }
                if (!ok) break;
                if (rank == 0) {
                    if (!wait(bar(CL), (uint32_t)it & 1u, abort_flag)) { fail(17); break; }
                    idx = launch_control_answer(smem_base + CL_OFF);
                    if (idx >= 0) idx >>= 1;
                }
            }
        }
    } else if (warp < C::NSW) {
        // ------------------------------------------------------------------ softmax / quantize
        const int grp = warp >> 2, quarter = warp & 3;
        const int r_loc = quarter * 32 + lane;                    // row inside the block = TMEM lane
        const uint32_t t_o = tmem + ((uint32_t)(quarter * 32) << 16);
        const float LOG2E = 1.4426950408889634f;
        const uint32_t mx_own = smem_base + C::MX_OFF + grp * 512 + r_loc * 4;
        const uint32_t rs_own = smem_base + C::RS_OFF + grp * 512 + r_loc * 4;
        const uint32_t r_own = at_rank(bars + 8 * grp, 0), r_sfr = at_rank(bar(SFR), 0);     // barriers in CTA 0
        int t0 = 0;                                               // tiles before the current pair (even)
        bool ok = true;
        for (int it = 0; ok; ++it) {
            if (!wait<true>(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(18); break; }
            volatile Work& w = work[it & 1];
            const int n_tiles = 2 * w.n_max, q0 = w.q0[rank];     // the last tile may lie past the last key: all masked
            if (n_tiles == 0) break;
            const int row = q0 + r_loc;
            float m_run = -INFINITY;
            const float mu_row = (QM && row < N) ? args.q_mu[(size_t)w.bh_q[rank] * N + row] : 0.f;

            for (int jt = grp; jt < n_tiles; jt += 2) {
                const int t = t0 + jt, u = t >> 1, j0 = jt * BC;   // t % 2 == grp; step u
                if (!wait(bar(SF), (uint32_t)u & 1u, abort_flag)) { fail(8); ok = false; break; }
                tc_fence_after();
                float p[BC];
                {
                    uint32_t r[BC];
                    tmem_ld32(t_o + C::S_COL + grp * 64, reinterpret_cast<uint32_t(&)[32]>(r[0]));
                    tmem_ld32(t_o + C::S_COL + grp * 64 + 32, reinterpret_cast<uint32_t(&)[32]>(r[32]));
                    tmem_wait_ld();
#pragma unroll
                    for (int i = 0; i < BC; ++i) p[i] = __uint_as_float(r[i]);
                }
                tc_fence_before();                                 // S(t) is in registers
                __syncwarp();
                arrive_remote0(r_sfr, lane);

                if (QM) {                                          // Q-Mean correction (line 6): + mu_i * sum_c k~_jc
                    if (!wait(bar(KSF + (u & 3)), (uint32_t)(u >> 2) & 1u, abort_flag)) { fail(15); ok = false; break; }
                    const uint32_t ks_s = smem_base + C::KSUM_OFF + (u & 3) * 512 + grp * 256;
                    const uint64_t mu2 = pack2(mu_row, mu_row);
#pragma unroll
                    for (int i = 0; i < BC / 4; ++i) {
                        float4 ks;
                        asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                                     : "=f"(ks.x), "=f"(ks.y), "=f"(ks.z), "=f"(ks.w) : "r"(ks_s + 16 * i));
                        unpack2(fma2(mu2, pack2(ks.x, ks.y), pack2(p[4 * i], p[4 * i + 1])), p[4 * i], p[4 * i + 1]);
                        unpack2(fma2(mu2, pack2(ks.z, ks.w), pack2(p[4 * i + 2], p[4 * i + 3])), p[4 * i + 2], p[4 * i + 3]);
                    }
                }
                if ((args.causal && (j0 + BC - 1 > q0)) || (j0 + BC > N)) {   // masked scores become -inf: exp gives exact zeros
                    const int key_lim = args.causal ? min(row, N - 1) : N - 1;
#pragma unroll
                    for (int i = 0; i < BC; ++i) p[i] = (j0 + i > key_lim) ? -INFINITY : p[i];
                }
                const float mx = max64(p);                         // row maximum = maximum of the tile's single 64-key group
                // running maximum after the previous tile, from its owner (at a pair's first tile the wait only says that the
                // owner of the pair before has read the slot that is written next)
                if (t > 0 && !wait(bar(MR + ((t - 1) & 3)), (uint32_t)((t - 1) >> 2) & 1u, abort_flag)) { fail(12); ok = false; break; }
                if (jt > 0) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(m_run) : "r"(mx_own ^ 512u) : "memory");
                // running maximum and rescale factor (lines 7-8), both FP16 values; r = 1 exactly when the maximum did
                // not move; at jt = 0 (m = -inf) r = 0 is never applied
                const float m_new = fmaxf(m_run, f16_round(mx * args.c0));
                const float rsc = f16_round(ex2_approx((m_run - m_new) * LOG2E));
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(mx_own), "f"(m_new) : "memory");   // for the owner of the next tile
                // slot t % 4 held the factors of tile t-4: P V(t-4), waited for during tile t-2, came after their use
                asm volatile("st.shared.f32 [%0], %1;" ::"r"(rs_own + (t & 2) * 512), "f"(rsc) : "memory");
                __syncwarp();
                arrive_local0(bar(MR + (t & 3)), lane);
                m_run = m_new;
                const float mL = m_run * LOG2E;
                const float A = p_of_score<false>(mx, args.c1, mL); // = max of P over the group (monotone map)

                // P = exp(S - m) in FP16 (line 9), P-hat = HIF4(P) (line 10)
                uint32_t pw[NU * 4];
                const auto qc = p_quant_const<false>(args.c1c1, mL, A);
                exp_quantize_units<NU, 0, NU, false, false>(p, qc, false, pw, nullptr, nullptr);
                // this P-hat buffer is free once P V(t-2) has completed
                if (t >= 2) {
                    if (!wait(bar(PV + ((t - 2) & 3)), (uint32_t)((t - 2) >> 2) & 1u, abort_flag)) { fail(10); ok = false; break; }
                    tc_fence_after();
                }
                tmem_st32(t_o + C::P_COL + grp * 32, pw);
                tmem_wait_st();
                tc_fence_before();
                __syncwarp();
                arrive_remote0(r_own + 8 * GL, lane);
                arrive_remote0(r_own + 8 * GH, lane);
            }
            if (!ok) break;
            t0 += n_tiles;
            __syncwarp();
            arrive_remote0(at_rank(bar(WE + (it & 1)), 0), lane);
        }
    } else if (warp < C::W_HIST + 4) {
        // ------------------------------------------------------------------ history: rescale, finalize
        const int quarter = warp & 3, r_loc = quarter * 32 + lane;
        const uint32_t t_o = tmem + ((uint32_t)(quarter * 32) << 16);
        const uint32_t rs_s = smem_base + C::RS_OFF + r_loc * 4, r_gl = at_rank(bar(GL), 0), r_gh = at_rank(bar(GH), 0);
        int t = 0;
        auto wait_pv = [&](int tile) { return wait(bar(PV + (tile & 3)), (uint32_t)(tile >> 2) & 1u, abort_flag); };
        // a part of P V(t-1)
        auto wait_part = [&](int part) { return wait(bar(part + ((t - 1) & 1)), (uint32_t)((t - 1) >> 1) & 1u, abort_flag); };
        bool ok = true;
        for (int it = 0; ok; ++it) {
            if (!wait<true>(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(18); break; }
            volatile Work& w = work[it & 1];
            const int n_tiles = 2 * w.n_max, q0 = w.q0[rank];
            if (n_tiles == 0) break;
            for (int jt = 0; jt < n_tiles; ++jt, ++t) {
                float rsc = 1.f;
                if (jt > 0) {
                    if (!wait(bar(MR + (t & 3)), (uint32_t)(t >> 2) & 1u, abort_flag)) { fail(12); ok = false; break; }
                    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(rsc) : "r"(rs_s + (t & 3) * 512) : "memory");
                }
                // P V(t-2) complete: the arrivals below belong to tile t, and no wait on PL or PH can be two phases behind
                if (t >= 2 && !wait_pv(t - 2)) { fail(10); ok = false; break; }
                // rescale (line 8), each part as soon as P V(t-1) of it has completed
                const bool any = __any_sync(0xffffffffu, rsc != 1.f);
                if (any) {
                    if (!wait_part(PL)) { fail(13); ok = false; break; }
                    tc_fence_after();
                    scale_columns<D / 2>(t_o, rsc);
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                }
                arrive_remote0(r_gl + 8 * (t & 1), lane);
                if (any) {
                    if (!wait_part(PH)) { fail(14); ok = false; break; }
                    tc_fence_after();
                    uint32_t rl[1];
                    tmem_ld1(t_o + C::L_COL, rl);
                    scale_columns<C::V_ROWS>(t_o + C::HI_COL, rsc);
                    scale_columns<C::V_ROWS>(t_o + C::L_COL + 16, rsc);
                    rl[0] = __float_as_uint(__uint_as_float(rl[0]) * rsc);
                    tmem_st1(t_o + C::L_COL, rl);
                    tmem_wait_st();
                    tc_fence_before();
                    __syncwarp();
                }
                arrive_remote0(r_gh + 8 * (t & 1), lane);
            }
            if (!ok) break;

            // finalize: out = O / l with l rounded to FP16 (line 13)
            // (P V(t-2) first: only then can the other barrier not be two phases behind)
            if (!wait_pv(t - 2) || !wait_pv(t - 1)) { fail(11); ok = false; break; }
            tc_fence_after();
            uint32_t lr[1];
            tmem_ld1(t_o + C::L_COL, lr);
            tmem_wait_ld();
            const float l16 = f16_round(__uint_as_float(lr[0]));
            // O / l as the correctly rounded quotient from the correctly rounded reciprocal and one correction step
            // (no value here is near the ends of the FP32 range: l >= 2^-24 is an FP16 value and |O| <= l * max|V|)
            const float rl = __frcp_rn(l16);
            const size_t orow = (size_t)w.bh_q[rank] * N + q0 + quarter * 32;        // first row of this warp
            const int rows = w.store[rank] ? N - q0 - quarter * 32 : 0;  // rows of the warp inside the sequence (may exceed 32)
            const uint32_t stage = smem_base + C::STG_OFF + (uint32_t)quarter * 2048u;
#pragma unroll 1
            for (int cc = 0; cc < D / 32; ++cc) {
                const int col = cc * 32;
                uint32_t r[32];
                tmem_ld32(t_o + col + (col >= C::L_COL ? 16 : 0), r);
                tmem_wait_ld();
                float o[32];
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    const float a = __uint_as_float(r[i]);
                    const float x0 = a * rl;
                    o[i] = fmaf(fmaf(-x0, l16, a), rl, x0);
                }
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
            tc_fence_before();                                // the arrivals at the next pair's first tile follow these reads
            __syncwarp();
            arrive_remote0(at_rank(bar(WE + (it & 1)), 0), lane);
        }
    } else if (rank == 0 && warp == C::W_QK) {
        // ------------------------------------------------------------------ issuer of S = Q K^T (CTA 0)
        if (elect_one()) {
            constexpr uint32_t idesc_s = umma_idesc_bf16(256, 2 * BC);
            const uint32_t q_lo = umma_desc_lo(smem_base), k_lo = umma_desc_lo(k_s);
            int st = 0, u = 0, sc = 0;                        // ring stage; steps, pieces of S issued
            uint32_t ph = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                if (!wait<true>(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(19); break; }
                const int n = work[it & 1].n_max;
                if (n == 0) break;
                arrive_remote(at_rank(bar(WE + (it & 1)), 0));
                if (!wait(bar(QF), (uint32_t)it & 1u, abort_flag)) { fail(3); break; }
                for (int j = 0; ok && j < n; ++j, ++u) {      // K halves landed, S(u-1) in registers
                    if (!wait(bar(KF + st), ph, abort_flag)) { fail(4); ok = false; break; }
                    if (u > 0 && !wait(bar(SFR), (uint32_t)(u - 1) & 1u, abort_flag)) { fail(6); ok = false; break; }
                    // in pieces of 64 channels, at most two in flight: a P V that becomes ready meanwhile must not wait for all of S
                    for (int ch = 0; ch < C::QSUB; ++ch, ++sc) {
                        if (sc >= 2 && !wait(bar(SC + (sc & 1)), (uint32_t)((sc >> 1) - 1) & 1u, abort_flag)) { fail(2); ok = false; break; }
                        tc_fence_after();
                        const uint32_t a0 = q_lo + ch * (16384 >> 4), b0 = k_lo + st * (C::K_STAGE >> 4) + ch * (C::K_SUB >> 4);
#pragma unroll
                        for (int kk = 0; kk < 4; ++kk)        // 16 channels per step
                            mma_ss(tmem + C::S_COL, a0 + kk * 2, b0 + kk * 2, idesc_s, (ch | kk) ? 1u : 0u);
                        commit_local(bar(SC + (sc & 1)));
                    }
                    if (!ok) break;
                    commit(bar(SF));
                    commit(bar(KE + st));
                    if (++st == C::K_STAGES) { st = 0; ph ^= 1u; }
                }
                if (ok) commit(bar(QD));
            }
        }
    } else if (rank == 0) {
        // ------------------------------------------------------------------ issuers of [O | l] += P-hat [V | 1] (CTA 0), a part each
        if (elect_one()) {
            const int hi = warp - C::W_PV;
            const uint32_t idesc = hi ? umma_idesc_bf16(256, D / 2 + 32) : umma_idesc_bf16(256, D / 2);
            const uint32_t d = tmem + (hi ? C::HI_COL : 0), b_lo = umma_desc_lo(v_s + (hi ? C::V_HI : 0));
            const uint32_t go = bar(hi ? GH : GL), part = bar(hi ? PH : PL);
            int st = 0, t = 0;                                // ring stage, tile
            uint32_t ph = 0;
            bool ok = true;
            for (int it = 0; ok; ++it) {
                if (!wait<true>(bar(WF + (it & 1)), (uint32_t)(it >> 1) & 1u, abort_flag)) { fail(22); break; }
                const int n_tiles = 2 * work[it & 1].n_max;
                if (n_tiles == 0) break;
                arrive_remote(at_rank(bar(WE + (it & 1)), 0));
                for (int jt = 0; jt < n_tiles; ++jt, ++t) {   // V^T halves landed; P-hat stored and this part rescaled
                    if (!wait(bar(VF + st), ph, abort_flag)) { fail(9); ok = false; break; }
                    if (!wait(go + 8 * (t & 1), (uint32_t)(t >> 1) & 1u, abort_flag)) { fail(7); ok = false; break; }
                    tc_fence_after();
                    const uint32_t a = tmem + C::P_COL + (t & 1) * 32, b0 = b_lo + st * (C::V_STAGE >> 4), acc0 = jt > 0 ? 1u : 0u;
#pragma unroll
                    for (int kk = 0; kk < 4; ++kk) mma_ts(d, a + kk * 8, b0 + kk * 2, idesc, kk ? 1u : acc0);      // 16 keys per step
                    commit(part + 8 * (t & 1));
                    commit(bar(PV + st));
                    if (++st == C::V_STAGES) { st = 0; ph ^= 1u; }
                }
            }
        }
    }

    tc_fence_before();
    __syncthreads();
    cluster_sync();                                           // the partner may still arrive on this CTA's barriers
    if (warp == C::W_LD) {
        __syncwarp();
        if (flag(abort_flag) == 1) let_copies_land();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS) : "memory");
    }
}

template <bool QM>
static int launch_cta2(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st)
{
    using C = Cta2Cfg;
    CUtensorMap mq, mk, mv;
    if (!make_bf16_map(&mq, qkv.q_mma, (uint64_t)sh.B * sh.Hq, sh.N, C::D, 128)) return HIFA4_ERR_CUDA;
    if (!make_bf16_map(&mk, qkv.k_mma, (uint64_t)sh.B * sh.Hkv, sh.N, C::D, 64)) return HIFA4_ERR_CUDA;
    if (!make_bf16_map(&mv, qkv.v_mma, (uint64_t)sh.B * sh.Hkv, C::D, sh.N, C::V_ROWS)) return HIFA4_ERR_CUDA;
    auto kern = attention_fwd_cta2_kernel<QM>;
    static SmemOptIn opt_in;
    if (!opt_in.ensure(kern, C::SMEM_BYTES)) return HIFA4_ERR_CUDA;
    const int blocks = (sh.N + 127) / 128 * args.unit_heads;
    const unsigned grid = 2u * (unsigned)(((blocks + 1) / 2) * (sh.Hq / args.unit_heads) * sh.B);
    return launch_dependent(kern, grid, C::THREADS, C::SMEM_BYTES, st, mq, mk, mv, args) == cudaSuccess ? HIFA4_OK : HIFA4_ERR_CUDA;
}

// Whether this kernel is the faster one: as soon as the 64-key kernel, one block per SM, no longer runs all blocks at once
// (d = 256, causal and not: 128 blocks 23-38 us there and 1-2 us more here; 256 blocks N = 1024 45.4 against 43.0 and, causal,
// 29.5 against 29.1, N = 2048 76 against 72 and 43 against 41, 512 blocks N = 4096 150 against 137), unless odd numbers of
// blocks per KV head leave many pairs without a second block.
bool attention_cta2_pays(const hifa4_shape& sh, const hifa4_attn_params& prm, int unit_heads)
{
    if (sh.d != 256 || prm.Bc != 64 || prm.normalizer || prm.p_dtype == HIFA4_F32) return false;
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0)
        return false;
    const long long unit_blocks = (long long)((sh.N + 127) / 128) * unit_heads, units = (long long)(sh.Hq / unit_heads) * sh.B;
    return unit_blocks * units > sms && 20 * ((unit_blocks + 1) / 2) <= 11 * unit_blocks;
}

int launch_attention_cta2(const hifa4_shape& sh, const hifa4_qkv& qkv, const AttnArgs& args, cudaStream_t st)
{
    if (sh.d != 256) return HIFA4_ERR_UNSUPPORTED;
    return args.qmean ? launch_cta2<true>(sh, qkv, args, st) : launch_cta2<false>(sh, qkv, args, st);
}

}  // namespace hifa4
