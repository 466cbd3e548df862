// lla_prefill.cu -- causal pass-2 prefill attention over latents (App. A, two-pass prefill;
// App. J absorbed attention).
//
// For a prompt of L tokens whose latents are all in the cache, query i at loop t attends to
// keys 0..i:
//   q~_i = W_up,t^K^T q_i                       (the constant q_i . mu^K_t cancels in softmax)
//   s_ij = scale * q~_i . c_k,j,   p_i = softmax_j<=i(s_i)
//   o_i  = W_up,t^V (sum_j p_ij c_v,j) + mu^V_t
//
// Tensor-core path (bf16 storage, d = 128, the ranks of launch_prefill): one CTA per (one or two
// 128-query tiles, sequence, head), four warps that move data and issue products, and two softmax
// groups of four warps with a thread per query row:
//   warp 0      K producer: W_up,t^K by TMA, then per page of 64 keys the K-plane (one bulk copy: its
//               granule-interleaved layout is already the core-matrix layout of a K-major MMA operand),
//               and W_up,t^V for the epilogue (TMA; into room of its own or, at (192, 320), over q~ and
//               the K ring once the last score product has read them)
//   warp 2      V producer, decoupled from the K-planes so that neither ring waits on the other: one TMA
//               load with 128-byte swizzle per 64 latent columns of a page (an MN-major operand)
//   warp 1      Q~ and S issuer and TMEM owner:
//                 Q~ = Q W_up,t^K             M=128, N=r_k, K=d
//                 S_j = Q~ C_k,j^T            M=128, N=64,  K=r_k
//   warp 3      PV and output issuer, so that neither MMA stream waits behind the other's barriers:
//                 O += P_j C_v,j              M=128, N=r_v (split at 256), K=64, P_j in TMEM
//                 out = (O/l) W_up,t^V^T      M=128, N=2 x 64, K=r_v, O/l as hi + lo in TMEM
//               The issuing warps run converged, one elected thread per product, on uniform values
//               (page counts broadcast from one lane, TMEM address 0): issued from a one-thread branch a
//               product cost that thread about 80 cycles, more than the product itself
//   warps 4-11  the softmax groups: Q and Q~ into bf16 operands, causal mask on diagonal pages, online
//               softmax in the exp2 domain, P to TMEM as packed bf16 (no shared memory, no proxy fence),
//               O rescaled in TMEM only when a row maximum grows by more than 2^8, V rows past the
//               prompt zeroed on its last page, then the epilogue.
// With two tiles per CTA each group owns one.  With one tile the groups take its pages in turn, so that
// one's softmax (about 1000 cycles from scores to weights) runs beside the other's: the running maximum
// goes from page to page through shared memory and a named barrier per warp pair, each group keeps its
// own row sums, and they meet after the last page.
// Accumulators are fp32 in TMEM; operands are bf16 (q~ carries scale * log2 e).  At (72, 120) q~, P
// and O / l are sums of three bf16 parts (24 significant bits; three times the products): that shape was
// served in fp32 by the CUDA cores, and its results stay as exact.  (Two parts, 16 bits, took 56 us instead
// of 70 for 3 ragged prompts, but with scores in the hundreds five times as many outputs were rounded the
// wrong way as with fp32 sums.)  So at (18, 30), whose rows are not whole 16-byte words: there the producer
// warps move pages and W_up through registers.
//
// Bound by the tensor pipe and the shared memory that feeds it: a (192, 320) page takes 640 cycles of PV
// products and 576 of score products (a 128 x 64 x 16 product reads 6 KB, 48 cycles of shared memory for
// 32 of arithmetic).  Measured, 16 heads, from the kernel with one tile, eight softmax warps in pairs and
// one-thread issue: 4 x 8192 tokens at (192, 320) 1955 -> 1656 us (1370 TFLOP/s; the clock falls under
// the power limit), at (96, 160) 1445 -> 919 us, at (128, 128) 1445 -> 975 us; a tile of 2 pages from
// launch to output 18 -> 10 us (W_up was staged by one warp's cp.async, W_up,t^V only after the last
// page, and the hi and lo projections followed each other through shared memory).  From the CUDA cores:
// (72, 120), 300 tokens 265 -> 11.2 us, 3 ragged prompts of 3531 tokens 8330 -> 70 us; (18, 30), 1000 tokens
// 720 -> 25.2 us, 8192 tokens 43.1 -> 0.53 ms (its producer warps bound it: their pairs' places kept in
// registers changed nothing; three pages in flight spilled and cost 15 %).
//
// CUDA-core path (fp32 storage, other ranks, d != 128, fp32 inputs at (72, 120) and (18, 30)): one CTA
// per (query, sequence, head), fp32 throughout.
#include <cuda_runtime.h>

#include <algorithm>

#include "lla_device.cuh"
#include "lla_internal.h"
#include "lla_tcgen05.cuh"
#include "lla_tmap.h"
#include "lla_units.cuh"

namespace lla {
namespace {

constexpr int kBM = 128;         // queries per tile
constexpr int kPT = 64;          // keys per page
constexpr int kGroup = 128;      // threads of a softmax group: one per query row of a tile
constexpr int kSWarp0 = 4;       // K producer, S issuer, V producer, PV issuer, then the two groups
constexpr int kPThreads = kSWarp0 * 32 + 2 * kGroup;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleLog2 = 8.f;  // rescale O only when a row maximum grows by more

struct PParams {
    int T, H, loop, io_bf16;
    float scale_log2;
    const float *mu_v;
    const void *w_up_k, *w_up_v;  // for NARROW rows (others come by tensor map)
    const char *pool;
    int64_t num_blocks;
    int head_page_bytes;
    const int32_t *block_table;
    int max_blocks;
    const int32_t *cu_seqlens;
    int max_len;
    const void *q;
    void *out;
    unsigned *err;
    // rotary positions after reconstruction: keys rebuilt and rotated, [B][kpps][H] pages of
    // 64 keys x d in the K-plane layout, and queries rotated and scaled, [Ntok][H][d], bf16
    const char *krot;
    const void *qrot;
    int kpps;
    int64_t qrows;  // rows of the rotated-query buffer (B * max_len)
    int B, first;   // prompts; (head, prompt) pairs that run one after the other, before the last ones together
    FastDiv by_tiles, by_rest, by_prompts;  // by the tiles of a pair, the pairs that run together, the prompts
};

// Shared-memory and TMEM plan of the tensor-core kernel for ranks (RK, RV), d = 128, NT query tiles
// per CTA and QP bf16 parts of q~ and of the softmax weights.  Offsets are multiples of 1024 bytes
// from a 1024-byte aligned base (128-byte swizzle atoms).  With ROPE the scores are formed from
// rebuilt, rotated keys of width d instead of latents of width RK.
template <int RK, int RV, int NT, bool ROPE, int QP>
struct PF {
    static constexpr int D = 128;
    // rows that are not whole 16-byte words have no bulk layout and no tensor map: the producer warps move
    // them through registers into the layouts that the copies would leave
    static constexpr bool NARROW = RK % 8 != 0 || RV % 8 != 0;
    static constexpr int RKX = (RK + 15) / 16 * 16;  // padded with zero columns of q~ and zero granules
    static constexpr int RS = ROPE ? D : RKX;        // contraction width of the scores
    static constexpr int ORV = (RV + 15) / 16 * 16;  // O columns of a tile
    static constexpr int VATOMS = (RV + 63) / 64;    // 64-column boxes of a V page, of W_up,t^V
    static constexpr int KATOMS = (RK + 63) / 64;    // 64-column boxes of W_up,t^K
    static constexpr int N0 = ORV > 256 ? 256 : ORV; // PV MMA split on atom boundaries
    static constexpr int N1 = ORV - N0;
    static constexpr int KPAGE = kPT * RS * 2;
    static constexpr int KCOPY = ROPE ? KPAGE : NARROW ? 0 : kPT * RK * 2;  // the rest of a stage is zeroed once
    static constexpr int VPAGE = VATOMS * kPT * 128;
    static constexpr int QT1 = kBM * RS * 2;         // q~ (or rotated q) operand: one part of one tile
    static constexpr int QT = NT * QP * QT1;
    static constexpr int QA1 = kBM * D * 2;          // q operand of one tile (prologue)
    static constexpr int WK = KATOMS * D * 128;      // W_up,t^K operand (prologue)
    static constexpr int WV = VATOMS * D * 128;      // W_up,t^V operand (epilogue)
    static constexpr int OP = QP > 1 ? 3 : 2;        // bf16 parts of O / l in the epilogue
    static constexpr int BUDGET = 222 * 1024;
    // W_up,t^V has room of its own, or takes q~'s and the K ring's once every score product is done
    static constexpr bool WVOWN = QT + 2 * KPAGE + 3 * VPAGE + WV <= BUDGET;
    static constexpr int WKOWN = NARROW ? WK : 0;  // NARROW: W_up,t^K has room of its own too
    static constexpr int LEFT = BUDGET - QT - (WVOWN ? WV : 0) - WKOWN;
    static constexpr int STV0 = (LEFT - 2 * KPAGE) / VPAGE;
    static constexpr int STV = STV0 > 4 ? 4 : STV0;
    static constexpr int STK0 = (LEFT - STV * VPAGE) / KPAGE;
    static constexpr int STK = STK0 > 4 ? 4 : STK0;
    static constexpr int oQT = 0;
    static constexpr int oK = oQT + QT;
    static constexpr int oV = oK + STK * KPAGE;
    static constexpr int oW = oV + STV * VPAGE;
    static constexpr int oEnd = oW + WKOWN + (WVOWN ? WV : 0);
    static constexpr int oQA = oV;                        // the prologue's q operands alias the V ring
    static constexpr int oWK = WVOWN ? oW : oV + NT * QA1;
    static constexpr int oWV = WVOWN ? oW + WKOWN : oQT;
    static constexpr int oM = oEnd;                       // NT = 1: [128] running maxima
    static constexpr int oX = oM + kBM * 4;               // NT = 1: [2 groups][128] (maximum, sum)
    static constexpr int oBar = oX + 2 * kBM * 8;
    static constexpr int NBAR = 48;
    static constexpr int SMEM = 1024 + oBar + NBAR * 8;
    // TMEM columns: S of each group, P of each group (packed pairs), O of each tile; q~ starts in O
    static constexpr uint32_t TM_S = 0, TM_P = 2 * kPT, TM_O = TM_P + 2 * QP * (kPT / 2), TM_COLS = 512;
    static_assert(RK % 2 == 0 && RV % 2 == 0 && RKX <= 256 && RKX <= ORV, "ranks");
    static_assert(!NARROW || (RK <= 64 && RV <= 64 && WVOWN && !ROPE), "one 64-column box per row");
    static_assert(TM_O + NT * ORV <= TM_COLS && N1 <= 256 && N1 % 16 == 0, "TMEM columns");
    static_assert(OP == 2 || (NT == 1 && VATOMS * 32 <= 2 * QP * (kPT / 2)), "the third part over the weights");
    static_assert(STK >= 2 && STV >= 2, "pipeline depth");
    static_assert(KPAGE % 1024 == 0 && QT1 % 1024 == 0, "align");
    static_assert(NT * QA1 <= STV * VPAGE && (WVOWN ? WK <= WV : NT * QA1 + WK <= STV * VPAGE), "prologue operands fit");
    static_assert(WVOWN || WV <= QT + STK * KPAGE, "epilogue operand fits");
    static_assert(SMEM <= 227 * 1024, "shared memory");
};

// barrier indices ([2]: by softmax group, which is the tile for NT = 2)
enum {
    kBWk = 0, kBWv, kBSfin, kBOfin /* [2] */, kBQa = 5 /* [2] */, kBQt = 7 /* [2] */, kBQs = 9 /* [2] */,
    kBOa = 11 /* [2] */, kBOut = 13 /* [2] */, kBOfree = 15 /* [2] */,
    kBSfull = 17 /* [2] */, kBSfree = 19, kBPfull = 21, kBPfree = 23,
    kBKfull = 25 /* [4] */, kBKempty = 29, kBVfull = 33, kBVempty = 37,
    kBAbort = 41,  // slot used as the CTA's abort flag
    kBTmem = 42    // and as the TMEM address
};

// Two consecutive TMEM loads of 32 columns each, waited for once.
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float (&v)[64]) {
    uint32_t a[32], b[32];
    tmem_ld32_nowait(taddr, a);
    tmem_ld32_nowait(taddr + 32, b);
    tmem_wait_ld(a);
    tmem_wait_ld(b);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
        v[i] = __uint_as_float(a[i]);
        v[32 + i] = __uint_as_float(b[i]);
    }
}

// NARROW rows through registers, by a whole warp: R columns (pairs of bf16) of 64 or 128 rows.
// A page's plane is loaded as 16-byte words (load), then its pairs are stored (store) at
//   K-plane (4-byte granules, pair c of row i at c*256 + i*4): granule c / 4 of row i at
//           (c / 4)*1024 + i*16, the core-matrix layout of a K-major operand;
//   V-plane and W_up rows (row-major): row i of 128 bytes, 16-byte chunk c / 4 at (c / 4) ^ (i % 8), the
//           128-byte swizzle of a tensor load.
template <int R, int ROWS>
struct NarrowRows {
    static constexpr int WORDS = ROWS * (R / 2);         // pairs
    static constexpr int NV = (WORDS / 4 + 31) / 32;     // 16-byte words per lane
    uint4 v[NV];
    __device__ __forceinline__ void load(const char *src, int lane) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
            if (k * 32 + lane < WORDS / 4) v[k] = reinterpret_cast<const uint4 *>(src)[k * 32 + lane];
    }
    template <bool KPLANE>
    __device__ __forceinline__ void store(char *dst, int lane) const {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const int w0 = (k * 32 + lane) * 4;
            if (w0 >= WORDS) break;
            const uint32_t w[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int x = w0 + e;
                const int c = KPLANE ? x / ROWS : x % (R / 2), i = KPLANE ? x % ROWS : x / (R / 2);
                char *at = KPLANE ? dst + (c >> 2) * (ROWS * 16) + i * 16 + (c & 3) * 4
                                  : dst + i * 128 + (((c >> 2) ^ (i & 7)) << 4) + (c & 3) * 4;
                *reinterpret_cast<uint32_t *>(at) = w[e];
            }
        }
    }
};

template <int RK, int RV, int NT, bool ROPE, int QP>
__global__ void __launch_bounds__(kPThreads, 1)
    prefill_tc_kernel(const __grid_constant__ CUtensorMap tv, const __grid_constant__ CUtensorMap twk,
                      const __grid_constant__ CUtensorMap twv, const __grid_constant__ PParams p) {
    using F = PF<RK, RV, NT, ROPE, QP>;
    constexpr int D = F::D;
    extern __shared__ __align__(1024) char sm_raw[];
    char *sm = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + F::oBar);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(bar + kBAbort);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + kBTmem);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;

    const int nqt = (p.max_len + NT * kBM - 1) / (NT * kBM);
    int qt = blockIdx.x, b = blockIdx.y, h = blockIdx.z;
    if (p.first >= 0) {  // pair after pair, then tile by tile every pair of the rest
        int pair = div_by(blockIdx.x, p.by_tiles);
        qt = blockIdx.x - pair * nqt;
        if (pair >= p.first) {
            const int r = blockIdx.x - p.first * nqt;
            qt = div_by(r, p.by_rest);
            pair = p.first + r - qt * (p.H * p.B - p.first);
        }
        h = div_by(pair, p.by_prompts);
        b = pair - h * p.B;
    }
    qt = nqt - 1 - qt;  // longest causal ranges first
    pdl_wait();
    const int q0 = p.cu_seqlens[b];
    const int L = p.cu_seqlens[b + 1] - q0;
    if (L > p.max_len || L < 0 || (ROPE && static_cast<int64_t>(q0) + L > p.qrows)) {
        if (tid == 0 && qt == nqt - 1) atomicOr(p.err, LLA_DEVERR_CONTEXT);
        return;
    }
    const int i0 = qt * NT * kBM;
    if (i0 >= L) return;  // uniform over the CTA, before any barrier or TMEM use
    // pages 0 .. np(g) - 1 hold every key of tile g (none past the prompt); NP: of the CTA
    auto np = [&](int g) { return i0 + g * kBM < L ? (min(L, i0 + (g + 1) * kBM) - 1) / kPT + 1 : 0; };
    const int NP = max(np(0), NT == 2 ? np(1) : 0);
    const int wrow = (h * p.T + p.loop) * D;  // first row of W_up,t of this head
    const int32_t *bt = p.block_table + static_cast<int64_t>(b) * p.max_blocks;

    if (tid == 0) {
        constexpr uint32_t fills = F::NARROW ? 32 : 1;  // arrivals of a filled stage
        mbar_init(&bar[kBWk], fills);
        mbar_init(&bar[kBWv], fills);
        mbar_init(&bar[kBSfin], 1);
        for (int g = 0; g < 2; ++g) {
            mbar_init(&bar[kBOfin + g], 1);
            mbar_init(&bar[kBQa + g], kGroup);
            mbar_init(&bar[kBQt + g], 1);
            mbar_init(&bar[kBQs + g], NT == 1 ? 2 * kGroup : kGroup);
            mbar_init(&bar[kBOa + g], NT == 1 ? 2 * kGroup : kGroup);
            mbar_init(&bar[kBOut + g], 1);
            mbar_init(&bar[kBOfree + g], kGroup);
            mbar_init(&bar[kBSfull + g], 1);
            mbar_init(&bar[kBSfree + g], kGroup);
            mbar_init(&bar[kBPfull + g], kGroup);
            mbar_init(&bar[kBPfree + g], 1);
        }
        for (int s = 0; s < F::STK; ++s) {
            mbar_init(&bar[kBKfull + s], fills);
            mbar_init(&bar[kBKempty + s], 1);
        }
        for (int s = 0; s < F::STV; ++s) {
            mbar_init(&bar[kBVfull + s], fills);
            mbar_init(&bar[kBVempty + s], 1);
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc(tslot, F::TM_COLS);
    if constexpr (F::KPAGE > F::KCOPY) {  // the K granules past r_k, against zero columns of q~
        for (int s = 0; s < F::STK; ++s)
            for (int i = tid; i < (F::KPAGE - F::KCOPY) / 16; i += kPThreads)
                reinterpret_cast<uint4 *>(sm + F::oK + s * F::KPAGE + F::KCOPY)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    if constexpr (F::NARROW) {  // the columns past the ranks of W_up (W_up,t^V after W_up,t^K) and of the V ring
        for (int i = tid; i < (F::WK + F::WV) / 16; i += kPThreads)
            reinterpret_cast<uint4 *>(sm + F::oWK)[i] = make_uint4(0, 0, 0, 0);
        fence_proxy_async_smem();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // the whole of TMEM is allocated, so its address is 0: a constant, and the page counts broadcast
    // from one lane, keep the issuing warps' code uniform
    constexpr uint32_t tmem = 0;
    const int np0 = __shfl_sync(0xffffffffu, np(0), 0), np1 = __shfl_sync(0xffffffffu, NT == 2 ? np(1) : 0, 0);
    auto npu = [&](int g) { return g ? np1 : np0; };
    const int NPU = max(np0, np1);

    if (warp == 0) {
        // ----------------------------------------------- producer: W_up,t^K, K-planes, W_up,t^V
        if constexpr (F::NARROW) {
            {
                NarrowRows<RK, F::D> wk;
                wk.load(static_cast<const char *>(p.w_up_k) + static_cast<int64_t>(wrow) * RK * 2, lane);
                wk.template store<false>(sm + F::oWK, lane);
                fence_proxy_async_smem();
                mbar_arrive(&bar[kBWk]);
            }
            // page j + 1 is on its way while page j waits for its stage
            NarrowRows<RK, kPT> cur, nxt;
            auto page = [&](int j) {
                int32_t blk = bt[j];
                if (blk < 0 || blk >= p.num_blocks) {
                    if (lane == 0) atomicOr(p.err, LLA_DEVERR_BLOCK_ID);
                    blk = 0;
                }
                return p.pool + (static_cast<int64_t>(blk) * p.H + h) * p.head_page_bytes;
            };
            cur.load(page(0), lane);
            for (int j = 0; j < NPU; ++j) {
                if (j + 1 < NPU) nxt.load(page(j + 1), lane);
                const int s = j % F::STK;
                // (after a failed wait the phases go on: no copy is in flight that could land late)
                mbar_wait(&bar[kBKempty + s], ((j / F::STK) & 1) ^ 1u, abort_flag, p.err);
                cur.template store<true>(sm + F::oK + s * F::KPAGE, lane);
                fence_proxy_async_smem();
                mbar_arrive(&bar[kBKfull + s]);
                cur = nxt;
                if (j == min(F::STK, NPU) - 1) {
                    NarrowRows<RV, F::D> wv;
                    wv.load(static_cast<const char *>(p.w_up_v) + static_cast<int64_t>(wrow) * RV * 2, lane);
                    wv.template store<false>(sm + F::oWV, lane);
                    fence_proxy_async_smem();
                    mbar_arrive(&bar[kBWv]);
                }
            }
        } else if (lane == 0) {
            if constexpr (!ROPE) {  // rows e of W_up,t^K as the MN-major operand of Q~
                mbar_arrive_expect_tx(&bar[kBWk], F::WK);
#pragma unroll
                for (int a = 0; a < F::KATOMS; ++a)
                    tma_load_2d(sm + F::oWK + a * (D * 128), &twk, a * 64, wrow, &bar[kBWk]);
            }
            const uint64_t pol = policy_evict_first();
            int nk = 0;  // copies issued
            auto load_wv = [&] {
                mbar_arrive_expect_tx(&bar[kBWv], F::WV);
#pragma unroll
                for (int a = 0; a < F::VATOMS; ++a)
                    tma_load_2d(sm + F::oWV + a * (D * 128), &twv, a * 64, wrow, &bar[kBWv]);
            };
            bool wv = false;
            for (int j = 0; j < NP; ++j) {
                const int s = j % F::STK;
                const uint32_t ph = (j / F::STK) & 1;
                int32_t blk = bt[j];
                if (blk < 0 || blk >= p.num_blocks) {
                    atomicOr(p.err, LLA_DEVERR_BLOCK_ID);
                    blk = 0;
                }
                const int64_t hp = static_cast<int64_t>(blk) * p.H + h;  // head page index
                // the latent K-plane of the page, or its rebuilt and rotated keys
                const char *src = ROPE ? p.krot + ((static_cast<int64_t>(b) * p.kpps + j) * p.H + h) * F::KPAGE
                                       : p.pool + hp * p.head_page_bytes;
                if (!mbar_wait(&bar[kBKempty + s], ph ^ 1u, abort_flag, p.err) || *abort_flag) break;
                mbar_arrive_expect_tx(&bar[kBKfull + s], F::KCOPY);
                bulk_g2s(sm + F::oK + s * F::KPAGE, src, F::KCOPY, &bar[kBKfull + s], pol);
                ++nk;
                // W_up,t^V's own room held W_up,t^K until every q~ was formed
                if (F::WVOWN && !wv && j == min(F::STK, NP) - 1) {
                    bool ok = true;
                    if constexpr (!ROPE) {
                        for (int g = 0; g < NT; ++g)
                            if (np(g) > 0) ok = mbar_wait(&bar[kBQt + g], 0, abort_flag, p.err) && ok;
                    }
                    if (ok) {
                        load_wv();
                        wv = true;
                    }
                }
            }
            // every copy has landed before the ring is reused or the CTA exits, even after an
            // abort (no copy is issued once a wait has failed)
            volatile int never = 0;
            for (int j = max(0, nk - F::STK); j < nk; ++j)
                mbar_wait(&bar[kBKfull + j % F::STK], (j / F::STK) & 1, &never, p.err);
            if constexpr (!ROPE) mbar_wait(&bar[kBWk], 0, &never, p.err);
            if (!F::WVOWN && mbar_wait(&bar[kBSfin], 0, abort_flag, p.err) && !*abort_flag) {
                load_wv();  // over q~ and the K ring, which every score product has read
                wv = true;
            }
            if (wv) mbar_wait(&bar[kBWv], 0, &never, p.err);
        }
        __syncwarp();
    } else if (warp == 2) {
        // ---------------------------------------------------------------------- V producer
        if constexpr (F::NARROW) {
            for (int g = 0; g < NT; ++g)
                if (npu(g) > 0) mbar_wait(&bar[kBQt + g], 0, abort_flag, p.err);
            // the ring held the prologue's q operands: its columns past r_v become zeros again
            for (int i = lane; i < F::STV * F::VPAGE / 16; i += 32)
                reinterpret_cast<uint4 *>(sm + F::oV)[i] = make_uint4(0, 0, 0, 0);
            __syncwarp();
            NarrowRows<RV, kPT> cur, nxt;
            auto page = [&](int j) {
                int32_t blk = bt[j];
                if (blk < 0 || blk >= p.num_blocks) blk = 0;  // flagged by the K producer
                return p.pool + (static_cast<int64_t>(blk) * p.H + h) * p.head_page_bytes + kPT * RK * 2;
            };
            cur.load(page(0), lane);
            for (int j = 0; j < NPU; ++j) {
                if (j + 1 < NPU) nxt.load(page(j + 1), lane);
                const int s = j % F::STV;
                mbar_wait(&bar[kBVempty + s], ((j / F::STV) & 1) ^ 1u, abort_flag, p.err);
                cur.template store<false>(sm + F::oV + s * F::VPAGE, lane);
                fence_proxy_async_smem();
                mbar_arrive(&bar[kBVfull + s]);
                cur = nxt;
            }
        } else if (lane == 0) {  // V-planes: one TMA tensor load with 128-byte swizzle per 64 columns
            // the V ring aliases the prologue operands: wait until q~ has been computed
            bool ok = true;
            if constexpr (!ROPE) {
                for (int g = 0; g < NT; ++g)
                    if (np(g) > 0) ok = mbar_wait(&bar[kBQt + g], 0, abort_flag, p.err) && ok;
            }
            int nv = 0;  // copies issued
            for (int j = 0; j < NP && ok; ++j) {
                const int s = j % F::STV;
                const uint32_t ph = (j / F::STV) & 1;
                int32_t blk = bt[j];
                if (blk < 0 || blk >= p.num_blocks) blk = 0;  // flagged by the K producer
                const int64_t hp = static_cast<int64_t>(blk) * p.H + h;
                if (!mbar_wait(&bar[kBVempty + s], ph ^ 1u, abort_flag, p.err) || *abort_flag) break;
                mbar_arrive_expect_tx(&bar[kBVfull + s], F::VPAGE);
                char *vs = sm + F::oV + s * F::VPAGE;
#pragma unroll
                for (int a = 0; a < F::VATOMS; ++a)
                    tma_load_3d(vs + a * (kPT * 128), &tv, a * 64, 0, static_cast<int>(hp), &bar[kBVfull + s]);
                ++nv;
            }
            volatile int never = 0;  // as for the K ring
            for (int j = max(0, nv - F::STV); j < nv; ++j)
                mbar_wait(&bar[kBVfull + j % F::STV], (j / F::STV) & 1, &never, p.err);
        }
        __syncwarp();
    } else if (warp == 1) {
        // -------------------------------------------------------------- Q~ and S MMA issuer
        {
            const uint32_t base = smem_addr(sm);
            if constexpr (!ROPE) {
                mbar_wait_warp(&bar[kBWk], 0, abort_flag, p.err);
                constexpr uint32_t idq = umma_idesc_bf16(128, F::RKX, 0, 1);
                const uint64_t dwk = umma_desc_sw128_mn(base + F::oWK, D * 128);
                for (int g = 0; g < NT; ++g) {
                    if (npu(g) == 0) continue;
                    mbar_wait_warp(&bar[kBQa + g], 0, abort_flag, p.err);
                    tc_fence_after();
                    const uint64_t dqa = umma_desc(base + F::oQA + g * F::QA1, 2048, 128);
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        umma_bf16_warp(tmem + F::TM_O + g * F::ORV, dqa + ks * (4096 >> 4), dwk + ks * (2048 >> 4), idq, ks > 0);
                    umma_commit_warp(&bar[kBQt + g]);
                }
            }
            constexpr uint32_t ids = umma_idesc_bf16(128, kPT, 0, 0);
            // descriptors are built once; a byte offset moves the start-address field by offset/16
            const uint64_t dq0 = umma_desc(base + F::oQT, 2048, 128);
            const uint64_t dk0 = umma_desc(base + F::oK, 1024, 128);
#pragma unroll 1
            for (int j = 0; j < NPU; ++j) {
                const int sk = j % F::STK;
                mbar_wait_warp(&bar[kBKfull + sk], (j / F::STK) & 1, abort_flag, p.err);
                const uint64_t dk = dk0 + static_cast<uint64_t>(sk * (F::KPAGE >> 4));
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    // NT = 2: tile i's softmax group takes page j; NT = 1: the groups take turns
                    const int g = NT == 2 ? i : (j & 1), jj = NT == 2 ? j : (j >> 1);
                    if (NT == 2 && j >= npu(i)) continue;
                    if (j == 0) mbar_wait_warp(&bar[kBQs + (NT == 2 ? g : 0)], 0, abort_flag, p.err);
                    if (jj > 0) mbar_wait_warp(&bar[kBSfree + g], (jj - 1) & 1, abort_flag, p.err);
                    tc_fence_after();
                    const uint32_t ds = tmem + F::TM_S + g * kPT;
#pragma unroll
                    for (int part = 0; part < QP; ++part) {
                        const uint64_t dq = dq0 + static_cast<uint64_t>((i * QP + part) * (F::QT1 >> 4));
#pragma unroll
                        for (int ks = 0; ks < F::RS / 16; ++ks)
                            umma_bf16_warp(ds, dq + ks * (4096 >> 4), dk + ks * (2048 >> 4), ids, part > 0 || ks > 0);
                    }
                    umma_commit_warp(&bar[kBSfull + g]);
                }
                umma_commit_warp(&bar[kBKempty + sk]);
            }
            umma_commit_warp(&bar[kBSfin]);
            // every product of this thread has completed before TMEM is released, even after an
            // abort (when the softmax warps stop waiting for them)
            volatile int never = 0;
            mbar_wait_warp(&bar[kBSfin], 0, &never, p.err);
        }
        __syncwarp();
    } else if (warp == 3) {
        // ----------------------------------------------------------- PV and output MMA issuer
        {
            const uint32_t base = smem_addr(sm);
            constexpr uint32_t idv0 = umma_idesc_bf16(128, F::N0, 0, 1);
            constexpr uint32_t idv1 = umma_idesc_bf16(128, F::N1 > 0 ? F::N1 : 16, 0, 1);
            const uint64_t dv0 = umma_desc_sw128_mn(base + F::oV, kPT * 128);
#pragma unroll 1
            for (int j = 0; j < NPU; ++j) {
                const int sv = j % F::STV;
                mbar_wait_warp(&bar[kBVfull + sv], (j / F::STV) & 1, abort_flag, p.err);
                const uint64_t dv = dv0 + static_cast<uint64_t>(sv * (F::VPAGE >> 4));
#pragma unroll
                for (int i = 0; i < NT; ++i) {
                    const int g = NT == 2 ? i : (j & 1), jj = NT == 2 ? j : (j >> 1);
                    if (NT == 2 && j >= npu(i)) continue;
                    mbar_wait_warp(&bar[kBPfull + g], jj & 1, abort_flag, p.err);
                    tc_fence_after();
                    const uint32_t to = tmem + F::TM_O + i * F::ORV;
                    const bool acc = j > 0;
#pragma unroll
                    for (int part = 0; part < QP; ++part)
#pragma unroll
                        for (int ks = 0; ks < kPT / 16; ++ks) {
                            const uint32_t tp = tmem + F::TM_P + (g * QP + part) * (kPT / 2) + ks * 8;
                            umma_bf16_ts_warp(to, tp, dv + ks * (2048 >> 4), idv0, acc || part > 0 || ks > 0);
                            if constexpr (F::N1 > 0)
                                umma_bf16_ts_warp(to + F::N0, tp, dv + ((F::N0 / 64) * (kPT * 128) >> 4) + ks * (2048 >> 4), idv1,
                                             acc || part > 0 || ks > 0);
                        }
                    umma_commit_warp(&bar[kBPfree + g]);
                    if (NT == 2 && j == npu(i) - 1) umma_commit_warp(&bar[kBOfin + i]);
                }
                umma_commit_warp(&bar[kBVempty + sv]);
            }
            if constexpr (NT == 1) umma_commit_warp(&bar[kBOfin]);
            // out = (O / l) W_up,t^V^T in two halves of 64 output columns, with O / l = hi + lo as two
            // bf16 operands in TMEM, so that the projection sees O / l to about 16 significant bits.
            // Chunk c of 64 latent columns: hi in the first half of its columns, lo in the second.
            mbar_wait_warp(&bar[kBWv], 0, abort_flag, p.err);
            constexpr uint32_t ido = umma_idesc_bf16(128, D / 2, 0, 0);
            const uint64_t dwv = umma_desc_sw128_k(base + F::oWV);
            auto project = [&](int tile, int half, uint32_t ds, uint64_t *done) {
                bool acc = false;
#pragma unroll
                for (int c = 0; c < F::VATOMS; ++c) {
                    constexpr int last = F::ORV - (F::VATOMS - 1) * 64;  // columns of the last chunk
                    const int cols = c == F::VATOMS - 1 ? last : 64;
#pragma unroll
                    for (int part = 0; part < F::OP; ++part)
#pragma unroll
                        for (int ks = 0; ks < 4; ++ks) {
                            if (ks * 16 >= cols) continue;
                            const uint32_t at = part == 2 ? F::TM_P + c * 32 : F::TM_O + tile * F::ORV + c * 64 + part * (cols / 2);
                            umma_bf16_ts_warp(ds, tmem + at + ks * 8,
                                         dwv + ((c * (D * 128) + half * (64 * 128) + ks * 32) >> 4), ido, acc);
                            acc = true;
                        }
                }
                umma_commit_warp(done);
            };
            if constexpr (NT == 1) {
                mbar_wait_warp(&bar[kBOa], 0, abort_flag, p.err);
                tc_fence_after();
                for (int g = 0; g < 2; ++g) project(0, g, tmem + F::TM_S + g * kPT, &bar[kBOut + g]);
            } else {
                for (int half = 0; half < 2; ++half)
                    for (int g = 0; g < 2; ++g) {
                        if (npu(g) == 0) continue;
                        // the first half has been read (so its product's phase has passed; after a failed
                        // wait that product is awaited itself, so that the phases stay in step)
                        if (!mbar_wait_warp(half ? &bar[kBOfree + g] : &bar[kBOa + g], 0, abort_flag, p.err) && half) {
                            volatile int never = 0;
                            mbar_wait_warp(&bar[kBOut + g], 0, &never, p.err);
                        }
                        tc_fence_after();
                        project(g, half, tmem + F::TM_S + g * kPT, &bar[kBOut + g]);
                    }
            }
            // as for the S issuer: this thread's last commits
            volatile int never = 0;
            for (int g = 0; g < 2; ++g) {
                if (NT == 2 && npu(g) == 0) continue;
                mbar_wait_warp(&bar[kBOut + g], NT == 1 ? 0 : 1, &never, p.err);
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------------------ softmax and epilogue
        // warps 4..7 are group 0, 8..11 group 1; thread = query row (TMEM lane) of the group's tile.
        // NT = 2: group g owns tile g.  NT = 1: the groups take the tile's pages in turn.
        const int quarter = warp & 3;
        const int g = (warp - kSWarp0) >> 2;
        const int tile = NT == 2 ? g : 0;
        const int row = quarter * 32 + lane;
        const uint32_t tl = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
        const uint32_t ts = tl + F::TM_S + g * kPT, to = tl + F::TM_O + tile * F::ORV;
        const uint32_t tp = tl + F::TM_P + g * QP * (kPT / 2);
        const int qi = i0 + tile * kBM + row;
        const bool valid_row = qi < L;
        const int64_t qrow = (static_cast<int64_t>(q0) + qi) * p.H + h;
        const int NPg = np(tile);
        if (NT == 1 || NPg > 0) {
        if constexpr (ROPE) {
            // the rotated, scaled q row -> the score operand directly (NT = 1: half a row per group)
            char *qt_ = sm + F::oQT + tile * F::QT1 + row * 16;
            const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const char *>(p.qrot) + qrow * D * 2);
            constexpr int NC = NT == 1 ? D / 16 : D / 8;
            const int c0 = NT == 1 ? g * NC : 0;
            uint4 v[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) v[c] = valid_row ? src[c0 + c] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int c = 0; c < NC; ++c) *reinterpret_cast<uint4 *>(qt_ + (c0 + c) * 2048) = v[c];
            fence_proxy_async_smem();
            mbar_arrive(&bar[kBQs + (NT == 2 ? g : 0)]);
        } else {
            // q row -> bf16 K-major operand: chunk c at c*2048 + row*16 (NT = 1: group 0)
            if (NT == 2 || g == 0) {
                char *qa = sm + F::oQA + tile * F::QA1 + row * 16;
                if (p.io_bf16) {
                    const uint4 *src = reinterpret_cast<const uint4 *>(static_cast<const char *>(p.q) + qrow * D * 2);
                    uint4 v[D / 8];
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) v[c] = valid_row ? src[c] : make_uint4(0, 0, 0, 0);
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) *reinterpret_cast<uint4 *>(qa + c * 2048) = v[c];
                } else {
                    const float4 *src = reinterpret_cast<const float4 *>(static_cast<const char *>(p.q) + qrow * D * 4);
#pragma unroll
                    for (int c = 0; c < D / 8; ++c) {
                        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b2 = a;
                        if (valid_row) {
                            a = src[2 * c];
                            b2 = src[2 * c + 1];
                        }
                        *reinterpret_cast<uint4 *>(qa + c * 2048) =
                            make_uint4(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w), pack_bf16x2(b2.x, b2.y),
                                       pack_bf16x2(b2.z, b2.w));
                    }
                }
                fence_proxy_async_smem();
                mbar_arrive(&bar[kBQa + g]);
            }
            // q~ (scaled into the exp2 domain) -> bf16 K-major operand, in QP parts (each the rounding
            // of what the part before leaves); NT = 1: the groups take its 16-column chunks in turn
            mbar_wait(&bar[kBQt + tile], 0, abort_flag, p.err);
            tc_fence_after();
            char *qt_ = sm + F::oQT + tile * QP * F::QT1 + row * 16;
            const float sc = p.scale_log2;
#pragma unroll 1
            for (int c0 = (NT == 1 ? g * 16 : 0); c0 < F::RKX; c0 += (NT == 1 ? 32 : 16)) {
                float v[16];
                tmem_ld16(to + c0, v);
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] *= sc;
#pragma unroll
                for (int part = 0; part < QP; ++part) {
#pragma unroll
                    for (int k = 0; k < 16; k += 8) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            w[e] = pack_bf16x2(v[k + 2 * e], v[k + 2 * e + 1]);
                            if (part + 1 < QP) {
                                const float2 f = bf2_to_f2(w[e]);
                                v[k + 2 * e] -= f.x;
                                v[k + 2 * e + 1] -= f.y;
                            }
                        }
                        *reinterpret_cast<uint4 *>(qt_ + part * F::QT1 + ((c0 + k) / 8) * 2048) = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
            fence_proxy_async_smem();
            tc_fence_before();
            mbar_arrive(&bar[kBQs + (NT == 2 ? g : 0)]);
        }

        const int lim = min(qi, L - 1);  // keys 0..lim are visible to this row
        float *mrun = reinterpret_cast<float *>(sm + F::oM);
        float m = -INFINITY, l = 0.f;
        // jj counts this group's pages
#pragma unroll 1
        for (int j = NT == 1 ? g : 0, jj = 0; j < NPg; j += NT == 1 ? 2 : 1, ++jj) {
            const int kb = j * kPT;
            mbar_wait(&bar[kBSfull + g], jj & 1, abort_flag, p.err);
            tc_fence_after();
            float x[kPT];
            tmem_ld64(ts, x);
            tc_fence_before();
            mbar_arrive(&bar[kBSfree + g]);
            if (kb + kPT - 1 > i0 + tile * kBM) {  // a page on the diagonal (or past the prompt): mask
                const int nv = lim - kb;           // keys c <= nv are visible
#pragma unroll
                for (int c = 0; c < kPT; ++c) x[c] = c <= nv ? x[c] : -INFINITY;
            }
            float mx;
            {
                float t[4];
#pragma unroll
                for (int c = 0; c < 4; ++c) t[c] = x[c];
#pragma unroll
                for (int c = 4; c < kPT; c += 8)
#pragma unroll
                    for (int e = 0; e < 4; ++e) t[e] = c + 4 + e < kPT ? fmaxf(fmaxf(t[e], x[c + e]), x[c + 4 + e]) : fmaxf(t[e], x[c + e]);
                mx = fmaxf(fmaxf(t[0], t[1]), fmaxf(t[2], t[3]));
            }
            if constexpr (NT == 1) {
                // the running maximum after page j - 1, from the other group's thread of this row; every
                // page's weights are relative to the running maximum its own step leaves
                if (j > 0) {
                    named_bar_sync(1 + quarter * 2 + ((j - 1) & 1), 64);
                    const float mp = mrun[row];
                    if (mp != m) {
                        l *= ex2_approx(m - mp);  // (m = -inf: no page yet, l = 0)
                        m = mp;
                    }
                }
            }
            const float m_new = fmaxf(m, mx);
            const bool need = m_new > m + kRescaleLog2;  // also the first finite maximum
            const float factor = need ? ex2_approx(m - m_new) : 1.f;
            if (need) {
                l *= factor;
                m = m_new;
            }
            if constexpr (NT == 1) {
                if (j + 1 < NPg) {
                    mrun[row] = m;
                    named_bar_arrive(1 + quarter * 2 + (j & 1), 64);
                }
            }
            const bool any = __any_sync(0xffffffffu, need && j > 0);
            // this group's previous page has been read by its product (and O holds it)
            auto wait_own = [&] {
                if (jj > 0) mbar_wait(&bar[kBPfree + g], (jj - 1) & 1, abort_flag, p.err);
            };
            if (any) {
                // O holds pages 0..j-1: wait for the last of them, then rescale.  For NT = 1 that page
                // is the other group's; this group's own, one page earlier, is waited for first: products
                // complete in order, so the other group's barrier is then at most one phase behind
                // and its parity test cannot pass a phase early.
                wait_own();
                if constexpr (NT == 1) mbar_wait(&bar[kBPfree + (g ^ 1)], ((j - 1) >> 1) & 1, abort_flag, p.err);
                tc_fence_after();
#pragma unroll 1
                for (int c0 = 0; c0 < F::ORV; c0 += 16) {
                    float v[16];
                    tmem_ld16(to + c0, v);
#pragma unroll
                    for (int c = 0; c < 16; ++c) v[c] *= factor;
                    tmem_st16(to + c0, v);
                }
            }
            {
                const float2 mm = make_float2(-m, -m);
                float2 s4[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) s4[e] = make_float2(0.f, 0.f);
                uint32_t w[kPT / 2];
#pragma unroll
                for (int c = 0; c < kPT; c += 2) {
                    float2 y = __fadd2_rn(make_float2(x[c], x[c + 1]), mm);
                    y.x = ex2_approx(y.x);
                    y.y = ex2_approx(y.y);
                    s4[(c >> 1) & 3] = __fadd2_rn(s4[(c >> 1) & 3], y);
                    w[c / 2] = pack_bf16x2(y.x, y.y);
                    if constexpr (QP > 1) {
                        const float2 f = bf2_to_f2(w[c / 2]);
                        x[c] = y.x - f.x;
                        x[c + 1] = y.y - f.y;
                    }
                }
                const float2 sa = __fadd2_rn(s4[0], s4[1]), sb = __fadd2_rn(s4[2], s4[3]);
                l += (sa.x + sa.y) + (sb.x + sb.y);
                if (!any) wait_own();
                tc_fence_after();
                tmem_st32u_nowait(tp, w);
#pragma unroll
                for (int part = 1; part < QP; ++part) {
#pragma unroll
                    for (int c = 0; c < kPT; c += 2) {
                        w[c / 2] = pack_bf16x2(x[c], x[c + 1]);
                        if (part + 1 < QP) {
                            const float2 f = bf2_to_f2(w[c / 2]);
                            x[c] -= f.x;
                            x[c + 1] -= f.y;
                        }
                    }
                    tmem_st32u_nowait(tp + part * (kPT / 2), w);
                }
            }
            if (j == NPg - 1 && kb + kPT > L) {
                // last page of the prompt: V rows past it hold no latents; zero them before the
                // PV product reads them (0 * NaN would poison the sum)
                const int sv = j % F::STV;
                mbar_wait(&bar[kBVfull + sv], (j / F::STV) & 1, abort_flag, p.err);
                char *vs = sm + F::oV + sv * F::VPAGE;
                const int valid = L - kb;
                const int nz = (kPT - valid) * F::VATOMS * 8;  // 16-byte words to clear
                for (int w = row; w < nz; w += kGroup) {
                    const int c = w & 7, r2 = w >> 3;
                    const int a = r2 % F::VATOMS, i = valid + r2 / F::VATOMS;
                    *reinterpret_cast<uint4 *>(vs + a * (kPT * 128) + i * 128 + c * 16) = make_uint4(0, 0, 0, 0);
                }
                fence_proxy_async_smem();
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(&bar[kBPfull + g]);
        }
        if constexpr (NT == 1) {
            // the row's sum over both groups, relative to the later maximum
            float2 *xs = reinterpret_cast<float2 *>(sm + F::oX);
            xs[g * kBM + row] = make_float2(m, l);
            named_bar_sync(9 + quarter, 64);
            const float2 o = xs[(g ^ 1) * kBM + row];
            const float mf = fmaxf(m, o.x);
            l = (m == mf ? l : l * ex2_approx(m - mf)) + (o.x == mf ? o.y : o.y * ex2_approx(o.x - mf));
        }
        // epilogue: O / l -> hi and lo = O/l - hi as packed bf16 pairs in the chunk's own columns
        mbar_wait(&bar[kBOfin + tile], 0, abort_flag, p.err);
        tc_fence_after();
        const float inv = l > 0.f ? 1.f / l : 0.f;
        // (a loop of its own code, not unrolled over the chunks: straight-line code run once is
        // fetched at every instruction)
        constexpr int last = F::ORV - (F::VATOMS - 1) * 64;
        static_assert(last == 64 || last == 32, "columns of the last chunk");
#pragma unroll 1
        for (int c = NT == 1 ? g : 0; c < F::VATOMS; c += NT == 1 ? 2 : 1) {
            const uint32_t half = c == F::VATOMS - 1 ? last / 2 : 32;  // packed columns of hi, of lo
            // 32 columns at a time: a chunk's first 32 hold its hi, so its second half is read first
            float v[32], u[32];
            tmem_ld32(to + c * 64, v);
            if (half == 32) tmem_ld32(to + c * 64 + 32, u);
            uint32_t hi[16], lo[16], lo2[16];
            auto convert = [&](const float (&v)[32]) {
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    float a = v[2 * k] * inv, bb = v[2 * k + 1] * inv;
                    hi[k] = pack_bf16x2(a, bb);
                    float2 f = bf2_to_f2(hi[k]);
                    a -= f.x;
                    bb -= f.y;
                    lo[k] = pack_bf16x2(a, bb);
                    if constexpr (F::OP == 3) {
                        f = bf2_to_f2(lo[k]);
                        lo2[k] = pack_bf16x2(a - f.x, bb - f.y);
                    }
                }
            };
            const uint32_t t2 = tl + F::TM_P + c * 32;  // every product has read the weights there
            convert(v);
            tmem_st16u(to + c * 64, hi);
            tmem_st16u(to + c * 64 + half, lo);
            if constexpr (F::OP == 3) tmem_st16u(t2, lo2);
            if (half == 32) {
                convert(u);
                tmem_st16u(to + c * 64 + 16, hi);
                tmem_st16u(to + c * 64 + 48, lo);
                if constexpr (F::OP == 3) tmem_st16u(t2 + 16, lo2);
            }
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(&bar[kBOa + tile]);
        const float *muv = p.mu_v ? p.mu_v + wrow : nullptr;
        // NT = 1: group g stores half g of the output columns; NT = 2: both halves, one after the other
#pragma unroll 1
        for (int half = NT == 1 ? g : 0; half < (NT == 1 ? g + 1 : 2); ++half) {
            mbar_wait(&bar[kBOut + g], NT == 1 ? 0 : half, abort_flag, p.err);
            tc_fence_after();
            float v[64];
            tmem_ld64(ts, v);
            if (NT == 2 && half == 0) {
                tc_fence_before();
                mbar_arrive(&bar[kBOfree + g]);
            }
            if (muv) {
#pragma unroll
                for (int c = 0; c < 64; ++c) v[c] += muv[half * 64 + c];
            }
            if (valid_row) {
                char *dst = static_cast<char *>(p.out) + (qrow * D + half * 64) * (p.io_bf16 ? 2 : 4);
                if (p.io_bf16) {
#pragma unroll
                    for (int k = 0; k < 64; k += 8)
                        *reinterpret_cast<uint4 *>(dst + k * 2) =
                            make_uint4(pack_bf16x2(v[k], v[k + 1]), pack_bf16x2(v[k + 2], v[k + 3]),
                                       pack_bf16x2(v[k + 4], v[k + 5]), pack_bf16x2(v[k + 6], v[k + 7]));
                } else {
#pragma unroll
                    for (int k = 0; k < 64; k += 4)
                        *reinterpret_cast<float4 *>(dst + k * 4) = make_float4(v[k], v[k + 1], v[k + 2], v[k + 3]);
                }
            }
        }
        }
    }
    pdl_trigger();
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, F::TM_COLS);
    }
}

// ------------------------------------------------------------------------- CUDA-core path

struct GParams {
    int T, H, d, r_k, r_v, loop, storage_bf16, io_bf16;
    float scale_log2;
    const void *w_up_k, *w_up_v;
    const float *mu_v;
    const char *pool;
    int64_t num_blocks, block_bytes;
    int head_page_bytes, kplane_bytes;
    const int32_t *block_table;
    int max_blocks;
    const int32_t *cu_seqlens;
    int max_len;
    const void *q;
    void *out;
    unsigned *err;
};

constexpr int kGThreads = 128;
constexpr int kGKeys = 128;  // keys per step

// One CTA per (query, sequence, head), fp32 accumulation.  Shared memory: q [d], q~ [r_k],
// o~ [r_v], p [kGKeys], reduction scratch.
__global__ void __launch_bounds__(kGThreads) prefill_generic_kernel(const GParams p) {
    extern __shared__ __align__(16) float gs[];
    const int qi = blockIdx.x, b = blockIdx.y, h = blockIdx.z, tid = threadIdx.x;
    pdl_wait();
    const int q0 = p.cu_seqlens[b];
    const int L = p.cu_seqlens[b + 1] - q0;
    if (L > p.max_len || L < 0) {
        if (tid == 0 && qi == 0) atomicOr(p.err, LLA_DEVERR_CONTEXT);
        return;
    }
    if (qi >= L) return;
    const int es = p.storage_bf16 ? 2 : 4;
    float *qv = gs, *qt = qv + p.d, *ov = qt + p.r_k, *pv = ov + p.r_v, *red = pv + kGKeys;
    const int64_t qrow = (static_cast<int64_t>(q0) + qi) * p.H + h;
    const int64_t wofs = (static_cast<int64_t>(h) * p.T + p.loop) * p.d;
    for (int e = tid; e < p.d; e += kGThreads) qv[e] = load_elem(p.q, qrow * p.d + e, p.io_bf16);
    for (int j = tid; j < p.r_v; j += kGThreads) ov[j] = 0.f;
    __syncthreads();
    for (int j = tid; j < p.r_k; j += kGThreads) {  // q~ = W_up,t^K^T q
        float acc = 0.f;
        for (int e = 0; e < p.d; ++e)
            acc = fmaf(load_elem(p.w_up_k, (wofs + e) * p.r_k + j, p.storage_bf16), qv[e], acc);
        qt[j] = acc * p.scale_log2;
    }
    __syncthreads();
    const int gk = granule_bytes(p.r_k, es);
    const int32_t *bt = p.block_table + static_cast<int64_t>(b) * p.max_blocks;
    float m = -INFINITY, l = 0.f;
    for (int k0 = 0; k0 <= qi; k0 += kGKeys) {
        const int kj = k0 + tid;
        float s = -INFINITY;
        if (kj <= qi) {
            int32_t blk = bt[kj / kPT];
            if (blk < 0 || blk >= p.num_blocks) {
                atomicOr(p.err, LLA_DEVERR_BLOCK_ID);
                blk = 0;
            }
            const char *page = p.pool + blk * p.block_bytes + static_cast<int64_t>(h) * p.head_page_bytes;
            float acc = 0.f;
            for (int j = 0; j < p.r_k; ++j) {
                const char *e = page + kplane_offset(kj % kPT, j, es, gk);
                acc = fmaf(qt[j], es == 2 ? bf_to_f(*reinterpret_cast<const uint16_t *>(e))
                                          : *reinterpret_cast<const float *>(e), acc);
            }
            s = acc;
        }
        // block maximum
        float mx = warp_max(s);
        if ((tid & 31) == 0) red[tid >> 5] = mx;
        __syncthreads();
        mx = red[0];
        for (int w = 1; w < kGThreads / 32; ++w) mx = fmaxf(mx, red[w]);
        const float m_new = fmaxf(m, mx);
        const float alpha = exp2f(m - m_new);
        const float pj = kj <= qi ? exp2f(s - m_new) : 0.f;
        pv[tid] = pj;
        float ps = warp_sum(pj);
        __syncthreads();  // every thread has read red[] for the maximum
        if ((tid & 31) == 0) red[tid >> 5] = ps;
        __syncthreads();
        float psum = 0.f;
        for (int w = 0; w < kGThreads / 32; ++w) psum += red[w];
        l = l * alpha + psum;
        m = m_new;
        const int nk = min(kGKeys, qi + 1 - k0);
        for (int j = tid; j < p.r_v; j += kGThreads) {
            float acc = ov[j] * alpha;
            for (int t = 0; t < nk; ++t) {
                const int kk = k0 + t;
                int32_t blk = bt[kk / kPT];
                if (blk < 0 || blk >= p.num_blocks) blk = 0;
                const char *e = p.pool + blk * p.block_bytes + static_cast<int64_t>(h) * p.head_page_bytes +
                                p.kplane_bytes + (static_cast<int64_t>(kk % kPT) * p.r_v + j) * es;
                acc = fmaf(pv[t], es == 2 ? bf_to_f(*reinterpret_cast<const uint16_t *>(e))
                                          : *reinterpret_cast<const float *>(e), acc);
            }
            ov[j] = acc;
        }
        __syncthreads();
    }
    const float inv = 1.f / l;
    for (int e = tid; e < p.d; e += kGThreads) {
        float acc = 0.f;
        for (int j = 0; j < p.r_v; ++j)
            acc = fmaf(load_elem(p.w_up_v, (wofs + e) * p.r_v + j, p.storage_bf16), ov[j], acc);
        float o = acc * inv;
        if (p.mu_v) o += p.mu_v[wofs + e];
        store_elem(p.out, qrow * p.d + e, o, p.io_bf16);
    }
    pdl_trigger();
}

// ------------------------------------------------- rotary positions: rebuild and rotate keys
//
// Sec. 3 "RoPE and reconstruction": keys are rebuilt by Eq. decode and rotated at their
// positions before attention.  One CTA per (sequence, page of 64 prompt tokens, group of heads)
// loops over its heads: Khat (64 tokens x d) = C_k W_up,t^K^T + mu^K_t on tcgen05 (M = 64 tokens, N = d,
// K = r_k, plus one K step for mu^K_t), then each token's pairs are rotated in registers and
// written as a bf16 page in the K-plane layout (granule g of 8 dimensions at g*1024 + token*16),
// and the page's queries are rotated and scaled by scale * log2 e into a bf16 copy of q.  Four warps
// rebuild the keys and four others rotate the queries (the next head's already loading), sharing the
// page's table of turns: one after the other in the same warps, the two chains of loads added up.

// 32 consecutive elements (bf16 or fp32, 16-byte aligned) as floats, loads issued together.
__device__ __forceinline__ void load32(const void *src, int is_bf16, float (&v)[32]) {
    if (is_bf16) {
        uint4 u[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) u[i] = reinterpret_cast<const uint4 *>(src)[i];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 a = bf2_to_f2(u[i].x), b = bf2_to_f2(u[i].y), c = bf2_to_f2(u[i].z), d = bf2_to_f2(u[i].w);
            v[8 * i] = a.x; v[8 * i + 1] = a.y; v[8 * i + 2] = b.x; v[8 * i + 3] = b.y;
            v[8 * i + 4] = c.x; v[8 * i + 5] = c.y; v[8 * i + 6] = d.x; v[8 * i + 7] = d.y;
        }
    } else {
        float4 f[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = reinterpret_cast<const float4 *>(src)[i];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            v[4 * i] = f[i].x; v[4 * i + 1] = f[i].y; v[4 * i + 2] = f[i].z; v[4 * i + 3] = f[i].w;
        }
    }
}

// 32 floats as bf16 (round to nearest even) with 16-byte stores.
__device__ __forceinline__ void store32_bf16(void *dst, const float (&v)[32]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
        reinterpret_cast<uint4 *>(dst)[i] =
            make_uint4(pack_bf16x2(v[8 * i], v[8 * i + 1]), pack_bf16x2(v[8 * i + 2], v[8 * i + 3]),
                       pack_bf16x2(v[8 * i + 4], v[8 * i + 5]), pack_bf16x2(v[8 * i + 6], v[8 * i + 7]));
}

struct RParams {
    int T, H, loop, io_bf16, kpps, pairing;
    float scale_log2;
    const void *w_up_k;
    const float *mu_k;
    const char *pool;
    int64_t num_blocks;
    int head_page_bytes;
    const int32_t *block_table;
    int max_blocks;
    const int32_t *cu_seqlens;
    int max_len;
    const void *q;
    char *krot;
    void *qrot;
    int64_t qrows;  // rows of the rotated-query buffer: B * max_len
    unsigned *err;
    unsigned long long phi[64];  // theta_j / (2 pi) * 2^64
};

template <int RK>
struct RB {
    static constexpr int D = 128;
    static constexpr int NG = RK / 8;                 // 16-byte granules of a latent row
    static constexpr int oTab = 0;                    // [64 tokens][65] (cos, sin) per pair
    static constexpr int TAB = 64 * 65 * 8;
    static constexpr int oB = (TAB + 1023) & ~1023;   // (mu_hi, mu_lo) granule, then W_up,t^K
    static constexpr int oW = oB + D * 16;
    static constexpr int oA = oW + NG * D * 16;       // the page's K-plane, then ones and zeros
    static constexpr int oOnes = oA + NG * 64 * 16;
    static constexpr int oBar = oOnes + 2 * 64 * 16;
    static constexpr int SMEM = oBar + 16 + 1024;     // + alignment slack
    static constexpr uint32_t IDESC = umma_idesc_bf16(64, D, 0, 0);
    static_assert(RK % 16 == 0, "K steps");
};

constexpr int kRKeys = 128;      // threads that rebuild keys; as many rotate queries
constexpr int kRThreads = 2 * kRKeys;

template <int RK>
__global__ void __launch_bounds__(kRThreads, 2) rope_rebuild_kernel(const __grid_constant__ RParams p) {
    using Z = RB<RK>;
    constexpr int D = Z::D;
    extern __shared__ __align__(1024) char rb_raw[];
    char *sm = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(rb_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    float2 *tab = reinterpret_cast<float2 *>(sm + Z::oTab);
    uint64_t *bar = reinterpret_cast<uint64_t *>(sm + Z::oBar);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int pg = blockIdx.x, b = blockIdx.y;
    const int hpg = (p.H + gridDim.z - 1) / gridDim.z;  // heads of this CTA: [h0, h1)
    const int h0 = blockIdx.z * hpg, h1 = min(p.H, h0 + hpg);
    pdl_wait();
    const int q0 = p.cu_seqlens[b];
    const int L = p.cu_seqlens[b + 1] - q0;
    if (L > p.max_len || L < 0 || static_cast<int64_t>(q0) + L > p.qrows) {
        if (tid == 0 && pg == 0) atomicOr(p.err, LLA_DEVERR_CONTEXT);
        return;
    }
    if (pg * kPT >= L || h0 >= h1) return;  // uniform, before any barrier
    const int nvalid = min(kPT, L - pg * kPT);
    int32_t blk = p.block_table[static_cast<int64_t>(b) * p.max_blocks + pg];
    if (blk < 0 || blk >= p.num_blocks) {
        if (tid == 0) atomicOr(p.err, LLA_DEVERR_BLOCK_ID);
        blk = 0;
    }
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
    }
    if (warp == 0) tmem_alloc(tslot, 128);
    // rotation of each token of the page at each pair's frequency, from exact turns
    for (int i = tid; i < 64 * 64; i += kRThreads) {
        const int r = i >> 6, j = i & 63;
        const unsigned long long turns = static_cast<unsigned long long>(pg * kPT + r) * p.phi[j];
        const float tf = __uint2float_rn(static_cast<uint32_t>(turns >> 32)) * 2.3283064365386963e-10f;
        float sa, ca;
        sincospif(2.f * tf, &sa, &ca);
        tab[r * 65 + j] = make_float2(ca, sa);
    }
    // A of the mu step: a (1, 1) pair per token, then a zero granule
    for (int i = tid; i < 128; i += kRThreads)
        reinterpret_cast<uint4 *>(sm + Z::oOnes)[i] = i < 64 ? make_uint4(0x3f803f80u, 0u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tslot;
    const uint32_t base = smem_addr(sm);
    if (tid >= kRKeys) {
        // the page's queries, head by head: rotated at their positions, scaled into the exp2 domain;
        // thread (r, hf) rotates pairs 32 hf .. 32 hf + 31 of query r
        const int r = (tid - kRKeys) >> 1, hf = tid & 1;
        if (r < nvalid) {
            const float2 *tr = tab + r * 65 + 32 * hf;
            const int es = p.io_bf16 ? 2 : 4;
            const int64_t row = (static_cast<int64_t>(q0) + pg * kPT + r) * p.H;
            // the thread's two runs of 32 elements: pairs (j, j + 64), or 64 consecutive elements
            const int oa = p.pairing == 0 ? 32 * hf : 64 * hf, ob = p.pairing == 0 ? 64 + 32 * hf : 64 * hf + 32;
            const char *qs = static_cast<const char *>(p.q);
            uint4 na[4], nb[4];  // the next head's elements, bf16
            auto prefetch = [&](int h) {
                const uint4 *a = reinterpret_cast<const uint4 *>(qs + ((row + h) * D + oa) * 2);
                const uint4 *b2 = reinterpret_cast<const uint4 *>(qs + ((row + h) * D + ob) * 2);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    na[k] = a[k];
                    nb[k] = b2[k];
                }
            };
            if (p.io_bf16) prefetch(h0);
            for (int h = h0; h < h1; ++h) {
                float xa[32], xb[32];
                if (p.io_bf16) {
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t wa[4] = {na[k].x, na[k].y, na[k].z, na[k].w}, wb[4] = {nb[k].x, nb[k].y, nb[k].z, nb[k].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const float2 fa = bf2_to_f2(wa[e]), fb = bf2_to_f2(wb[e]);
                            xa[8 * k + 2 * e] = fa.x; xa[8 * k + 2 * e + 1] = fa.y;
                            xb[8 * k + 2 * e] = fb.x; xb[8 * k + 2 * e + 1] = fb.y;
                        }
                    }
                    if (h + 1 < h1) prefetch(h + 1);
                } else {
                    load32(qs + ((row + h) * D + oa) * es, 0, xa);
                    load32(qs + ((row + h) * D + ob) * es, 0, xb);
                }
                char *qo = static_cast<char *>(p.qrot) + (row + h) * D * 2;
                if (p.pairing == 0) {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const float2 cs = tr[i];
                        const float a = xa[i], bb = xb[i];
                        xa[i] = (a * cs.x - bb * cs.y) * p.scale_log2;
                        xb[i] = (a * cs.y + bb * cs.x) * p.scale_log2;
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < 32; ++i) {
                        const float2 cs = tr[i];
                        float *pr = i < 16 ? xa + 2 * i : xb + 2 * (i - 16);
                        const float a = pr[0], bb = pr[1];
                        pr[0] = (a * cs.x - bb * cs.y) * p.scale_log2;
                        pr[1] = (a * cs.y + bb * cs.x) * p.scale_log2;
                    }
                }
                store32_bf16(qo + oa * 2, xa);
                store32_bf16(qo + ob * 2, xb);
            }
        }
    } else {
    // epilogue geometry (16x256b fragments of the M = 64 accumulator): warp w holds tokens
    // 16w + lane/4 and 16w + lane/4 + 8; columns 8k + 2c and 8k + 2c + 1, c = lane % 4
    const int c = lane & 3;
    const int tok0 = 16 * warp + (lane >> 2);
    const uint32_t tq = tmem + (static_cast<uint32_t>(32 * warp) << 16);
    // W_up,t^K of head h (B: row e = dimension, K-major) and the page's K-plane of head h (A, as
    // stored), by cp.async; the (mu_hi, mu_lo) granule of head h before W
    auto stage = [&](int h) {
        const int64_t hl = (static_cast<int64_t>(h) * p.T + p.loop) * D;
        const char *W = static_cast<const char *>(p.w_up_k) + hl * RK * 2;
        for (int i = tid; i < D * Z::NG; i += kRKeys) {
            const int e = i / Z::NG, g = i - e * Z::NG;
            cp_async16(sm + Z::oW + g * (D * 16) + e * 16, W + (static_cast<int64_t>(e) * RK + g * 8) * 2);
        }
        const char *K = p.pool + (static_cast<int64_t>(blk) * p.H + h) * p.head_page_bytes;
        for (int i = tid; i < Z::NG * 64; i += kRKeys) cp_async16(sm + Z::oA + i * 16, K + i * 16);
        cp_async_commit();
        const float mu = p.mu_k ? p.mu_k[hl + tid] : 0.f;
        const __nv_bfloat16 hi = __float2bfloat16_rn(mu);
        const __nv_bfloat16 lo = __float2bfloat16_rn(mu - __bfloat162float(hi));
        *reinterpret_cast<uint4 *>(sm + Z::oB + tid * 16) =
            make_uint4(static_cast<uint32_t>(__bfloat16_as_ushort(hi)) |
                           (static_cast<uint32_t>(__bfloat16_as_ushort(lo)) << 16),
                       0u, 0u, 0u);
    };
    stage(h0);
    for (int h = h0; h < h1; ++h) {
        cp_async_wait_all();
        fence_proxy_async_smem();
        tc_fence_before();
        named_bar_sync(1, kRKeys);
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int st = 0; st < RK / 16; ++st)
                umma_bf16(tmem, umma_desc(base + Z::oA + st * 2048, 1024, 128),
                          umma_desc(base + Z::oW + st * 4096, 2048, 128), Z::IDESC, st > 0);
            // mu: the ones pair of every token against (mu_hi, mu_lo) of every dimension; the
            // second granules are zeros (A) and W_up,t^K (B, finite)
            umma_bf16(tmem, umma_desc(base + Z::oOnes, 1024, 128), umma_desc(base + Z::oB, 2048, 128),
                      Z::IDESC, true);
            umma_commit(bar);
        }
        {
            volatile int never = 0;
            mbar_wait(bar, (h - h0) & 1, &never, p.err);
        }
        tc_fence_after();
        // the MMA has read its operands: the next head's travel while this one's epilogue runs
        if (h + 1 < h1) stage(h + 1);
        uint32_t r0[32], r1[32];  // dimensions 0..63 (k = 0..7) and 64..127 (k = 8..15)
        tmem_ld16x256_x8_nowait(tq, r0);
        tmem_ld16x256_x8_nowait(tq + 64, r1);
        tmem_wait_ld(r0);
        tmem_wait_ld(r1);
        // rotate each token's pairs and write the page: dims (8k + 2c, +1) of token t at
        // granule k, byte 4c
        char *kout = p.krot + ((static_cast<int64_t>(b) * p.kpps + pg) * p.H + h) * (kPT * D * 2);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int t = tok0 + 8 * u;
            const float2 *tr = tab + t * 65;
            const bool ok = t < nvalid;
            float y[32];  // y[2k + e]: dimension 8k + 2c + e
            if (p.pairing == 0) {  // pairs (j, j + 64): k and k + 8
#pragma unroll
                for (int k = 0; k < 8; ++k)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const float xa = __uint_as_float(r0[4 * k + 2 * u + e]);
                        const float xb = __uint_as_float(r1[4 * k + 2 * u + e]);
                        const float2 cs = tr[8 * k + 2 * c + e];
                        y[2 * k + e] = xa * cs.x - xb * cs.y;
                        y[2 * (k + 8) + e] = xa * cs.y + xb * cs.x;
                    }
            } else {  // pairs (2j, 2j + 1), j = 4k + c
#pragma unroll
                for (int k = 0; k < 16; ++k) {
                    const uint32_t *rr = k < 8 ? r0 : r1;
                    const int kk = k & 7;
                    const float xa = __uint_as_float(rr[4 * kk + 2 * u]);
                    const float xb = __uint_as_float(rr[4 * kk + 2 * u + 1]);
                    const float2 cs = tr[4 * k + c];
                    y[2 * k] = xa * cs.x - xb * cs.y;
                    y[2 * k + 1] = xa * cs.y + xb * cs.x;
                }
            }
#pragma unroll
            for (int k = 0; k < 16; ++k)
                *reinterpret_cast<uint32_t *>(kout + k * 1024 + t * 16 + c * 4) =
                    ok ? pack_bf16x2(y[2 * k], y[2 * k + 1]) : 0u;
        }
        tc_fence_before();
        named_bar_sync(1, kRKeys);  // the operands and the accumulator may take the next head
        tc_fence_after();
    }
    }
    pdl_trigger();
    if (warp == 0) tmem_dealloc(tmem, 128);
}

template <typename K, typename P>
lla_status launch_pf(K kern, dim3 grid, int threads, int smem, cudaStream_t stream, const P &prm) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, kern, prm) != cudaSuccess) return LLA_ERR_CUDA;
    return LLA_OK;
}

template <int RK, int RV, int NT, bool ROPE, int QP>
lla_status launch_tiles(const PParams &prm0, const PrefillArgs &a, cudaStream_t stream) {
    using F = PF<RK, RV, NT, ROPE, QP>;
    static DeviceOnce configured;
    if (raise_smem_limit(prefill_tc_kernel<RK, RV, NT, ROPE, QP>, F::SMEM, configured) != LLA_OK) return LLA_ERR_CUDA;
    // the V-planes of every head page: [pages][64 tokens][r_v] bf16, one page = one head page
    CUtensorMap tv = {}, twk = {}, twv = {};
    if constexpr (!F::NARROW) {
    const uint64_t dims[3] = {static_cast<uint64_t>(RV), static_cast<uint64_t>(kPT),
                              static_cast<uint64_t>(prm0.num_blocks) * prm0.H};
    const uint64_t strides[2] = {static_cast<uint64_t>(RV) * 2, static_cast<uint64_t>(prm0.head_page_bytes)};
    const uint32_t box[3] = {64, kPT, 1};
    if (!encode_tmap_bf16(&tv, prm0.pool + kPT * RK * 2, 3, dims, strides, box, true)) return LLA_ERR_CUDA;
    // W_up of both axes: [H T d][r] bf16, the d rows of one (head, loop) at a time
    const uint64_t wk[2] = {static_cast<uint64_t>(RK), static_cast<uint64_t>(prm0.H) * prm0.T * F::D};
    const uint64_t wv[2] = {static_cast<uint64_t>(RV), wk[1]};
    const uint64_t sk[1] = {static_cast<uint64_t>(RK) * 2}, sv[1] = {static_cast<uint64_t>(RV) * 2};
    const uint32_t wbox[2] = {64, F::D};
    if (!encode_tmap_bf16(&twk, a.w_up_k, 2, wk, sk, wbox, true) || !encode_tmap_bf16(&twv, a.w_up_v, 2, wv, sv, wbox, true))
        return LLA_ERR_CUDA;
    }
    cudaLaunchConfig_t cfg = {};
    // The launch order.  One (head, prompt) pair after the other, its longest tiles first, shares the pair's
    // pages in L2, but ends on the last pair's long tiles; the longest tiles of all pairs first ends evenly
    // but reads all pages at once.  So pair after pair, and then the last three waves of CTAs' pairs, or
    // as many as half of L2 holds, together.  Pair after pair only / this rule / all together: 3 ragged
    // prompts at (72, 120) 127 / 115 / 113 us, 8 x 2048 tokens at (96, 160) 207 / 195 / 186, 4 x 2000 at
    // (18, 30) 235 / 169 / 171 (both with two bf16 parts of q~ and P), 4 x 8192 at (192, 320) 1679 / 1652 / 2047, six ragged rotary prompts 396 /
    // 357 / 356.  (Six and ten waves: 1693 and 1770 us at (192, 320).)
    const int tiles = (a.max_len + NT * kBM - 1) / (NT * kBM);
    const int64_t pairs = static_cast<int64_t>(a.B) * a.H;
    PParams prm = prm0;
    prm.first = -1;
    cfg.gridDim = dim3(tiles, a.B, a.H);
    if (pairs * tiles < (int64_t(1) << 31)) {
        const int sms = num_sms();
        if (sms <= 0) return LLA_ERR_CUDA;
        const int64_t pair_bytes = static_cast<int64_t>(a.max_len) * ((ROPE ? F::D : RK) + RV) * 2;
        const int64_t last = std::max<int64_t>((3ll * sms + tiles - 1) / tiles, (64ll << 20) / pair_bytes);
        prm.first = static_cast<int>(std::max<int64_t>(0, pairs - last));
        // divisions by multiplication: a tile past its prompt is little else (32 prompts of 100 tokens at
        // (192, 320), launched for 8192 each: 212 us with divisions, 187 so)
        prm.by_tiles = fast_div(tiles);
        prm.by_rest = fast_div(static_cast<uint32_t>(pairs - prm.first));
        prm.by_prompts = fast_div(a.B);
        cfg.gridDim = dim3(static_cast<unsigned>(pairs * tiles));
    }
    cfg.blockDim = dim3(kPThreads);
    cfg.dynamicSmemBytes = F::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaLaunchKernelEx(&cfg, prefill_tc_kernel<RK, RV, NT, ROPE, QP>, tv, twk, twv, prm) != cudaSuccess) return LLA_ERR_CUDA;
    return LLA_OK;
}

// One query tile per CTA, or two that share every page.  Two halve the pages' way through L2 and need no
// hand-over of maxima, but a CTA's work is twice as long, so that few CTAs end unevenly.  Measured with one
// and with two (us, 16 heads; pairs of tiles over the whole batch at its longest prompt):
//   (96, 160):  1 x 2048 tokens (128 pairs) 28 and 36, 2 x 2048 (256) 56 and 51, 32 x 250 (512) 66 and 61,
//               1 x 8192 (512) 231 and 220, 4 x 8192 (2048) 1005 and 919
//   (128, 128): 1 x 2048 29 and 38, 2 x 2048 58 and 52, 32 x 250 65 and 60, 4 x 8192 1031 and 975
//   rotated keys, (96, 160): 1 x 2048 47 and 57, 4 x 600 (192) 54 and 51, 1 x 4096 (256) 115 and 101, 2 x 8192
//               (1024) 723 and 579: they are 128 wide instead of 96, so that the pages weigh more
// From 160 to 400 pairs the two come within a few percent where the prompts differ in length (4 x 700 to
// 1050 tokens, 256 pairs, 35 and 36; 8 x 64 to 2048, 384 pairs of which half exist, 25 and 28), so that
// two start above that; with rotated keys those two cases take 63 and 61, 50 and 51, and two start at 256.
// Prompts of one tile leave the second empty (32 x 100: 34 and 37).  The pairs are counted from max_len, an
// upper bound; where it is far above the prompts, half as many CTAs past their ends weigh more than empty
// tiles (one and two tiles: 32 x 100 tokens under max_len 1024 47 and 40, 8192 179 and 109; 8 x 500 to 900
// under 8192 91 and 78; rotated keys, 16 x 100 under 4096 94 and 76).  With two bf16 parts the products bound
// it either way (2 x 8192 at (72, 120): 630 and 644), and three leave no TMEM for a second O: one tile.
template <int RK, int RV, bool ROPE, int QP = 1>
lla_status launch_tc(const PParams &prm, const PrefillArgs &a, cudaStream_t stream) {
    if constexpr (RV <= 160 && QP == 1) {
        const int64_t pairs = static_cast<int64_t>((a.max_len + 2 * kBM - 1) / (2 * kBM)) * a.B * a.H;
        if (a.max_len > kBM && pairs >= (ROPE ? 256 : 400)) return launch_tiles<RK, RV, 2, ROPE, QP>(prm, a, stream);
    }
    return launch_tiles<RK, RV, 1, ROPE, QP>(prm, a, stream);
}

PParams tc_params(const PrefillArgs &a, int hpb, unsigned *err) {
    PParams p = {};
    p.T = a.T; p.H = a.H; p.loop = a.loop; p.io_bf16 = a.io_bf16;
    p.scale_log2 = a.scale * kLog2e;
    p.mu_v = a.mu_v;
    p.w_up_k = a.w_up_k; p.w_up_v = a.w_up_v;
    p.pool = static_cast<const char *>(a.pool);
    p.num_blocks = a.num_blocks;
    p.head_page_bytes = hpb;
    p.block_table = a.block_table; p.max_blocks = a.max_blocks;
    p.cu_seqlens = a.cu_seqlens; p.B = a.B; p.max_len = a.max_len;
    p.q = a.q; p.out = a.out; p.err = err;
    return p;
}

}  // namespace

lla_status launch_prefill(const PrefillArgs &a, cudaStream_t stream) {
    lla_status st = LLA_OK;
    unsigned *err = device_error_word(&st);
    if (st != LLA_OK) return st;
    const int es = a.storage_bf16 ? 2 : 4;
    const int hpb = static_cast<int>(head_page_bytes(a.r_k, a.r_v, es));
    if (a.B > 65535 || a.H > 65535) return LLA_ERR_UNSUPPORTED;
    // the tensor-core kernel addresses head pages with a 32-bit TMA coordinate
    if (a.storage_bf16 && a.d == 128 && a.num_blocks * a.H < (int64_t(1) << 31)) {
        const PParams p = tc_params(a, hpb, err);
        if (a.r_k == 96 && a.r_v == 160) return launch_tc<96, 160, false>(p, a, stream);
        if (a.r_k == 192 && a.r_v == 320) return launch_tc<192, 320, false>(p, a, stream);
        if (a.r_k == 128 && a.r_v == 128) return launch_tc<128, 128, false>(p, a, stream);
        if (a.r_k == 72 && a.r_v == 120 && a.io_bf16) return launch_tc<72, 120, false, 3>(p, a, stream);
        if (a.r_k == 18 && a.r_v == 30 && a.io_bf16) return launch_tc<18, 30, false, 3>(p, a, stream);
    }
    GParams g = {};
    g.T = a.T; g.H = a.H; g.d = a.d; g.r_k = a.r_k; g.r_v = a.r_v; g.loop = a.loop;
    g.storage_bf16 = a.storage_bf16; g.io_bf16 = a.io_bf16;
    g.scale_log2 = a.scale * kLog2e;
    g.w_up_k = a.w_up_k; g.w_up_v = a.w_up_v; g.mu_v = a.mu_v;
    g.pool = static_cast<const char *>(a.pool);
    g.num_blocks = a.num_blocks;
    g.head_page_bytes = hpb;
    g.block_bytes = static_cast<int64_t>(hpb) * a.H;
    g.kplane_bytes = kPT * a.r_k * es;
    g.block_table = a.block_table; g.max_blocks = a.max_blocks;
    g.cu_seqlens = a.cu_seqlens; g.max_len = a.max_len;
    g.q = a.q; g.out = a.out; g.err = err;
    const int smem = (a.d + a.r_k + a.r_v + kGKeys + 32) * 4;
    return launch_pf(prefill_generic_kernel, dim3(a.max_len, a.B, a.H), kGThreads, smem, stream, g);
}


size_t prefill_rope_workspace_bytes(int B, int max_len, int H) {
    const size_t kpps = (static_cast<size_t>(max_len) + kPT - 1) / kPT;
    const size_t krot = static_cast<size_t>(B) * kpps * H * kPT * 128 * 2;
    const size_t qrot = static_cast<size_t>(B) * max_len * H * 128 * 2;
    return krot + qrot;
}

bool prefill_rope_supported(int es, int d, int r_k, int r_v) {
    return es == 2 && d == 128 &&
           ((r_k == 96 && r_v == 160) || (r_k == 192 && r_v == 320) || (r_k == 128 && r_v == 128));
}

namespace {
template <int RK>
lla_status launch_rebuild(const RParams &rp, int kpps, int B, cudaStream_t stream) {
    static DeviceOnce configured;
    if (raise_smem_limit(rope_rebuild_kernel<RK>, RB<RK>::SMEM, configured) != LLA_OK) return LLA_ERR_CUDA;
    // heads split over a few CTAs per page, so that more CTAs hide each other's load latency
    const int groups = rp.H >= 8 ? 4 : 1;
    return launch_pf(rope_rebuild_kernel<RK>, dim3(kpps, B, groups), kRThreads, RB<RK>::SMEM, stream, rp);
}
}  // namespace

lla_status launch_prefill_rope(const PrefillArgs &a, double base, int pairing, void *workspace,
                               size_t workspace_bytes, cudaStream_t stream) {
    const int es = a.storage_bf16 ? 2 : 4;
    if (!prefill_rope_supported(es, a.d, a.r_k, a.r_v)) return LLA_ERR_UNSUPPORTED;
    if (a.B > 65535 || a.H > 65535 || a.num_blocks * a.H >= (int64_t(1) << 31)) return LLA_ERR_UNSUPPORTED;
    if (workspace_bytes < prefill_rope_workspace_bytes(a.B, a.max_len, a.H)) return LLA_ERR_WORKSPACE;
    lla_status st = LLA_OK;
    unsigned *err = device_error_word(&st);
    if (st != LLA_OK) return st;
    const int hpb = static_cast<int>(head_page_bytes(a.r_k, a.r_v, es));
    const int kpps = (a.max_len + kPT - 1) / kPT;
    char *krot = static_cast<char *>(workspace);
    void *qrot = krot + static_cast<size_t>(a.B) * kpps * a.H * kPT * 128 * 2;

    RParams r = {};
    r.T = a.T; r.H = a.H; r.loop = a.loop; r.io_bf16 = a.io_bf16; r.kpps = kpps; r.pairing = pairing;
    r.scale_log2 = a.scale * kLog2e;
    r.w_up_k = a.w_up_k; r.mu_k = a.mu_k;
    r.pool = static_cast<const char *>(a.pool); r.num_blocks = a.num_blocks;
    r.head_page_bytes = hpb;
    r.block_table = a.block_table; r.max_blocks = a.max_blocks;
    r.cu_seqlens = a.cu_seqlens; r.max_len = a.max_len;
    r.q = a.q; r.krot = krot; r.qrot = qrot; r.err = err;
    r.qrows = static_cast<int64_t>(a.B) * a.max_len;
    const double two_pi = 6.283185307179586476925286766559;
    for (int j = 0; j < 64; ++j)
        r.phi[j] = static_cast<unsigned long long>(ldexp(pow(base, -2.0 * j / a.d) / two_pi, 64));
    lla_status rs = LLA_ERR_UNSUPPORTED;
    if (a.r_k == 96) rs = launch_rebuild<96>(r, kpps, a.B, stream);
    else if (a.r_k == 192) rs = launch_rebuild<192>(r, kpps, a.B, stream);
    else if (a.r_k == 128) rs = launch_rebuild<128>(r, kpps, a.B, stream);
    if (rs != LLA_OK) return rs;

    PParams p = tc_params(a, hpb, err);
    p.krot = krot; p.qrot = qrot; p.kpps = kpps;
    p.qrows = static_cast<int64_t>(a.B) * a.max_len;
    if (a.r_k == 96) return launch_tc<96, 160, true>(p, a, stream);
    if (a.r_k == 192) return launch_tc<192, 320, true>(p, a, stream);
    return launch_tc<128, 128, true>(p, a, stream);
}

}  // namespace lla
