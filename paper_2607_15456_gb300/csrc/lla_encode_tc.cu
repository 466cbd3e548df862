// lla_encode_tc.cu -- Eq. encode (Sec. 3) of a prompt on tcgen05 tensor cores, both axes in one
// persistent launch.
//
// A unit is (head h, tile of 128 tokens, column group g of one axis):
//   C[128 x R] = (X - m)[128 x T*d] W_down[T*d x R] - (mu - m) W_down,   m: mu rounded to bf16
// with X the stacked loop vectors of the tile's tokens (row n, column t*d + e = x_t[n][h][e]).
// LLA-2D is the case of one head of width H*d.  An axis of rank r is cut into ceil(r / 192) column
// groups of equal width (a multiple of 16; the columns of the last group past r read as zeros and
// are not stored).  Units are numbered head-major, then tile, then group (K groups first): one CTA
// per SM takes an equal contiguous range of them, so the groups of a tile follow one another on the
// same SM and the second read of a tile's x_v hits L2, and a CTA meets few heads (the bias
// (mu - m) W_down of a group is computed once per head the CTA meets).  bf16 operands, fp32 accumulation
// in TMEM, latents rounded to bf16 and scattered to each token's slot.  Warp roles:
//   warp 0     x producer: per slab of 64 reduction rows, a TMA tensor load with 128-byte swizzle
//              of the x tile (one box of 128 tokens x 64 elements: a K-major operand) into its
//              own ring, which runs on across units
//   warp 2     W producer: the slab's W_down (boxes of 64 rows x 64 columns: an MN-major
//              operand) into a second ring; the two rings let the x stream from HBM run ahead
//              of the W_down stream from L2 (one shared ring of 40 KB stages gave x only 16 of
//              every 40 bytes in flight)
//   warp 1     MMA issuer and TMEM owner: 4 MMAs (K = 16) per slab, M = 128, N = R, into one of
//              two accumulator slots; the next piece of four slabs takes the other
//   warps 3-10 epilogue: each piece's accumulators are added to the unit's sum, in registers (one token
//              row and every other chunk of 32 columns per thread); then bias -> bf16 -> the paged cache
//              (V-plane rows pass through a per-warp staging buffer, so a store writes 8 rows of 64
//              bytes).  Sums inside the tensor core are cut off, not rounded: over 512 rows and more
//              they lost up to six times what fp32 sums lose (latents rounded the wrong way, LLA-2D
//              (1152, 1920): 2.5e-3 in chains of 4096 rows, 2.0e-4 in pieces, 3.9e-4 on the CUDA cores).
//              Pieces of two slabs, 9.5e-5 and not 1.5e-4 at (72, 120), cost (96, 160) 4 % and LLA-2D 10 %
//   warps 11-14 (with mu only) x - m of a slab, exactly, as two bf16 parts in TMEM (one token row per
//              thread), two slabs deep: the products then take their operand A from there, twice as many,
//              so that a piece is two slabs.  x W_down - mu W_down instead lost what the two large sums
//              round off where mu is far above the spread of x (mu 64 times the spread: 1.2 % of the
//              latents rounded the wrong way, here 0.005 %)
// Tokens past N read as zeros (tensor-map fill) and are not stored.
//
// Few units with a long reduction (LLA-2D prompts: T*H*d = 8192 rows, N/128 tiles) are split over
// clusters of up to 8 CTAs: each CTA reduces its share of the rows, then writes its accumulators,
// column range by column range, into the shared memory of the CTA that owns the range (the rings
// are idle by then), which adds the parts in rank order and stores.
//
// Rows of W_down that are not a multiple of 16 bytes (r = 18, 30) have no tensor map: with WRES the
// epilogue warps copy the head's whole W_down of an axis (ranks up to 64, T*d up to 512) into
// shared memory, zero-padded to a multiple of 32 columns, in the layout the boxes would have, when
// the CTA first meets that head and axis.
//
// Bound: HBM for per-head prompts (x is read once; 41.7 us of bytes for 7208 tokens at (72, 120)),
// the L2 -> shared memory stream for LLA-2D (a 128 x 192 unit moves 40 KB per 64 rows).  Measured
// against the CUDA-core kernel, which these shapes took before: 7208 tokens at (72, 120) 1352 -> 53 us,
// with mu 1690 -> 85 us; 8000 tokens at (18, 30) 516 -> 61 us, with mu 593 -> 92 us (150 tokens 19.7 ->
// 7.6 us); LLA-2D (288, 480), 1500 tokens 4862 -> 30 us, with mu 5028 -> 82 us.  8000 tokens at (96, 160),
// here before too: 62 -> 60 us, with mu 191 -> 99 us.  With mu the chain of one slab through a converting
// warp (about 1500 cycles, from its landing to its products) is the bound.
#include <cuda_runtime.h>

#include "lla_device.cuh"
#include "lla_internal.h"
#include "lla_tcgen05.cuh"
#include "lla_tmap.h"

namespace lla {
namespace {

constexpr int kEM = 128;             // tokens per tile
constexpr int kES = 64;              // reduction rows per slab
constexpr int kEpi0 = 3;              // x producer, MMA issuer, W producer, then eight epilogue warps
constexpr int kEpi = 256;
constexpr int kConv0 = kEpi0 + kEpi / 32;  // and with mu four converting warps
constexpr int kMaxGroup = 192;       // columns of a group
constexpr int kMaxGroups = 20;       // groups of both axes (LLA-2D (1152, 1920): 6 + 10)
constexpr int kMaxSplit = 8;         // CTAs that share one unit's reduction
constexpr int kLongReduction = 4096; // reduction rows from which small batches take this kernel too
constexpr int kLongestStack = 24576; // T*d of one fp32 token in 96 KB
constexpr int kResSlabs = 8;         // WRES: most slabs (T*d = 512 rows) kept resident
constexpr int kASlab = kEM * kES * 2;   // x slab (16 KB)
constexpr int kBAtom = kES * 128;       // one W_down atom of 64 columns (8 KB)
constexpr int kWStage = 3 * kBAtom;          // 24 KB
constexpr int kWStages = 5;                 // W_down slabs in flight (from L2)
constexpr uint32_t kTmemCols = 512, kAT = 2 * kMaxGroup;
template <bool WRES, bool MU>
struct EL {  // shared-memory plan: x ring, W_down (ring or resident), biases, V staging, mu, barriers
    static constexpr int THREADS = kConv0 * 32 + (MU ? 128 : 0);
    // slabs whose products add up in TMEM (16 sums there either way) before fp32 adds in registers
    static constexpr int PIECE = MU ? 2 : 4;
    static constexpr int XST = MU || WRES ? 4 : 5;          // x slabs in flight (from HBM)
    // TMEM: accumulator slot s at s * SLOT; with mu two buffers of x - m as operand A (hi, then lo, 32
    // columns each) at kAT
    static constexpr uint32_t SLOT = MU ? kMaxGroup : 256;
    static constexpr int oW = XST * kASlab;
    static constexpr int GROUPS = !MU ? 0 : WRES ? 2 : kMaxGroups;
    static constexpr int NC = WRES ? 1 : 3;  // chunks of 32 columns of an epilogue warp
    static constexpr int oBias = oW + (WRES ? 2 * kResSlabs * kBAtom : kWStages * kWStage);
    static constexpr int oStg = oBias + GROUPS * kMaxGroup * 4;  // 8 warps x 32 rows x 80 B
    static constexpr int oMu = oStg + 8 * 32 * 80;               // 4 warps x 2 buffers x 64 bf16
    static constexpr int oBar = oMu + (MU ? 4 * 2 * 128 : 0);
    static constexpr int NBAR = 2 * XST + 2 * kWStages + 4 + 1 + (MU ? 4 : 0);
    static constexpr int SMEM = 1024 + oBar + NBAR * 8 + 16;  // + alignment slack, abort flag, TMEM slot
    static_assert(SMEM <= 227 * 1024, "shared memory");
};
// split units: parts of one column range, [rank][column / 4][row] float4 (over the idle rings)
static_assert(kMaxSplit * kEM * 32 * 4 <= EL<false, true>::oBias && 2 * kEM * 96 * 4 <= EL<false, true>::oBias, "exchange area");

struct ETParams {
    int T, H, d, N;
    int r_k, r_v;
    int nk, nv;      // column groups of each axis
    int gk, gv;      // columns per group of each axis (the last group of an axis may hold fewer)
    int split;       // CTAs per unit (a cluster); 1: no split
    int tiles;       // ceil(N / 128)
    int64_t units;   // H * tiles * (nk + nv)
    const float *mu_k, *mu_v;           // [H][T*d] or NULL
    const void *w_down_k, *w_down_v;    // [H][T*d][r] bf16 (for the bias)
    char *pool;
    int64_t num_blocks, block_bytes;
    int head_page_bytes, kplane_bytes;
    int gran;        // bytes of a K-plane granule: 16, or 4 when a K row is not whole 16-byte words
    const int64_t *slot_mapping;
    unsigned *err;
};

struct Unit {
    int h, n0, axis, col0, R, cols, g;  // R: columns of the product, cols: columns that exist
};

__device__ __forceinline__ Unit unit_of(const ETParams &p, int64_t u) {
    const int G = p.nk + p.nv;
    const int64_t per_head = static_cast<int64_t>(p.tiles) * G;
    Unit U;
    U.h = static_cast<int>(u / per_head);
    const int rem = static_cast<int>(u - U.h * per_head);
    const int tile = rem / G;
    U.g = rem - tile * G;
    U.n0 = tile * kEM;
    U.axis = U.g < p.nk ? 0 : 1;
    const int ga = U.axis ? U.g - p.nk : U.g;
    const int w = U.axis ? p.gv : p.gk;
    U.col0 = ga * w;
    U.cols = min(w, (U.axis ? p.r_v : p.r_k) - U.col0);
    U.R = (U.cols + 15) & ~15;
    return U;
}

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void st_cluster_f4(uint32_t local_addr, uint32_t rank, float4 v) {
    asm volatile(
        "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "st.shared::cluster.v4.f32 [ra], {%2, %3, %4, %5};\n\t}" ::"r"(local_addr),
        "r"(rank), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
        : "memory");
}

// (mu - m) W_down over reduction rows [k0, k1) for the columns of unit U, into bs[0 .. cols): EPL columns
// (8, or 2 when the rows of W_down are not whole 16-byte words) per thread and the rows cut into as
// many slices as the 256 epilogue threads allow, eight rows' loads in flight each (one thread per
// eight columns over all rows took tens of microseconds).  scr: at least 256 * EPL floats.
template <int EPL>
__device__ void group_bias(const uint16_t *W, const float *mu, int r, const Unit &U, int k0, int k1, int et,
                           float *scr, float *bs) {
    const int nch = (U.cols + EPL - 1) / EPL;  // at most 24 (EPL = 8), 32 (EPL = 2)
    const int nsl = kEpi / nch;
    const int ch = et % nch, sl = et / nch;
    float acc[EPL];
#pragma unroll
    for (int i = 0; i < EPL; ++i) acc[i] = 0.f;
    if (sl < nsl) {
        const uint16_t *Wc = W + U.col0 + ch * EPL;
#pragma unroll 8
        for (int k = k0 + sl; k < k1; k += nsl) {
            const float mk = bf16_rest(mu[k]);
            uint32_t w[EPL / 2];
            if constexpr (EPL == 8) {
                const uint4 q = *reinterpret_cast<const uint4 *>(Wc + static_cast<int64_t>(k) * r);
                w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
            } else {
                w[0] = *reinterpret_cast<const uint32_t *>(Wc + static_cast<int64_t>(k) * r);
            }
#pragma unroll
            for (int i = 0; i < EPL / 2; ++i) {
                const float2 f = bf2_to_f2(w[i]);
                acc[2 * i] = fmaf(mk, f.x, acc[2 * i]);
                acc[2 * i + 1] = fmaf(mk, f.y, acc[2 * i + 1]);
            }
        }
    }
    named_bar_sync(1, kEpi);  // scr and bs are free
#pragma unroll
    for (int i = 0; i < EPL; ++i) scr[et * EPL + i] = acc[i];
    named_bar_sync(1, kEpi);
    for (int c = et; c < U.cols; c += kEpi) {
        float v = 0.f;
        for (int q = 0; q < nsl; ++q) v += scr[(q * nch + c / EPL) * EPL + c % EPL];
        bs[c] = v;
    }
    named_bar_sync(1, kEpi);
}

// Where token row `row` of unit U goes: its K-plane row or V-plane row in the page of its slot (NULL:
// past N, skipped, or outside the pool).
__device__ __forceinline__ char *row_dst(const ETParams &p, const Unit &U, int row, bool flag) {
    const int n = U.n0 + row;
    if (n >= p.N) return nullptr;
    const int64_t slot_id = p.slot_mapping[n];
    if (slot_id < 0) return nullptr;
    const int64_t blk = slot_id / kBlockTokens;
    const int r_in = static_cast<int>(slot_id % kBlockTokens);
    if (blk >= p.num_blocks) {
        if (flag) atomicOr(p.err, LLA_DEVERR_SLOT);
        return nullptr;
    }
    char *page = p.pool + blk * p.block_bytes + static_cast<int64_t>(U.h) * p.head_page_bytes;
    return U.axis == 0 ? page + r_in * p.gran : page + p.kplane_bytes + static_cast<int64_t>(r_in) * p.r_v * 2;
}

template <bool WRES, bool MU>
__global__ void __launch_bounds__(EL<WRES, MU>::THREADS, 1)
    encode_tc_kernel(const __grid_constant__ CUtensorMap txk, const __grid_constant__ CUtensorMap txv,
                     const __grid_constant__ CUtensorMap twk, const __grid_constant__ CUtensorMap twv,
                     const ETParams p) {
    using L = EL<WRES, MU>;
    constexpr int oW = L::oW;
    extern __shared__ __align__(1024) char sm_raw[];
    // 128-byte swizzle atoms need a 1024-byte aligned base
    char *sm = reinterpret_cast<char *>((reinterpret_cast<uintptr_t>(sm_raw) + 1023) & ~static_cast<uintptr_t>(1023));
    float *bias = reinterpret_cast<float *>(sm + L::oBias);  // [group][192] of the current head
    uint64_t *full = reinterpret_cast<uint64_t *>(sm + L::oBar);
    uint64_t *empty = full + L::XST;
    uint64_t *wfull = empty + L::XST;
    uint64_t *wempty = wfull + kWStages;
    uint64_t *accfull = wempty + kWStages;  // [2]
    uint64_t *accempty = accfull + 2;     // [2]
    uint64_t *done = accempty + 2;
    uint64_t *afull = done + 1, *aempty = afull + 2;  // MU: [2] each
    uint64_t *after = full + L::NBAR;
    volatile int *abort_flag = reinterpret_cast<volatile int *>(after);
    uint32_t *tslot = reinterpret_cast<uint32_t *>(after) + 1;
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const bool split = p.split > 1;
    const int64_t u0 = split ? blockIdx.x / p.split : static_cast<int64_t>(blockIdx.x) * p.units / gridDim.x;
    const int64_t u1 = split ? u0 + 1 : static_cast<int64_t>(blockIdx.x + 1) * p.units / gridDim.x;
    const int Td = p.T * p.d;
    // slabs of the reduction of this CTA
    const int crank = split ? static_cast<int>(cluster_rank()) : 0;
    const int S0 = crank * (Td / kES) / p.split, S1 = (crank + 1) * (Td / kES) / p.split;
    const int NS = S1 - S0;

    if (tid == 0) {
        for (int s = 0; s < L::XST; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], MU ? 4 : 1);  // the converting warps, or the products
        }
        for (int s = 0; s < kWStages; ++s) {
            mbar_init(&wfull[s], WRES ? kEpi : 1);  // resident: the epilogue warps' copy (one per axis)
            mbar_init(&wempty[s], 1);
        }
        for (int s = 0; s < 2; ++s) {
            mbar_init(&accfull[s], 1);
            mbar_init(&accempty[s], 8);  // one arrival per epilogue warp
        }
        mbar_init(done, 1);
        if constexpr (MU) {
            for (int s = 0; s < 2; ++s) {
                mbar_init(&afull[s], 4);
                mbar_init(&aempty[s], 1);
            }
        }
        *abort_flag = 0;
        fence_mbar_init();
    }
    if (warp == 1) tmem_alloc(tslot, kTmemCols);
    if constexpr (WRES) {  // the padding columns of the resident W_down
        for (int i = tid; i < 2 * kResSlabs * kBAtom / 16; i += L::THREADS)
            reinterpret_cast<uint4 *>(sm + oW)[i] = make_uint4(0, 0, 0, 0);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    constexpr uint32_t tmem = 0;  // all of TMEM is allocated; a constant keeps the issuing warp's code uniform
    // epilogue: token row `row` of the tile, and of its columns the even or the odd chunks of 32
    const int wt = tid - kEpi0 * 32, half = (warp - kEpi0) >> 2, quarter = warp & 3, row = quarter * 32 + lane;
    float sum[L::NC][32];
    pdl_wait();  // x, slots and the pool may come from the previous kernel

    if (warp == 0 || (warp == 2 && !WRES)) {
        // ------------------------------------------------------------ producers: x (0), W (2)
        const bool isx = warp == 0;
        const int NST = isx ? L::XST : kWStages;
        uint64_t *F = isx ? full : wfull;
        uint64_t *E = isx ? empty : wempty;
        int q = 0;  // slabs issued
        bool stop = false;
        for (int64_t u = u0; u < u1 && !stop; ++u) {
            const Unit U = unit_of(p, u);
            const int atoms = (U.cols + 63) / 64;
            const CUtensorMap *tx = U.axis ? &txv : &txk;
            const CUtensorMap *tw = U.axis ? &twv : &twk;
            for (int s = 0; s < NS; ++s) {
                const int st = q % NST;
                const uint32_t ph = (q / NST) & 1;
                int halt = 0;
                if (lane == 0) {
                    halt = !mbar_wait(&E[st], ph ^ 1u, abort_flag, p.err) || *abort_flag;
                    if (!halt) mbar_arrive_expect_tx(&F[st], isx ? kASlab : atoms * kBAtom);
                }
                if (__shfl_sync(0xffffffffu, halt, 0)) {
                    stop = true;
                    break;
                }
                __syncwarp();
                const int k0 = (S0 + s) * kES, t = k0 / p.d, e0 = k0 - t * p.d;
                if (isx) {
                    if (lane == 0) tma_load_4d(sm + st * kASlab, tx, e0, U.h, U.n0, t, &F[st]);
                } else {
                    if (lane < atoms) tma_load_3d(sm + oW + st * kWStage + lane * kBAtom, tw, U.col0 + lane * 64, k0, U.h, &F[st]);
                }
                ++q;
            }
        }
        if (lane == 0 && *abort_flag) {
            volatile int never = 0;
            for (int j = q > NST ? q - NST : 0; j < q; ++j)
                mbar_wait(&F[j % NST], (j / NST) & 1, &never, p.err);
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------------ MMA issuer
        {
            const uint32_t base = smem_addr(sm);
            int q = 0, head = -1;
            uint32_t piece = 0;
            int nres[2] = {0, 0};               // WRES: copies of each axis's W_down seen
            bool wax[2] = {false, false};
            for (int64_t u = u0; u < u1; ++u) {
                const Unit U = unit_of(p, u);
                if constexpr (WRES) {  // the head's W_down of this axis is in shared memory
                    if (U.h != head) {
                        head = U.h;
                        wax[0] = wax[1] = false;
                    }
                    if (!wax[U.axis]) {
                        wax[U.axis] = true;
                        if (!mbar_wait_warp(&wfull[U.axis], nres[U.axis]++ & 1, abort_flag, p.err)) break;
                    }
                }
                const uint32_t idesc = umma_idesc_bf16(128, U.R, 0, 1);
                bool ok = true;
#pragma unroll 1
                for (int s = 0; s < NS; ++s, ++q) {
                    const int st = q % L::XST, sw = q % kWStages, slot = piece & 1;
                    const bool fresh = s % L::PIECE == 0;  // the epilogue has read this slot's piece before last
                    if (fresh && !mbar_wait_warp(&accempty[slot], ((piece >> 1) & 1) ^ 1u, abort_flag, p.err)) {
                        ok = false;
                        break;
                    }
                    const uint32_t d = tmem + slot * L::SLOT;
                    if (!(MU ? mbar_wait_warp(&afull[q & 1], (q >> 1) & 1, abort_flag, p.err)
                             : mbar_wait_warp(&full[st], (q / L::XST) & 1, abort_flag, p.err)) ||
                        (!WRES && !mbar_wait_warp(&wfull[sw], (q / kWStages) & 1, abort_flag, p.err))) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t a = base + st * kASlab, b = base + oW + (WRES ? (U.axis * kResSlabs + s) * kBAtom : sw * kWStage);
                    if constexpr (MU) {
#pragma unroll
                        for (int part = 0; part < 2; ++part)
#pragma unroll
                            for (int ks = 0; ks < kES / 16; ++ks)
                                umma_bf16_ts_warp(d, tmem + kAT + (q & 1) * 64 + part * 32 + ks * 8,
                                                  umma_desc_sw128_mn(b + ks * 2048, kBAtom), idesc, !fresh || part > 0 || ks > 0);
                        umma_commit_warp(&aempty[q & 1]);
                    } else {
#pragma unroll
                        for (int ks = 0; ks < kES / 16; ++ks)
                            umma_bf16_warp(d, umma_desc_sw128_k(a + ks * 32), umma_desc_sw128_mn(b + ks * 2048, kBAtom),
                                           idesc, !fresh || ks > 0);
                        umma_commit_warp(&empty[st]);
                    }
                    if (!WRES) umma_commit_warp(&wempty[sw]);
                    if (s % L::PIECE == L::PIECE - 1 || s == NS - 1) {
                        umma_commit_warp(&accfull[slot]);
                        ++piece;
                    }
                }
                if (!ok) break;
            }
            // every product has completed before TMEM is released
            umma_commit_warp(done);
            volatile int never = 0;
            mbar_wait_warp(done, 0, &never, p.err);
        }
        __syncwarp();
    } else if (warp >= kEpi0 && warp < kConv0) {
        // --------------------------------------------------------------------------- epilogue
        int head = -1;
        uint32_t have = 0;             // groups whose bias of this head is in `bias`
        bool wax[2] = {false, false};  // WRES: axes whose W_down of this head is resident
        uint32_t piece = 0;
        for (int64_t u = u0; u < u1; ++u) {
            const Unit U = unit_of(p, u);
            if (U.h != head) {
                head = U.h;
                have = 0;
                wax[0] = wax[1] = false;
            }
            if (WRES && !wax[U.axis]) {
                // this axis's W_down of the head, pairs of columns (zeros past r from the start): slab s at
                // s * kBAtom, row k % 64 of 128 bytes, 16-byte chunk c at c ^ (k % 8).  Every product
                // of the previous head has completed: its last accumulator has been read.
                wax[U.axis] = true;
                const int r = U.axis ? p.r_v : p.r_k, hp = r / 2;
                // 16-byte loads of the contiguous rows, up to eight in flight per thread, and four
                // 4-byte stores each (4-byte loads of padded rows took 8 us a head: 15 -> 8 us a call)
                const uint4 *W = reinterpret_cast<const uint4 *>(static_cast<const uint16_t *>(U.axis ? p.w_down_v : p.w_down_k) +
                                                                 static_cast<int64_t>(U.h) * Td * r);
                char *dst = sm + oW + U.axis * (kResSlabs * kBAtom);
                const uint32_t inv = (1u << 20) / hp + 1;  // q / hp = q * inv >> 20 below 512 rows of 32 pairs
                for (int i0 = wt; i0 < Td * r / 8; i0 += kEpi * 8) {
                    uint4 v[8];
#pragma unroll
                    for (int b = 0; b < 8; ++b)
                        if (i0 + b * kEpi < Td * r / 8) v[b] = W[i0 + b * kEpi];
#pragma unroll
                    for (int b = 0; b < 8; ++b) {
                        if (i0 + b * kEpi >= Td * r / 8) break;
                        const uint32_t wd[4] = {v[b].x, v[b].y, v[b].z, v[b].w};
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const uint32_t q = (i0 + b * kEpi) * 4 + e;  // pair q: row q / hp
                            const uint32_t k = static_cast<uint32_t>((static_cast<uint64_t>(q) * inv) >> 20), c = q - k * hp;
                            *reinterpret_cast<uint32_t *>(dst + k * 128 + (((c >> 2) ^ (k & 7)) << 4) + (c & 3) * 4) = wd[e];
                        }
                    }
                }
                fence_proxy_async_smem();
                mbar_arrive(&wfull[U.axis]);
            }
            const bool use_bias = MU && (U.axis ? p.mu_v : p.mu_k) != nullptr;
            float *bs = bias + U.g * kMaxGroup;
            if (MU && use_bias && !(have >> U.g & 1u)) {
                have |= 1u << U.g;
                const int r = U.axis ? p.r_v : p.r_k;
                const uint16_t *W = static_cast<const uint16_t *>(U.axis ? p.w_down_v : p.w_down_k) +
                                    static_cast<int64_t>(U.h) * Td * r;
                group_bias<WRES ? 2 : 8>(W, (U.axis ? p.mu_v : p.mu_k) + static_cast<int64_t>(U.h) * Td, r, U, S0 * kES,
                                         S1 * kES, wt, reinterpret_cast<float *>(sm + L::oStg), bs);
            }
            // the sum of the unit's pieces
#pragma unroll
            for (int i = 0; i < L::NC; ++i)
#pragma unroll
                for (int k = 0; k < 32; ++k) sum[i][k] = 0.f;
#pragma unroll 1
            for (int s = 0; s < NS; s += L::PIECE, ++piece) {
                const int slot = piece & 1;
                mbar_wait_warp(&accfull[slot], (piece >> 1) & 1, abort_flag, p.err);
                tc_fence_after();
                const uint32_t tl = tmem + slot * L::SLOT + (static_cast<uint32_t>(quarter * 32) << 16);
#pragma unroll
                for (int i = 0; i < L::NC; ++i) {
                    const int c0 = 64 * i + 32 * half;
                    if (c0 >= U.cols) break;
                    if constexpr (MU) {  // fewer registers
#pragma unroll
                        for (int k0 = 0; k0 < 32; k0 += 16) {
                            float v[16];
                            tmem_ld16(tl + c0 + k0, v);  // warp-collective
#pragma unroll
                            for (int k = 0; k < 16; ++k) sum[i][k0 + k] += v[k];
                        }
                    } else {
                        float v[32];
                        tmem_ld32(tl + c0, v);
#pragma unroll
                        for (int k = 0; k < 32; ++k) sum[i][k] += v[k];
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&accempty[slot]);  // this slot may take the piece after next
            }
            if (split) break;  // the parts meet below
            char *stg = sm + L::oStg + (warp - kEpi0) * (32 * 80);
            char *dst = row_dst(p, U, row, U.g == 0 && half == 0);
#pragma unroll
            for (int i = 0; i < L::NC; ++i) {
                const int c0 = 64 * i + 32 * half;
                if (c0 >= U.cols) break;
                const float (&v)[32] = sum[i];
                if constexpr (WRES) {
                    // rows that are not whole 16-byte words: pairs of columns.  K: consecutive rows
                    // are consecutive granules.  V: the warp's 32 rows through the staging buffer, so
                    // that a store writes neighbouring pairs.
                    const int np = min(32, U.cols - c0) / 2;
                    uint32_t w[16];
#pragma unroll
                    for (int k = 0; k < 16; ++k) {
                        const int c = c0 + 2 * k;
                        w[k] = use_bias ? pack_bf16(v[2 * k] - bs[c], v[2 * k + 1] - bs[c + 1]) : pack_bf16(v[2 * k], v[2 * k + 1]);
                    }
                    if (U.axis == 0) {
#pragma unroll
                        for (int k = 0; k < 16; ++k) {
                            const int c = c0 + 2 * k;
                            if (dst && k < np)
                                *reinterpret_cast<uint32_t *>(dst + (p.gran == 16 ? (c >> 3) * (kBlockTokens * 16) + (c & 7) * 2
                                                                                  : (c >> 1) * (kBlockTokens * 4))) = w[k];
                        }
                    } else {
                        uint32_t *sw = reinterpret_cast<uint32_t *>(stg);  // 17 words a row
#pragma unroll
                        for (int k = 0; k < 16; ++k) sw[lane * 17 + k] = w[k];
                        __syncwarp();
                        const uint32_t inv = 65536u / np + 1;  // i / np for i < 512
                        for (int i = lane; i < 32 * np; i += 32) {
                            const int rr = static_cast<int>(i * inv >> 16), c = i - rr * np;
                            char *d = reinterpret_cast<char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), rr));
                            if (d) *reinterpret_cast<uint32_t *>(d + (c0 + 2 * c) * 2) = sw[rr * 17 + c];
                        }
                        __syncwarp();
                    }
                    continue;
                }
                if (U.axis == 1) {
                    // V-plane rows are r_v * 2 bytes apart: stage the warp's 32 rows x 64 bytes and
                    // store 8 rows of 64 contiguous bytes per instruction
#pragma unroll
                    for (int k = 0; k < 32; k += 8) {
                        const int c = c0 + k;
                        float b8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                        if (use_bias) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) b8[i] = bs[c + i];
                        }
                        *reinterpret_cast<uint4 *>(stg + lane * 80 + (k / 8) * 16) =
                            make_uint4(pack_bf16(v[k] - b8[0], v[k + 1] - b8[1]), pack_bf16(v[k + 2] - b8[2], v[k + 3] - b8[3]),
                                       pack_bf16(v[k + 4] - b8[4], v[k + 5] - b8[5]), pack_bf16(v[k + 6] - b8[6], v[k + 7] - b8[7]));
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int rr = 8 * i + (lane >> 2), cc = lane & 3;
                        char *d = reinterpret_cast<char *>(__shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(dst), rr));
                        const uint4 val = *reinterpret_cast<const uint4 *>(stg + rr * 80 + cc * 16);
                        if (d && c0 + cc * 8 < U.cols) *reinterpret_cast<uint4 *>(d + (U.col0 + c0 + cc * 8) * 2) = val;
                    }
                    __syncwarp();
                } else if (dst) {
#pragma unroll
                    for (int k = 0; k < 32; k += 8) {
                        const int c = c0 + k, jc = U.col0 + c;  // column in the group, in the axis
                        if (c >= U.cols) break;
                        float b8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                        if (use_bias) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) b8[i] = bs[c + i];
                        }
                        const uint4 w = make_uint4(pack_bf16(v[k] - b8[0], v[k + 1] - b8[1]),
                                                   pack_bf16(v[k + 2] - b8[2], v[k + 3] - b8[3]),
                                                   pack_bf16(v[k + 4] - b8[4], v[k + 5] - b8[5]),
                                                   pack_bf16(v[k + 6] - b8[6], v[k + 7] - b8[7]));
                        // K-plane: granule jc/8 of 16 bytes at (jc/8) * 64 * 16 + row * 16
                        *reinterpret_cast<uint4 *>(dst + (jc / 8) * (kBlockTokens * 16)) = w;
                    }
                }
            }
        }
    } else if (MU && warp >= kConv0) {
        // ------------------------------------------------------- x - m into TMEM (one row per thread)
        uint32_t *mws = reinterpret_cast<uint32_t *>(sm + L::oMu) + quarter * 64;  // [2][32] pairs of m
        const char *xr = sm + row * 128;
        const uint32_t ta = tmem + kAT + (static_cast<uint32_t>(quarter * 32) << 16);
        const int total = static_cast<int>(u1 - u0) * NS;
        int64_t u = u0;
        int s = 0;
        const float *mu = nullptr;
        float m0 = 0.f, m1 = 0.f;  // mu of the slab to come
        auto next_mu = [&] {       // of slab s of unit u, then on to the next
            if (s == 0 && u < u1) {
                const Unit U = unit_of(p, u);
                mu = U.axis ? p.mu_v : p.mu_k;
                if (mu) mu += static_cast<int64_t>(U.h) * Td + S0 * kES + 2 * lane;
                else m0 = m1 = 0.f;
            }
            if (u < u1 && mu) {
                m0 = mu[s * kES];
                m1 = mu[s * kES + 1];
            }
            if (++s == NS) {
                s = 0;
                ++u;
            }
        };
        next_mu();
#pragma unroll 1
        for (int q = 0; q < total; ++q) {
            const int st = q % L::XST, buf = q & 1;
            mws[buf * 32 + lane] = pack_bf16(m0, m1);
            next_mu();
            __syncwarp();
            mbar_wait_warp(&full[st], (q / L::XST) & 1, abort_flag, p.err);
            uint32_t hi[32], lo[32];
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 x = *reinterpret_cast<const uint4 *>(xr + st * kASlab + ((c ^ (row & 7)) << 4));
                hi[4 * c] = x.x; hi[4 * c + 1] = x.y; hi[4 * c + 2] = x.z; hi[4 * c + 3] = x.w;
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&empty[st]);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const uint4 m = *reinterpret_cast<const uint4 *>(mws + buf * 32 + 4 * c);
                sub_exact_bf16x2(hi[4 * c], m.x, hi[4 * c], lo[4 * c]);
                sub_exact_bf16x2(hi[4 * c + 1], m.y, hi[4 * c + 1], lo[4 * c + 1]);
                sub_exact_bf16x2(hi[4 * c + 2], m.z, hi[4 * c + 2], lo[4 * c + 2]);
                sub_exact_bf16x2(hi[4 * c + 3], m.w, hi[4 * c + 3], lo[4 * c + 3]);
            }
            // the products of two slabs ago have read this buffer
            mbar_wait_warp(&aempty[buf], ((q >> 1) & 1) ^ 1u, abort_flag, p.err);
            tc_fence_after();
            tmem_st32u_nowait(ta + buf * 64, hi);
            tmem_st32u_nowait(ta + buf * 64 + 32, lo);
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&afull[buf]);
        }
    }
    pdl_trigger();
    if (split) {
        // every CTA of the cluster has finished its products: the rings may take the parts
        __syncthreads();
        cluster_sync();
        const Unit U = unit_of(p, u0);
        const int own = ((U.cols + p.split - 1) / p.split + 7) & ~7;  // columns each rank stores
        const bool ep = warp >= kEpi0 && warp < kConv0;
        const float *bs = bias + U.g * kMaxGroup;
        const bool use_bias = MU && (U.axis ? p.mu_v : p.mu_k) != nullptr;
        if (ep) {
#pragma unroll
            for (int i = 0; i < L::NC; ++i)
#pragma unroll
                for (int k = 0; k < 32; k += 8) {
                    const int c0 = 64 * i + 32 * half + k;
                    if (c0 >= U.cols) break;
                    float v[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[e] = use_bias ? sum[i][k + e] - bs[c0 + e] : sum[i][k + e];
                    const uint32_t to = c0 / own;
                    const uint32_t at = smem_addr(sm) + ((crank * (own / 4) + (c0 - to * own) / 4) * kEM + row) * 16;
                    st_cluster_f4(at, to, make_float4(v[0], v[1], v[2], v[3]));
                    st_cluster_f4(at + kEM * 16, to, make_float4(v[4], v[5], v[6], v[7]));
                }
        }
        cluster_sync();
        if (ep) {
            char *dst = row_dst(p, U, row, U.g == 0 && crank == 0 && half == 0);
            for (int c0 = crank * own + 8 * half; c0 < min(U.cols, (crank + 1) * own); c0 += 16) {
                float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                for (int q = 0; q < p.split; ++q) {
                    const float4 *src = reinterpret_cast<const float4 *>(sm) + (q * (own / 4) + (c0 - crank * own) / 4) * kEM + row;
                    const float4 a = src[0], b = src[kEM];
                    v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w;
                    v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
                }
                if (dst) {
                    const int jc = U.col0 + c0;
                    *reinterpret_cast<uint4 *>(U.axis == 0 ? dst + (jc / 8) * (kBlockTokens * 16) : dst + jc * 2) =
                        make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, kTmemCols);
    }
}

bool make_maps(const EncodeArgs &a, int axis, bool wres, CUtensorMap *tx, CUtensorMap *tw) {
    const int Td = a.T * a.d;
    const int r = axis ? a.r_v : a.r_k;
    const void *x = axis ? a.x_v : a.x_k;
    const void *w = axis ? a.w_down_v : a.w_down_k;
    {
        const uint64_t dims[4] = {static_cast<uint64_t>(a.d), static_cast<uint64_t>(a.H),
                                  static_cast<uint64_t>(a.N), static_cast<uint64_t>(a.T)};
        const uint64_t strides[3] = {static_cast<uint64_t>(a.d) * 2, static_cast<uint64_t>(a.H) * a.d * 2,
                                     static_cast<uint64_t>(a.N) * a.H * a.d * 2};
        const uint32_t box[4] = {kES, 1, kEM, 1};
        if (!encode_tmap_bf16(tx, x, 4, dims, strides, box, true)) return false;
    }
    if (wres) {  // W_down goes through registers: the map is never used
        *tw = *tx;
        return true;
    }
    const uint64_t dims[3] = {static_cast<uint64_t>(r), static_cast<uint64_t>(Td), static_cast<uint64_t>(a.H)};
    const uint64_t strides[2] = {static_cast<uint64_t>(r) * 2, static_cast<uint64_t>(Td) * r * 2};
    const uint32_t box[3] = {64, kES, 1};
    return encode_tmap_bf16(tw, w, 3, dims, strides, box, true);
}

// Column groups of an axis of rank r: ceil(r / 192) groups of `width` columns (a multiple of 16).
int axis_groups(int r, int *width) {
    const int n = (r + kMaxGroup - 1) / kMaxGroup;
    *width = ((r + n - 1) / n + 15) & ~15;
    return (r + *width - 1) / *width;
}

// Equal groups of a multiple of 32 columns, at most 192 (7: r has no such split).
int groups_of_32(int r) {
    const int n = (r + kMaxGroup - 1) / kMaxGroup;
    return r % n == 0 && (r / n) % 32 == 0 ? n : 7;
}

// W_down rows of whole 16-byte words travel by tensor map; others (even ranks) only resident.
bool wide_rows(const EncodeArgs &a) { return a.r_k % 8 == 0 && a.r_v % 8 == 0; }
bool fits_resident(const EncodeArgs &a) { return a.r_k <= 64 && a.r_v <= 64 && a.T * a.d <= kResSlabs * kES; }

template <bool WRES, bool MU>
lla_status launch_tc(const EncodeArgs &a, const ETParams &p, int grid, cudaStream_t stream) {
    CUtensorMap txk, txv, twk, twv;
    if (!make_maps(a, 0, WRES, &txk, &twk) || !make_maps(a, 1, WRES, &txv, &twv)) return LLA_ERR_CUDA;
    static DeviceOnce configured;
    if (raise_smem_limit(encode_tc_kernel<WRES, MU>, EL<WRES, MU>::SMEM, configured) != LLA_OK) return LLA_ERR_CUDA;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(grid));
    cfg.blockDim = dim3(EL<WRES, MU>::THREADS);
    cfg.dynamicSmemBytes = EL<WRES, MU>::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(p.split);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = p.split > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, encode_tc_kernel<WRES, MU>, txk, txv, twk, twv, p) != cudaSuccess) return LLA_ERR_CUDA;
    return LLA_OK;
}

}  // namespace

bool encode_tc_supported(const EncodeArgs &a) {
    int w = 0;
    // stacks that no token tile of the CUDA-core kernel holds are taken where they always were
    if (a.T * a.d > kLongestStack && !(a.N >= kEM && groups_of_32(a.r_k) + groups_of_32(a.r_v) <= 6)) return false;
    // From half a tile of tokens on (what encode_step_kernel leaves): 130 tokens at (72, 120) take 7.5 us here and 34 us on the CUDA
    // cores, 100 tokens at (96, 160) 28 us there.  With a long reduction (LLA-2D) always: the CUDA-core
    // kernel holds only 96 KB / (4 T*d) tokens per CTA and reads all of W_down again for each such
    // tile (one token at 8192 rows: 59 us there, 16 us here; at 4096 rows 35 and 16 us).
    return a.storage_bf16 && a.x_bf16 && !a.dense && a.d % kES == 0 && (a.N > kEM / 2 || a.T * a.d >= kLongReduction) &&
           (wide_rows(a) ? axis_groups(a.r_k, &w) + axis_groups(a.r_v, &w) <= kMaxGroups : fits_resident(a));
}

lla_status launch_encode_tc(const EncodeArgs &a, cudaStream_t stream) {
    lla_status st = LLA_OK;
    unsigned *err = device_error_word(&st);
    if (st != LLA_OK) return st;
    ETParams p = {};
    p.T = a.T; p.H = a.H; p.d = a.d; p.N = a.N; p.r_k = a.r_k; p.r_v = a.r_v;
    p.nk = axis_groups(a.r_k, &p.gk);
    p.nv = axis_groups(a.r_v, &p.gv);
    p.tiles = (a.N + kEM - 1) / kEM;
    p.units = static_cast<int64_t>(a.H) * p.tiles * (p.nk + p.nv);
    p.mu_k = a.mu_k; p.mu_v = a.mu_v;
    p.w_down_k = a.w_down_k; p.w_down_v = a.w_down_v;
    p.pool = static_cast<char *>(a.pool);
    p.num_blocks = a.num_blocks;
    p.head_page_bytes = static_cast<int>(head_page_bytes(a.r_k, a.r_v, 2));
    p.block_bytes = static_cast<int64_t>(p.head_page_bytes) * a.H;
    p.kplane_bytes = LLA_BLOCK_TOKENS * a.r_k * 2;
    p.gran = granule_bytes(a.r_k, 2);
    p.slot_mapping = a.slot_mapping;
    p.err = err;
    const int sms = num_sms();
    if (sms <= 0) return LLA_ERR_CUDA;
    // split the reduction while the clusters fit the SMs and each CTA keeps at least 8 slabs
    p.split = 1;
    const int slabs = a.T * a.d / kES;
    while (wide_rows(a) && p.split < kMaxSplit && p.units * p.split * 2 <= sms && slabs / (p.split * 2) >= 8) p.split *= 2;
    const int grid = static_cast<int>(p.split > 1 ? p.units * p.split : p.units < sms ? p.units : sms);
    if (a.mu_k || a.mu_v)
        return wide_rows(a) ? launch_tc<false, true>(a, p, grid, stream) : launch_tc<true, true>(a, p, grid, stream);
    return wide_rows(a) ? launch_tc<false, false>(a, p, grid, stream) : launch_tc<true, false>(a, p, grid, stream);
}

}  // namespace lla
