// lla_encode_step.cu -- Eq. encode (Sec. 3) of a decode step's completed tokens: few tokens, every
// layer in one launch, bf16 inputs and storage.
//
// c = (x - mu) W_down for N tokens reads all of W_down once (4 MB per layer at rho = 4, 101 MB for 24
// layers) for 16 multiply-adds per weight and token: a stream of W_down from HBM.  The CUDA-core
// kernel (lla_encode.cu) spent the time on multiply-adds, on unpacking bf16 and on staging x as fp32
// once per 32 columns.  Here each weight goes from global memory straight into an mma.sync fragment:
//   * a CTA takes 16 or 32 tokens x up to 64 columns of one axis of one head, its four warps a
//     quarter of the reduction each (partial sums meet in shared memory);
//   * lane (g, q) = (lane / 4, lane % 4) loads 16 bytes (columns 8g .. 8g + 7) of the eight rows
//     8q .. 8q + 7 of a block of 32 rows, and 16 bytes (those eight k) of x of tokens g and g + 8.
//     The reduction index is permuted to fit: step s of the block gives the fragment's k pairs
//     (2q, 2q + 1) and (2q + 8, 2q + 9) the rows 8q + 4s + {0, 1} and + {2, 3}, so the words of x
//     are A registers as loaded, and two rows' words interleave (prmt) into B registers.  Column g
//     of n-tile j is column 8g + j, so a lane ends with whole 8-column chunks of its tokens.
//   * with mu, x - m for the bf16 rounding m of mu is formed exactly as two bf16 parts, each an operand A,
//     and the rest mu - m enters as two more rows of A (its 16 significant bits): (mu - m) W_down, in
//     accumulators of its own, is subtracted at the end.  (x W_down - mu W_down instead, with mu in three
//     parts, lost what the two large sums round off where mu is far above the spread of x: with mu 64
//     times the spread thirty times as many latents were rounded the wrong way.)
// No shared memory holds operands, so five CTAs fit an SM and about 80 KB of loads are in flight.
// mma.sync and not tcgen05: with 16 tokens the products are 3 % of the tensor rate, and W_down rows
// need no staging, no tensor maps (four per layer) and no TMEM.
//
// Measured (replayed from a graph, cold weights) against the kernels that took these calls before: 24
// layers of 16 tokens at (96, 160) 90.5 -> 25.6 us (bytes: 17 us), with mu 113.6 -> 41 us, 64 tokens
// 337 -> 73 us (with mu 420 -> 119), 128 tokens 216 -> 133 us (1738 -> 227); 48 layers of 64 tokens at (72, 120) 584 -> 112 us; 48 layers
// of 128 tokens at (18, 30) 397 -> 90 us; one layer of 16 tokens at (96, 160) 7.3 -> 5.2 us.  What
// bounds it: the latency of one block of W_down per warp at few tokens; the loads of x (16 bytes of a
// token per lane, again for every 64 columns) at many, so that the prompt kernel takes over where
// tokens x ranks pass kStepWork (100 tokens at (192, 320): 9.2 us a layer there, 10.4 here).
#include <cuda_runtime.h>

#include "lla_device.cuh"
#include "lla_internal.h"

namespace lla {
namespace {

constexpr int kWarps = 4;
constexpr int kThreadsS = kWarps * 32;
constexpr int kStepTokens = 256;      // beyond these, and beyond tokens x ranks of kStepWork, the prompt kernel
constexpr int kStepWork = 128 * 256;
constexpr int kLongReduction = 4096;  // LLA-2D stacks: the prompt kernel splits them over clusters

struct StepLayer {
    const void *w_down_k, *w_down_v;
    const float *mu_k, *mu_v;
    const void *x_k, *x_v;
    char *pool;
    int64_t num_blocks;
};
struct StepParams {
    int T, H, d, r_k, r_v, N;
    int gk, gv;  // column groups of each axis
    int ck, cv;  // chunks per group of each axis
    int64_t block_bytes;
    int head_page_bytes, kplane_bytes, gran;
    const int64_t *slot_mapping;
    unsigned *err;
    StepLayer l[kMaxEncodeLayers];
};

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 ldg_stream(const uint4 *p) {
    uint4 v;
    // (not .nc: the previous kernel on the stream may still write it when this one starts)
    asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p)
                 : "memory");
    return v;
}

// Chunks of W_down columns: 8 columns (16 bytes), one per lane; or, for ranks whose rows are not whole
// 16-byte words, 2 columns (4 bytes), two per lane (chunks g and g + 8).
template <int CW>
struct Chunks {
    static constexpr int SLOTS = CW == 8 ? 1 : 2;
    static constexpr int PER = 8 * SLOTS;      // most chunks of a CTA
    static constexpr int COLS = CW * PER;      // and columns
    static constexpr int NT = CW * SLOTS;      // n-tiles: column i of slot u is n-tile u * CW + i
    static constexpr int WORDS = CW / 2;       // 32-bit words of a chunk
};

// The words of one block of 32 reduction rows held by a lane.
template <int MT, bool MU, int CW>
struct Block {
    uint32_t w[8][Chunks<CW>::SLOTS * Chunks<CW>::WORDS];  // rows 8q .. 8q + 7
    uint4 x[2 * MT];      // tokens g, g + 8 (, g + 16, g + 24)
    float m[MU ? 8 : 1];  // mu of the eight rows
};

// Resident CTAs per SM the registers are held to.  One block of 32 rows in flight per warp and more
// warps beat two blocks per warp: 24 layers of 16 tokens at (96, 160) take 25.3 us with five CTAs
// and one block, 28.2 with four, 30.5 with three and two blocks each.  (64 tokens per CTA, which reads
// W_down half as often as two CTAs of 32, was slower: 78.8 against 73.3 us for 64 tokens.)
// With mu: three and two CTAs, whose registers hold everything (one more each spilled: 24 layers of 16
// tokens 40.7 and 45.4 us, of 64 tokens 119 and 133; mu - m as constant rows into the tokens' own
// accumulators instead, 33.5 and 101 us, took four roundings per 16 rows where this takes two, and more
// latents were rounded the wrong way than with fp32 sums).
constexpr int step_ctas(int mt, bool mu) { return mt == 1 ? (mu ? 3 : 5) : (mu ? 2 : 3); }

template <int MT, bool MU, int CW>
__global__ void __launch_bounds__(kThreadsS, step_ctas(MT, MU)) encode_step_kernel(const __grid_constant__ StepParams p) {
    using C = Chunks<CW>;
    constexpr int ROWS = 16 * MT + (MU ? 2 : 0);
    constexpr int kRowF = C::COLS + 4;  // floats of a partial row (padded)
    __shared__ __align__(16) float red[kWarps][ROWS][kRowF];
    __shared__ float bias[64];
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
    const int layer = blockIdx.z / p.H, h = blockIdx.z - layer * p.H;
    const StepLayer &L = p.l[layer];
    const int axis = static_cast<int>(blockIdx.y) < p.gk ? 0 : 1;
    const int grp = axis ? blockIdx.y - p.gk : blockIdx.y;
    const int r = axis ? p.r_v : p.r_k, per = axis ? p.cv : p.ck;
    const int chunk0 = grp * per, nch = min(per, r / CW - chunk0);
    const int n0 = blockIdx.x * 16 * MT;
    const int Td = p.T * p.d;
    const int nblk = Td / 32;  // blocks of 32 rows; this warp takes [b0, b1)
    const int b0 = warp * nblk / kWarps, b1 = (warp + 1) * nblk / kWarps;
    const char *W = static_cast<const char *>(axis ? L.w_down_v : L.w_down_k) +
                    (static_cast<int64_t>(h) * Td * r + (chunk0 + g) * CW) * 2;
    const char *x = static_cast<const char *>(axis ? L.x_v : L.x_k) + static_cast<int64_t>(h) * p.d * 2;
    const float *mu = axis ? L.mu_v : L.mu_k;
    const bool use_mu = MU && mu != nullptr;

    Block<MT, MU, CW> blk;
    auto load_w = [&](Block<MT, MU, CW> &B, int b) {
        const int k = b * 32 + 8 * q;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const char *row = W + static_cast<int64_t>(k + i) * r * 2;
            if constexpr (CW == 8) {
                const uint4 v = g < nch ? ldg_stream(reinterpret_cast<const uint4 *>(row)) : make_uint4(0, 0, 0, 0);
                B.w[i][0] = v.x; B.w[i][1] = v.y; B.w[i][2] = v.z; B.w[i][3] = v.w;
            } else {
#pragma unroll
                for (int u = 0; u < C::SLOTS; ++u)
                    B.w[i][u] = g + 8 * u < nch ? *reinterpret_cast<const uint32_t *>(row + u * 8 * CW * 2) : 0u;
            }
        }
        if constexpr (MU) {
            const float *s = mu + static_cast<int64_t>(h) * Td + k;
#pragma unroll
            for (int i = 0; i < 8; ++i) B.m[i] = use_mu ? s[i] : 0.f;
        }
    };
    auto load_x = [&](Block<MT, MU, CW> &B, int b) {
        const int k = b * 32 + 8 * q, t = k / p.d, e = k - t * p.d;
#pragma unroll
        for (int i = 0; i < 2 * MT; ++i) {
            const int n = n0 + g + 8 * i;
            B.x[i] = n < p.N ? *reinterpret_cast<const uint4 *>(x + ((static_cast<int64_t>(t) * p.N + n) * p.H * p.d + e) * 2)
                             : make_uint4(0, 0, 0, 0);
        }
    };
    float acc[MT + (MU ? 1 : 0)][C::NT][4];
#pragma unroll
    for (int m = 0; m < MT + (MU ? 1 : 0); ++m)
#pragma unroll
        for (int j = 0; j < C::NT; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[m][j][i] = 0.f;
    auto compute = [&](const Block<MT, MU, CW> &B) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            uint32_t am[2] = {0u, 0u};
            uint32_t xa[MT][4], xl[MU ? MT : 1][4];  // A of each m-tile: x, or hi and lo of x - m
#pragma unroll
            for (int m = 0; m < MT; ++m) {
                const uint4 &u = B.x[2 * m], &v = B.x[2 * m + 1];
                xa[m][0] = s ? u.z : u.x; xa[m][1] = s ? v.z : v.x; xa[m][2] = s ? u.w : u.y; xa[m][3] = s ? v.w : v.y;
            }
            if constexpr (MU) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const float m0 = B.m[4 * s + 2 * i], m1 = B.m[4 * s + 2 * i + 1];
                    const __nv_bfloat162 mb = __floats2bfloat162_rn(m0, m1);
                    const uint32_t mh = *reinterpret_cast<const uint32_t *>(&mb);
#pragma unroll
                    for (int m = 0; m < MT; ++m) {
                        sub_exact_bf16x2(xa[m][2 * i], mh, xa[m][2 * i], xl[m][2 * i]);
                        sub_exact_bf16x2(xa[m][2 * i + 1], mh, xa[m][2 * i + 1], xl[m][2 * i + 1]);
                    }
                    // rows 0 and 1 of the mu tile: the upper eight bits of mu - m, and the lower (exact)
                    float r0 = g < 2 ? bf16_rest(m0) : 0.f, r1 = g < 2 ? bf16_rest(m1) : 0.f;
                    if (g == 1) {
                        r0 -= __uint_as_float(__float_as_uint(r0) & 0xffff0000u);
                        r1 -= __uint_as_float(__float_as_uint(r1) & 0xffff0000u);
                    }
                    am[i] = __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
                }
            }
#pragma unroll
            for (int j = 0; j < C::NT; ++j) {
                const uint32_t sel = (j & 1) ? 0x7632u : 0x5410u;
                const uint32_t f0 = __byte_perm(B.w[4 * s][j / 2], B.w[4 * s + 1][j / 2], sel);
                const uint32_t f1 = __byte_perm(B.w[4 * s + 2][j / 2], B.w[4 * s + 3][j / 2], sel);
#pragma unroll
                for (int m = 0; m < MT; ++m) {
                    mma_bf16(acc[m][j], xa[m][0], xa[m][1], xa[m][2], xa[m][3], f0, f1);
                    if constexpr (MU) mma_bf16(acc[m][j], xl[m][0], xl[m][1], xl[m][2], xl[m][3], f0, f1);
                }
                if constexpr (MU) mma_bf16(acc[MT][j], am[0], 0u, am[1], 0u, f0, f1);
            }
        }
    };
    // any input, the codec's too, may come from the previous kernel: only addresses come before the wait
    pdl_wait();
    if (b0 < b1) {
        load_w(blk, b0);
        load_x(blk, b0);
    }
#pragma unroll 1
    for (int b = b0; b < b1; ++b) {
        compute(blk);
        if (b + 1 < b1) {
            load_w(blk, b + 1);
            load_x(blk, b + 1);
        }
    }
    pdl_trigger();
    // partial sums: token row g (+ 8) of each m-tile, columns 2q and 2q + 1 of every n-tile: column i
    // of chunk c sits at c * CW + i
    auto put = [&](int row, const float (&a)[C::NT][4], int hf) {
#pragma unroll
        for (int u = 0; u < C::SLOTS; ++u)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                float *dst = &red[warp][row][(8 * u + 2 * q + c) * CW];
                const int i = 2 * hf + c;
                if constexpr (CW == 8) {
                    reinterpret_cast<float4 *>(dst)[0] = make_float4(a[0][i], a[1][i], a[2][i], a[3][i]);
                    reinterpret_cast<float4 *>(dst)[1] = make_float4(a[4][i], a[5][i], a[6][i], a[7][i]);
                } else {
                    *reinterpret_cast<float2 *>(dst) = make_float2(a[u * CW][i], a[u * CW + 1][i]);
                }
            }
    };
#pragma unroll
    for (int m = 0; m < MT; ++m) {
        put(16 * m + g, acc[m], 0);
        put(16 * m + 8 + g, acc[m], 1);
    }
    if constexpr (MU) {
        if (g < 2) put(16 * MT + g, acc[MT], 0);
    }
    __syncthreads();
    if constexpr (MU) {
        if (tid < C::COLS) {
            float v = 0.f;
#pragma unroll
            for (int w = 0; w < kWarps; ++w)
#pragma unroll
                for (int i = 0; i < 2; ++i) v += red[w][16 * MT + i][tid];
            bias[tid] = v;
        }
        __syncthreads();
    }
    // thread (token, chunk): sum of the warps' parts, minus the bias, rounded and scattered
    for (int o = tid; o < 16 * MT * C::PER; o += kThreadsS) {
        const int row = o / C::PER, c = o % C::PER, n = n0 + row;
        if (n >= p.N || c >= nch) continue;
        float v[CW];
#pragma unroll
        for (int i = 0; i < CW; ++i) v[i] = MU ? -bias[c * CW + i] : 0.f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
#pragma unroll
            for (int i = 0; i < CW; i += 2) {
                const float2 a = *reinterpret_cast<const float2 *>(&red[w][row][c * CW + i]);
                v[i] += a.x;
                v[i + 1] += a.y;
            }
        }
        const int64_t slot = p.slot_mapping[n];
        if (slot < 0) continue;
        const int64_t blk = slot / kBlockTokens;
        const int ri = static_cast<int>(slot % kBlockTokens);
        if (blk >= L.num_blocks) {
            atomicOr(p.err, LLA_DEVERR_SLOT);
            continue;
        }
        char *page = L.pool + blk * p.block_bytes + static_cast<int64_t>(h) * p.head_page_bytes;
        char *dst = axis == 0 ? page + kplane_offset(ri, (chunk0 + c) * CW, 2, p.gran)
                              : page + p.kplane_bytes + (static_cast<int64_t>(ri) * p.r_v + (chunk0 + c) * CW) * 2;
        uint32_t wd[C::WORDS];
#pragma unroll
        for (int i = 0; i < C::WORDS; ++i) {
            const __nv_bfloat162 t = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
            wd[i] = *reinterpret_cast<const uint32_t *>(&t);
        }
        if constexpr (CW == 8) *reinterpret_cast<uint4 *>(dst) = make_uint4(wd[0], wd[1], wd[2], wd[3]);
        else *reinterpret_cast<uint32_t *>(dst) = wd[0];
    }
}

template <int CW>
lla_status launch_step(const cudaLaunchConfig_t &cfg, int tokens, bool mu, const StepParams &p) {
    const auto kern = tokens == 16 ? (mu ? encode_step_kernel<1, true, CW> : encode_step_kernel<1, false, CW>)
                                   : (mu ? encode_step_kernel<2, true, CW> : encode_step_kernel<2, false, CW>);
    return cudaLaunchKernelEx(&cfg, kern, p) == cudaSuccess ? LLA_OK : LLA_ERR_CUDA;
}

}  // namespace

bool encode_step_supported(const EncodeArgs &a) {
    return a.storage_bf16 && a.x_bf16 && !a.dense && a.d % 32 == 0 && a.T * a.d < kLongReduction &&
           (a.N <= 64 || (a.N <= kStepTokens && a.N * (a.r_k + a.r_v) <= kStepWork));
}

lla_status launch_encode_step(const EncodeArgs *a, int L, cudaStream_t stream) {
    const EncodeArgs &a0 = a[0];
    lla_status st = LLA_OK;
    unsigned *err = device_error_word(&st);
    if (st != LLA_OK) return st;
    StepParams p = {};
    p.T = a0.T; p.H = a0.H; p.d = a0.d; p.r_k = a0.r_k; p.r_v = a0.r_v; p.N = a0.N;
    const int cw = a0.r_k % 8 == 0 && a0.r_v % 8 == 0 ? 8 : 2, most = cw == 8 ? Chunks<8>::PER : Chunks<2>::PER;
    p.gk = (a0.r_k / cw + most - 1) / most;
    p.gv = (a0.r_v / cw + most - 1) / most;
    p.ck = (a0.r_k / cw + p.gk - 1) / p.gk;
    p.cv = (a0.r_v / cw + p.gv - 1) / p.gv;
    p.gran = granule_bytes(a0.r_k, 2);
    p.head_page_bytes = static_cast<int>(head_page_bytes(a0.r_k, a0.r_v, 2));
    p.block_bytes = static_cast<int64_t>(p.head_page_bytes) * a0.H;
    p.kplane_bytes = LLA_BLOCK_TOKENS * a0.r_k * 2;
    p.slot_mapping = a0.slot_mapping;
    p.err = err;
    bool mu = false;
    for (int l = 0; l < L; ++l) {
        p.l[l] = StepLayer{a[l].w_down_k, a[l].w_down_v, a[l].mu_k, a[l].mu_v, a[l].x_k, a[l].x_v,
                           static_cast<char *>(a[l].pool), a[l].num_blocks};
        mu = mu || a[l].mu_k || a[l].mu_v;
    }
    if (static_cast<int64_t>(a0.H) * L > 65535) return LLA_ERR_UNSUPPORTED;
    const int tokens = a0.N > 16 ? 32 : 16;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a0.N + tokens - 1) / tokens, p.gk + p.gv, a0.H * L);
    cfg.blockDim = dim3(kThreadsS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cw == 8 ? launch_step<8>(cfg, tokens, mu, p) : launch_step<2>(cfg, tokens, mu, p);
}

}  // namespace lla
