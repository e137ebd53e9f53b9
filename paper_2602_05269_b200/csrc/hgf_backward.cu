// Straight-through backward pass of the HGF layer (paper, Section 2.2, Definition "Straight-Through
// Estimator"; the forward pass it differentiates is Algorithm 1 with both quantisers treated as the
// identity):
//     dW = dY^T Xd,  dX = dY Wd + dZ A^T,  dZ = ((dY (.) g) B^T) (.) SiLU'(x A),
//     dA = x^T dZ,   dB = g (.) (H^T dY),   dg = sum_m dY (.) (H B)
// with Xd = x~ gamma_x / 127 and Wd = gamma_W t.  Seven matrix products on one generic tcgen05 bf16 GEMM
// (C = A B^T, each operand read in the form it is stored in), plus preparation kernels: Xd as a bf16 matrix (the
// quantiser again, its codes times their scale), the ternary codes as a bf16 matrix of exact -1 / 0 / +1, A and
// g (.) B in bf16.  gamma_W is applied to the fp32 accumulator.
#include <algorithm>
#include <vector>

#include "hgf_tc.cuh"
#include "hgf_warp.cuh"

namespace hgf {

// Every launch of the backward pass is chained to the one before by programmatic dependent launch: its blocks are set up
// under the predecessor's tail and wait for its completion before they touch memory (a step of the 2048 x 5632 layer at
// M = 8192 had seventeen such launches, most of them of 2 to 3 us: 662 -> 646 us together with bw_quant_kernel; now twelve).
template <typename... Params, typename... Args>
static cudaError_t launch_chained(void (*kernel)(Params...), unsigned grid, unsigned block, size_t smem, cudaStream_t stream, Args... args) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, Params(args)...);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}
__device__ __forceinline__ void chain() {  // first thing of a kernel that is all loads and stores
    pdl_launch_dependents();
    pdl_wait();
}

// ---- generic GEMM on the 5th-generation tensor cores: C[I][J] (fp32) = alpha * sum_c A[i][c] B[j][c] (+ C) ----
// Either operand may be stored with the contraction index contiguous ([rows][Cn], "K-major") or with its
// row index contiguous ([Cn][rows], "MN-major"): tcgen05.mma reads both forms from shared memory (the
// instruction descriptor says which), so no operand of the backward pass is ever transposed in memory.
// A K-major tile of R rows x 64 contraction elements is one TMA box of R rows of 128 bytes; an MN-major
// tile is R / 64 boxes of 64 contraction rows of 128 bytes (64 operand rows each), 8 KiB apart; both use
// the 128-byte swizzle.  The contraction may continue over a second pair of operands (A2, B2: the
// low-rank term of dX), and may be split over several CTAs that write partial sums which a second
// kernel adds up in a fixed order.
// Persistent, one CTA per SM, six warps: warp 0 stages operand tiles with TMA, warp 1 issues (elect.sync)
// tcgen05.mma.kind::f16 (bf16 inputs, 128 x BN x 16 per instruction, fp32 accumulators in tensor memory,
// two of them so that a tile's epilogue runs under the next tile's main loop), warps 2-5 read the
// accumulator back (tcgen05.ld) and write C.  Rows and columns past the matrices, and contraction
// elements past Cn, are zeros from TMA's out-of-bounds fill; stores are guarded.  Every wait is bounded.
constexpr int kTBM = 128, kTBK = 64, kTThreads = 192, kTBox = 64 * 128;

struct TcGemmArgs {
    float *C;          // output, or the partial sums [splits][I][ldc] when splits > 1
    int I, J, ldc;
    int kb1, kb2;      // 64-element contraction blocks of the first and of the second operand pair
    int splits, kb_per_split;
    int n_half;        // splits == 1 only: the last n_half / 2 tiles are worked as halves of BN / 2 columns (see tc_gemm)
    int a_mn, b_mn;    // operand forms (both pairs alike); 2: by blocks of 64 rows, two a copy (tc_map)
    float alpha;
    int accumulate;
};

// A product with one extent of at most 64 that rides in a launch by pairs (tc_pair_gemm_kernel): output tiles of 256 x 64, the
// contraction in `splits` parts, each of one or several partial sums of kb_per_sum blocks: those of a launch of its own (tc_split_blocks), added
// in the same order, so the results are the same bits either way.  The sums of the first part are added before they are written; the
// others are left to the reader.  B is stored with its row index contiguous.
struct TcThin {
    float *P;                    // [1 + sums of the parts past the first][I][J], or [..][J][I] when `across`
    int I, J, kb, splits, kb_per_split, kb_per_sum;  // (kb_per_split a multiple of kb_per_sum)
    int a_mn, across;            // (a_mn as in TcGemmArgs)
};
constexpr int kTcThinMax = 2;
struct TcThinArgs {
    TcThin job[kTcThinMax];
    int items, items0;           // tiles times splits of all jobs, of the first
    int busy, c_idle, c_busy;    // pairs 0 .. busy - 1, which have a product tile more than the others, take c_busy items each, the others c_idle
};

template <int BN>
struct TcCfg {
    static constexpr int STAGES = BN == 256 ? 4 : 6;
    static constexpr int A_BYTES = kTBM * 128, B_BYTES = BN * 128, STAGE_BYTES = A_BYTES + B_BYTES;
    static constexpr int OFF_BAR = STAGES * STAGE_BYTES;
    static constexpr int BAR_FULL = 0, BAR_EMPTY = STAGES, BAR_ACCFULL = 2 * STAGES, BAR_ACCEMPTY = 2 * STAGES + 2, BAR_COUNT = 2 * STAGES + 4;
    static constexpr int SMEM_BYTES = OFF_BAR + 256 + 1024;
    static constexpr uint32_t IDESC = (1u << 4) /*f32*/ | (1u << 7) /*A bf16*/ | (1u << 10) /*B bf16*/ |
                                      ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(kTBM >> 4) << 24);
    static constexpr int TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;
};

template <int BN>
__global__ void __launch_bounds__(kTThreads, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
               const __grid_constant__ CUtensorMap tmap_a2, const __grid_constant__ CUtensorMap tmap_b2, const TcGemmArgs g,
               unsigned int *status) {
    using C = TcCfg<BN>;
    extern __shared__ uint8_t tc_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem), bar0 = sbase + C::OFF_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_BAR + C::BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_BAR + C::BAR_COUNT * 8 + 4);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int tiles_i = (g.I + kTBM - 1) / kTBM, tiles_j = (g.J + BN - 1) / BN, tiles_ij = tiles_i * tiles_j;
    const int n_full = tiles_ij - g.n_half / 2;  // tiles worked whole (all of them unless n_half > 0)
    const int num_work = g.n_half ? n_full + g.n_half : tiles_ij * g.splits, kb_all = g.kb1 + g.kb2;
    // work item w: output tile w % tiles_ij, contraction blocks [kb_lo, kb_hi) of split w / tiles_ij; with
    // half tiles (one split): items past n_full are the two halves of the remaining tiles, in turn
    auto kb_lo = [&](int w) { return g.n_half ? 0 : (w / tiles_ij) * g.kb_per_split; };
    auto kb_hi = [&](int w) {
        if (g.n_half) return kb_all;
        const int e = (w / tiles_ij + 1) * g.kb_per_split;
        return e < kb_all ? e : kb_all;
    };
    auto tile_of = [&](int w, int &i0, int &j0, int &bn) {
        int tile = w % tiles_ij, half = 0;
        bn = BN;
        if (g.n_half && w >= n_full) {
            tile = n_full + (w - n_full) / 2;
            half = (w - n_full) & 1;
            bn = BN / 2;
        }
        i0 = (tile / tiles_j) * kTBM;
        j0 = (tile % tiles_j) * BN + half * (BN / 2);
    };

    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(bar(C::BAR_FULL + s), 1);
            mbar_init(bar(C::BAR_EMPTY + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(C::BAR_ACCFULL + b), 1);
            mbar_init(bar(C::BAR_ACCEMPTY + b), 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(C::TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);  // (warp-uniform)
    chain();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        int s = 0;
        uint32_t ph = 0;
        uint32_t issued[C::STAGES] = {};
        bool ok = true;
        for (int w = blockIdx.x; ok && w < num_work; w += gridDim.x) {
            int i0, j0, bn;
            tile_of(w, i0, j0, bn);
            for (int kb = kb_lo(w); kb < kb_hi(w); ++kb) {
                ok = mbar_wait(bar(C::BAR_EMPTY + s), ph ^ 1u, abort_flag, status, 0x800u + s);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    const bool second = kb >= g.kb1;
                    const CUtensorMap *ma = second ? &tmap_a2 : &tmap_a, *mb = second ? &tmap_b2 : &tmap_b;
                    const int c0 = (second ? kb - g.kb1 : kb) * kTBK;
                    const uint32_t dst_a = sbase + s * C::STAGE_BYTES, dst_b = dst_a + C::A_BYTES, full = bar(C::BAR_FULL + s);
                    mbar_arrive_expect_tx(full, C::A_BYTES + (g.b_mn ? bn * 128 : C::B_BYTES));  // (a K-major box always has BN rows)
                    if (g.a_mn == 2) {
                        tma_load_3d(dst_a, ma, 0, c0, i0 / 64, full);
                    } else if (g.a_mn) {
                        for (int h = 0; h < kTBM / 64; ++h) tma_load_2d(dst_a + h * kTBox, ma, i0 + 64 * h, c0, full);
                    } else {
                        tma_load_2d(dst_a, ma, c0, i0, full);
                    }
                    if (g.b_mn == 2) {
                        for (int h = 0; h < bn / 128; ++h) tma_load_3d(dst_b + 2 * h * kTBox, mb, 0, c0, j0 / 64 + 2 * h, full);
                    } else if (g.b_mn) {
                        for (int h = 0; h < bn / 64; ++h) tma_load_2d(dst_b + h * kTBox, mb, j0 + 64 * h, c0, full);
                    } else {
                        tma_load_2d(dst_b, mb, c0, j0, full);
                    }
                }
                ++issued[s];
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
        for (int q = 0; q < C::STAGES; ++q)  // never leave with a copy in flight
            if (issued[q]) {
                const uint32_t par = (issued[q] - 1u) & 1u;
                for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_FULL + q), par); ++i) {}
            }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // (the whole warp walks the loop: see the wrappers)
        {
            auto wait = [&](int i, uint32_t par, unsigned int code) { return __all_sync(0xffffffffu, mbar_wait_poll(bar(i), par, abort_flag, status, code)) != 0; };
            int s = 0, it = 0;
            uint32_t ph = 0;
            bool ok = true;
            const uint32_t idesc = C::IDESC | (g.a_mn ? 1u << 15 : 0u) | (g.b_mn ? 1u << 16 : 0u);
            const uint32_t a_step = g.a_mn ? (16 * 128) >> 4 : 32 >> 4, b_step = g.b_mn ? (16 * 128) >> 4 : 32 >> 4;  // 16 contraction elements
            for (int w = blockIdx.x; ok && w < num_work; w += gridDim.x, ++it) {
                const int b = it & 1;
                const uint32_t acc = tmem_base + b * BN;
                if (it >= 2 && !(ok = wait(C::BAR_ACCEMPTY + b, (uint32_t)((it >> 1) - 1) & 1u, 0x810u)))
                    break;
                tc_fence_after();
                const int lo = kb_lo(w), hi = kb_hi(w);
                int ti0, tj0, bn;
                tile_of(w, ti0, tj0, bn);
                const uint32_t idesc_w = (idesc & ~(0x3fu << 17)) | ((uint32_t)(bn >> 3) << 17);
                for (int kb = lo; kb < hi; ++kb) {
                    if (!(ok = wait(C::BAR_FULL + s, ph, 0x820u + s))) break;
                    tc_fence_after();
                    const uint32_t sa = sbase + s * C::STAGE_BYTES, sb = sa + C::A_BYTES;
                    const uint64_t adesc = g.a_mn ? make_sw128_mn_desc(sa, kTBox) : make_sw128_desc(sa);
                    const uint64_t bdesc = g.b_mn ? make_sw128_mn_desc(sb, kTBox) : make_sw128_desc(sb);
#pragma unroll
                    for (int kk = 0; kk < kTBK / 16; ++kk)
                        warp_mma_f16(acc, adesc + (uint64_t)(a_step * kk), bdesc + (uint64_t)(b_step * kk), idesc_w, (kb > lo || kk) ? 1u : 0u);
                    warp_commit(bar(C::BAR_EMPTY + s));
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                warp_commit(bar(C::BAR_ACCFULL + b));
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int q = warp & 3;  // tensor-memory lane quarter this warp may access
        bool ok = true;
        int it = 0;
        for (int w = blockIdx.x; ok && w < num_work; w += gridDim.x, ++it) {
            int i0, j0, bn;
            tile_of(w, i0, j0, bn);
            float *Cw = g.C + (g.n_half ? (size_t)0 : (size_t)(w / tiles_ij) * g.I * g.ldc);
            const int b = it & 1;
            ok = mbar_wait(bar(C::BAR_ACCFULL + b), (uint32_t)(it >> 1) & 1u, abort_flag, status, 0x830u);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const int i = i0 + 32 * q + lane;  // this thread's row of C = its tensor-memory lane
            const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16) + b * BN;
            const bool empty = kb_lo(w) >= kb_hi(w);  // a split past the end of the contraction: zeros
            for (int cc = 0; cc < bn; cc += 32) {
                if (j0 + cc >= g.J) break;  // (warp-uniform)
                uint32_t v[32];
                tmem_ld32(lane_base + cc, v);
                tmem_ld_wait();
                if (i < g.I) {
                    float *row = Cw + (size_t)i * g.ldc + j0 + cc;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (j0 + cc + 4 * u < g.J) {  // J is a multiple of 4
                            float4 o = make_float4(g.alpha * __uint_as_float(v[4 * u]), g.alpha * __uint_as_float(v[4 * u + 1]),
                                                   g.alpha * __uint_as_float(v[4 * u + 2]), g.alpha * __uint_as_float(v[4 * u + 3]));
                            if (empty) o = make_float4(0.f, 0.f, 0.f, 0.f);
                            float4 *dst = reinterpret_cast<float4 *>(row + 4 * u);
                            if (g.accumulate) { const float4 c = *dst; o.x += c.x; o.y += c.y; o.z += c.z; o.w += c.w; }
                            *dst = o;
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_ACCEMPTY + b));
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(C::TMEM_COLS) : "memory");
    }
}

// ---- the same by pairs of CTAs: 256 x 256 tiles ------------------------------------------------------------
// tcgen05.mma.cta_group::2: the pair's first CTA issues for both; each CTA stages 128 rows of A and half of B's rows, and keeps 128
// rows of C in its tensor memory.  An instruction of 128 x 256 x 16 reads 12 KiB of operands from an SM's shared memory, one of the
// pair 8 KiB on each SM, and a tile's operands are fetched once for 256 rows instead of 128.
// Barriers: both CTAs' copies count on the first one's FULL; its commits reach both CTAs' EMPTY and ACCFULL; both epilogues
// arrive on its ACCEMPTY.
// Which products it takes: tc_pairs_pay.  The tiles of 128 x 256 by single CTAs held the two large products of
// 2048 x 5632 at M = 8192 at 1.14 and 1.22 PFLOP/s (166, 155 us), pairs at 1.25 and 1.42 (152, 133 us; 143 and 127 since a stage comes in
// fewer copies: tc_map), where the power limit is near (library bf16 products for seconds on end: 1.37).  Whole backward pass in a captured chain: 425 -> 380 us, 8192 x 5632 -> 2048
// 547 -> 451, 2048 -> 2048 215 -> 186, 1500 x 3200 -> 2000 93 -> 75.
struct TpCfg {
    static constexpr int STAGES = 6, A_BYTES = kTBM * 128, STAGE_BYTES = 2 * A_BYTES;
    static constexpr int OFF_BAR = STAGES * STAGE_BYTES;
    static constexpr int BAR_FULL = 0, BAR_EMPTY = STAGES, BAR_ACCFULL = 2 * STAGES, BAR_ACCEMPTY = 2 * STAGES + 2, BAR_COUNT = 2 * STAGES + 4;
    static constexpr int SMEM_BYTES = OFF_BAR + 256 + 1024;
    static constexpr uint32_t IDESC = (1u << 4) /*f32*/ | (1u << 7) /*A bf16*/ | (1u << 10) /*B bf16*/ | ((uint32_t)(256 >> 4) << 24);
};
constexpr int kTpTile = 256;
constexpr int kTpMinBlocks = 7, kTpMinBlocksRounds = 10;  // 64-element blocks of the contraction: one round of tiles, several (see tc_pairs_pay)

__device__ __forceinline__ uint32_t cluster_address(uint32_t addr, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Into this CTA's shared memory, counted by a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t cluster_bar) {
    asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n"
                 ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t cluster_bar) {
    asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];\n"
                 ::"r"(dst), "l"(map), "r"(cluster_bar), "r"(x), "r"(y), "r"(z)
                 : "memory");
}
__device__ __forceinline__ void warp_mma_f16_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
    asm volatile("{\n.reg .pred p, e;\nelect.sync _|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\n"
                 "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
                 : "memory");
}
__device__ __forceinline__ void warp_commit_pair(uint32_t bar) {  // arrives at this place in both CTAs
    asm volatile("{\n.reg .pred e;\nelect.sync _|e, 0xffffffff;\n"
                 "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;\n}\n" ::"r"(bar), "h"((uint16_t)3)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_bar) : "memory");
}

struct TcThinMaps { CUtensorMap a[kTcThinMax], b[kTcThinMax]; };

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTThreads, 1)
tc_pair_gemm_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                    const __grid_constant__ CUtensorMap tmap_a2, const __grid_constant__ CUtensorMap tmap_b2, const TcGemmArgs g,
                    const __grid_constant__ TcThinMaps thin_maps, const __grid_constant__ TcThinArgs thin, unsigned int *status) {
    using C = TpCfg;
    extern __shared__ uint8_t tp_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)tp_smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem), bar0 = sbase + C::OFF_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_BAR + C::BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_BAR + C::BAR_COUNT * 8 + 4);
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31, rank = (int)blockIdx.x & 1;
    const int pair = (int)blockIdx.x >> 1, pairs = (int)gridDim.x >> 1;
    const int tiles_i = (g.I + kTpTile - 1) / kTpTile, tiles_j = (g.J + kTpTile - 1) / kTpTile, tiles = tiles_i * tiles_j;
    const int n_full = tiles - g.n_half / 2, num_work = n_full + g.n_half, kb_all = g.kb1 + g.kb2;
    auto tile_of = [&](int w, int &i0, int &j0, int &bn) {  // (halves of the last tiles: as in tc_gemm_kernel)
        int tile = w, half = 0;
        bn = kTpTile;
        if (w >= n_full) {
            tile = n_full + (w - n_full) / 2;
            half = (w - n_full) & 1;
            bn = kTpTile / 2;
        }
        i0 = (tile / tiles_j) * kTpTile;
        j0 = (tile % tiles_j) * kTpTile + half * (kTpTile / 2);
    };
    // The pair's pieces of the thin products, after its tiles.  (Loops of their own in every role: as one loop over both kinds of work the
    // products themselves took 3 % longer, the operands of their MMAs no longer being uniform to the compiler.)
    struct Piece { int i0, kb0, kb1, job, part; };
    auto piece_of = [&](int q, Piece &t) {
        const bool busy = pair < thin.busy;
        int e = (busy ? (pairs - thin.busy) * thin.c_idle + pair * thin.c_busy : (pair - thin.busy) * thin.c_idle) + q;
        if (q >= (busy ? thin.c_busy : thin.c_idle) || e >= thin.items) return false;
        t.job = e >= thin.items0 ? 1 : 0;
        if (t.job) e -= thin.items0;
        const TcThin &T = thin.job[t.job];
        const int tiles_t = (T.I + kTpTile - 1) / kTpTile;
        t.i0 = (e % tiles_t) * kTpTile;
        t.part = e / tiles_t;
        t.kb0 = t.part * T.kb_per_split;
        t.kb1 = t.kb0 + T.kb_per_split < T.kb ? t.kb0 + T.kb_per_split : T.kb;
        return true;
    };
    constexpr int kThinCols = kTpTile / 2;  // (the second CTA's half of the columns lies past the matrix: zeros)

    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            mbar_init(bar(C::BAR_FULL + s), 1);
            mbar_init(bar(C::BAR_EMPTY + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(C::BAR_ACCFULL + b), 1);
            mbar_init(bar(C::BAR_ACCEMPTY + b), 8);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    cluster_arrive_release();  // both CTAs' barriers are there before either is reached from the other
    cluster_wait_acquire();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);  // (warp-uniform)
    chain();

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        int s = 0;
        uint32_t ph = 0, issued = 0;
        bool ok = true;
        for (int w = pair; ok && w < num_work; w += pairs) {
            int i0, j0, bn;
            tile_of(w, i0, j0, bn);
            i0 += rank * kTBM;
            j0 += rank * (bn / 2);
            for (int kb = 0; kb < kb_all; ++kb) {
                ok = mbar_wait(bar(C::BAR_EMPTY + s), ph ^ 1u, abort_flag, status, 0x840u + s);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    const bool second = kb >= g.kb1;
                    const CUtensorMap *ma = second ? &tmap_a2 : &tmap_a, *mb = second ? &tmap_b2 : &tmap_b;
                    const int c0 = (second ? kb - g.kb1 : kb) * kTBK;
                    const uint32_t dst_a = sbase + s * C::STAGE_BYTES, dst_b = dst_a + C::A_BYTES, full = cluster_address(bar(C::BAR_FULL + s), 0);
                    if (rank == 0)  // (a K-major box always has 128 rows, one by blocks two of them)
                        mbar_arrive_expect_tx(bar(C::BAR_FULL + s), 2 * (C::A_BYTES + (g.b_mn == 1 ? bn / 2 * 128 : C::A_BYTES)));
                    if (g.a_mn == 2) {
                        tma_load_3d_pair(dst_a, ma, 0, c0, i0 / 64, full);
                    } else if (g.a_mn) {
                        for (int h = 0; h < kTBM / 64; ++h) tma_load_2d_pair(dst_a + h * kTBox, ma, i0 + 64 * h, c0, full);
                    } else {
                        tma_load_2d_pair(dst_a, ma, c0, i0, full);
                    }
                    if (g.b_mn == 2) {
                        tma_load_3d_pair(dst_b, mb, 0, c0, j0 / 64, full);
                    } else if (g.b_mn) {
                        for (int h = 0; h < bn / 128; ++h) tma_load_2d_pair(dst_b + h * kTBox, mb, j0 + 64 * h, c0, full);
                    } else {
                        tma_load_2d_pair(dst_b, mb, c0, j0, full);
                    }
                }
                ++issued;
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
        Piece t;
        for (int q = 0; ok && piece_of(q, t); ++q) {
            const int i0 = t.i0 + rank * kTBM, a_mn = thin.job[t.job].a_mn;
            for (int kb = t.kb0; kb < t.kb1; ++kb) {
                ok = mbar_wait(bar(C::BAR_EMPTY + s), ph ^ 1u, abort_flag, status, 0x880u + s);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    const CUtensorMap *ma = &thin_maps.a[t.job];
                    const int c0 = kb * kTBK;
                    const uint32_t dst_a = sbase + s * C::STAGE_BYTES, dst_b = dst_a + C::A_BYTES, full = cluster_address(bar(C::BAR_FULL + s), 0);
                    if (rank == 0) mbar_arrive_expect_tx(bar(C::BAR_FULL + s), 2 * (C::A_BYTES + kTBox));
                    if (a_mn == 2) {
                        tma_load_3d_pair(dst_a, ma, 0, c0, i0 / 64, full);
                    } else if (a_mn) {
                        for (int h = 0; h < kTBM / 64; ++h) tma_load_2d_pair(dst_a + h * kTBox, ma, i0 + 64 * h, c0, full);
                    } else {
                        tma_load_2d_pair(dst_a, ma, c0, i0, full);
                    }
                    tma_load_2d_pair(dst_b, &thin_maps.b[t.job], rank * (kThinCols / 2), c0, full);
                }
                ++issued;
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
        // Never leave with a copy in flight: a stage's MMAs, which follow its copies, reach this CTA's EMPTY.
        for (uint32_t q = 0; q < (uint32_t)C::STAGES; ++q) {
            const uint32_t rounds = (issued + C::STAGES - 1 - q) / C::STAGES;
            if (rounds)
                for (uint32_t i = 0; i < (ok ? kSpinLimit : 1u << 12) && !mbar_try_wait(bar(C::BAR_EMPTY + q), (rounds - 1u) & 1u); ++i)
                    if (!ok) __nanosleep(1000);  // (after a time-out nothing may come: some milliseconds, which a copy does not take)
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer (the first CTA's, for both)
        if (rank == 0) {
            auto wait = [&](int i, uint32_t par, unsigned int code) { return __all_sync(0xffffffffu, mbar_wait_poll(bar(i), par, abort_flag, status, code)) != 0; };
            int s = 0, it = 0;
            uint32_t ph = 0;
            bool ok = true;
            const uint32_t idesc = C::IDESC | (g.a_mn ? 1u << 15 : 0u) | (g.b_mn ? 1u << 16 : 0u);
            const uint32_t a_step = g.a_mn ? (16 * 128) >> 4 : 32 >> 4, b_step = g.b_mn ? (16 * 128) >> 4 : 32 >> 4;  // 16 contraction elements
            for (int w = pair; ok && w < num_work; w += pairs, ++it) {
                const int b = it & 1;
                const uint32_t acc = tmem_base + b * kTpTile;
                if (it >= 2 && !(ok = wait(C::BAR_ACCEMPTY + b, (uint32_t)((it >> 1) - 1) & 1u, 0x850u))) break;
                tc_fence_after();
                int ti0, tj0, bn;
                tile_of(w, ti0, tj0, bn);
                const uint32_t idesc_w = idesc | ((uint32_t)(bn >> 3) << 17);
                for (int kb = 0; kb < kb_all; ++kb) {
                    if (!(ok = wait(C::BAR_FULL + s, ph, 0x860u + s))) break;
                    tc_fence_after();
                    const uint32_t sa = sbase + s * C::STAGE_BYTES, sb = sa + C::A_BYTES;
                    const uint64_t adesc = g.a_mn ? make_sw128_mn_desc(sa, kTBox) : make_sw128_desc(sa);
                    const uint64_t bdesc = g.b_mn ? make_sw128_mn_desc(sb, kTBox) : make_sw128_desc(sb);
#pragma unroll
                    for (int kk = 0; kk < kTBK / 16; ++kk)
                        warp_mma_f16_pair(acc, adesc + (uint64_t)(a_step * kk), bdesc + (uint64_t)(b_step * kk), idesc_w, (kb || kk) ? 1u : 0u);
                    warp_commit_pair(bar(C::BAR_EMPTY + s));
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
                if (!ok) break;
                warp_commit_pair(bar(C::BAR_ACCFULL + b));
            }
            Piece t;
            for (int q = 0; ok && piece_of(q, t); ++q) {
                const bool a_mn = thin.job[t.job].a_mn != 0;
                const uint32_t idesc_w = C::IDESC | (a_mn ? 1u << 15 : 0u) | (1u << 16) | ((uint32_t)(kThinCols >> 3) << 17), step = a_mn ? (16 * 128) >> 4 : 32 >> 4;
                for (int k0 = t.kb0; ok && k0 < t.kb1; k0 += thin.job[t.job].kb_per_sum, ++it) {
                    const int b = it & 1, k1 = min(k0 + thin.job[t.job].kb_per_sum, t.kb1);
                    const uint32_t acc = tmem_base + b * kTpTile;
                    if (it >= 2 && !(ok = wait(C::BAR_ACCEMPTY + b, (uint32_t)((it >> 1) - 1) & 1u, 0x890u))) break;
                    tc_fence_after();
                    for (int kb = k0; kb < k1; ++kb) {
                        if (!(ok = wait(C::BAR_FULL + s, ph, 0x8a0u + s))) break;
                        tc_fence_after();
                        const uint32_t sa = sbase + s * C::STAGE_BYTES, sb = sa + C::A_BYTES;
                        const uint64_t adesc = a_mn ? make_sw128_mn_desc(sa, kTBox) : make_sw128_desc(sa), bdesc = make_sw128_mn_desc(sb, kTBox);
#pragma unroll
                        for (int kk = 0; kk < kTBK / 16; ++kk)
                            warp_mma_f16_pair(acc, adesc + (uint64_t)(step * kk), bdesc + (uint64_t)(((16 * 128) >> 4) * kk), idesc_w, (kb > k0 || kk) ? 1u : 0u);
                        warp_commit_pair(bar(C::BAR_EMPTY + s));
                        if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                    }
                    if (!ok) break;
                    warp_commit_pair(bar(C::BAR_ACCFULL + b));
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ epilogue warps
        const int q = warp & 3;  // tensor-memory lane quarter this warp may access
        bool ok = true;
        int it = 0;
        for (int w = pair; ok && w < num_work; w += pairs, ++it) {
            int i0, j0, bn;
            tile_of(w, i0, j0, bn);
            const int b = it & 1;
            ok = mbar_wait(bar(C::BAR_ACCFULL + b), (uint32_t)(it >> 1) & 1u, abort_flag, status, 0x870u);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const int i = i0 + rank * kTBM + 32 * q + lane;  // this thread's row of C = its tensor-memory lane
            const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16) + b * kTpTile;
            for (int cc = 0; cc < bn; cc += 32) {
                if (j0 + cc >= g.J) break;  // (warp-uniform)
                uint32_t v[32];
                tmem_ld32(lane_base + cc, v);
                tmem_ld_wait();
                if (i < g.I) {
                    float *row = g.C + (size_t)i * g.ldc + j0 + cc;
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        if (j0 + cc + 4 * u < g.J) {  // J is a multiple of 4
                            float4 o = make_float4(g.alpha * __uint_as_float(v[4 * u]), g.alpha * __uint_as_float(v[4 * u + 1]),
                                                   g.alpha * __uint_as_float(v[4 * u + 2]), g.alpha * __uint_as_float(v[4 * u + 3]));
                            float4 *dst = reinterpret_cast<float4 *>(row + 4 * u);
                            if (g.accumulate) { const float4 c = *dst; o.x += c.x; o.y += c.y; o.z += c.z; o.w += c.w; }
                            *dst = o;
                        }
                    }
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(cluster_address(bar(C::BAR_ACCEMPTY + b), 0));
        }
        Piece t;
        for (int n = 0; ok && piece_of(n, t); ++n) {
            const TcThin &T = thin.job[t.job];
            int out = t.part ? 1 + (t.kb0 - T.kb_per_split) / T.kb_per_sum : 0;
            float run[64];
            for (int k0 = t.kb0; ok && k0 < t.kb1; k0 += T.kb_per_sum, ++it) {
                const int b = it & 1;
                ok = mbar_wait(bar(C::BAR_ACCFULL + b), (uint32_t)(it >> 1) & 1u, abort_flag, status, 0x8b0u);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
                const int i = t.i0 + rank * kTBM + 32 * q + lane;
                const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16) + b * kTpTile;
                const bool add = t.part == 0 && k0 > 0, store = t.part > 0 || k0 + T.kb_per_sum >= t.kb1;
#pragma unroll
                for (int cc = 0; cc < 64; cc += 16) {
                    if (cc >= T.J) break;  // (J is a multiple of 16)
                    uint32_t v[16];
                    tmem_ld16(lane_base + cc, v);
                    tmem_ld_wait();
#pragma unroll
                    for (int u = 0; u < 16; ++u) run[cc + u] = add ? run[cc + u] + __uint_as_float(v[u]) : __uint_as_float(v[u]);
                    if (store && i < T.I) {
                        if (T.across) {
#pragma unroll
                            for (int u = 0; u < 16; ++u) T.P[((size_t)out * T.J + cc + u) * T.I + i] = run[cc + u];
                        } else {
                            float4 *dst = reinterpret_cast<float4 *>(T.P + ((size_t)out * T.I + i) * T.J + cc);
#pragma unroll
                            for (int u = 0; u < 4; ++u) dst[u] = make_float4(run[cc + 4 * u], run[cc + 4 * u + 1], run[cc + 4 * u + 2], run[cc + 4 * u + 3]);
                        }
                    }
                }
                out += store;
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive_cluster(cluster_address(bar(C::BAR_ACCEMPTY + b), 0));
            }
        }
    }

    tc_fence_before();
    __syncwarp();
    cluster_arrive_release();  // no CTA leaves while the other may still reach its barriers or its shared memory
    cluster_wait_acquire();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// Sum of the partial results of a split contraction, in split order: C = alpha * sum_s P[s] (+ C).
__global__ void __launch_bounds__(256) tc_reduce_kernel(const float4 *P, int splits, size_t n4, float alpha, int accumulate, float4 *C) {
    chain();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n4) return;
    float4 a = P[i];
    for (int s = 1; s < splits; ++s) {
        const float4 b = P[(size_t)s * n4 + i];
        a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    a.x *= alpha; a.y *= alpha; a.z *= alpha; a.w *= alpha;
    if (accumulate) { const float4 c = C[i]; a.x += c.x; a.y += c.y; a.z += c.z; a.w += c.w; }
    C[i] = a;
}

// One operand: `rows` x `cn` values; mn = stored [cn][rows] (row index contiguous), else [rows][cn]; ld in elements.
struct TcOperand {
    const __nv_bfloat16 *p;
    int ld;
    bool mn;
};

// *form: 0 for a K-major operand, 1 for one whose row index is contiguous, 2 where two blocks of 64 of its rows come with one copy (their number
// a multiple of 64, tiles of 128 rows and more).  The TMA unit works a copy of 64 rows of 128 bytes hardly faster than one of 128, and a
// stage of dW was four of them: 2048 x 5632 at M = 8192 dW 167 -> 143 us, dX 142 -> 127, a training step 596 -> 577.
static bool tc_map(CUtensorMap *m, const TcOperand &o, int rows, int cn, int tile_rows, int *form = nullptr) {
    if (form && o.mn && tile_rows >= 128 && make_map_blocks(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, o.p, (uint64_t)rows, (uint64_t)cn, (uint64_t)o.ld * 2, kTBK, 2)) {
        *form = 2;
        return true;
    }
    if (form) *form = o.mn ? 1 : 0;
    if (o.mn) return make_map_2d(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, o.p, (uint64_t)rows, (uint64_t)cn, (uint64_t)o.ld * 2, 64, kTBK, CU_TENSOR_MAP_SWIZZLE_128B);
    return make_map_2d(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, o.p, (uint64_t)cn, (uint64_t)rows, (uint64_t)o.ld * 2, kTBK, (uint32_t)tile_rows, CU_TENSOR_MAP_SWIZZLE_128B);
}

template <int BN>
static cudaError_t tc_gemm_bn(const CUtensorMap *maps, const TcGemmArgs &g, cudaStream_t stream) {
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = ensure_dynamic_smem(tc_gemm_kernel<BN>, TcCfg<BN>::SMEM_BYTES, attr_done);
    if (e != cudaSuccess) return e;
    const int sms = device_sm_count();
    if (!sms) return cudaErrorInvalidDevice;
    const int tiles = ((g.I + kTBM - 1) / kTBM) * ((g.J + BN - 1) / BN);
    const int work = g.n_half ? tiles + g.n_half / 2 : tiles * g.splits;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    return launch_chained(tc_gemm_kernel<BN>, (unsigned)(work < sms ? work : sms), kTThreads, TcCfg<BN>::SMEM_BYTES, stream, maps[0], maps[1], maps[2], maps[3], g, status);
}

// Pairs of CTAs that run at once with one CTA an SM.
static int tc_pairs_at_once() {
    static std::atomic<int> cache[kMaxDevices];
    const int dev = current_device();
    if (dev < 0 || dev >= kMaxDevices) return 0;
    int n = cache[dev].load(std::memory_order_acquire);
    if (n) return n;
    static std::atomic<unsigned long long> attr_done{0};
    if (ensure_dynamic_smem(tc_pair_gemm_kernel, TpCfg::SMEM_BYTES, attr_done) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2);
    cfg.blockDim = dim3(kTThreads);
    cfg.dynamicSmemBytes = TpCfg::SMEM_BYTES;
    if (cudaOccupancyMaxActiveClusters(&n, tc_pair_gemm_kernel, &cfg) != cudaSuccess || n <= 0) {
        cudaGetLastError();  // (single CTAs take the product: their launch is not to report this call's error)
        return 0;
    }
    cache[dev].store(n, std::memory_order_release);
    return n;
}

// Rounds of the persistent schedule for that many tiles, in halves: the last tiles are worked as twice as many of half the width
// where that fills their round (`halves`: the operand forms and the width allow it).
static int tc_half_rounds(int tiles, int at_once, bool halves) {
    const int rest = tiles % at_once;
    return 2 * (tiles / at_once) + (rest == 0 ? 0 : (halves && tiles > at_once && 2 * rest <= at_once ? 1 : 2));
}
// Whether pairs of CTAs take an I x J product over kb_all blocks of 64.  An output has to be more than 128 x 128.  A short contraction
// does not repay a pair's start and its hand-overs: over 1300 products (I 136 to 4096, J 192 to 12544; dW or dX alone in a captured
// chain, single CTAs' time over pairs') 64 to 256 gave 0.85 to 1.03, 448 to 576 gave 0.95 to 1.06 in one round of tiles and 0.93 to 1.08
// in several, 640 and more 0.97 to 1.54.  And 256-row tiles may need more rounds than 128-row ones: one and a half
// instead of one gave 0.86 to 0.98 at any contraction, two and a half instead of two 0.91 to 0.99 up to 1024 and 0.98 to 1.14 from
// 2048 on.  4096 x 4096 over 300: 32.4 us, by pairs 35.3; 384 x 9984 over 640: 21.7, 25.3; 8192 x 2048 over 5632: 155, 133.
static bool tc_pairs_pay(int I, int J, int kb_all, bool b_mn, int sms, int pairs) {
    if (I <= kTBM || J <= 128 || pairs <= 0 || sms <= 0) return false;
    const int tiles_j = (J + 255) / 256, tiles = (I + kTpTile - 1) / kTpTile * tiles_j;
    if (kb_all < (tiles <= pairs ? kTpMinBlocks : kTpMinBlocksRounds)) return false;
    const bool halves = b_mn && J % 256 == 0;
    const int by_pairs = tc_half_rounds(tiles, pairs, halves), by_one = tc_half_rounds((I + kTBM - 1) / kTBM * tiles_j, sms, halves);
    return by_pairs <= by_one || (kb_all >= 16 && 4 * by_pairs <= 5 * by_one);
}
// (for the tests)
extern "C" int hgf_internal_tc_pairs_pay(int32_t I, int32_t J, int32_t contraction, int32_t sms, int32_t pairs) {
    return tc_pairs_pay(I, J, (contraction + kTBK - 1) / kTBK, true, sms, pairs) ? 1 : 0;
}

constexpr int kBwSplitsMax = 16;  // partial sums of a product that may be split

// Output columns of a single CTA's tile.
static int tc_tile_columns(int J) { return J > 128 ? 256 : (J > 64 ? 128 : 64); }
// An I x J product over kb blocks of 64 by single CTAs that may split its contraction: blocks of a partial sum.
static int tc_split_blocks(int I, int J, int kb, int sms) {
    const int BN = tc_tile_columns(J), tiles = ((I + kTBM - 1) / kTBM) * ((J + BN - 1) / BN);
    int splits = 1;
    if (sms > 0 && tiles * 2 <= sms) splits = std::max(1, std::min({sms / tiles, kBwSplitsMax, kb / 4}));  // at least four blocks per split
    return (kb + splits - 1) / splits;
}

// A thin product as the caller describes it: P as in TcThin, room for all of its partial sums; `rides` is set by tc_gemm: to how many sums
// there are in P then, 0 if it did not ride.
struct TcThinProduct {
    TcOperand A, B;      // B.mn
    int I, J, Cn;
    bool across;
    float *P;
    int kb_per_sum;      // those of a launch of its own
    int rides;
    int sums() const { return ((Cn + kTBK - 1) / kTBK + kb_per_sum - 1) / kb_per_sum; }
    int sums_left(const TcThin &t) const { return 1 + std::max(0, sums() - t.kb_per_split / kb_per_sum); }
};

// The thin products' pieces over the pairs; false where launches of their own are the better way.  In half blocks of the product (64 of the
// contraction for half a tile, 0.22 us): a piece costs 1.1 a block - its first operand is staged whole, of the second nearly nothing - and 10
// for its start and end.  The pairs that have a tile of the last round less take pieces first; contractions are split, up to four
// times, where that brings the last pair's end forward.  A launch of its own takes 4 us and its first operand's bytes at 4.5 TB/s; the
// estimate has to stay below three quarters of that, since a pair streams what has left L2 by then more slowly than all SMs together do.
// Backward passes in a captured chain, launches of their own / this: 700 x 1024 -> 3000, r = 32 72 / 54 us, 2048 x 2048 -> 2048 91 / 76,
// 1500 x 3200 -> 2000, r = 64 129 / 106, 8000 x 768 -> 1536, r = 64 133 / 106, 4096 x 4096 -> 4096, r = 16 287 / 268, 8192 x 4096 -> 1024, r = 64
// 228 / 220, 8192 x 2048 -> 5632 391 / 390.  A part is whole partial sums of a launch of its own, for the same bits.  Parts of any size would be 0 to
// 11 per cent faster (geometric mean of 30 passes 2.8), but their longer sums are others: gradients moved by 1e-4.
static bool tc_deal_thin(TcThinArgs *t, const TcThinProduct *thin, int n, int num_work, int n_half, int kb_all, int pairs) {
    const int rest = num_work % pairs, idle = pairs - rest;
    const double extra = rest ? (n_half ? kb_all : 2.0 * kb_all) : 0.0;
    double best = -1.0, alone = 0.0;
    int longest = 0;
    for (int i = 0; i < n; ++i) {
        longest = std::max(longest, (thin[i].Cn + kTBK - 1) / kTBK);
        alone += 4.0 + 2.0 * thin[i].I * thin[i].Cn / 4.5e6;
    }
    for (int parts = 1; parts <= 4; ++parts) {
        const int share = (longest + parts - 1) / parts;
        int piece = 0;  // blocks of the longest
        TcThinArgs c = {};
        for (int i = 0; i < n; ++i) {
            TcThin &T = c.job[i];
            T.P = thin[i].P;
            T.I = thin[i].I; T.J = thin[i].J;
            T.kb = (thin[i].Cn + kTBK - 1) / kTBK;
            T.kb_per_sum = thin[i].kb_per_sum;
            T.splits = (T.kb + share - 1) / share;
            T.kb_per_split = ((T.kb + T.splits - 1) / T.splits + T.kb_per_sum - 1) / T.kb_per_sum * T.kb_per_sum;  // whole partial sums
            T.splits = (T.kb + T.kb_per_split - 1) / T.kb_per_split;  // no empty part
            piece = std::max(piece, std::min(T.kb_per_split, T.kb));
            T.across = thin[i].across ? 1 : 0;
            c.items += (T.I + kTpTile - 1) / kTpTile * T.splits;
            if (i == 0) c.items0 = c.items;
        }
        c.busy = rest;
        for (c.c_busy = 0; c.c_busy <= (rest > 0 ? 1 : 0); ++c.c_busy) {
            c.c_idle = std::max(0, (c.items - c.c_busy * rest + idle - 1) / idle);
            if (c.c_idle > 2) continue;
            const double cost = 10.0 + 1.1 * piece, end = std::max(c.c_idle * cost, c.c_busy ? extra + c.c_busy * cost : extra);
            if (best >= 0.0 && end >= best) continue;
            best = end;
            *t = c;
        }
    }
    if (best >= 0.0 && 0.22 * (best - extra) <= 0.75 * alone) return true;
    *t = TcThinArgs{};
    return false;
}

// (for the tests: how n thin products of I[i] rows over contractions Cn[i] are dealt behind num_work tiles of kb_all blocks, the last n_half of
// them halves; out: items, items0, busy, c_idle, c_busy, then splits and kb_per_split of each)
extern "C" int hgf_internal_tc_deal_thin(const int32_t *I, const int32_t *Cn, int32_t n, int32_t num_work, int32_t n_half, int32_t kb_all, int32_t pairs, int32_t *out) {
    TcThinProduct thin[kTcThinMax] = {};
    for (int i = 0; i < n && i < kTcThinMax; ++i) {
        thin[i].I = I[i]; thin[i].Cn = Cn[i]; thin[i].J = 16;
        thin[i].kb_per_sum = tc_split_blocks(I[i], 16, (Cn[i] + kTBK - 1) / kTBK, 2 * pairs);
    }
    TcThinArgs t = {};
    const bool ride = tc_deal_thin(&t, thin, n, num_work, n_half, kb_all, pairs);
    out[0] = t.items; out[1] = t.items0; out[2] = t.busy; out[3] = t.c_idle; out[4] = t.c_busy;
    for (int i = 0; i < n; ++i) { out[5 + 2 * i] = t.job[i].splits; out[6 + 2 * i] = t.job[i].kb_per_split; }
    return ride ? 1 : 0;
}

// (for the tests) What a pass does with its room for partial sums, in the order of its launches, of which none is enqueued.
struct BwTrace {
    int sms, pairs;
    const float *room;
    struct Use { bool write; int64_t first, end; };
    std::vector<Use> uses;
    struct Rides { bool dx; int n, n_half, c_idle, c_busy; };
    std::vector<Rides> rides;  // of each launch by pairs
    void use(bool write, const float *p, size_t n) { uses.push_back({write, p - room, p - room + (int64_t)n}); }
};

// C[I][J] = alpha * (A B^T + A2 B2^T) (+ C).  A2.p == nullptr: one pair only.  Both pairs have the same
// operand forms.  `partials` (kBwSplitsMax * I * ldc floats) enables splitting the contraction when the
// output has fewer tiles than the device has SMs; ldc must then be J.  With `splits_out` they are left there for the kernel that
// reads the product next (*splits_out of them; 1: the product is in C).  `thin`: products that may ride in a launch by pairs; those that
// did have `rides` afterwards.  Bases 16-byte aligned, ld % 8 == 0.
static cudaError_t tc_gemm(TcOperand A, TcOperand B, int Cn, TcOperand A2, TcOperand B2, int Cn2, float *C, int ldc, int I, int J,
                           float alpha, bool accumulate, float *partials, int *splits_out, TcThinProduct *thin, int n_thin, cudaStream_t stream, BwTrace *trace) {
    const int BN = tc_tile_columns(J), sms = trace ? trace->sms : device_sm_count();
    const int kb1 = (Cn + kTBK - 1) / kTBK, kb2 = A2.p ? (Cn2 + kTBK - 1) / kTBK : 0, kb_all = kb1 + kb2;
    int pairs = I > kTBM && J > 128 && kb_all >= kTpMinBlocks && sms > 0 ? (trace ? trace->pairs : tc_pairs_at_once()) : 0;
    if (!tc_pairs_pay(I, J, kb_all, B.mn, sms, pairs)) pairs = 0;
    CUtensorMap maps[4];
    const int rows_b = pairs ? 128 : BN;
    TcGemmArgs g = {};
    if (!trace) {
        if (!tc_map(&maps[0], A, I, Cn, kTBM, &g.a_mn) || !tc_map(&maps[1], B, J, Cn, rows_b, &g.b_mn)) return cudaErrorInvalidValue;
        maps[2] = maps[0];
        maps[3] = maps[1];
        int form_a = g.a_mn, form_b = g.b_mn;  // (by the extents I and J and the row pitches' alignment: alike for both pairs)
        if (A2.p && (!tc_map(&maps[2], A2, I, Cn2, kTBM, &form_a) || !tc_map(&maps[3], B2, J, Cn2, rows_b, &form_b))) return cudaErrorInvalidValue;
        if (form_a != g.a_mn || form_b != g.b_mn) return cudaErrorInvalidValue;
    }
    g.I = I; g.J = J; g.ldc = ldc;
    g.kb1 = kb1;
    g.kb2 = kb2;
    if (pairs) {
        const int tiles = ((I + kTpTile - 1) / kTpTile) * ((J + kTpTile - 1) / kTpTile);
        if (B.mn && tiles > pairs && tiles % pairs != 0 && 2 * (tiles % pairs) <= pairs && J % kTpTile == 0) g.n_half = 2 * (tiles % pairs);
        g.splits = 1;
        g.C = C; g.alpha = alpha; g.accumulate = accumulate ? 1 : 0;
        if (splits_out) *splits_out = 1;
        const int work = tiles + g.n_half / 2;
        TcThinArgs t = {};
        TcThinMaps thin_maps;
        if (n_thin && !tc_deal_thin(&t, thin, n_thin, work, g.n_half, kb_all, pairs)) n_thin = 0;
        if (trace) {
            for (int i = 0; i < n_thin; ++i) {
                thin[i].rides = thin[i].sums_left(t.job[i]);
                trace->use(true, thin[i].P, (size_t)thin[i].rides * thin[i].I * thin[i].J);
            }
            trace->rides.push_back({!A.mn, n_thin, g.n_half, t.c_idle, t.c_busy});
            return cudaSuccess;
        }
        for (int i = 0; i < kTcThinMax; ++i) {
            thin_maps.a[i] = maps[0];
            thin_maps.b[i] = maps[1];
            if (i >= n_thin) continue;
            if (!tc_map(&thin_maps.a[i], thin[i].A, thin[i].I, thin[i].Cn, kTBM, &t.job[i].a_mn) || !tc_map(&thin_maps.b[i], thin[i].B, thin[i].J, thin[i].Cn, 0))
                return cudaErrorInvalidValue;
            thin[i].rides = thin[i].sums_left(t.job[i]);
        }
        unsigned int *status = device_status_word();
        if (!status) return cudaErrorMemoryAllocation;
        return launch_chained(tc_pair_gemm_kernel, 2u * (unsigned)(work < pairs && !n_thin ? work : pairs), kTThreads, TpCfg::SMEM_BYTES, stream, maps[0], maps[1],
                              maps[2], maps[3], g, thin_maps, t, status);
    }
    const int tiles = ((I + kTBM - 1) / kTBM) * ((J + BN - 1) / BN);
    g.kb_per_split = partials && ldc == J ? tc_split_blocks(I, J, kb_all, sms) : kb_all;
    g.splits = (kb_all + g.kb_per_split - 1) / g.kb_per_split;  // no empty split
    // Tail of the tile schedule: when the tiles left for the last round of the persistent CTAs would keep at most
    // half of the SMs busy, they are worked as twice as many tiles of half the width, which fills the round.
    if (g.splits == 1 && BN == 256 && B.mn && sms > 0 && tiles > sms && tiles % sms != 0 && 2 * (tiles % sms) <= sms &&
        J % 256 == 0)
        g.n_half = 2 * (tiles % sms);
    if (g.splits == 1) {
        g.C = C; g.alpha = alpha; g.accumulate = accumulate ? 1 : 0;
    } else {
        g.C = partials; g.alpha = 1.0f; g.accumulate = 0;
    }
    if (splits_out) *splits_out = g.splits;  // the caller adds the partial sums
    const size_t n4 = (size_t)I * J / 4;
    if (trace) {
        if (g.splits > 1) trace->use(true, partials, 4 * n4 * g.splits);
        if (g.splits > 1 && !splits_out) trace->use(false, partials, 4 * n4 * g.splits);
        return cudaSuccess;
    }
    cudaError_t e = BN == 256 ? tc_gemm_bn<256>(maps, g, stream) : (BN == 128 ? tc_gemm_bn<128>(maps, g, stream) : tc_gemm_bn<64>(maps, g, stream));
    if (e != cudaSuccess || g.splits == 1 || splits_out) return e;
    return launch_chained(tc_reduce_kernel, (unsigned)((n4 + 255) / 256), 256, 0, stream, (const float4 *)partials, g.splits, n4, alpha, accumulate ? 1 : 0, (float4 *)C);
}

// ---- operand preparation ---------------------------------------------------------------------------
// Xd = x~ gamma_x / 127 as bf16 [M][K] (eight values per thread).
__global__ void __launch_bounds__(256) bw_dequant_kernel(const int8_t *xq, const float *gamma_x, int K, size_t n8, __nv_bfloat16 *xd) {
    chain();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n8) return;
    const float s = gamma_x[(i * 8) / (size_t)K] * (1.0f / 127.0f);
    const uint2 w = reinterpret_cast<const uint2 *>(xq)[i];
    const uint32_t ww[2] = {w.x, w.y};
    uint32_t o[4];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
        const int c0 = (int)(int8_t)(ww[h >> 1] >> (16 * (h & 1))), c1 = (int)(int8_t)(ww[h >> 1] >> (16 * (h & 1) + 8));
        const __nv_bfloat162 v = __floats2bfloat162_rn((float)c0 * s, (float)c1 * s);
        o[h] = *reinterpret_cast<const uint32_t *>(&v);
    }
    reinterpret_cast<uint4 *>(xd)[i] = make_uint4(o[0], o[1], o[2], o[3]);
}

// Algorithm 1, steps 1-2, and Xd in one pass over x for rows of up to 256 U columns: one warp per row, the row in
// registers between the maximum and the rounding, the codes turned into values without touching memory.  Bound by HBM
// (2 + 2 bytes an element): 8192 x 2048 in 11.9 us, against 11.9 + 8.8 us through int8 codes in memory.
template <int U>
__global__ void __launch_bounds__(256) bw_quant_kernel(const __nv_bfloat16 *x, int M, int K, __nv_bfloat16 *xd) {
    chain();
    const int lane = threadIdx.x & 31, m = blockIdx.x * 8 + (threadIdx.x >> 5), nv = K / 8;
    if (m >= M) return;
    const uint4 *xv = reinterpret_cast<const uint4 *>(x + (size_t)m * K);
    uint4 v[U];
    uint32_t abits = 0u;
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = lane + 32 * u < nv ? xv[lane + 32 * u] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < U; ++u) abits = absmax8_bits(abits, v[u]);
    const float g = fmaxf(warp_max(absmax_bits_to_float(abits)), 1e-5f), s = g * (1.0f / 127.0f);
    const QuantScale qs = make_quant_scale(g);
    uint4 *dst = reinterpret_cast<uint4 *>(xd + (size_t)m * K);
    int sum = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (lane + 32 * u < nv) {
            const uint2 c = quant8<true>(v[u], qs, sum);
            const uint32_t w[2] = {c.x ^ 0x80808080u, c.y ^ 0x80808080u};  // code + 128
            uint32_t o[4];
#pragma unroll
            for (int h = 0; h < 4; ++h) {
                // the byte as the low mantissa bits of 2^23, minus (2^23 + 128): the code as a float, exactly
                const float c0 = __uint_as_float(__byte_perm(w[h >> 1], 0x4b000000u, 0x7650 + 2 * (h & 1))) - 8388736.0f;
                const float c1 = __uint_as_float(__byte_perm(w[h >> 1], 0x4b000000u, 0x7651 + 2 * (h & 1))) - 8388736.0f;
                const __nv_bfloat162 p = __floats2bfloat162_rn(c0 * s, c1 * s);
                o[h] = *reinterpret_cast<const uint32_t *>(&p);
            }
            dst[lane + 32 * u] = make_uint4(o[0], o[1], o[2], o[3]);
        }
    }
}

// The weights' side of the products, one launch: a small layer's pass is a chain of launches of 2 to 3 us (this one as three, and the
// partial sums of three products added by launches of their own: 64 x 512 -> 512 42.1 us, now 38.8; 2048 -> 5632 at M = 2048
// 137.9 / 136.8).  The ternary codes of the packed matrix as a bf16 matrix T [N][K] of -1 / 0 / +1 (one packed word = 16 columns
// per thread), A^T in bf16, and B^T in bf16 with the gate folded in (an element per thread).
struct BwWeights {
    const uint32_t *packed;
    const __half *At, *Bt;
    const float *gate;
    __nv_bfloat16 *T, *At_b, *gBt;
    size_t n_words, n_at, n_bt;      // 0: not wanted
    unsigned blocks_t, blocks_at;    // blocks of the first two parts
    int N, K, r, steps;
};
__global__ void __launch_bounds__(256) bw_weights_kernel(const BwWeights p) {
    chain();
    if (blockIdx.x >= p.blocks_t) {
        const unsigned b = blockIdx.x - p.blocks_t;
        if (b < p.blocks_at) {
            const size_t i = (size_t)b * 256 + threadIdx.x;
            if (i < p.n_at) p.At_b[i] = __float2bfloat16_rn(__half2float(p.At[i]));
        } else {
            const size_t i = (size_t)(b - p.blocks_at) * 256 + threadIdx.x;
            if (i < p.n_bt) p.gBt[i] = __float2bfloat16_rn(__half2float(p.Bt[i]) * p.gate[i / (size_t)p.r]);
        }
        return;
    }
    const size_t w = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (w >= p.n_words) return;
    const int kw = (int)(w & 15), r = (int)((w >> 4) & 15);
    const size_t tile = w >> 8;
    const int n = (int)(tile / p.steps) * 16 + r, k0 = (int)(tile % p.steps) * 256 + kw * 16;
    if (n >= p.N || k0 >= p.K) return;
    const uint32_t word = p.packed[w];
    uint32_t o[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const uint32_t e = (word >> (2 * j)) & 0x03030303u;
#pragma unroll
        for (int b = 0; b < 4; b += 2) {
            const int c0 = (e >> (8 * b)) & 0xff, c1 = (e >> (8 * b + 8)) & 0xff;
            const __nv_bfloat162 v = __floats2bfloat162_rn((float)(c0 == 3 ? 0 : c0 - 1), (float)(c1 == 3 ? 0 : c1 - 1));
            o[2 * j + (b >> 1)] = *reinterpret_cast<const uint32_t *>(&v);
        }
    }
    uint4 *dst = reinterpret_cast<uint4 *>(p.T + (size_t)n * p.K + k0);
    dst[0] = make_uint4(o[0], o[1], o[2], o[3]);
    dst[1] = make_uint4(o[4], o[5], o[6], o[7]);
}

// Element i of a product: the sum of its partial results in split order (n elements each), or the product itself.
__device__ __forceinline__ float split_sum(const float *P, int splits, size_t n, size_t i) {
    float v = P[i];
    for (int s = 1; s < splits; ++s) v += P[(size_t)s * n + i];
    return v;
}

// Z (fp32 [M][r], in `splits` partial sums) -> H = act(Z) as bf16 [M][r] and SiLU'(Z) as fp32.
__global__ void __launch_bounds__(256) bw_act_kernel(const float *P, int splits, size_t n, int no_silu, float *dact, __nv_bfloat16 *h) {
    chain();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float v = split_sum(P, splits, n, i);
    const float sg = 1.0f / (1.0f + expf(-v));
    h[i] = __float2bfloat16_rn(no_silu ? v : v * sg);
    dact[i] = no_silu ? 1.0f : sg * (1.0f + v * (1.0f - sg));
}

// dZ = dH * SiLU'(Z), rounded to bf16, and dZ * scale (the copy that enters dX next to gamma_W dY T); dH in partial sums.
__global__ void __launch_bounds__(256) bw_dz_kernel(const float *P, int splits, const float *dact, size_t n, float scale, __nv_bfloat16 *dz,
                                                    __nv_bfloat16 *dz_scaled) {
    chain();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n) return;
    const float v = split_sum(P, splits, n, i) * dact[i];
    dz[i] = __float2bfloat16_rn(v);
    dz_scaled[i] = __float2bfloat16_rn(v * scale);
}

// From G[n][j] = sum_m dY[m][n] H[m][j] (in partial sums): dBt[n][j] = gate[n] G[n][j], dgate[n] = sum_j G[n][j] Bt[n][j].
// One warp per output channel n (its r values are contiguous).
__global__ void __launch_bounds__(256) bw_gate_kernel(const float *P, int splits, const __half *Bt, const float *gate, int N, int r, float *dBt,
                                                      float *dgate) {
    chain();
    const int n = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (n >= N) return;
    float dg = 0.0f;
    const float gn = gate[n];
    for (int j = lane; j < r; j += 32) {
        const float v = split_sum(P, splits, (size_t)N * r, (size_t)n * r + j);
        dg = fmaf(v, __half2float(Bt[(size_t)n * r + j]), dg);
        dBt[(size_t)n * r + j] = gn * v;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dg += __shfl_xor_sync(0xffffffffu, dg, o);
    if (dgate && lane == 0) dgate[n] = dg;
}

constexpr int kBwQuantMaxK = 4096;  // up to here a row fits a warp's registers (bw_quant_kernel): no codes and scales in memory

struct BwLayout {
    size_t xq, gamma_x, xd, T, At_b, gBt, z, h_b, dh, dz_b, dzs_b, G, partials, total;
};
static BwLayout bw_layout(int64_t M, int64_t K, int64_t N, int32_t r) {
    BwLayout L;
    size_t off = 0;
    auto take = [&](size_t bytes) { const size_t o = off; off += align_up(bytes, 256); return o; };
    const size_t rr = (size_t)(r > 0 ? r : 16);
    L.xq = take(K > kBwQuantMaxK ? (size_t)M * K : 0);
    L.gamma_x = take(K > kBwQuantMaxK ? (size_t)M * 4 : 0);
    L.xd = take((size_t)M * K * 2);
    L.T = take((size_t)N * K * 2);
    L.At_b = take(rr * K * 2);
    L.gBt = take((size_t)N * rr * 2);
    L.z = take((size_t)M * rr * 4);
    L.h_b = take((size_t)M * rr * 2);
    L.dh = take((size_t)M * rr * 4);
    L.dz_b = take((size_t)M * rr * 2);
    L.dzs_b = take((size_t)M * rr * 2);
    L.G = take((size_t)N * rr * 4);
    const size_t big = (size_t)(M > N ? (M > K ? M : K) : (N > K ? N : K));
    L.partials = take((size_t)kBwSplitsMax * big * rr * 4);  // split contractions all have r as one output extent
    L.total = off;
    return L;
}

}  // namespace hgf

using namespace hgf;

extern "C" size_t hgf_backward_workspace_bytes(int64_t M, int64_t d_in, int64_t d_out, int32_t r) {
    if (M <= 0 || d_in <= 0 || d_out <= 0 || r < 0) return 256;
    return bw_layout(M, d_in, d_out, r).total;
}

static hgf_status backward(const void *x, int64_t M, const void *packed, float gamma, int64_t d_in, int64_t d_out, const void *At, const void *Bt,
                           int32_t r, const float *gate, const void *dy, const hgf_grads *grads, void *workspace, size_t workspace_bytes,
                           uint32_t flags, void *stream_, BwTrace *trace) {
    if (!x || !packed || !dy || !grads || M <= 0 || d_in <= 0 || d_out <= 0 || r < 0) return HGF_ERR_INVALID_ARG;
    if (flags & ~HGF_FLAG_NO_SILU) return HGF_ERR_INVALID_ARG;
    if (!At || !Bt || !gate) r = 0;
    if (d_in % 64 != 0 || d_out % 8 != 0 || d_in > 65536 || d_out > (1 << 24) || M > (1 << 22)) return HGF_ERR_UNSUPPORTED_SHAPE;
    if (r != 0 && r != 16 && r != 32 && r != 48 && r != 64) return HGF_ERR_UNSUPPORTED_SHAPE;
    const uintptr_t bits = (uintptr_t)x | (uintptr_t)packed | (uintptr_t)dy | (uintptr_t)At | (uintptr_t)Bt | (uintptr_t)gate |
                           (uintptr_t)grads->dx | (uintptr_t)grads->dW | (uintptr_t)grads->dAt | (uintptr_t)grads->dBt |
                           (uintptr_t)grads->dgate;
    if (bits & 15u) return HGF_ERR_MISALIGNED;
    const BwLayout L = bw_layout(M, d_in, d_out, r);
    if (!workspace || workspace_bytes < L.total) return HGF_ERR_WORKSPACE;
    if (((uintptr_t)workspace) & 255u) return HGF_ERR_MISALIGNED;
    cudaStream_t stream = (cudaStream_t)stream_;
    char *ws = (char *)workspace;
    const int Mi = (int)M, K = (int)d_in, N = (int)d_out;
    auto bf = [&](size_t off) { return (__nv_bfloat16 *)(ws + off); };
    auto blocks1 = [](size_t n) { return (unsigned)((n + 255) / 256); };
    const TcOperand none = {nullptr, 0, false};
    float *partials = (float *)(ws + L.partials);
    if (trace) trace->room = partials;
    bool ok = true;
    auto launch = [&](auto *kernel, unsigned blocks, auto... args) {
        if (!trace) ok = ok && launch_chained(kernel, blocks, 256, 0, stream, args...) == cudaSuccess;
    };
    auto done = [&] { return ok && (trace || cudaGetLastError() == cudaSuccess) ? HGF_OK : HGF_ERR_CUDA; };
    auto gemm = [&](TcOperand A, TcOperand B, int Cn, TcOperand A2, TcOperand B2, int Cn2, float *C, int ldc, int I, int J, float alpha,
                    bool acc, bool may_split, int *splits_out = nullptr, TcThinProduct *thin = nullptr, int n_thin = 0) {
        ok = ok && tc_gemm(A, B, Cn, A2, B2, Cn2, C, ldc, I, J, alpha, acc, may_split ? partials : nullptr, splits_out, thin, n_thin, stream, trace) == cudaSuccess;
    };
    // The partial sums of a product, or the product itself, for the launch that comes next; the room may be used again after it.
    auto read = [&](const float *sums, const float *product, int splits, size_t n) {
        if (trace && splits > 0 && sums != product) trace->use(false, sums, n * splits);
        return sums;
    };
    const TcOperand dy_k = {(const __nv_bfloat16 *)dy, N, false};  // dY as [M rows][N contraction]
    const TcOperand dy_mn = {(const __nv_bfloat16 *)dy, N, true};  // dY as [N rows] contracted over its M stored rows
    const TcOperand x_k = {(const __nv_bfloat16 *)x, K, false}, x_mn = {(const __nv_bfloat16 *)x, K, true};

    {
        BwWeights p = {};
        p.packed = (const uint32_t *)packed;
        p.T = bf(L.T);
        p.N = N; p.K = K; p.r = r;
        p.steps = (int)(padded_k(d_in) / 256);
        p.n_words = grads->dx ? (size_t)row_tiles(d_out) * p.steps * 256 : 0;
        p.blocks_t = blocks1(p.n_words);
        if (r) {
            p.At = (const __half *)At; p.At_b = bf(L.At_b); p.n_at = (size_t)r * K;
            p.Bt = (const __half *)Bt; p.gate = gate; p.gBt = bf(L.gBt); p.n_bt = (size_t)N * r;
            p.blocks_at = blocks1(p.n_at);
        }
        const unsigned blocks = p.blocks_t + p.blocks_at + blocks1(p.n_bt);
        if (blocks) launch(bw_weights_kernel, blocks, p);
    }
    float *z = (float *)(ws + L.z), *dh = (float *)(ws + L.dh), *G = grads->dBt ? grads->dBt : (float *)(ws + L.G);
    const TcOperand At_k = {bf(L.At_b), K, false}, At_mn = {bf(L.At_b), K, true};
    int sp = 1;
    if (r) {                                                                                                 // Z = x A
        gemm(x_k, At_k, K, none, none, 0, z, r, Mi, r, 1.0f, false, true, &sp);
        launch(bw_act_kernel, blocks1((size_t)M * r), read(sp > 1 ? partials : z, z, sp, (size_t)M * r), sp, (size_t)M * r, (flags & HGF_FLAG_NO_SILU) ? 1 : 0, z, bf(L.h_b));
    }
    // The products with dY and H: dH = dY (g (.) B^T), and G[n][j] = sum_m dY[m][n] H[m][j], behind dW's tiles where tc_deal_thin has room there,
    // else as launches of their own.
    const bool want_g = r && (grads->dBt || grads->dgate);
    const int sms = trace ? trace->sms : device_sm_count();
    auto blocks64 = [](int n) { return (n + kTBK - 1) / kTBK; };
    TcThinProduct with_dw[2] = {{dy_k, TcOperand{bf(L.gBt), r, true}, Mi, r, N, false, partials, r ? tc_split_blocks(Mi, r, blocks64(N), sms) : 1, 0},
                                {dy_mn, TcOperand{bf(L.h_b), r, true}, N, r, Mi, false, nullptr, r ? tc_split_blocks(N, r, blocks64(Mi), sms) : 1, 0}};
    // G's partial sums lie behind dH's; where there is no room for both (M just above N, both above K: 2261 x 1024 -> 2048) G has a launch of its own.
    const size_t h_floats = (size_t)with_dw[0].sums() * Mi * r, g_floats = (size_t)with_dw[1].sums() * N * r;
    const bool both = want_g && h_floats + g_floats <= (size_t)kBwSplitsMax * std::max({Mi, N, K}) * r;
    with_dw[1].P = partials + h_floats;
    if (grads->dW) {  // Algorithm 1, steps 1-2 again, then dW[n][k] = sum_m dY[m][n] Xd[m][k]
        if (K <= kBwQuantMaxK) {
            const unsigned rows8 = (unsigned)((Mi + 7) / 8);
            const __nv_bfloat16 *xp = (const __nv_bfloat16 *)x;
            launch(K <= kBwQuantMaxK / 2 ? bw_quant_kernel<8> : bw_quant_kernel<16>, rows8, xp, Mi, K, bf(L.xd));
        } else {
            PrologueParams pp = {};
            pp.x = (const __nv_bfloat16 *)x;
            pp.xq = (int8_t *)(ws + L.xq);
            pp.gamma_x = (float *)(ws + L.gamma_x);
            pp.M = Mi;
            pp.K = K;
            pp.flags = HGF_FLAG_NO_PDL;
            if (!trace && launch_quant(pp, GemmPrologueExtra{}, stream) != cudaSuccess) return HGF_ERR_CUDA;
            const size_t n8 = (size_t)M * K / 8;
            launch(bw_dequant_kernel, blocks1(n8), pp.xq, pp.gamma_x, K, n8, bf(L.xd));
        }
        gemm(dy_mn, TcOperand{bf(L.xd), K, true}, Mi, none, none, 0, grads->dW, K, N, K, 1.0f, false, false, nullptr, with_dw, r ? (both ? 2 : 1) : 0);
    }
    const bool fold = gamma > 1e-20f;  // the low-rank term of dX rides in the same contraction, pre-divided by gamma_W
    const TcOperand T_mn = {bf(L.T), K, true};  // T [N][K]: rows k of the product, contracted over n
    if (!r) {
        if (grads->dx) gemm(dy_k, T_mn, N, none, none, 0, grads->dx, K, Mi, K, gamma, false, false);
        return done();
    }
    const float *dh_sums = partials;
    sp = with_dw[0].rides;
    if (!sp) {
        gemm(dy_k, TcOperand{bf(L.gBt), r, true}, N, none, none, 0, dh, r, Mi, r, 1.0f, false, true, &sp);
        if (sp == 1) dh_sums = dh;
    }
    launch(bw_dz_kernel, blocks1((size_t)M * r), read(dh_sums, dh, sp, (size_t)M * r), sp, z, (size_t)M * r, fold ? 1.0f / gamma : 1.0f, bf(L.dz_b), bf(L.dzs_b));
    auto from_g = [&](const float *sums, int splits) {  // dBt and dgate
        launch(bw_gate_kernel, (unsigned)((N + 7) / 8), read(sums, G, splits, (size_t)N * r), splits, (const __half *)Bt, gate, N, r, G, grads->dgate);
    };
    if (with_dw[1].rides) from_g(with_dw[1].P, with_dw[1].rides);  // (ahead of dA, whose partial sums may take all of the room)
    // dA^T[j][k] = sum_m dZ[m][j] x[m][k]
    TcThinProduct with_dx = {x_mn, TcOperand{bf(L.dz_b), r, true}, K, r, Mi, true, partials, tc_split_blocks(r, K, blocks64(Mi), sms), 0};
    if (grads->dx) {                                                                                         // dX = gamma_W dY T + dZ A^T
        const TcOperand dzs_k = {bf(L.dzs_b), r, false};
        if (fold) {
            gemm(dy_k, T_mn, N, dzs_k, At_mn, r, grads->dx, K, Mi, K, gamma, false, false, nullptr, &with_dx, grads->dAt ? 1 : 0);
        } else {
            gemm(dy_k, T_mn, N, none, none, 0, grads->dx, K, Mi, K, gamma, false, false);
            gemm(dzs_k, At_mn, r, none, none, 0, grads->dx, K, Mi, K, 1.0f, true, false);
        }
    }
    if (grads->dAt) {
        if (!with_dx.rides) {
            gemm(TcOperand{bf(L.dz_b), r, true}, x_mn, Mi, none, none, 0, grads->dAt, K, r, K, 1.0f, false, true);
        } else {
            const size_t n4 = (size_t)r * K / 4;
            launch(tc_reduce_kernel, blocks1(n4), (const float4 *)read(partials, nullptr, with_dx.rides, 4 * n4), with_dx.rides, n4, 1.0f, 0, (float4 *)grads->dAt);
        }
    }
    if (want_g && !with_dw[1].rides) {
        gemm(dy_mn, TcOperand{bf(L.h_b), r, true}, Mi, none, none, 0, G, r, N, r, 1.0f, false, true, &sp);
        from_g(sp > 1 ? partials : G, sp);
    }
    return done();
}

extern "C" hgf_status hgf_linear_backward(const void *x, int64_t M, const void *packed, float gamma, int64_t d_in, int64_t d_out,
                                          const void *At, const void *Bt, int32_t r, const float *gate, const void *dy,
                                          const hgf_grads *grads, void *workspace, size_t workspace_bytes, uint32_t flags,
                                          void *stream) {
    return backward(x, M, packed, gamma, d_in, d_out, At, Bt, r, gate, dy, grads, workspace, workspace_bytes, flags, stream, nullptr);
}

// (for the tests, without a GPU: what the pass does with its room for partial sums, `floats` of it, on a device of that many SMs and pairs;
// want: bits 0 to 4 for dx, dW, dAt, dBt, dgate.  uses: [write, first, end] each, at most `most`, their number is returned, -1 if the call is
// refused; rides: [thin products taken, half tiles, c_idle, c_busy] of dW's launch by pairs and of dX's, zeros where there is none)
extern "C" int hgf_internal_backward_trace(int64_t M, int64_t d_in, int64_t d_out, int32_t r, float gamma, int32_t want, int32_t sms, int32_t pairs,
                                           int64_t *floats, int64_t *uses, int32_t most, int32_t *rides) {
    BwTrace trace = {};
    trace.sms = sms;
    trace.pairs = pairs;
    char *at = (char *)((uintptr_t)1 << 40);  // (addresses that nothing reads)
    const hgf_grads g = {(float *)(want & 1 ? at : nullptr), (float *)(want & 2 ? at : nullptr), (float *)(want & 4 ? at : nullptr),
                         (float *)(want & 8 ? at : nullptr), (float *)(want & 16 ? at : nullptr)};
    const size_t bytes = hgf_backward_workspace_bytes(M, d_in, d_out, r);
    if (backward(at, M, at, gamma, d_in, d_out, at, at, r, (const float *)at, at, &g, at, bytes, 0, nullptr, &trace) != HGF_OK) return -1;
    *floats = (int64_t)((bytes - bw_layout(M, d_in, d_out, r).partials) / 4);
    int n = 0;
    for (const BwTrace::Use &u : trace.uses) {
        if (n == most) break;
        uses[3 * n] = u.write; uses[3 * n + 1] = u.first; uses[3 * n + 2] = u.end;
        ++n;
    }
    for (int k = 0; k < 8; ++k) rides[k] = 0;
    for (const BwTrace::Rides &t : trace.rides) {
        int32_t *to = rides + (t.dx ? 4 : 0);
        to[0] = t.n; to[1] = t.n_half; to[2] = t.c_idle; to[3] = t.c_busy;
    }
    return n;
}
