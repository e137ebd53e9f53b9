// Causal differential attention forward (paper, Section 2.4, Definition "Differential Attention"):
//     O = ( Softmax(Q1 K1^T / sqrt(d_h)) - lambda * Softmax(Q2 K2^T / sqrt(d_h)) ) V
// on the outputs of the HGF attention projections (Definition "HGF Attention Projections": Q, K of
// width d, V of width d / 2), per batch element and head.
//
#include <cmath>

#include "hgf_tc.cuh"

namespace hgf {

struct AttnParams {
    const __nv_bfloat16 *q, *k, *v;  // q, k [B*L][2*h*dh]; v [B*L][h*dh]
    void *out;                       // [B*L][h*dh] fp32 or bf16
    int B, L, h;
    float lambda, out_scale, scale_log2;  // scale_log2 = log2(e) / sqrt(dh)
    uint32_t flags;
};

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// Persistent, one CTA of twelve warps per SM; a tile is 128 queries of a (batch element, head), both streams, worked in
// steps of 64 keys:
//   warp 0      TMA producer: a tile's two query tiles, then per step K of both streams (one ring) and V (another)
//   warps 1, 2  issue the tcgen05.mma.kind::f16 of a stream each: S_s = Q_s K_s^T (128 x 64, fp32, tensor memory), and
//               O_s += P_s V with P_s (bf16) read from tensor memory and V read from its stored form
//               (key rows of 128 bytes: the second operand with its row index contiguous)
//   warps 4-7   softmax of stream 1, warps 8-11 of stream 2: a thread owns one query row; it takes the step's 64 scores
//               into registers (tcgen05.ld), keeps a reference maximum and the sum, rescales its row of O_s in tensor
//               memory when the maximum moved far, and writes P_s = exp2(scale (s - reference)) as bf16 pairs
//               (tcgen05.st) over the scores
// The special-function pipe bounds it (2 x 128 x 64 exponentials a step at 16 a clock and SM: 1024 clocks) and, at the
// rate that is reached, the power limit (1.7 of 1.965 GHz).  So a softmax warp must not wait for a product: each stream
// has two score buffers, and its issuer puts the scores of step j + 2 behind P V of step j, in the buffer that P of
// step j just left - when a softmax warp ends step j the scores of j + 1 have been there for most of a step.  The steps of
// all tiles are one sequence, so the next tile's scores are formed under this tile's last exponentials.
// Measured at B = 4, L = 4096, 16 heads of 64 and at B = 2, L = 1500, 16 heads of 128: one score buffer of 128 (64) keys
// a stream, one issuing thread, a CTA per tile 502 and 79 us; two buffers, one issuing thread 645 and 80 (a thread in a
// divergent branch takes 80 to 125 clocks an MMA, and a step of 64 keys has as many as one of 128); issued by a whole warp
// with elect.sync 540 and 68; a warp per stream 455 and 62.5; persistent 448 and 61 to 63.  1360 clocks a step at
// head_dim 64, 1725 at 128.  Slower: every fourth or second pair of exponentials as a polynomial on the FMA pipe (issue
// slots are short too), four sets of softmax warps, the two streams' exponentials in turns or half a step apart.
// Tensor-memory columns: 4 score buffers of 64, O_1, O_2 (2 head_dim, twice for head_dim 64).  At the end O_1 / l_1 -
// lambda O_2 / l_2 is formed from the two accumulators by the thread pair that owns the row.  Every wait is bounded.
constexpr int kTaBM = 128, kTaThreads = 384, kTaKV = 64;
constexpr float kTaSlack = 8.0f;

template <int DH>
struct TaCfg {
    static constexpr int NBLK = DH / 64;
    static constexpr int KST = DH == 64 ? 5 : 3, VST = DH == 64 ? 5 : 3;  // ring stages
    static constexpr int NQ = DH == 64 ? 2 : 1, NO = DH == 64 ? 2 : 1;    // buffers of the query tiles and of O_1, O_2
    static constexpr int Q_BYTES = NBLK * kTaBM * 128;                    // one stream's query tile
    static constexpr int K_BYTES = NBLK * kTaKV * 128, V_BLOCK = kTaKV * 128, V_BYTES = NBLK * V_BLOCK;
    static constexpr int OFF_K = NQ * 2 * Q_BYTES, OFF_V = OFF_K + KST * 2 * K_BYTES, OFF_BAR = OFF_V + VST * V_BYTES;
    static constexpr int BAR_QFULL = 0, BAR_QEMPTY = 2, BAR_OEMPTY = 4, BAR_KFULL = 6, BAR_KEMPTY = BAR_KFULL + KST, BAR_VFULL = BAR_KEMPTY + KST, BAR_VEMPTY = BAR_VFULL + VST,
                         BAR_SFULL = BAR_VEMPTY + VST,    // [stream][buffer]
                         BAR_PFULL = BAR_SFULL + 4, BAR_L = BAR_PFULL + 4, BAR_END = BAR_L + 2,  // [parity of the tile], [stream]
                         BAR_COUNT = BAR_END + 2;
    static constexpr int OFF_L = OFF_BAR + 384;                           // [parity of the tile][2][128] floats
    static constexpr int SMEM_BYTES = OFF_L + 2 * 2 * kTaBM * 4 + 1024;
    static constexpr int COL_S = 0, COL_O = 4 * kTaKV;                    // scores: + (2 stream + buffer) 64; O: + (2 buffer + stream) DH
    static constexpr uint32_t IDESC_S = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTaKV >> 3) << 17) | ((uint32_t)(kTaBM >> 4) << 24);
    static constexpr uint32_t IDESC_PV = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(DH >> 3) << 17) | ((uint32_t)(kTaBM >> 4) << 24);
    static_assert(BAR_COUNT * 8 + 16 <= 384, "barrier block");
    static_assert(COL_O + NO * 2 * DH <= 512 && SMEM_BYTES <= 227 * 1024, "tensor and shared memory");
};

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
    return y;
}
// Four lanes (lane / 4 alike) with four 16-byte blocks each: afterwards block q of lane 4 i + t is what block t of lane
// 4 i + q was.
__device__ __forceinline__ void exchange_blocks(uint32_t (&v)[16], int lane) {
#pragma unroll
    for (int step = 1; step <= 2; step *= 2) {
        const bool upper = (lane & step) != 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            if (b & step) continue;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                uint32_t &lo = v[4 * b + e], &hi = v[4 * (b + step) + e];
                const uint32_t got = __shfl_xor_sync(0xffffffffu, upper ? lo : hi, step);
                if (upper) lo = got; else hi = got;
            }
        }
    }
}

template <int DH>
__global__ void __launch_bounds__(kTaThreads, 1)
ta_diff_attention_kernel(const __grid_constant__ CUtensorMap tmap_q, const __grid_constant__ CUtensorMap tmap_k,
                         const __grid_constant__ CUtensorMap tmap_v, const AttnParams p, unsigned int *status) {
    using C = TaCfg<DH>;
    constexpr int KV = kTaKV;
    extern __shared__ uint8_t ta_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)ta_smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem), bar0 = sbase + C::OFF_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_BAR + C::BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_BAR + C::BAR_COUNT * 8 + 4);
    float *s_l = reinterpret_cast<float *>(smem + C::OFF_L);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int L = p.L, h = p.h, nqt = (L + kTaBM - 1) / kTaBM, bhs = p.B * h, items = nqt * bhs, G = (int)gridDim.x;
    // The CTA's k-th tile: the tiles in order of falling length (late queries first) are dealt in rounds, every other
    // round backwards, so that the CTAs' sums stay close.
    struct Tile { int q0, tok0, hd, J; };
    auto tile_of = [&](int k, Tile &t) {
        const int i = k * G + ((k & 1) ? G - 1 - (int)blockIdx.x : (int)blockIdx.x);
        if (i >= items) return false;
        const int qt = nqt - 1 - i / bhs, bh = i % bhs, keys = (qt + 1) * kTaBM < L ? (qt + 1) * kTaBM : L;  // keys visible to the tile
        t.q0 = qt * kTaBM;
        t.tok0 = (bh / h) * L;
        t.hd = bh % h;
        t.J = (keys + KV - 1) / KV;
        return true;
    };

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bar(C::BAR_QFULL + i), 1);
            mbar_init(bar(C::BAR_QEMPTY + i), 2);
            mbar_init(bar(C::BAR_OEMPTY + i), 8);
            mbar_init(bar(C::BAR_L + i), 8);
            mbar_init(bar(C::BAR_END + i), 1);
        }
        for (int s = 0; s < C::KST; ++s) {
            mbar_init(bar(C::BAR_KFULL + s), 1);
            mbar_init(bar(C::BAR_KEMPTY + s), 2);  // a commit from each issuer
        }
        for (int s = 0; s < C::VST; ++s) {
            mbar_init(bar(C::BAR_VFULL + s), 1);
            mbar_init(bar(C::BAR_VEMPTY + s), 2);
        }
        for (int i = 0; i < 4; ++i) {
            mbar_init(bar(C::BAR_SFULL + i), 1);
            mbar_init(bar(C::BAR_PFULL + i), 4);
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)), "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);  // (warp-uniform)

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        uint32_t k_issued[C::KST] = {}, v_issued[C::VST] = {}, q_issued[C::NQ] = {};
        bool ok = true;
        int ks = 0, vs = 0, qb = 0;
        uint32_t kph = 1, vph = 1, qph = 1;
        Tile t;
        for (int k = 0; ok && tile_of(k, t); ++k) {
            ok = mbar_wait(bar(C::BAR_QEMPTY + qb), qph, abort_flag, status, 0xa04u + qb);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            if (lane == 0) {
                const uint32_t full = bar(C::BAR_QFULL + qb);
                mbar_arrive_expect_tx(full, 2 * C::Q_BYTES);
                for (int st = 0; st < 2; ++st)
                    for (int blk = 0; blk < C::NBLK; ++blk)
                        tma_load_2d(sbase + (2 * qb + st) * C::Q_BYTES + blk * kTaBM * 128, &tmap_q, (st * h + t.hd) * DH + 64 * blk, t.tok0 + t.q0, full);
            }
            ++q_issued[qb];
            if (++qb == C::NQ) { qb = 0; qph ^= 1u; }
            for (int j = 0; j < t.J; ++j) {
                ok = mbar_wait(bar(C::BAR_KEMPTY + ks), kph, abort_flag, status, 0xa00u + ks);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    const uint32_t dst = sbase + C::OFF_K + ks * 2 * C::K_BYTES, full = bar(C::BAR_KFULL + ks);
                    mbar_arrive_expect_tx(full, 2 * C::K_BYTES);
                    for (int blk = 0; blk < C::NBLK; ++blk) {
                        tma_load_2d(dst + blk * KV * 128, &tmap_k, t.hd * DH + 64 * blk, t.tok0 + j * KV, full);
                        tma_load_2d(dst + C::K_BYTES + blk * KV * 128, &tmap_k, (h + t.hd) * DH + 64 * blk, t.tok0 + j * KV, full);
                    }
                }
                ++k_issued[ks];
                if (++ks == C::KST) { ks = 0; kph ^= 1u; }
                ok = mbar_wait(bar(C::BAR_VEMPTY + vs), vph, abort_flag, status, 0xa08u + vs);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    const uint32_t full = bar(C::BAR_VFULL + vs);
                    mbar_arrive_expect_tx(full, C::V_BYTES);
                    for (int blk = 0; blk < C::NBLK; ++blk)
                        tma_load_2d(sbase + C::OFF_V + vs * C::V_BYTES + blk * C::V_BLOCK, &tmap_v, t.hd * DH + 64 * blk, t.tok0 + j * KV, full);
                }
                ++v_issued[vs];
                if (++vs == C::VST) { vs = 0; vph ^= 1u; }
            }
        }
        // never leave with a copy in flight
        for (int q = 0; q < C::KST; ++q)
            if (k_issued[q])
                for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_KFULL + q), (k_issued[q] - 1u) & 1u); ++i) {}
        for (int q = 0; q < C::VST; ++q)
            if (v_issued[q])
                for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_VFULL + q), (v_issued[q] - 1u) & 1u); ++i) {}
        for (int q = 0; q < C::NQ; ++q)
            if (q_issued[q])
                for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_QFULL + q), (q_issued[q] - 1u) & 1u); ++i) {}
    } else if (warp < 3) {
        // ------------------------------------------------------------------ MMA issuers, one warp per stream
        // The whole warp walks the loop, so that descriptors live in uniform registers; elect.sync picks the issuing
        // lane (one thread in a divergent branch took 80 to 125 clocks an MMA).  A warp per stream, because the
        // book-keeping of a step shares its scheduler with the exponentials.
        const int st = warp - 1;
        auto wait = [&](int i, uint32_t par, unsigned int code) {
            return __all_sync(0xffffffffu, mbar_wait_poll(bar(i), par, abort_flag, status, code)) != 0;
        };
        const uint64_t q_desc = make_sw128_desc(sbase + st * C::Q_BYTES), k_desc = make_sw128_desc(sbase + C::OFF_K + st * C::K_BYTES);
        const uint64_t v_desc = make_sw128_mn_desc(sbase + C::OFF_V, C::V_BLOCK);
        const uint32_t s_col = tmem_base + C::COL_S + 2 * st * KV;
        auto issue_s = [&](int buf, int s, int qb) {  // the stream's scores from K stage s
            const uint64_t qd = q_desc + (uint64_t)(qb * (2 * C::Q_BYTES >> 4)), kd = k_desc + (uint64_t)(s * (2 * C::K_BYTES >> 4));
#pragma unroll
            for (int blk = 0; blk < C::NBLK; ++blk)
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    warp_mma_f16(s_col + buf * KV, qd + (uint64_t)(blk * (kTaBM * 128 >> 4) + 2 * kk), kd + (uint64_t)(blk * (KV * 128 >> 4) + 2 * kk),
                                 C::IDESC_S, (blk | kk) ? 1u : 0u);
        };
        auto issue_pv = [&](int buf, int s, int ob, bool first) {  // O (+)= P V from V stage s
            const uint32_t o_col = tmem_base + C::COL_O + (2 * ob + st) * DH;
            const uint64_t vd = v_desc + (uint64_t)(s * (C::V_BYTES >> 4));
#pragma unroll
            for (int kk = 0; kk < KV / 16; ++kk)
                warp_mma_f16_ts(o_col, s_col + buf * KV + 8 * kk, vd + (uint64_t)(128 * kk), C::IDESC_PV, (!first || kk) ? 1u : 0u);
        };
        // The steps of all tiles are one sequence, g: the scores of step g + 2 follow P V of step g also across
        // the end of a tile, while its outputs are still being written.  (sj, sk, stile: the score side, two steps ahead.)
        bool ok = true, s_more, p_more;
        int ks = 0, vs = 0, sqb = 0, sk = 0, sj = 0, pk_ = 0, pob = 0, g = 0;
        uint32_t kph = 0, vph = 0, sqph = 0, poph = 1;
        Tile stile, ptile;
        s_more = tile_of(0, stile);
        p_more = tile_of(0, ptile);
        auto next_scores = [&](int buf) {  // false if a wait gave up
            if (sj == 0 && !wait(C::BAR_QFULL + sqb, sqph, 0xa10u + sqb)) return false;
            if (!wait(C::BAR_KFULL + ks, kph, 0xa30u + ks)) return false;
            tc_fence_after();
            issue_s(buf, ks, sqb);
            warp_commit(bar(C::BAR_SFULL + 2 * st + buf));  // also: P V of two steps before is complete
            warp_commit(bar(C::BAR_KEMPTY + ks));
            if (++ks == C::KST) { ks = 0; kph ^= 1u; }
            if (++sj == stile.J) {
                warp_commit(bar(C::BAR_QEMPTY + sqb));
                if (++sqb == C::NQ) { sqb = 0; sqph ^= 1u; }
                sj = 0;
                s_more = tile_of(++sk, stile);
            }
            return true;
        };
        for (int i = 0; ok && i < 2 && s_more; ++i) ok = next_scores(i);
        while (ok && p_more) {
            if (!(ok = wait(C::BAR_OEMPTY + pob, poph, 0xa18u + pob))) break;
            for (int j = 0; j < ptile.J; ++j, ++g) {
                const int buf = g & 1;
                if (!(ok = wait(C::BAR_VFULL + vs, vph, 0xa28u + vs))) break;
                if (!(ok = wait(C::BAR_PFULL + 2 * st + buf, (uint32_t)(g >> 1) & 1u, 0xa20u + st))) break;
                tc_fence_after();
                issue_pv(buf, vs, pob, j == 0);
                warp_commit(bar(C::BAR_VEMPTY + vs));
                if (C::NQ == 1 && j + 1 == ptile.J) warp_commit(bar(C::BAR_END + st));
                if (++vs == C::VST) { vs = 0; vph ^= 1u; }
                // the products execute in issue order: P of this step has been read when those scores replace it
                if (s_more) { if (!(ok = next_scores(buf))) break; }
                else warp_commit(bar(C::BAR_SFULL + 2 * st + buf));
            }
            if (++pob == C::NO) { pob = 0; poph ^= 1u; }
            p_more = tile_of(++pk_, ptile);
        }
    } else if (warp >= 4) {
        // ------------------------------------------------------------------ softmax of one stream, one row per thread
        const int st = warp >= 8 ? 1 : 0, quarter = warp & 3, row = 32 * quarter + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(32 * quarter) << 16);
        const float c = p.scale_log2;
        bool ok = true;
        int g = 0, ob = 0;
        Tile t;
        for (int k = 0; ok && tile_of(k, t); ++k) {
            const int qi = t.q0 + row, w0 = t.q0 + 32 * quarter;  // w0: the warp's first query
            const uint32_t o_addr = lane_base + C::COL_O + (2 * ob + st) * DH;
            float m = -1e30f;
            uint64_t l2a = 0, l2b = 0;  // the row's sum, four partial sums
            if constexpr (DH == 64) if (t.J > 1 && KV <= w0 + 31) {
                // The first reference point is the maximum of the first 128 keys: the scores of the second step are there
                // by now (they follow the last product of the tile before).  A row's largest probability is then mostly 1,
                // which bf16 holds exactly: relative error at L = 4096 1.82e-3, with the first 64 keys alone 1.85e-3.
                const int ahead = (g & 1) ^ 1;
                ok = mbar_wait_poll(bar(C::BAR_SFULL + 2 * st + ahead), (uint32_t)((g + 1) >> 1) & 1u, abort_flag, status, 0xa4cu + st);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
                uint32_t v0[32], v1[32];
                tmem_ld32(lane_base + C::COL_S + (2 * st + ahead) * KV, v0);
                tmem_ld32(lane_base + C::COL_S + (2 * st + ahead) * KV + 32, v1);
                tmem_ld_wait();
                if (2 * KV - 1 > w0) {  // some key of the step lies after some query of the warp
#pragma unroll
                    for (int u = 0; u < 32; ++u) {
                        if (KV + u > qi) v0[u] = 0xff800000u;
                        if (KV + 32 + u > qi) v1[u] = 0xff800000u;
                    }
                }
                float m0 = m, m1 = m, m2 = m, m3 = m;
#pragma unroll
                for (int u = 0; u < 32; u += 4) {
                    m0 = fmaxf(m0, fmaxf(__uint_as_float(v0[u]), __uint_as_float(v0[u + 1])));
                    m1 = fmaxf(m1, fmaxf(__uint_as_float(v0[u + 2]), __uint_as_float(v0[u + 3])));
                    m2 = fmaxf(m2, fmaxf(__uint_as_float(v1[u]), __uint_as_float(v1[u + 1])));
                    m3 = fmaxf(m3, fmaxf(__uint_as_float(v1[u + 2]), __uint_as_float(v1[u + 3])));
                }
                m = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
            }
            for (int j = 0; j < t.J; ++j, ++g) {
                const int buf = g & 1, k0 = j * KV;
                const uint32_t s_addr = lane_base + C::COL_S + (2 * st + buf) * KV;
                ok = mbar_wait_poll(bar(C::BAR_SFULL + 2 * st + buf), (uint32_t)(g >> 1) & 1u, abort_flag, status, 0xa40u + st);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
                uint32_t pk[32];
                if (k0 > w0 + 31) {  // every key of the step lies after every query of the warp
#pragma unroll
                    for (int u = 0; u < 32; ++u) pk[u] = 0u;
                } else {
                    uint32_t v0[32], v1[32];
                    tmem_ld32(s_addr, v0);
                    tmem_ld32(s_addr + 32, v1);
                    tmem_ld_wait();
                    if (k0 + KV - 1 > w0) {  // some key of the step lies after some query of the warp
#pragma unroll
                        for (int u = 0; u < 32; ++u) {
                            if (k0 + u > qi) v0[u] = 0xff800000u;       // -inf: probability 0
                            if (k0 + 32 + u > qi) v1[u] = 0xff800000u;
                        }
                    }
                    float m0 = -1e30f, m1 = -1e30f, m2 = -1e30f, m3 = -1e30f;
#pragma unroll
                    for (int u = 0; u < 32; u += 4) {
                        m0 = fmaxf(m0, fmaxf(__uint_as_float(v0[u]), __uint_as_float(v0[u + 1])));
                        m1 = fmaxf(m1, fmaxf(__uint_as_float(v0[u + 2]), __uint_as_float(v0[u + 3])));
                        m2 = fmaxf(m2, fmaxf(__uint_as_float(v1[u]), __uint_as_float(v1[u + 1])));
                        m3 = fmaxf(m3, fmaxf(__uint_as_float(v1[u + 2]), __uint_as_float(v1[u + 3])));
                    }
                    const float mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
                    // The reference point of the exponentials follows the maximum only when the maximum has moved by more
                    // than kTaSlack (in log2 units): probabilities then stay below 2^kTaSlack, and O and l are rescaled
                    // rarely instead of at nearly every tile.  (The final O / l does not depend on the reference point.)
                    float m_new = m;
                    if ((mx - m) * c > (j == 0 ? (DH == 64 ? 0.0f : -1.0f) : kTaSlack)) m_new = mx;
                    if (j > 0 && __any_sync(0xffffffffu, m_new != m)) {
                        // O_s is at rest once P V of the step before is complete: the barrier of the next step's scores follows it
                        ok = mbar_wait_poll(bar(C::BAR_SFULL + 2 * st + (buf ^ 1)), (uint32_t)((g + 1) >> 1) & 1u, abort_flag, status, 0xa48u + st);
                        if (!(ok = __all_sync(0xffffffffu, ok))) break;
                        tc_fence_after();
                        const float alpha = ex2_approx((m - m_new) * c);
                        const uint64_t a2 = pack_f32x2(alpha, alpha);
                        l2a = fma_f32x2(l2a, a2, 0ull);
                        l2b = fma_f32x2(l2b, a2, 0ull);
#pragma unroll
                        for (int cc = 0; cc < DH; cc += 16) {
                            uint32_t o[16];
                            tmem_ld16(o_addr + cc, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int u = 0; u < 16; ++u) o[u] = __float_as_uint(__uint_as_float(o[u]) * alpha);
                            tmem_st16(o_addr + cc, o);
                        }
                    }
                    m = m_new;
                    // probabilities as bf16 pairs
                    const uint64_t c2 = pack_f32x2(c, c), nmc2 = pack_f32x2(-m_new * c, -m_new * c);
                    auto pair = [&](uint32_t a, uint32_t b, uint64_t &sum) {
                        float x0, x1;
                        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(a), __uint_as_float(b)), c2, nmc2), x0, x1);
                        const float p0 = ex2_approx(x0), p1 = ex2_approx(x1);
                        sum = add_f32x2(sum, pack_f32x2(p0, p1));
                        return pack_bf16(p0, p1);
                    };
#pragma unroll
                    for (int u = 0; u < 32; u += 2) {
                        pk[u >> 1] = pair(v0[u], v0[u + 1], l2a);
                        pk[16 + (u >> 1)] = pair(v1[u], v1[u + 1], l2b);
                    }
                }
                tmem_st32(s_addr, pk);
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(C::BAR_PFULL + 2 * st + buf));
            }
            if (!ok) break;
            // ---- outputs of the tile: (O_1 / l_1 - lambda O_2 / l_2) out_scale; stream s's thread of a row writes half s
            // of the row's columns.  This stream's last P V is complete when the barrier of the scores two steps on says so (with one
            // query buffer those wait for the next tile's queries, so it has a barrier of its own); of the other stream's barriers
            // this warp does not know the phase: both streams' are complete when all eight warps have said so.
            if (C::NQ == 1) ok = mbar_wait_poll(bar(C::BAR_END + st), (uint32_t)k & 1u, abort_flag, status, 0xa50u + st);
            else ok = mbar_wait_poll(bar(C::BAR_SFULL + 2 * st + ((g - 1) & 1)), (uint32_t)((g + 1) >> 1) & 1u, abort_flag, status, 0xa50u + st);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            float la, lb, lc, ld;
            unpack_f32x2(l2a, la, lb);
            unpack_f32x2(l2b, lc, ld);
            float *sl = s_l + (k & 1) * 2 * kTaBM;
            sl[st * kTaBM + row] = (la + lb) + (lc + ld);
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_L + (k & 1)));
            ok = mbar_wait_poll(bar(C::BAR_L + (k & 1)), (uint32_t)(k >> 1) & 1u, abort_flag, status, 0xa52u);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;
            tc_fence_after();
            const float w1 = p.out_scale / sl[row], w2 = p.out_scale * p.lambda / sl[kTaBM + row];
            const uint32_t o_base = lane_base + C::COL_O + 2 * ob * DH;
#pragma unroll
            for (int cc = st * (DH / 2); cc < (st + 1) * (DH / 2); cc += 32) {
                uint32_t v1[32], v2[32];
                tmem_ld32(o_base + cc, v1);
                tmem_ld32(o_base + DH + cc, v2);
                tmem_ld_wait();
                if (cc + 32 == (st + 1) * (DH / 2)) {  // all of the accumulators is in registers
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(C::BAR_OEMPTY + ob));
                }
                if constexpr (DH == 128) {
                    // Four neighbouring rows exchange 16-byte blocks, so that four lanes store 64 consecutive bytes of one row:
                    // a lane storing along its own row touches 32 lines with every instruction.  (With the barrier above
                    // 59.7 -> 56.3 us at B = 2, L = 1500, 16 heads of 128, fp32; at head_dim 64, half the bytes a row, the exchange
                    // cost 1 to 5 %.)
                    const int quad = t.q0 + 32 * quarter + (lane & ~3);  // the first of the four rows
                    const size_t at = (size_t)(t.tok0 + quad) * ((size_t)h * DH) + (size_t)t.hd * DH + cc;
                    if (p.flags & HGF_FLAG_OUT_BF16) {
                        uint32_t o[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e)
                            o[e] = pack_bf16(__uint_as_float(v1[2 * e]) * w1 - __uint_as_float(v2[2 * e]) * w2,
                                             __uint_as_float(v1[2 * e + 1]) * w1 - __uint_as_float(v2[2 * e + 1]) * w2);
                        exchange_blocks(o, lane);
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            if (quad + e < L)
                                *reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(p.out) + at + (size_t)e * h * DH + 8 * (lane & 3)) =
                                    make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
                    } else {
#pragma unroll
                        for (int u = 0; u < 32; u += 16) {
                            uint32_t o[16];
#pragma unroll
                            for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(v1[u + e]) * w1 - __uint_as_float(v2[u + e]) * w2);
                            exchange_blocks(o, lane);
#pragma unroll
                            for (int e = 0; e < 4; ++e)
                                if (quad + e < L)
                                    *reinterpret_cast<uint4 *>(reinterpret_cast<float *>(p.out) + at + (size_t)e * h * DH + u + 4 * (lane & 3)) =
                                        make_uint4(o[4 * e], o[4 * e + 1], o[4 * e + 2], o[4 * e + 3]);
                        }
                    }
                } else {
                    const size_t obase = (size_t)(t.tok0 + qi) * ((size_t)h * DH) + (size_t)t.hd * DH;
                    if (qi < L) {
                        if (p.flags & HGF_FLAG_OUT_BF16) {
                            uint4 *dst = reinterpret_cast<uint4 *>(reinterpret_cast<__nv_bfloat16 *>(p.out) + obase + cc);
#pragma unroll
                            for (int u = 0; u < 32; u += 8) {
                                uint32_t o[4];
#pragma unroll
                                for (int e = 0; e < 4; ++e)
                                    o[e] = pack_bf16(__uint_as_float(v1[u + 2 * e]) * w1 - __uint_as_float(v2[u + 2 * e]) * w2,
                                                     __uint_as_float(v1[u + 2 * e + 1]) * w1 - __uint_as_float(v2[u + 2 * e + 1]) * w2);
                                dst[u >> 3] = make_uint4(o[0], o[1], o[2], o[3]);
                            }
                        } else {
                            float4 *dst = reinterpret_cast<float4 *>(reinterpret_cast<float *>(p.out) + obase + cc);
#pragma unroll
                            for (int u = 0; u < 32; u += 4)
                                dst[u >> 2] = make_float4(__uint_as_float(v1[u]) * w1 - __uint_as_float(v2[u]) * w2,
                                                          __uint_as_float(v1[u + 1]) * w1 - __uint_as_float(v2[u + 1]) * w2,
                                                          __uint_as_float(v1[u + 2]) * w1 - __uint_as_float(v2[u + 2]) * w2,
                                                          __uint_as_float(v1[u + 3]) * w1 - __uint_as_float(v2[u + 3]) * w2);
                        }
                    }
                }
            }
            if (++ob == C::NO) ob = 0;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

template <int DH>
static cudaError_t launch_attention_tc(const AttnParams &p, cudaStream_t stream) {
    using C = TaCfg<DH>;
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = ensure_dynamic_smem(ta_diff_attention_kernel<DH>, C::SMEM_BYTES, attr_done);
    if (e != cudaSuccess) return e;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    const uint64_t rows = (uint64_t)p.B * p.L, dq = (uint64_t)2 * p.h * DH, dv = (uint64_t)p.h * DH;
    CUtensorMap mq, mk, mv;
    if (!make_map_2d(&mq, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.q, dq, rows, dq * 2, 64, kTaBM, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&mk, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.k, dq, rows, dq * 2, 64, kTaKV, CU_TENSOR_MAP_SWIZZLE_128B) ||
        !make_map_2d(&mv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, p.v, dv, rows, dv * 2, 64, kTaKV, CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    const int sms = device_sm_count();
    if (!sms) return cudaErrorInvalidDevice;
    const unsigned items = (unsigned)(((p.L + kTaBM - 1) / kTaBM) * p.B * p.h), grid = items < (unsigned)sms ? items : (unsigned)sms;
    ta_diff_attention_kernel<DH><<<grid, kTaThreads, C::SMEM_BYTES, stream>>>(mq, mk, mv, p, status);
    count_launch();
    return cudaGetLastError();
}

}  // namespace hgf

using namespace hgf;

extern "C" hgf_status hgf_diff_attention_forward(const void *q, const void *k, const void *v, int64_t B, int64_t L,
                                                 int32_t n_heads, int32_t head_dim, float lambda, float out_scale, void *out,
                                                 uint32_t flags, void *stream) {
    if (!q || !k || !v || !out || B <= 0 || L <= 0 || n_heads <= 0) return HGF_ERR_INVALID_ARG;
    if (flags & ~HGF_FLAG_OUT_BF16) return HGF_ERR_INVALID_ARG;
    if ((head_dim != 64 && head_dim != 128) || B > 65535 || n_heads > 65535 || L > (1 << 24)) return HGF_ERR_UNSUPPORTED_SHAPE;
    // token rows and CTAs are counted in 32 bits
    if (B * L > 0x7fffffffll || (uint64_t)B * (uint64_t)n_heads * (uint64_t)((L + kTaBM - 1) / kTaBM) > 0x7fffffffull) return HGF_ERR_UNSUPPORTED_SHAPE;
    if ((((uintptr_t)q) | ((uintptr_t)k) | ((uintptr_t)v) | ((uintptr_t)out)) & 15u) return HGF_ERR_MISALIGNED;
    AttnParams p = {};
    p.q = (const __nv_bfloat16 *)q;
    p.k = (const __nv_bfloat16 *)k;
    p.v = (const __nv_bfloat16 *)v;
    p.out = out;
    p.B = (int)B;
    p.L = (int)L;
    p.h = n_heads;
    p.lambda = lambda;
    p.out_scale = out_scale;
    p.scale_log2 = (float)(1.4426950408889634 / sqrt((double)head_dim));
    p.flags = flags;
    const cudaError_t e = head_dim == 64 ? launch_attention_tc<64>(p, (cudaStream_t)stream) : launch_attention_tc<128>(p, (cudaStream_t)stream);
    return e == cudaSuccess ? HGF_OK : HGF_ERR_CUDA;
}

extern "C" double hgf_diff_lambda0(double head_dim) { return 0.8 - 0.6 * exp(-0.3 * head_dim); }
