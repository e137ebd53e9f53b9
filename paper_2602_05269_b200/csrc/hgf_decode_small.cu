// Decode path for launches whose packed weights fit the shared memory of the chip: one launch per layer call (or per
// small group), where the prologue / GEMV pair of hgf_prologue.cu and hgf_decode.cu takes two.  Algorithm 1 whole:
// quantisation, H = SiLU(x A), the ternary contraction, dequantisation, up-projection, gate.
//
// Such a call moves 0.1 to 20 MB, a few microseconds of HBM time; what it waits for is the chain of launches and
// dependent memory round trips.  So everything that does not depend on the preceding launch (the CTA's weight
// tiles, its part of A^T, its rows of B^T) is requested into shared memory at once, before the kernel waits for that
// launch (programmatic dependent launch), and after the wait there is one trip to memory (x) and three barriers to
// the result (2048 -> 2048, r = 32, M = 1: 3.7 us of 5.2 a call in a chain; the rest is the hand-over between launches):
//  - a CTA owns whole row tiles of one problem and quantises all of x for itself (from L2) instead of reading codes
//    that another launch wrote;
//  - x A needs all of A^T, too much for every CTA: the CTAs of a cluster take one slice of K each and
//    exchange their partial sums through distributed shared memory, in rank order.  The cluster barrier runs under
//    the integer products.
//  - the sixteen warps split K (column tiles of 256) and, where K is short, the row tiles; their integer sums meet in
//    shared memory (exact, so in any order).
// Two CTAs fit an SM when a share is small, so the next call's CTAs can be fetching their weights while this one
// works.
#include "hgf_warp.cuh"

namespace hgf {

constexpr int kSmThreads = 512, kSmWarps = kSmThreads / 32;
constexpr int kSmSmemLimit = 113 * 1024;  // two CTAs on an SM (228 KB, 1 KB of each CTA's reserved)
constexpr int kSmSmemMax = 200 * 1024;
constexpr int kSmHPitch = 72;  // halves per row of H in shared memory (r <= 64, + 8 bank spread)

struct SmHead {                // per-token values at the start of shared memory
    unsigned long long bar_a, bar_w, bar_x, bar_h;
    uint32_t amax[16];         // pattern of the largest |x| (or |xn|), an unsigned maximum
    int row_sum[16];
    float mean[16], rstd[16];
};

template <int NT, int NP>
__global__ void __launch_bounds__(kSmThreads, NT == 1 ? 2 : 1)
decode_small_kernel(const __grid_constant__ SmallLaunch<NP> L, unsigned int *status) {
    extern __shared__ __align__(128) uint8_t smem[];
    pdl_launch_dependents();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const int C = 1 << L.cluster_log2, cid = (int)blockIdx.x >> L.cluster_log2, rank = (int)blockIdx.x & (C - 1);
    int pi = 0;
    if constexpr (NP > 1)
        while (pi + 1 < L.n && cid >= L.p[pi + 1].cluster_begin) ++pi;
    const SmallProblem &P = L.p[pi];
    const int K = P.K, M = P.M, N = P.N, r = P.r, steps = (K + 255) >> 8, Kp = steps << 8, pitch = Kp + 64, xpitch = 2 * K + 64;
    const int ci = (cid - P.cluster_begin) * C + rank;
    const uint32_t tiles = (uint32_t)(N + 15) >> 4;  // (plan_small: tiles * ctas fits 32 bits)
    const int tile0 = (int)(tiles * (uint32_t)ci / (uint32_t)P.ctas), nt = (int)(tiles * (uint32_t)(ci + 1) / (uint32_t)P.ctas) - tile0;
    const int jts = r >> 4, E = jts * NT * 128;  // values of the CTA's partial sums of x A, in the tf32 MMA's accumulator layout

    SmHead *head = reinterpret_cast<SmHead *>(smem);
    const uint32_t s0 = dsmem_u32(smem), bar_a = s0 + 0, bar_w = s0 + 8, bar_x = s0 + 16, bar_h = s0 + 24;
    __half *h_hi = reinterpret_cast<__half *>(smem + L.off_h), *h_lo = h_hi + NT * 8 * kSmHPitch;
    float *slots = reinterpret_cast<float *>(smem + L.off_slots);   // [cluster rank][E]
    float *part = reinterpret_cast<float *>(smem + L.off_part);     // [warp / J][E]
    int *red = reinterpret_cast<int *>(smem + L.off_red);           // [row tile][NT * 4][32]
    int8_t *xq_s = reinterpret_cast<int8_t *>(smem + L.off_xq);
    const uint8_t *at_s = smem + L.off_at, *bt_s = smem + L.off_bt, *w_s = smem + L.off_w, *x_s = smem + L.off_x;

    // this CTA's slice of K in 32-column chunks, for x A
    const int chunks = K >> 5, per = (chunks + C - 1) >> L.cluster_log2, ch0 = rank * per < chunks ? rank * per : chunks;
    const int nch = chunks - ch0 < per ? chunks - ch0 : per;
    const int at_pitch = per * 64 + ((per & 1) ? 0 : 64);  // rows g and g + 1 on different halves of the banks

    if (warp == 0) {
        if (lane == 0) {
            dmbar_init(bar_a, 1);
            dmbar_init(bar_w, 1);
            dmbar_init(bar_x, 1);
            dmbar_init(bar_h, 1);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            const int n_rows = N - 16 * tile0 < 16 * nt ? N - 16 * tile0 : 16 * nt;
            const uint32_t bt_bytes = nt > 0 ? (uint32_t)(n_rows * r * 2) : 0u;
            announce(bar_a, (uint32_t)(r * nch * 64));
            announce(bar_w, (uint32_t)(nt * steps) * 1024u + bt_bytes);
            announce(bar_h, (uint32_t)(C * E * 4));
            if (bt_bytes) bulk_load_announced(s0 + L.off_bt, P.Bt + (size_t)16 * tile0 * r, bt_bytes, bar_w);
        }
        __syncwarp();
        if (nch > 0)
            for (int j = lane; j < r; j += 32)
                bulk_load_announced(s0 + L.off_at + j * at_pitch, P.At + (size_t)j * K + 32 * ch0, (uint32_t)(nch * 64), bar_a);
        for (int i = lane; i < nt; i += 32)
            bulk_load_announced(s0 + L.off_w + i * steps * 1024, P.packed + (size_t)(tile0 + i) * steps * 1024, (uint32_t)steps * 1024u, bar_w);
        __syncwarp();
        if (r > 0) cluster_arrive_relaxed();  // (the other warps below)
        pdl_wait();                           // x, the gates, the workspace and y belong to earlier work
        if (lane == 0) announce(bar_x, (uint32_t)(2 * M * K));
        __syncwarp();
        if (lane < M) bulk_load_announced(s0 + L.off_x + lane * xpitch, P.x + (size_t)lane * K, (uint32_t)(2 * K), bar_x);
        __syncwarp();
    }
    if (r > 0 && warp > 0) cluster_arrive_relaxed();  // (waited for before the first store into a peer's memory)
    if (tid < 16) { head->amax[tid] = 0u; head->row_sum[tid] = 0; }
    for (int i = tid; i < nt * NT * 128; i += kSmThreads) red[i] = 0;
    if (M < NT * 8)  // the row of zeros that stands in for absent tokens
        for (int i = tid; i < (Kp >> 4); i += kSmThreads) *reinterpret_cast<uint4 *>(xq_s + (size_t)M * pitch + 16 * i) = make_uint4(0u, 0u, 0u, 0u);
    const bool ln = P.ln_w != nullptr;
    if (ln && warp > 0)
        for (int i = tid - 32; i < (K >> 5); i += kSmThreads - 32) {
            prefetch_l2(P.ln_w + 32 * i);
            prefetch_l2(P.ln_b + 32 * i);
        }
    // the gates of the row tile whose epilogue this warp runs (its first one; a share rarely has more than 16)
    float gate_a = 0.0f, gate_b = 0.0f;
    auto load_gates = [&](int rt) {
        const int n0 = 16 * (tile0 + rt);
        if (P.gate_group > 1) {  // whole row tiles share a gate
            gate_a = gate_b = __ldg(P.gate + n0 / P.gate_group);
        } else {
            gate_a = __ldg(P.gate + (n0 + g < N ? n0 + g : N - 1));
            gate_b = __ldg(P.gate + (n0 + g + 8 < N ? n0 + g + 8 : N - 1));
        }
    };
    __syncthreads();
    pdl_wait();  // (every thread: what it stores to global memory may belong to earlier work)
    if (r > 0 && warp < nt) load_gates(warp);
    int32_t *group_dbg_y_int = nullptr;
    if constexpr (NP > 1) group_dbg_y_int = *P.dbg_y_int_at;
    bool ok = warp_wait(bar_x, status, 0x600u);

    // ---- x, in segments of 256 columns of one token (32 units of 16 bytes), dealt to the warps in turn -----------
    // At most one a warp (one token up to K = 4096, two up to 2048, ...): the first eight warps quantise while the others
    // compute x A; else every warp does both.
    const int segs = steps;
    const bool apart = r > 0 && M * segs <= kSmWarps;
    const int q_warps = apart ? kSmWarps / 2 : kSmWarps, a_warps = apart ? kSmWarps / 2 : kSmWarps, a_warp = warp - (kSmWarps - a_warps);
    const bool quantises = warp < q_warps, multiplies = r > 0 && a_warp >= 0;
    auto each_segment = [&](auto &&body) {
        int m = 0, seg = warp;
#pragma unroll 1
        for (;;) {
            while (seg >= segs) { seg -= segs; ++m; }
            if (m >= M) break;
            const int i = 32 * seg + lane;
            const bool in = 8 * i < K;
            body(m, seg, i, in, in ? *reinterpret_cast<const uint4 *>(x_s + m * xpitch + 16 * i) : make_uint4(0u, 0u, 0u, 0u));
            seg += q_warps;
        }
    };
    if (ln && quantises) {
        // Mean and variance in one pass, in double, of d = x - x[0] (exact): sum d and sum d^2.  x[0] is one of
        // the values, so (mean - x[0])^2 <= K var and the subtraction below loses at most a factor K of 2^-53.
        double2 *seg_sum = reinterpret_cast<double2 *>(smem + L.off_ln);
        each_segment([&](int m, int seg, int i, bool in, const uint4 &u) {
            double s = 0.0, ss = 0.0;
            if (in) {
                const double x0 = (double)__bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(x_s + m * xpitch));
                float f[8];
                unpack8(u, f);
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const double d = (double)f[k] - x0;
                    s += d;
                    ss = fma(d, d, ss);
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
            }
            if (lane == 0) seg_sum[m * segs + seg] = make_double2(s, ss);
        });
        bar_sync(1, 32 * q_warps);
        if (tid < M) {
            double s = 0.0, ss = 0.0;
            for (int k = 0; k < segs; ++k) {
                const double2 a = seg_sum[tid * segs + k];
                s += a.x;
                ss += a.y;
            }
            const double dm = s / (double)K, v0 = ss / (double)K - dm * dm, var = v0 < 0.0 ? 0.0 : v0;  // (NaN stays NaN)
            const double x0 = (double)__bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(x_s + tid * xpitch));
            const float mean = (float)(x0 + dm), rstd = (float)rsqrt(var + (double)P.eps);
            head->mean[tid] = mean;
            head->rstd[tid] = rstd;
            if (ci == 0) {
                if (P.mean_out) P.mean_out[tid] = mean;
                if (P.rstd_out) P.rstd_out[tid] = rstd;
            }
        }
        bar_sync(1, 32 * q_warps);
    }
    auto ln_unit = [&](int m, int i, const uint4 &u, float (&xn)[8]) {
        const float mean = head->mean[m], rstd = head->rstd[m];
        const float4 *w4 = reinterpret_cast<const float4 *>(P.ln_w + 8 * i), *b4 = reinterpret_cast<const float4 *>(P.ln_b + 8 * i);
        const float4 w0 = w4[0], w1 = w4[1], b0 = b4[0], b1 = b4[1];
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float f[8];
        unpack8(u, f);
#pragma unroll
        for (int k = 0; k < 8; ++k) xn[k] = ln_value(f[k], mean, rstd, w[k], b[k]);
    };

    // largest magnitude of each token (non-negative floats order like their patterns)
    if (quantises) each_segment([&](int m, int, int i, bool in, const uint4 &u) {
        uint32_t bits;
        if (ln) {
            float a = 0.0f;
            if (in) {
                float xn[8];
                ln_unit(m, i, u, xn);
#pragma unroll
                for (int k = 0; k < 8; ++k) a = fmaxf(a, fabsf(xn[k]));
            }
            bits = __float_as_uint(a);
        } else {
            bits = __float_as_uint(absmax_bits_to_float(absmax8_bits(0u, u)));
            if (bits > 0x7f800000u) bits = 0u;  // a NaN does not count, as in fmaxf
        }
        bits = __reduce_max_sync(0xffffffffu, bits);
        if (lane == 0) atomicMax(&head->amax[m], bits);
    });

    // ---- x A over the CTA's slice of K: rows of A^T are the 16-row operand, tokens the 8-column operand.  Warp w
    // takes 16 columns of H (jt = w mod J) and every (warps / J)-th chunk of the slice; then their sums, in warp order, to
    // every CTA of the cluster. ---------------------------------------------------------------------------------
    const int J = jts <= 1 ? 1 : (jts == 2 ? 2 : 4), parts = a_warps / J;
    if (multiplies) {
        ok = warp_wait(bar_a, status, 0x600u) && ok;
        const int jt = a_warp & (J - 1), cw = a_warp / J;
        if (jt < jts) {
            float acc[NT][4];
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int c = 0; c < 4; ++c) acc[n][c] = 0.0f;
            const uint8_t *arow = at_s + (16 * jt + g) * at_pitch + 16 * t;
            const uint8_t *xrow[NT];
#pragma unroll
            for (int n = 0; n < NT; ++n) xrow[n] = x_s + (g + 8 * n < M ? g + 8 * n : 0) * xpitch + 64 * ch0 + 16 * t;
#pragma unroll 2
            for (int c = cw; c < nch; c += parts) {
                const uint4 av = *reinterpret_cast<const uint4 *>(arow + 64 * c), bv = *reinterpret_cast<const uint4 *>(arow + 8 * at_pitch + 64 * c);
                const uint32_t aw[4] = {av.x, av.y, av.z, av.w}, bw[4] = {bv.x, bv.y, bv.z, bv.w};
                uint4 xv[NT];
#pragma unroll
                for (int n = 0; n < NT; ++n) xv[n] = g + 8 * n < M ? *reinterpret_cast<const uint4 *>(xrow[n] + 64 * c) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    // elements 2 k and 2 k + 1 of this lane's eight take the k slots t and t + 4 of the MMA
                    const float2 fa = __half22float2(*reinterpret_cast<const __half2 *>(&aw[k]));
                    const float2 fb = __half22float2(*reinterpret_cast<const __half2 *>(&bw[k]));
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const uint32_t xw = (&xv[n].x)[k];
                        mma_tf32(acc[n], __float_as_uint(fa.x), __float_as_uint(fb.x), __float_as_uint(fa.y), __float_as_uint(fb.y), xw << 16,
                                 xw & 0xffff0000u);
                    }
                }
            }
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int c = 0; c < 4; ++c) part[cw * E + (jt * NT * 4 + n * 4 + c) * 32 + lane] = acc[n][c];
        }
        bar_sync(2, 32 * a_warps);  // partial sums are there (and the maxima, where every warp does both)
        cluster_wait_acquire();     // every CTA of the cluster has started
#pragma unroll 1
        for (int e = 32 * a_warp + lane; e < E; e += 32 * a_warps) {
            float z = 0.0f;
#pragma unroll 4
            for (int w = 0; w < parts; ++w) z += part[w * E + e];
            const uint32_t dst = s0 + L.off_slots + (uint32_t)(rank * E + e) * 4u;
            for (int q = 0; q < C; ++q) st_async_f32(dst, bar_h, (uint32_t)q, z);
        }
        __syncwarp();
    }

    // codes, in the order the integer MMA reads them (hgf_decode.cu, staging of x~), and the tokens' sums; columns
    // past the matrix are zeros
    if (quantises && (apart || r == 0)) bar_sync(1, 32 * q_warps);  // the maxima are there
    if (quantises) each_segment([&](int m, int seg, int i, bool in, const uint4 &u) {
        int sum = 0;
        uint2 o = make_uint2(0u, 0u);
        const float gm = fmaxf(__uint_as_float(head->amax[m]), 1e-5f);
        if (in) {
            if (ln) {
                float xn[8];
                ln_unit(m, i, u, xn);
                const float scale = __fdiv_rn(127.0f, gm);
                o = ln_codes8(xn, scale, sum);
            } else {
                o = quant8(u, make_quant_scale(gm), sum);
            }
            if (ci == 0) {  // what the two-launch path leaves behind: hgf_group_debug's views, a contraction run on its own
                if (P.xq) *reinterpret_cast<uint2 *>(P.xq + (size_t)m * K + 8 * i) = o;
                if (P.dbg_xq) *reinterpret_cast<uint2 *>(P.dbg_xq + (size_t)m * K + 8 * i) = o;
            }
        }
        const int q = lane >> 2, j = lane & 3;
        uint32_t *dst = reinterpret_cast<uint32_t *>(xq_s + (size_t)m * pitch + 256 * seg + 16 * (q >> 1) + 128 * (q & 1) + 64 * (j & 1) + 4 * (j >> 1));
        dst[0] = o.x;
        dst[2] = o.y;
        sum = __reduce_add_sync(0xffffffffu, sum);
        if (lane == 0) atomicAdd(&head->row_sum[m], sum);
    });
    // the codes are there; the quantising warps go on without the others
    if (!apart) __syncthreads();
    else if (quantises) { bar_arrive(3, kSmThreads); bar_sync(1, 32 * q_warps); }
    else bar_sync(3, kSmThreads);

    // ---- the ternary contraction: warp (kw, rw) takes column tiles kw, kw + KS, ... of row tiles rw, rw + RS, ... --
    ok = warp_wait(bar_w, status, 0x600u) && ok;
    {
        const int ks_log2 = steps >= 16 ? 4 : 31 - __clz(steps), KS = 1 << ks_log2, RS = kSmWarps >> ks_log2;
        const int kw = warp & (KS - 1), rw = warp >> ks_log2;
        const int8_t *xrow[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) xrow[n] = xq_s + (size_t)(g + 8 * n < M ? g + 8 * n : M) * pitch + 16 * t;
#pragma unroll 1
        for (int rt = rw; rt < nt; rt += RS) {
            int acc[NT][4][4];
#pragma unroll
            for (int a = 0; a < NT; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[a][b][c] = 0;
#pragma unroll 1
            for (int s = kw; s < steps; s += KS) {
                const uint8_t *wt = w_s + ((size_t)rt * steps + s) * 1024 + 16 * lane;
                const uint4 pq = *reinterpret_cast<const uint4 *>(wt), qq = *reinterpret_cast<const uint4 *>(wt + 512);
                const uint32_t pw[4] = {pq.x, pq.y, pq.z, pq.w}, qw[4] = {qq.x, qq.y, qq.z, qq.w};
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    uint4 xa[NT], xb[NT];
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        xa[n] = *reinterpret_cast<const uint4 *>(xrow[n] + 256 * s + 128 * h);
                        xb[n] = *reinterpret_cast<const uint4 *>(xrow[n] + 256 * s + 128 * h + 64);
                    }
#pragma unroll
                    for (int jj = 0; jj < 4; ++jj) {
                        const uint32_t mask = 0x03030303u << (2 * jj);
                        const uint32_t a0 = pw[2 * h] & mask, a1 = qw[2 * h] & mask, a2 = pw[2 * h + 1] & mask, a3 = qw[2 * h + 1] & mask;
#pragma unroll
                        for (int n = 0; n < NT; ++n) {
                            const uint4 &xv = jj < 2 ? xa[n] : xb[n];
                            if (jj & 1) mma_u8s8(acc[n][jj], a0, a1, a2, a3, xv.z, xv.w);
                            else mma_u8s8(acc[n][jj], a0, a1, a2, a3, xv.x, xv.y);
                        }
                    }
                }
            }
            // the four scales' exact quotients; integer sums are exact in any order
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int c = 0; c < 4; ++c)
                    atomicAdd(&red[(rt * NT * 4 + n * 4 + c) * 32 + lane], acc[n][0][c] + (acc[n][1][c] >> 2) + (acc[n][2][c] >> 4) + (acc[n][3][c] >> 6));
        }
    }
    if (ci == 0 && tid < M) {
        const float gm = fmaxf(__uint_as_float(head->amax[tid]), 1e-5f);
        if (P.gamma_x) { P.gamma_x[tid] = gm; P.row_sum[tid] = head->row_sum[tid]; }
        if (P.dbg_gamma_x) P.dbg_gamma_x[tid] = gm;
    }

    // ---- H: the cluster's partial sums in rank order, SiLU, fp16 value and fp16 residual; by the warps that computed x A,
    // which have a smaller part in the products above (none where the CTA has one row tile) ----------------------------------
    if (multiplies) {
        ok = warp_wait(bar_h, status, 0x600u) && ok;
        const bool no_silu = (P.flags & HGF_FLAG_NO_SILU) != 0;
#pragma unroll 1
        for (int e = 32 * a_warp + lane; e < E; e += 32 * a_warps) {
            float z = 0.0f;
            for (int q = 0; q < C; ++q) z += slots[q * E + e];
            // accumulator register c of lane (g, t): row g + 8 (c >> 1), token 8 n + 2 t + (c & 1)
            const int ln_ = e & 31, idx = e >> 5, c = idx & 3, n = (idx >> 2) % NT, jt = idx / (4 * NT);
            const int j = 16 * jt + (ln_ >> 2) + 8 * (c >> 1), m = 8 * n + 2 * (ln_ & 3) + (c & 1);
            const float h = no_silu ? z : silu_f(z);
            const __half hi = __float2half_rn(h), lo = __float2half_rn(h - __half2float(hi));
            h_hi[m * kSmHPitch + j] = hi;
            h_lo[m * kSmHPitch + j] = lo;
            if (ci == 0) {
                if (P.hpart) {  // the sum in the first slice's place, zeros in the others'
                    float *dst = P.hpart + (size_t)jt * P.nslices * 256 + (4 * n + c) * 32 + ln_;
                    dst[0] = z;
                    for (int q = 1; q < P.nslices; ++q) dst[(size_t)q * 256] = 0.0f;
                } else if (P.h && m < M) {
                    P.h[(size_t)m * r + j] = h;
                    P.h_hi[(size_t)m * r + j] = hi;
                    P.h_lo[(size_t)m * r + j] = lo;
                }
                if (P.dbg_h && m < M) P.dbg_h[(size_t)m * r + j] = h;
            }
        }
    }
    __syncthreads();
    // A copy never landed (reported; what the call wrote is undefined): bounded drain, then leave.  Only warps that waited for it
    // know; telling the others through shared memory cost every call 0.1 us.
    if (!ok) {
        for (uint32_t i = 0; i < (1u << 16) && !(dmbar_try_wait(bar_a, 0) && dmbar_try_wait(bar_w, 0) && dmbar_try_wait(bar_x, 0) && dmbar_try_wait(bar_h, 0)); ++i) {}
        return;
    }

    // ---- epilogue: one warp per row tile ------------------------------------------------------------------
    const bool out_bf16 = (P.flags & HGF_FLAG_OUT_BF16) != 0;
#pragma unroll 1
    for (int rt = warp; rt < nt; rt += kSmWarps) {
        const int n0 = 16 * (tile0 + rt);
        float corr[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int c = 0; c < 4; ++c) corr[n][c] = 0.0f;
        if (r > 0) {
            if (rt != warp) load_gates(rt);
            const int rows = N - n0 < 16 ? N - n0 : 16;
            const uint32_t *b0 = reinterpret_cast<const uint32_t *>(bt_s) + (size_t)rt * 16 * (r >> 1);
            const uint32_t *bA = b0 + (g < rows ? g : rows - 1) * (r >> 1) + t, *bB = b0 + (g + 8 < rows ? g + 8 : rows - 1) * (r >> 1) + t;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                if (16 * kk < r) {
                    const uint32_t a0 = bA[8 * kk], a1 = bB[8 * kk], a2 = bA[8 * kk + 4], a3 = bB[8 * kk + 4];
#pragma unroll
                    for (int n = 0; n < NT; ++n) {
                        const uint32_t *hh = reinterpret_cast<const uint32_t *>(h_hi + (g + 8 * n) * kSmHPitch);
                        const uint32_t *hl = reinterpret_cast<const uint32_t *>(h_lo + (g + 8 * n) * kSmHPitch);
                        mma_f16(corr[n], a0, a1, a2, a3, hh[8 * kk + t], hh[8 * kk + 4 + t]);
                        mma_f16(corr[n], a0, a1, a2, a3, hl[8 * kk + t], hl[8 * kk + 4 + t]);
                    }
                }
            }
        }
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const int m = 8 * n + 2 * t + (c & 1), row = n0 + g + 8 * (c >> 1);
                if (m < M && row < N) {
                    const int y_int = red[(rt * NT * 4 + n * 4 + c) * 32 + lane] - head->row_sum[m];
                    const float scale = fmaxf(__uint_as_float(head->amax[m]), 1e-5f) * P.gw_over_127;
                    const float y = fmaf(c >> 1 ? gate_b : gate_a, corr[n][c], (float)y_int * scale);
                    const size_t o = (size_t)m * N + row;
                    if (out_bf16) reinterpret_cast<__nv_bfloat16 *>(P.y)[o] = __float2bfloat16_rn(y);
                    else reinterpret_cast<float *>(P.y)[o] = y;
                    if (int32_t *dbg = NP > 1 ? group_dbg_y_int : P.dbg_y_int) dbg[o] = y_int;
                }
            }
    }
}

// ---- host side ----------------------------------------------------------------------------------------------
// Clusters that run at the same time with one CTA an SM.  They do not fill the chip: a cluster stays within a part of it whose
// SM count is no multiple of its size.
static int clusters_at_once(int cluster_log2) {
    static std::atomic<int> cache[kMaxDevices][4];
    const int dev = current_device();
    if (dev < 0 || dev >= kMaxDevices) return 0;
    int n = cache[dev][cluster_log2].load(std::memory_order_acquire);
    if (n) return n;
    static std::atomic<unsigned long long> attr_done{0};
    auto kernel = decode_small_kernel<1, kSmallMax>;
    if (ensure_dynamic_smem(kernel, kSmSmemMax, attr_done) != cudaSuccess) return 0;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << cluster_log2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(1u << cluster_log2);
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = kSmSmemMax;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess || n <= 0) return 0;
    cache[dev][cluster_log2].store(n, std::memory_order_release);
    return n;
}

// Cuts the launch into clusters and lays out shared memory.  False where the two-launch path is the better one
// (microseconds a call in a captured chain of layers with weights of their own, this path / two launches):
//  - M K above 8192 (4096 behind a LayerNorm): every CTA quantises all of x, which the two-launch path does once.
//    2048 -> 2048, r = 32: 5.2 / 8.0 at M = 1, 6.0 / 7.8 at M = 2, 7.5 / 7.9 at M = 4, 9.6 / 7.9 at M = 8; with a
//    LayerNorm 6.7 / 9.0, 8.2 / 9.0, 10.9 / 9.0 at M = 1, 2, 4; 512 -> 512: 4.1 / 7.6 at M = 1, 6.4 / 9.1 at M = 16;
//  - more shared memory than lets two CTAs share an SM: the next call's copies then wait for this one's end.
//    2048 -> 5632 8.4 / 9.1 within (M = 4); Q, K and V of 2048 (three problems, LayerNorms) 7.7 / 14, two up-projections
//    2048 -> 5632 6.9 / 11.9 at M = 1.  Groups of four problems and more take it all the same: seven of 2048 -> 2048 12.5 / 16.3 at M = 1.
//  - base-3 weights (no such kernel).
// With one CTA an SM (that, and every launch of two token tiles, for its registers) a launch is cut into the clusters that run at
// once, 33 of four or 15 of eight on 148 SMs: 37 and 18 took a second round.  In two rounds / in one / two launches: 512 -> 5632,
// r = 32, M = 16 14.1 / 8.3 / 10.4; behind a LayerNorm 64 -> 5632 at M = 12 16.6 / 9.3 / 10.4; four of 2048 -> 2048, r = 64, M = 4 16.5 / 10.3 /
// 12.9; seven 11.4 in one round, 18.1 as two launches.  Where the larger shares don't fit, five problems and more run in
// two rounds: eight of 4096 -> 1536, r = 32 15.6 / - / 20.3; but four of 3072 -> 3072, r = 64 15.7 / - / 14.0.
template <int NP>
bool plan_small(SmallLaunch<NP> &L, uint32_t flags) {
    const int sms = device_sm_count();
    if (sms < 8 || (flags & HGF_FLAG_BASE3)) return false;
    long long lora = 0;
    bool any_ln = false;
    int max_M = 0, max_K = 0;
    for (int i = 0; i < L.n; ++i) {
        const SmallProblem &P = L.p[i];
        if (P.N > (1 << 20)) return false;
        any_ln = any_ln || P.ln_w;
        lora = (long long)P.r * P.K * 2 > lora ? (long long)P.r * P.K * 2 : lora;
        max_M = P.M > max_M ? P.M : max_M;
        max_K = P.K > max_K ? P.K : max_K;
    }
    if ((long long)max_M * max_K > (any_ln ? 4096 : 8192)) return false;
    L.nt = max_M <= 8 ? 1 : 2;
    L.cluster_log2 = lora <= 4 * 36 * 1024 ? 2 : 3;
    const int cluster = 1 << L.cluster_log2;
    // Clusters per problem: the largest remaining cost per cluster gets the next one; never more CTAs than row tiles.
    // Returns the shared memory that a CTA then needs.
    auto cut = [&](int total) -> size_t {
        if (L.n > total) return (size_t)-1;
        int cl[NP > 1 ? NP : 1], left = total - L.n;
        for (int i = 0; i < L.n; ++i) cl[i] = 1;
        if (NP == 1) {  // (what the loop comes to; this runs on every call)
            const int most = (int)((row_tiles(L.p[0].N) + cluster - 1) >> L.cluster_log2);
            cl[0] = most < total ? most : total;
            left = 0;
        }
        while (left > 0) {
            int best = -1;
            double most = 0.0;
            for (int i = 0; i < L.n; ++i) {
                const SmallProblem &P = L.p[i];
                const double per = (double)row_tiles(P.N) * ((P.K + 255) / 256) / cl[i];
                if ((long long)cl[i] * cluster < row_tiles(P.N) && per > most) { most = per; best = i; }
            }
            if (best < 0) break;
            ++cl[best];
            --left;
        }
        int begin = 0;
        size_t h = 0, slots = 0, part = 0, lnb = 0, red = 0, x = 0, xq = 0, at = 0, bt = 0, w = 0;
        auto up = [](size_t &v, size_t x) { v = x > v ? x : v; };
        for (int i = 0; i < L.n; ++i) {
            SmallProblem &P = L.p[i];
            P.cluster_begin = begin;
            P.ctas = cl[i] * cluster;
            begin += cl[i];
            const size_t steps = (size_t)((P.K + 255) / 256), tiles = (size_t)((row_tiles(P.N) + P.ctas - 1) / P.ctas);
            const size_t E = (size_t)(P.r / 16) * L.nt * 128, per = (size_t)((P.K / 32 + cluster - 1) / cluster);
            up(h, (size_t)2 * L.nt * 8 * kSmHPitch * 2);
            up(slots, (size_t)cluster * E * 4);
            up(part, (size_t)(kSmWarps / (P.r <= 16 ? 1 : (P.r == 32 ? 2 : 4))) * E * 4);
            if (P.ln_w) up(lnb, (size_t)P.M * steps * 16);
            up(x, (size_t)P.M * (2 * (size_t)P.K + 64));
            up(red, tiles * L.nt * 512);
            up(xq, (size_t)(P.M + (P.M < 8 * L.nt ? 1 : 0)) * (steps * 256 + 64));
            up(at, (size_t)P.r * (per * 64 + ((per & 1) ? 0 : 64)));
            up(bt, tiles * 16 * P.r * 2);
            up(w, tiles * steps * 1024);
        }
        L.clusters = begin;
        size_t off = align_up(sizeof(SmHead), 128);
        auto take = [&](size_t bytes) { const size_t o = off; off += align_up(bytes, 128); return (int)o; };
        L.off_h = take(h);
        L.off_slots = take(slots);
        L.off_part = take(part);
        L.off_ln = take(lnb);
        L.off_red = take(red);
        L.off_x = take(x);
        L.off_xq = take(xq);
        L.off_at = take(at);
        L.off_bt = take(bt);
        L.off_w = take(w);
        L.smem = (int)off;
        return off;
    };
    if (L.nt == 1 && cut(sms / cluster) <= (size_t)kSmSmemLimit) return true;  // two CTAs an SM
    if (L.nt == 1 && L.n < 4) return false;
    if (cut(clusters_at_once(L.cluster_log2)) <= (size_t)(L.n >= 4 ? kSmSmemMax : kSmSmemLimit)) return true;
    return L.n >= 5 && cut(sms / cluster) <= (size_t)kSmSmemMax;  // in two rounds
}
template bool plan_small<1>(SmallLaunch<1> &, uint32_t);
template bool plan_small<kSmallMax>(SmallLaunch<kSmallMax> &, uint32_t);

template <int NT, int NP>
static cudaError_t launch_small_nt(const SmallLaunch<NP> &L, bool pdl, cudaStream_t stream) {
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = ensure_dynamic_smem(decode_small_kernel<NT, NP>, kSmSmemMax, attr_done);
    if (e != cudaSuccess) return e;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(L.clusters << L.cluster_log2));
    cfg.blockDim = dim3(kSmThreads);
    cfg.dynamicSmemBytes = (size_t)L.smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << L.cluster_log2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 2 : 1;
    e = cudaLaunchKernelEx(&cfg, decode_small_kernel<NT, NP>, L, status);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}
template <int NP>
cudaError_t launch_small(const SmallLaunch<NP> &L, bool pdl, cudaStream_t stream) {
    return L.nt == 1 ? launch_small_nt<1, NP>(L, pdl, stream) : launch_small_nt<2, NP>(L, pdl, stream);
}
template cudaError_t launch_small<1>(const SmallLaunch<1> &, bool, cudaStream_t);
template cudaError_t launch_small<kSmallMax>(const SmallLaunch<kSmallMax> &, bool, cudaStream_t);

}  // namespace hgf
