// Prologue kernels: per-token absmax int8 quantisation (Algorithm 1, steps 1-2) and the LoRA
// down-projection H = SiLU(x A) (Algorithm 1, steps 5-6).
#include "hgf_warp.cuh"

namespace hgf {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// One block quantises one token row.
__device__ __forceinline__ void quant_row(const PrologueParams &p, int m, float *tok_sc = nullptr, float gw_over_127 = 0.0f) {
    __shared__ float s_red_f[kWarps];
    __shared__ int s_red_i[kWarps];
    const int K = p.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 *xv = reinterpret_cast<const uint4 *>(p.x + (size_t)m * K);
    const int nv = K / 8;

    uint32_t abits = 0u;
    for (int i = tid; i < nv; i += kThreads) abits = absmax8_bits(abits, xv[i]);
    float amax = warp_max(absmax_bits_to_float(abits));
    if (lane == 0) s_red_f[warp] = amax;
    __syncthreads();
    float g = s_red_f[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) g = fmaxf(g, s_red_f[w]);
    g = fmaxf(g, 1e-5f);
    const QuantScale qs = make_quant_scale(g);

    int sum = 0;
    uint2 *qv = reinterpret_cast<uint2 *>(p.xq + (size_t)m * K);
    uint2 *dq = p.dbg_xq ? reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * K) : nullptr;
    for (int i = tid; i < nv; i += kThreads) {
        const uint2 o = quant8(xv[i], qs, sum);
        qv[i] = o;
        if (dq) dq[i] = o;
    }
    sum = warp_sum_i(sum);
    if (lane == 0) s_red_i[warp] = sum;
    __syncthreads();
    if (tid == 0) {
        int tot = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) tot += s_red_i[w];
        if (p.row_sum) p.row_sum[m] = tot;
        if (tok_sc) tok_sc[m] = g * gw_over_127;
        p.gamma_x[m] = g;
        if (p.dbg_gamma_x) p.dbg_gamma_x[m] = g;
    }
}

// ---- LayerNorm front end (Appendix E, ScientificBitLinear.forward) -----------------------------------
__device__ __forceinline__ double block_sum_d(double v, double *s_red, int lane, int warp) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();  // the previous use of s_red is over
    if (lane == 0) s_red[warp] = v;
    __syncthreads();
    double t = 0.0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t += s_red[w];
    return t;
}
// One block normalises and quantises one token row: mean and variance (two passes, summed in double),
// the row's largest |xn|, then the codes - the listing's binary32 arithmetic: scale = 127 / gamma_x,
// code = rint(xn * scale).  The row is read from L1/L2 in every pass.
__device__ __forceinline__ void quant_row_ln(const PrologueParams &p, const FrontEnd &fe, int m, float *tok_sc, float gw_over_127) {
    __shared__ double s_red_d[kWarps];
    __shared__ float s_red_f[kWarps];
    __shared__ int s_red_i[kWarps];
    const int K = p.K, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint4 *xv = reinterpret_cast<const uint4 *>(p.x + (size_t)m * K);
    const int nv = K / 8;
    float f[8];

    double sum = 0.0;
    for (int i = tid; i < nv; i += kThreads) {
        unpack8(xv[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) sum += (double)f[e];
    }
    const double mean_d = block_sum_d(sum, s_red_d, lane, warp) / (double)K;
    double ss = 0.0;
    for (int i = tid; i < nv; i += kThreads) {
        unpack8(xv[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const double d = (double)f[e] - mean_d;
            ss += d * d;
        }
    }
    const double var = block_sum_d(ss, s_red_d, lane, warp) / (double)K;
    const float mean = (float)mean_d, rstd = (float)(1.0 / sqrt(var + (double)fe.eps));

    float amax = 0.0f;
    for (int i = tid; i < nv; i += kThreads) {
        unpack8(xv[i], f);
        const float4 w0 = *reinterpret_cast<const float4 *>(fe.ln_w + 8 * i), w1 = *reinterpret_cast<const float4 *>(fe.ln_w + 8 * i + 4);
        const float4 b0 = *reinterpret_cast<const float4 *>(fe.ln_b + 8 * i), b1 = *reinterpret_cast<const float4 *>(fe.ln_b + 8 * i + 4);
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) amax = fmaxf(amax, fabsf(ln_value(f[e], mean, rstd, w[e], b[e])));
    }
    amax = warp_max(amax);
    if (lane == 0) s_red_f[warp] = amax;
    __syncthreads();
    float g = s_red_f[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) g = fmaxf(g, s_red_f[w]);
    g = fmaxf(g, 1e-5f);
    const float scale = __fdiv_rn(127.0f, g);

    int sum_q = 0;
    uint2 *qv = reinterpret_cast<uint2 *>(p.xq + (size_t)m * K);
    uint2 *dq = p.dbg_xq ? reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * K) : nullptr;
    for (int i = tid; i < nv; i += kThreads) {
        unpack8(xv[i], f);
        const float4 w0 = *reinterpret_cast<const float4 *>(fe.ln_w + 8 * i), w1 = *reinterpret_cast<const float4 *>(fe.ln_w + 8 * i + 4);
        const float4 b0 = *reinterpret_cast<const float4 *>(fe.ln_b + 8 * i), b1 = *reinterpret_cast<const float4 *>(fe.ln_b + 8 * i + 4);
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float xn[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) xn[e] = ln_value(f[e], mean, rstd, w[e], b[e]);
        const uint2 o = ln_codes8(xn, scale, sum_q);
        qv[i] = o;
        if (dq) dq[i] = o;
    }
    sum_q = warp_sum_i(sum_q);
    if (lane == 0) s_red_i[warp] = sum_q;
    __syncthreads();
    if (tid == 0) {
        int tot = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) tot += s_red_i[w];
        if (p.row_sum) p.row_sum[m] = tot;
        if (tok_sc) tok_sc[m] = g * gw_over_127;
        p.gamma_x[m] = g;
        if (p.dbg_gamma_x) p.dbg_gamma_x[m] = g;
        if (fe.dbg_mean) fe.dbg_mean[m] = mean;
        if (fe.dbg_rstd) fe.dbg_rstd[m] = rstd;
    }
}

__device__ __forceinline__ uint4 ldg_nc_u4(const void *ptr) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(ptr));
    return v;
}

// One block computes 16 columns of H (rows 16 jt .. 16 jt + 15 of A^T) for up to 16 tokens:
// H[m][j] = act(sum_k x[m][k] A[k][j]) on the warp-level tf32 MMA.  bf16 and fp16 values are both
// exactly representable in tf32 (8 exponent, 10 mantissa bits), so the products are formed from
// exact inputs and accumulated in fp32.  The rows of A^T are the 16-row operand, the tokens the
// 8-column operand; the warps split K in 32-element chunks and their partial sums are added in a
// fixed order through shared memory.  NT = number of 8-token tiles.
// With `hpart` the block covers only the 32-column chunks [cbeg, cend) of K and parks its raw sums
// there (MMA accumulator layout: [register][lane]); the GEMV adds the slices and applies the SiLU.
template <int NT>
__device__ __forceinline__ void lora_down_tile(const PrologueParams &p, int jt, int cbeg, int cend, float *hpart) {
    __shared__ float s_red[kWarps][NT * 4][32];
    const int K = p.K, M = p.M, r = p.r, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const __half *rowA = p.At + (size_t)(16 * jt + g) * K + 8 * t;
    const __half *rowB = rowA + (size_t)8 * K;
    const __nv_bfloat16 *xr[NT];
    bool tok_ok[NT];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
        tok_ok[nt] = g + 8 * nt < M;
        xr[nt] = p.x + (size_t)(tok_ok[nt] ? g + 8 * nt : 0) * K + 8 * t;
    }
    float acc[NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[nt][c] = 0.0f;

    const int nchunks = cend;
    constexpr int U = 4;  // chunks in flight per warp
    for (int c0 = cbeg + warp; c0 < nchunks; c0 += U * kWarps) {
        uint4 av[U], bv[U], xv[U][NT];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int c = c0 + u * kWarps;
            av[u] = bv[u] = make_uint4(0u, 0u, 0u, 0u);
            if (c < nchunks) {
                av[u] = ldg_nc_u4(rowA + 32 * c);
                bv[u] = ldg_nc_u4(rowB + 32 * c);
            }
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) {
                xv[u][nt] = make_uint4(0u, 0u, 0u, 0u);
                if (c < nchunks && tok_ok[nt]) xv[u][nt] = *reinterpret_cast<const uint4 *>(xr[nt] + 32 * c);
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint32_t aw[4] = {av[u].x, av[u].y, av[u].z, av[u].w};
            const uint32_t bw[4] = {bv[u].x, bv[u].y, bv[u].z, bv[u].w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // elements 2 i and 2 i + 1 of this lane's eight take the k slots t and t + 4 of the MMA
                const float2 fa = __half22float2(*reinterpret_cast<const __half2 *>(&aw[i]));
                const float2 fb = __half22float2(*reinterpret_cast<const __half2 *>(&bw[i]));
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const uint32_t xw = (&xv[u][nt].x)[i];
                    mma_tf32(acc[nt], __float_as_uint(fa.x), __float_as_uint(fb.x), __float_as_uint(fa.y),
                             __float_as_uint(fb.y), xw << 16, xw & 0xffff0000u);
                }
            }
        }
    }
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int c = 0; c < 4; ++c) s_red[warp][nt * 4 + c][lane] = acc[nt][c];
    __syncthreads();
    if (tid < NT * 4 * 32) {
        const int idx = tid >> 5, ln = tid & 31, nt = idx >> 2, c = idx & 3;
        float z = 0.0f;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) z += s_red[w][idx][ln];
        // accumulator register c of lane (g, t): row g + 8 (c >> 1), token 8 nt + 2 t + (c & 1)
        const int j = 16 * jt + (ln >> 2) + 8 * (c >> 1), m = 8 * nt + 2 * (ln & 3) + (c & 1);
        if (hpart) {
            hpart[idx * 32 + ln] = z;
        } else if (m < M) {
            const float h = (p.flags & HGF_FLAG_NO_SILU) ? z : silu_f(z);
            const size_t o = (size_t)m * r + j;
            p.h[o] = h;
            if (p.dbg_h) p.dbg_h[o] = h;
            if (p.h_hi) {
                const __half hi = __float2half_rn(h);
                p.h_hi[o] = hi;
                p.h_lo[o] = __float2half_rn(h - __half2float(hi));
            }
        }
    }
}

__device__ __forceinline__ void lora_down_block(const PrologueParams &p, int jt, int cbeg, int cend, float *hpart) {
    if (p.M <= 8) lora_down_tile<1>(p, jt, cbeg, cend, hpart); else lora_down_tile<2>(p, jt, cbeg, cend, hpart);
}

// Many rows of up to 4096 elements (quantisation alone): one warp per token row, the row held in registers between the maximum and
// the rounding (U 16-byte units per lane), so a row costs one trip to memory, no block-wide
// synchronisation, and the per-row overhead (scale, reductions) is spread over 8 U elements per lane.
template <int U>
__global__ void __launch_bounds__(kThreads) quant_rows_kernel(const PrologueParams p, const GemmPrologueExtra x) {
    asm volatile("griddepcontrol.wait;\n" ::: "memory");  // see gemm_prologue_kernel
    const int lane = threadIdx.x & 31, m = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (m >= p.M) return;
    const int K = p.K, nv = K / 8;
    const uint4 *xv = reinterpret_cast<const uint4 *>(p.x + (size_t)m * K);
    uint4 v[U];
    uint32_t abits = 0u;
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = lane + 32 * u < nv ? xv[lane + 32 * u] : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int u = 0; u < U; ++u) abits = absmax8_bits(abits, v[u]);
    const float g = fmaxf(warp_max(absmax_bits_to_float(abits)), 1e-5f);
    const QuantScale qs = make_quant_scale(g);
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");  // the row is in registers: the next launch may be set up
    int sum = 0;
    uint2 *qv = reinterpret_cast<uint2 *>(p.xq + (size_t)m * K);
    uint2 *dq = p.dbg_xq ? reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * K) : nullptr;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        if (lane + 32 * u < nv) {
            const uint2 o = quant8<true>(v[u], qs, sum);
            qv[lane + 32 * u] = o;
            if (dq) dq[lane + 32 * u] = o;
        }
    }
    sum = warp_sum_i(sum);
    if (lane == 0) {
        if (p.row_sum) p.row_sum[m] = sum;
        if (x.tok_sc) x.tok_sc[m] = g * x.gw_over_127;
        p.gamma_x[m] = g;
        if (p.dbg_gamma_x) p.dbg_gamma_x[m] = g;
    }
}

__global__ void __launch_bounds__(kThreads) quant_kernel(const PrologueParams p, const GemmPrologueExtra x) {
    quant_row(p, blockIdx.x, x.tok_sc, x.gw_over_127);
}

// Decode prologue: blocks [0, M) quantise one token each; the others compute 16 columns of H each,
// over all of K, or - with a scratch for partial sums - over one K slice each (slice-major), which
// shortens the chain of dependent loads from K / 1024 rounds to one or two.
__global__ void __launch_bounds__(kThreads) decode_prologue_kernel(const PrologueParams p) {
    pdl_launch_dependents();  // the GEMV that follows may start streaming its weights
    pdl_wait();               // x, and the workspace this kernel overwrites, belong to earlier work
    if ((int)blockIdx.x < p.M)
        quant_row(p, blockIdx.x);
    else if (p.hpart) {
        const int lb = blockIdx.x - p.M, jts = p.r / 16, sl = lb / jts, jt = lb - sl * jts;
        const int per = prologue_slice_k(p.M) / 32, cbeg = sl * per, cend = cbeg + per < p.K / 32 ? cbeg + per : p.K / 32;
        lora_down_block(p, jt, cbeg, cend, p.hpart + ((size_t)jt * p.nslices + sl) * 256);
    } else {
        lora_down_block(p, blockIdx.x - p.M, 0, p.K / 32, nullptr);
    }
}

// The same with the LayerNorm front end: the row blocks normalise before they quantise; the
// correction path's blocks read the raw x as before.
__global__ void __launch_bounds__(kThreads) decode_prologue_ln_kernel(const PrologueParams p, const FrontEnd fe) {
    pdl_launch_dependents();
    pdl_wait();
    if ((int)blockIdx.x < p.M)
        quant_row_ln(p, fe, blockIdx.x, nullptr, 0.0f);
    else if (p.hpart) {
        const int lb = blockIdx.x - p.M, jts = p.r / 16, sl = lb / jts, jt = lb - sl * jts;
        const int per = prologue_slice_k(p.M) / 32, cbeg = sl * per, cend = cbeg + per < p.K / 32 ? cbeg + per : p.K / 32;
        lora_down_block(p, jt, cbeg, cend, p.hpart + ((size_t)jt * p.nslices + sl) * 256);
    } else {
        lora_down_block(p, blockIdx.x - p.M, 0, p.K / 32, nullptr);
    }
}

// GEMM path with the front end: one block per token row.
__global__ void __launch_bounds__(kThreads) ln_quant_kernel(const PrologueParams p, const GemmPrologueExtra x, const FrontEnd fe) {
    pdl_wait();
    quant_row_ln(p, fe, blockIdx.x, x.tok_sc, x.gw_over_127);
}

// ---- group prologue: persistent CTAs, one warp per work item ------------------------------------
// The rows of A^T are the bulk of what a decode prologue reads, and a group has thousands of small
// pieces of them, each behind a chain of dependent memory latencies.  Here the grid stays resident
// (one CTA of 8 warps per SM) and every warp walks the item tables with a grid-wide stride.  For a
// LoRA item the warp requests everything the item reads at once - per lane up to 32 + 16 asynchronous
// 16-byte copies into its own part of shared memory, which serves as a register extension: a lane
// reads back only what it requested itself - while the next item's descriptor is already on its
// way, then runs the tf32 MMAs (rows of A^T are the 16-row operand, tokens the 8-column operand) and
// parks the 16 x 16 partial sums; the GEMV adds a tile's K slices in slice order.
constexpr int kPgWarps = 8;
constexpr int kPgThreads = kPgWarps * 32;

// 16-byte asynchronous copy global -> shared; src_bytes = 0 writes zeros and reads nothing.
__device__ __forceinline__ void cp_async_16(uint32_t dst, const void *src, uint32_t src_bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ uint4 pg_lds_u4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// One warp quantises one token row (Algorithm 1, steps 1-2).  The row is brought into the warp's
// shared-memory buffer with asynchronous copies, all requested at once, so both passes (maximum,
// then rounding) read it from there; a row longer than the buffer goes through in pieces and is
// fetched a second time for the second pass.
__device__ void warp_quant_row(const QuantItem &q, uint32_t buf_u32, const uint8_t *buf, int buf_bytes, int lane) {
    const int K = q.K, piece = buf_bytes / 2;  // elements per piece (a multiple of 256)
    const int npieces = (K + piece - 1) / piece;
    auto fetch = [&](int pc) {  // units of 8 elements; lane-strided, so a lane reads back its own units
        const int n = (K - pc * piece < piece ? K - pc * piece : piece) / 8;
        for (int i = lane; i < n; i += 32) cp_async_16(buf_u32 + 16 * i, q.x + (size_t)pc * piece + 8 * i, 16u);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        return n;
    };
    uint32_t abits = 0u;
    int n = 0;
    for (int pc = 0; pc < npieces; ++pc) {
        n = fetch(pc);
        for (int i = lane; i < n; i += 32) abits = absmax8_bits(abits, *reinterpret_cast<const uint4 *>(buf + 16 * i));
    }
    const float g = fmaxf(warp_max(absmax_bits_to_float(abits)), 1e-5f);
    const QuantScale qs = make_quant_scale(g);
    int sum = 0;
    for (int pc = 0; pc < npieces; ++pc) {
        if (npieces > 1) n = fetch(pc);
        uint2 *qv = reinterpret_cast<uint2 *>(q.xq + (size_t)pc * piece);
        for (int i = lane; i < n; i += 32) qv[i] = quant8(*reinterpret_cast<const uint4 *>(buf + 16 * i), qs, sum);
    }
    sum = warp_sum_i(sum);
    if (lane == 0) {
        *q.row_sum = sum;
        *q.gamma_x = g;
    }
}

// The same for a row behind the LayerNorm front end (Appendix E of the paper): statistics in two passes
// summed in double, the largest |xn|, then the codes - the arithmetic of quant_row_ln, one warp per
// row, each pass reading the row from L1 / L2.
__device__ void warp_quant_row_ln(const QuantItem &q, int lane) {
    const int K = q.K, nv = K / 8;
    const uint4 *xv = reinterpret_cast<const uint4 *>(q.x);
    float f[8];
    double sum = 0.0;
    for (int i = lane; i < nv; i += 32) {
        unpack8(xv[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) sum += (double)f[e];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    const double mean_d = sum / (double)K;
    double ss = 0.0;
    for (int i = lane; i < nv; i += 32) {
        unpack8(xv[i], f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const double d = (double)f[e] - mean_d;
            ss += d * d;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    const float mean = (float)mean_d, rstd = (float)(1.0 / sqrt(ss / (double)K + (double)q.eps));
    auto load_wb = [&](int i, float (&w)[8], float (&b)[8]) {
        const float4 w0 = *reinterpret_cast<const float4 *>(q.ln_w + 8 * i), w1 = *reinterpret_cast<const float4 *>(q.ln_w + 8 * i + 4);
        const float4 b0 = *reinterpret_cast<const float4 *>(q.ln_b + 8 * i), b1 = *reinterpret_cast<const float4 *>(q.ln_b + 8 * i + 4);
        w[0] = w0.x; w[1] = w0.y; w[2] = w0.z; w[3] = w0.w; w[4] = w1.x; w[5] = w1.y; w[6] = w1.z; w[7] = w1.w;
        b[0] = b0.x; b[1] = b0.y; b[2] = b0.z; b[3] = b0.w; b[4] = b1.x; b[5] = b1.y; b[6] = b1.z; b[7] = b1.w;
    };
    float amax = 0.0f, w[8], b[8];
    for (int i = lane; i < nv; i += 32) {
        unpack8(xv[i], f);
        load_wb(i, w, b);
#pragma unroll
        for (int e = 0; e < 8; ++e) amax = fmaxf(amax, fabsf(ln_value(f[e], mean, rstd, w[e], b[e])));
    }
    const float g = fmaxf(warp_max(amax), 1e-5f);
    const float scale = __fdiv_rn(127.0f, g);
    int sum_q = 0;
    uint2 *qv = reinterpret_cast<uint2 *>(q.xq);
    for (int i = lane; i < nv; i += 32) {
        unpack8(xv[i], f);
        load_wb(i, w, b);
        float xn[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) xn[e] = ln_value(f[e], mean, rstd, w[e], b[e]);
        qv[i] = ln_codes8(xn, scale, sum_q);
    }
    sum_q = warp_sum_i(sum_q);
    if (lane == 0) {
        *q.row_sum = sum_q;
        *q.gamma_x = g;
        if (q.mean_out) *q.mean_out = mean;
        if (q.rstd_out) *q.rstd_out = rstd;
    }
}

// The LayerNorm front end for many rows (the GEMM path): one warp per token row, eight rows per block, the
// row's passes (mean, variance, largest |xn|, codes) all from L1 with warp shuffles between them - one block
// per row spent its time in block-wide barriers between the passes.
__global__ void __launch_bounds__(kThreads) ln_quant_rows_kernel(const PrologueParams p, const GemmPrologueExtra x, const FrontEnd fe) {
    pdl_wait();
    const int lane = threadIdx.x & 31, m = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (m >= p.M) return;
    QuantItem q;
    q.x = p.x + (size_t)m * p.K;
    q.xq = p.xq + (size_t)m * p.K;
    q.gamma_x = p.gamma_x + m;
    q.row_sum = p.row_sum + m;
    q.K = p.K;
    q.eps = fe.eps;
    q.ln_w = fe.ln_w;
    q.ln_b = fe.ln_b;
    q.mean_out = fe.dbg_mean ? fe.dbg_mean + m : nullptr;
    q.rstd_out = fe.dbg_rstd ? fe.dbg_rstd + m : nullptr;
    warp_quant_row_ln(q, lane);
    __syncwarp();
    if (lane == 0) {  // (reads back what this lane wrote)
        const float g = p.gamma_x[m];
        if (x.tok_sc) x.tok_sc[m] = g * x.gw_over_127;
        if (p.dbg_gamma_x) p.dbg_gamma_x[m] = g;
    }
    if (p.dbg_xq) {  // each lane copies the units it wrote itself
        const uint2 *qv = reinterpret_cast<const uint2 *>(q.xq);
        uint2 *dq = reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * p.K);
        for (int i = lane; i < p.K / 8; i += 32) dq[i] = qv[i];
    }
}

// A row behind the LayerNorm front end by a whole CTA: brought into shared memory once, mean and variance in one pass in
// double of x - x[0] (see hgf_decode_small.cu), the largest |xn|, the codes.  A decode launch has a few of these and
// one warp alone took 20 us over a row of 2048 (four passes, a memory latency in each of their steps).
__device__ void block_quant_row_ln(const QuantItem &q, uint8_t *buf, int tid) {
    __shared__ double2 s_sum[kPgWarps];
    __shared__ uint32_t s_max[kPgWarps];
    __shared__ int s_codes[kPgWarps];
    const int K = q.K, nv = K / 8, lane = tid & 31, warp = tid >> 5;
    const uint32_t buf_u32 = (uint32_t)__cvta_generic_to_shared(buf);
    for (int i = tid; i < nv; i += kPgThreads) cp_async_16(buf_u32 + 16 * i, q.x + 8 * i, 16u);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    const double first = (double)__bfloat162float(*reinterpret_cast<const __nv_bfloat16 *>(buf));
    double s = 0.0, ss = 0.0;
    for (int i = tid; i < nv; i += kPgThreads) {
        float f[8];
        unpack8(*reinterpret_cast<const uint4 *>(buf + 16 * i), f);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const double d = (double)f[e] - first;
            s += d;
            ss = fma(d, d, ss);
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, o);
        ss += __shfl_xor_sync(0xffffffffu, ss, o);
    }
    if (lane == 0) s_sum[warp] = make_double2(s, ss);
    __syncthreads();
    s = ss = 0.0;
#pragma unroll
    for (int w = 0; w < kPgWarps; ++w) { s += s_sum[w].x; ss += s_sum[w].y; }
    const double dm = s / (double)K, v0 = ss / (double)K - dm * dm, var = v0 < 0.0 ? 0.0 : v0;  // (NaN stays NaN)
    const float mean = (float)(first + dm), rstd = (float)rsqrt(var + (double)q.eps);
    auto normal = [&](int i, float (&xn)[8]) {
        const float4 *w4 = reinterpret_cast<const float4 *>(q.ln_w + 8 * i), *b4 = reinterpret_cast<const float4 *>(q.ln_b + 8 * i);
        const float4 w0 = w4[0], w1 = w4[1], b0 = b4[0], b1 = b4[1];
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
        float f[8];
        unpack8(*reinterpret_cast<const uint4 *>(buf + 16 * i), f);
#pragma unroll
        for (int e = 0; e < 8; ++e) xn[e] = ln_value(f[e], mean, rstd, w[e], b[e]);
    };
    float a = 0.0f, xn[8];
    for (int i = tid; i < nv; i += kPgThreads) {
        normal(i, xn);
#pragma unroll
        for (int e = 0; e < 8; ++e) a = fmaxf(a, fabsf(xn[e]));
    }
    const uint32_t most = __reduce_max_sync(0xffffffffu, __float_as_uint(a));
    if (lane == 0) s_max[warp] = most;
    __syncthreads();
    uint32_t top = s_max[0];
#pragma unroll
    for (int w = 1; w < kPgWarps; ++w) top = s_max[w] > top ? s_max[w] : top;
    const float g = fmaxf(__uint_as_float(top), 1e-5f), scale = __fdiv_rn(127.0f, g);
    int sum = 0;
    for (int i = tid; i < nv; i += kPgThreads) {
        normal(i, xn);
        reinterpret_cast<uint2 *>(q.xq)[i] = ln_codes8(xn, scale, sum);
    }
    sum = __reduce_add_sync(0xffffffffu, sum);
    if (lane == 0) s_codes[warp] = sum;
    __syncthreads();  // (also: the row's buffer is free)
    if (tid == 0) {
        int all = 0;
#pragma unroll
        for (int w = 0; w < kPgWarps; ++w) all += s_codes[w];
        *q.row_sum = all;
        *q.gamma_x = g;
        if (q.mean_out) *q.mean_out = mean;
        if (q.rstd_out) *q.rstd_out = rstd;
    }
}

// LN_WARPS: rows behind a LayerNorm are among the warps' rows (without them the kernel goes without their code).
template <int NT, bool LN_WARPS>
__global__ void __launch_bounds__(kPgThreads, 1)
decode_prologue_group_kernel(const QuantItem *quant_items, int n_ln, int n_quant, const LoraItem *lora, int n_lora) {
    constexpr int CH = 16 / NT;                       // 32-column chunks per item
    constexpr int kWarpBytes = CH * (1024 + 512 * NT);  // per chunk: two rows of A^T and NT rows of x, 16 bytes per lane
    extern __shared__ __align__(128) uint8_t pg_smem[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int gw = blockIdx.x * kPgWarps + warp, nw = gridDim.x * kPgWarps;
    const uint32_t buf = (uint32_t)__cvta_generic_to_shared(pg_smem) + warp * kWarpBytes + 16 * lane;

    pdl_launch_dependents();
    // the item tables are written at set-up, not by the preceding work
    uint4 d0 = make_uint4(0u, 0u, 0u, 0u), d1 = d0;
    if (gw < n_lora) {
        d0 = reinterpret_cast<const uint4 *>(lora + gw)[0];
        d1 = reinterpret_cast<const uint4 *>(lora + gw)[1];
    }
    // LoRA items are dealt from the first warp up, quantisation items from the last warp down, so the
    // warps with one LoRA item fewer take the rows
    const int q_first = n_ln + nw - 1 - gw;
    QuantItem q = {};
    if (q_first < n_quant) q = quant_items[q_first];
    pdl_wait();  // x, and the scratch this kernel overwrites, belong to earlier work

    // the first n_ln items, rows behind a LayerNorm: a CTA each, from the last CTA down
    for (int i = gridDim.x - 1 - blockIdx.x; i < n_ln; i += gridDim.x) {
        const QuantItem row = quant_items[i];
        block_quant_row_ln(row, pg_smem, threadIdx.x);
        __syncthreads();
    }

    for (int i = q_first; i < n_quant; i += nw) {
        QuantItem q_next = q;
        if (i + nw < n_quant) q_next = quant_items[i + nw];  // travels while this row is worked on
        if (LN_WARPS && q.ln_w) warp_quant_row_ln(q, lane);
        else warp_quant_row(q, buf - 16 * lane, pg_smem + warp * kWarpBytes, kWarpBytes, lane);
        q = q_next;
    }

    for (int i = gw; i < n_lora; i += nw) {
        const LoraItem it = {reinterpret_cast<const __half *>(((uint64_t)d0.y << 32) | d0.x),
                             reinterpret_cast<const __nv_bfloat16 *>(((uint64_t)d0.w << 32) | d0.z),
                             reinterpret_cast<float *>(((uint64_t)d1.y << 32) | d1.x), (int)d1.z, (int)d1.w};
        const int K = it.K, M = it.kvalid_M & 0xff, nchunks = (it.kvalid_M >> 8) / 32;
        // everything this item reads, requested at once
        const __half *rowA = it.At + (size_t)g * K + 8 * t;
        const __half *rowB = rowA + (size_t)8 * K;
#pragma unroll
        for (int c = 0; c < CH; ++c) {
            const bool in = c < nchunks;
            cp_async_16(buf + c * 1024, in ? rowA + 32 * c : it.At, in ? 16u : 0u);
            cp_async_16(buf + c * 1024 + 512, in ? rowB + 32 * c : it.At, in ? 16u : 0u);
        }
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            const bool tok = g + 8 * nt < M;
            const __nv_bfloat16 *xr = it.x + (size_t)(tok ? g + 8 * nt : 0) * K + 8 * t;
#pragma unroll
            for (int c = 0; c < CH; ++c) {
                const bool in = tok && c < nchunks;
                cp_async_16(buf + CH * 1024 + (c * NT + nt) * 512, in ? xr + 32 * c : it.x, in ? 16u : 0u);
            }
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        if (i + nw < n_lora) {  // the next item's descriptor travels meanwhile
            d0 = reinterpret_cast<const uint4 *>(lora + i + nw)[0];
            d1 = reinterpret_cast<const uint4 *>(lora + i + nw)[1];
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");

        float acc[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[nt][c] = 0.0f;
#pragma unroll 4
        for (int c = 0; c < CH; ++c) {
            const uint4 av = pg_lds_u4(buf + c * 1024), bv = pg_lds_u4(buf + c * 1024 + 512);
            uint4 xv[NT];
#pragma unroll
            for (int nt = 0; nt < NT; ++nt) xv[nt] = pg_lds_u4(buf + CH * 1024 + (c * NT + nt) * 512);
            const uint32_t aw[4] = {av.x, av.y, av.z, av.w};
            const uint32_t bw[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                // elements 2 e and 2 e + 1 of this lane's eight take the k slots t and t + 4 of the MMA
                const float2 fa = __half22float2(*reinterpret_cast<const __half2 *>(&aw[e]));
                const float2 fb = __half22float2(*reinterpret_cast<const __half2 *>(&bw[e]));
#pragma unroll
                for (int nt = 0; nt < NT; ++nt) {
                    const uint32_t xw = (&xv[nt].x)[e];
                    mma_tf32(acc[nt], __float_as_uint(fa.x), __float_as_uint(fb.x), __float_as_uint(fa.y),
                             __float_as_uint(fb.y), xw << 16, xw & 0xffff0000u);
                }
            }
        }
        // park the partial sums: [register 0..7][lane]
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int c = 0; c < 4; ++c) __stcg(it.hpart + (nt * 4 + c) * 32 + lane, acc[nt][c]);
    }
}

static cudaLaunchConfig_t prologue_cfg(int blocks, bool pdl, cudaStream_t stream, cudaLaunchAttribute *attr);
constexpr int kRpSmemLimit = 200 * 1024;

// ---- GEMM-path prologue in one kernel -------------------------------------------------------------
// Quantisation (Algorithm 1, steps 1-2) and the LoRA down-projection (steps 5-6) of a block of TOK
// tokens, reading x from HBM once.  First pass: x and the rows of A^T travel through a three-stage
// ring of 256-column chunks (16-byte asynchronous copies); every warp takes 32 columns of a chunk,
// feeds them to the tf32 MMA (tokens are the 16-row operand, 8 columns of H the 8-column operand;
// bf16 and fp16 values are exact in tf32) and, since every element of x passes through exactly one
// lane's registers on the way, keeps the running maximum of |x| of its rows.  Then the warps' partial
// sums of x A are added in a fixed order, and the block's rows - still in L2 - are read again and
// rounded with the now known scales.  JT = r / 8 column tiles of H; JT = 0 quantises only.
// W: eight warps of two token tiles each, two blocks an SM; from rank 48 on, where a block's ring takes an SM's shared memory, sixteen
// warps (the second eight take every other token tile), so that the MMA and its conversions have as many warps there.  Layer calls,
// eight / sixteen: r = 64, 6144 -> 1024 at M = 6000 119.1 / 115.5 us, 4096 -> 1024 with a LayerNorm at M = 8192 131.5 / 128.9, 1024 -> 1024 at M = 4000
// 23.3 / 21.2, 512 -> 512 at M = 300 11.7 / 10.75; r = 48, 512 -> 1024 at M = 4736 19.4 / 17.6, 768 -> 768 at M = 700 12.4 / 11.5.  Ranks up to 32 have sixteen warps
// an SM as it is and are bound by the MMA's rate: with 32 warps 2048 -> 5632 at M = 8192 117.9 / 119.6, 5632 -> 2048 135.0 / 140.4.
// TOK: 64 tokens a block halve the reads of A^T and need fewer rounds; that is worth it at rank 48 beyond one round of 32 tokens
// (3072 -> 1024 at M = 5000 58.0 / 50.0 us, 1024 -> 512 at M = 16384 53.1 / 47.8).  Rank 64 would spill at 128 registers (6144 -> 1024 at M = 6000
// 115.5 / 133.1), for ranks up to 32 it is the same time (2048 -> 5632 at M = 8192 118.6 / 119.3).
constexpr int kFpWarps = 8;                          // warps that share a chunk's columns
constexpr int kFpChunk = 256;                        // columns per stage
constexpr int kFpPitch = kFpChunk * 2 + 64;          // bytes per staged row: neighbouring rows on the other 16 banks
constexpr int kFpStages = 3;
__host__ __device__ constexpr int fp_stage_bytes(int tokens, int r) { return (tokens + r) * kFpPitch; }
__host__ __device__ constexpr int fp_smem_bytes(int tokens, int r) {
    return kFpStages * fp_stage_bytes(tokens, r) > kFpWarps * tokens * r * 4 ? kFpStages * fp_stage_bytes(tokens, r) : kFpWarps * tokens * r * 4;
}

// The up-projection's operand: row n of B^T times its channel's gate, fp16, padded to 64 columns; piece `idx` is 16 bytes.
__device__ __forceinline__ void gate_operand(const GemmPrologueExtra &x, int r, int idx) {
    const int n = idx >> 3, c = idx & 7;
    if (n >= x.N) return;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (c * 8 < r) {
        v = *reinterpret_cast<const uint4 *>(x.Bt + (size_t)n * r + c * 8);
        const float g = x.gate[x.gate_group > 1 ? n / x.gate_group : n];
        __half2 *h2 = reinterpret_cast<__half2 *>(&v);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float2 f = __half22float2(h2[k]);
            h2[k] = __floats2half2_rn(g * f.x, g * f.y);
        }
    }
    *reinterpret_cast<uint4 *>(x.gb16 + (size_t)n * 64 + c * 8) = v;
}

template <int JT, int W, int TOK>
__global__ void __launch_bounds__(32 * W, 1) gemm_prologue_kernel(const PrologueParams p, const GemmPrologueExtra x) {
    extern __shared__ __align__(128) uint8_t fp_smem[];
    constexpr int THREADS = 32 * W, SETS = W / kFpWarps, TILES = TOK / 16 / SETS;  // (token tiles a warp)
    __shared__ float s_amax[kFpWarps][TOK];
    __shared__ float s_gamma[TOK];
    constexpr int r = 8 * JT;
    pdl_wait();  // x, and the workspace this kernel overwrites, belong to earlier work
    const int tpb = x.tokens_per_block;  // tokens this launch gives a block (at most TOK)
    const int token_blocks = (p.M + tpb - 1) / tpb;
    if ((int)blockIdx.x >= token_blocks) {
        // the remaining blocks prepare the up-projection's operand
        if constexpr (JT > 0) {
            gate_operand(x, r, ((int)blockIdx.x - token_blocks) * THREADS + (int)threadIdx.x);
        }
        return;
    }
    const int K = p.K, M = p.M;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, part = warp % kFpWarps, mt0 = warp / kFpWarps, g = lane >> 2, t = lane & 3;
    const int m0 = blockIdx.x * tpb;
    const uint32_t smem_u32 = (uint32_t)__cvta_generic_to_shared(fp_smem);
    constexpr int kStage = fp_stage_bytes(TOK, r);
    const int nchunks = (K + kFpChunk - 1) / kFpChunk;

    // One chunk into one stage: TOK (+ r) rows of 32 16-byte units; rows past M and columns past K are
    // zeros.  A thread copies unit `lane` of rows warp, warp + W, ... (tokens first: TOK and r are multiples of 16): the same
    // ones in every chunk.
    constexpr int kRowsPerThread = (TOK + r) / W;
    const uint8_t *src_x = reinterpret_cast<const uint8_t *>(p.x + (size_t)(m0 + warp) * K) + 16 * lane;
    const uint8_t *src_a = JT > 0 ? reinterpret_cast<const uint8_t *>(p.At + (size_t)warp * K) + 16 * lane : nullptr;
    const int rows_x = M - m0 < tpb ? M - m0 : tpb;
    auto fetch = [&](int c, int stage) {
        const uint32_t dst = smem_u32 + stage * kStage + warp * kFpPitch + 16 * lane;
        const int k = c * kFpChunk + 8 * lane;
        const bool col_ok = k < K;
#pragma unroll
        for (int q = 0; q < kRowsPerThread; ++q) {
            constexpr int kTokenRows = TOK / W;
            const bool token = q < kTokenRows, in = col_ok && (!token || warp + W * q < rows_x);
            const uint8_t *src = token ? src_x + (size_t)(q * W) * K * 2 : src_a + (size_t)((q - kTokenRows) * W) * K * 2;
            cp_async_16(dst + q * W * kFpPitch, in ? src + (size_t)c * kFpChunk * 2 : reinterpret_cast<const uint8_t *>(p.x), in ? 16u : 0u);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };

    float acc[TILES][JT > 0 ? JT : 1][4];
#pragma unroll
    for (int a = 0; a < TILES; ++a)
#pragma unroll
        for (int b = 0; b < (JT > 0 ? JT : 1); ++b)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[a][b][c] = 0.0f;
    uint32_t amax[TILES][2] = {};  // rows 16 mt + 8 hh + g, packed maxima of the bit patterns

#pragma unroll
    for (int sg = 0; sg < kFpStages - 1; ++sg) {
        if (sg < nchunks) fetch(sg, sg);
        else asm volatile("cp.async.commit_group;\n" ::: "memory");
    }
    for (int c = 0; c < nchunks; ++c) {
        asm volatile("cp.async.wait_group %0;\n" ::"n"(kFpStages - 2) : "memory");
        __syncthreads();  // chunk c has landed for every thread, and everyone is done with chunk c - 1
        if (c + kFpStages - 1 < nchunks) fetch(c + kFpStages - 1, (c + kFpStages - 1) % kFpStages);
        else asm volatile("cp.async.commit_group;\n" ::: "memory");

        const uint32_t st = smem_u32 + (c % kFpStages) * kStage + 64 * part + 16 * t;
#pragma unroll
        for (int i_mt = 0; i_mt < TILES; ++i_mt) {
            const int mt = mt0 + SETS * i_mt;
            if (16 * mt >= tpb) break;  // a block of up to 16 tokens has no second tile
            const uint4 x0 = pg_lds_u4(st + (16 * mt + g) * kFpPitch), x1 = pg_lds_u4(st + (16 * mt + 8 + g) * kFpPitch);
            amax[i_mt][0] = absmax8_bits(amax[i_mt][0], x0);
            amax[i_mt][1] = absmax8_bits(amax[i_mt][1], x1);
            if constexpr (JT > 0) {
                // elements 2 i and 2 i + 1 of this lane's eight take the k slots t and t + 4 of MMA i
                uint32_t xs[4][4];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const uint32_t w0 = (&x0.x)[i], w1 = (&x1.x)[i];
                    xs[i][0] = w0 << 16; xs[i][1] = w1 << 16; xs[i][2] = w0 & 0xffff0000u; xs[i][3] = w1 & 0xffff0000u;
                }
#pragma unroll
                for (int jt = 0; jt < JT; ++jt) {
                    const uint4 a4 = pg_lds_u4(st + (TOK + 8 * jt + g) * kFpPitch);
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float2 bf = __half22float2(*reinterpret_cast<const __half2 *>(&(&a4.x)[i]));
                        mma_tf32(acc[i_mt][jt], xs[i][0], xs[i][1], xs[i][2], xs[i][3], __float_as_uint(bf.x), __float_as_uint(bf.y));
                    }
                }
            }
        }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");

    // the rows' maxima: over the four lanes that share a row, then over the warps
#pragma unroll
    for (int mt = 0; mt < TILES; ++mt)
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            float a = absmax_bits_to_float(amax[mt][hh]);
            a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 1));
            a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, 2));
            if (t == 0) s_amax[part][16 * (mt0 + SETS * mt) + 8 * hh + g] = a;
        }
    __syncthreads();  // also: every warp is done with the ring, which the partial sums now reuse
    if (tid < TOK) {
        float a = s_amax[0][tid];
#pragma unroll
        for (int w = 1; w < kFpWarps; ++w) a = fmaxf(a, s_amax[w][tid]);
        s_gamma[tid] = fmaxf(a, 1e-5f);
    }
    if constexpr (JT > 0) {
        float *s_acc = reinterpret_cast<float *>(fp_smem);  // [part of the columns, kFpWarps of them][TOK][r]
#pragma unroll
        for (int mt = 0; mt < TILES; ++mt)
#pragma unroll
            for (int jt = 0; jt < JT; ++jt) {
                float *base = s_acc + ((size_t)part * TOK + 16 * (mt0 + SETS * mt)) * r + 8 * jt;
                base[g * r + 2 * t] = acc[mt][jt][0];
                base[g * r + 2 * t + 1] = acc[mt][jt][1];
                base[(g + 8) * r + 2 * t] = acc[mt][jt][2];
                base[(g + 8) * r + 2 * t + 1] = acc[mt][jt][3];
            }
    }
    __syncthreads();
    if constexpr (JT > 0) {
        const float *s_acc = reinterpret_cast<const float *>(fp_smem);
        for (int e = tid; e < TOK * r; e += THREADS) {
            const int ml = e / r, j = e % r, m = m0 + ml;
            float z = 0.0f;
#pragma unroll
            for (int w = 0; w < kFpWarps; ++w) z += s_acc[w * TOK * r + e];
            const float h = (p.flags & HGF_FLAG_NO_SILU) ? z : silu_f(z);
            if (ml < tpb && m < M) {
                p.h[(size_t)m * r + j] = h;
                if (p.dbg_h) p.dbg_h[(size_t)m * r + j] = h;
                if (p.h16) p.h16[(size_t)m * 64 + j] = __float2half_rn(h);
            }
        }
        if constexpr (JT < 8) {  // zero padding of the fp16 copy up to 64 columns
            if (p.h16)
                for (int e = tid; e < TOK * (64 - r); e += THREADS) {
                    const int ml = e / (64 - r), j = r + e % (64 - r), m = m0 + ml;
                    if (ml < tpb && m < M) p.h16[(size_t)m * 64 + j] = __float2half_rn(0.0f);
                }
        }
    }

    // The launch that follows (the GEMM) may be set up from here on; it waits for this grid's completion
    // before it reads.  (Not earlier: blocks of a dependent launch that sit waiting on an SM slow the
    // blocks still working there.)
    pdl_launch_dependents();

    if (!p.xq) return;  // the LayerNorm front end quantises in a kernel of its own
    if (x.split_round) {  // the rounding pass is the next launch: leave it the scales
        if (tid < tpb && m0 + tid < M) {
            const float gm = s_gamma[tid];
            p.gamma_x[m0 + tid] = gm;
            if (x.tok_sc) x.tok_sc[m0 + tid] = gm * x.gw_over_127;
            if (p.dbg_gamma_x) p.dbg_gamma_x[m0 + tid] = gm;
        }
        return;
    }

    // second pass: the warps round the block's rows, warp w rows w, w + W, ...
    const int nv = K / 8;
#pragma unroll 1
    for (int rr = 0; rr < TOK / W; ++rr) {
        const int ml = warp + W * rr, m = m0 + ml;
        if (ml >= tpb || m >= M) break;
        const float gm = s_gamma[ml];
        const QuantScale qs = make_quant_scale(gm);
        const uint4 *xv = reinterpret_cast<const uint4 *>(p.x + (size_t)m * K);
        uint2 *qv = reinterpret_cast<uint2 *>(p.xq + (size_t)m * K);
        uint2 *dq = p.dbg_xq ? reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * K) : nullptr;
        int sum = 0;
        int i = lane;
        for (; i + 96 < nv; i += 128) {  // four units in flight per lane
            const uint4 v0 = xv[i], v1 = xv[i + 32], v2 = xv[i + 64], v3 = xv[i + 96];
            const uint2 o0 = quant8<true>(v0, qs, sum), o1 = quant8<true>(v1, qs, sum), o2 = quant8<true>(v2, qs, sum), o3 = quant8<true>(v3, qs, sum);
            qv[i] = o0; qv[i + 32] = o1; qv[i + 64] = o2; qv[i + 96] = o3;
            if (dq) { dq[i] = o0; dq[i + 32] = o1; dq[i + 64] = o2; dq[i + 96] = o3; }
        }
        for (; i < nv; i += 32) {
            const uint2 o = quant8<true>(xv[i], qs, sum);
            qv[i] = o;
            if (dq) dq[i] = o;
        }
        sum = warp_sum_i(sum);
        if (lane == 0) {
            if (p.row_sum) p.row_sum[m] = sum;
            if (x.tok_sc) x.tok_sc[m] = gm * x.gw_over_127;
            p.gamma_x[m] = gm;
            if (p.dbg_gamma_x) p.dbg_gamma_x[m] = gm;
        }
    }
}

// The rounding pass as a launch of its own: one warp per token row, the scale taken from gamma_x.  At 64
// registers a thread four blocks share an SM (32 warps), which this arithmetic-bound pass needs: inside the
// kernel above it runs at 16 warps per SM and takes twice as long.  The rows are read from L2.
__global__ void __launch_bounds__(kThreads, 4) round_rows_kernel(const PrologueParams p) {
    pdl_wait();               // the scales come from the launch before
    pdl_launch_dependents();  // the GEMM may set itself up; it waits for this grid before it reads
    const int lane = threadIdx.x & 31, m = blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (m >= p.M) return;
    const int K = p.K, nv = K / 8;
    const QuantScale qs = make_quant_scale(p.gamma_x[m]);
    const uint4 *xv = reinterpret_cast<const uint4 *>(p.x + (size_t)m * K);
    uint2 *qv = reinterpret_cast<uint2 *>(p.xq + (size_t)m * K);
    uint2 *dq = p.dbg_xq ? reinterpret_cast<uint2 *>(p.dbg_xq + (size_t)m * K) : nullptr;
    int sum = 0;
    int i = lane;
    for (; i + 96 < nv; i += 128) {  // four units in flight per lane
        const uint4 v0 = xv[i], v1 = xv[i + 32], v2 = xv[i + 64], v3 = xv[i + 96];
        const uint2 o0 = quant8<true>(v0, qs, sum), o1 = quant8<true>(v1, qs, sum), o2 = quant8<true>(v2, qs, sum), o3 = quant8<true>(v3, qs, sum);
        qv[i] = o0; qv[i + 32] = o1; qv[i + 64] = o2; qv[i + 96] = o3;
        if (dq) { dq[i] = o0; dq[i + 32] = o1; dq[i + 64] = o2; dq[i + 96] = o3; }
    }
    for (; i < nv; i += 32) {
        const uint2 o = quant8<true>(xv[i], qs, sum);
        qv[i] = o;
        if (dq) dq[i] = o;
    }
    sum = warp_sum_i(sum);
    if (lane == 0 && p.row_sum) p.row_sum[m] = sum;
}

// ---- GEMM-path prologue for batches that leave the kernel above short of blocks -----------------------
// A cluster takes 16 tokens and each of its C CTAs a slice of their columns, small enough to stay in shared memory: x is
// read once, by one bulk copy per row, and statistics, x A and rounding all work from there.  The CTAs exchange
// partial maxima (with a LayerNorm also sums), partial sums of x A and row sums through distributed shared memory
// (st.async, counted by the receiver's mbarrier); the 16 / C tokens a CTA owns get their H and scales from it.
// What it replaces there: a block walked its tokens' columns in a chain of 256-column chunks (a barrier and most of
// a memory latency each, K / 256 of them, on M / 8 blocks), rounded in a second pass from L2, and a LayerNorm took a
// launch of its own.
constexpr int kRpTokens = 16;
constexpr int kRpParts = 8;  // warps that share out the slice for x A; of sixteen warps two sets, half of the columns of H each
struct RpLayout {
    int per, pitch;              // columns of a slice (a multiple of 64), bytes per staged row
    int off_stat, off_amax, off_sum, off_slots, off_part, off_x, smem;
};
__host__ __device__ inline RpLayout rp_layout(int K, int r, int log2_c) {
    const int C = 1 << log2_c;
    RpLayout L;
    L.per = ((K / 64 + C - 1) >> log2_c) * 64;
    L.pitch = 2 * L.per + 64;    // neighbouring rows on different halves of the banks
    L.off_stat = 64;                                      // [rank][token] double2
    L.off_amax = L.off_stat + C * kRpTokens * 16;         // [rank][token] patterns
    L.off_sum = L.off_amax + C * kRpTokens * 4;           // [rank][token] ints
    L.off_slots = L.off_sum + C * kRpTokens * 4;          // [rank][token][r]
    L.off_part = L.off_slots + C * kRpTokens * r * 4;     // [part][token][r]
    L.off_x = (L.off_part + kRpParts * kRpTokens * r * 4 + 127) / 128 * 128;
    L.smem = L.off_x + kRpTokens * L.pitch;
    return L;
}

// PER_SM: CTAs an SM that its registers leave room for (0: as they come).  All forms fit two but the widest behind a LayerNorm, which takes 154 registers
// and spills 36 bytes at 128: in launches of more CTAs than SMs two an SM are worth that (r = 64, 2048 -> 1024: 26.3 -> 21.1 us
// at M = 1000, 34.5 -> 27.8 at M = 2048), in smaller ones not (22.1 -> 26.4 at M = 1184; they run sixteen warps a CTA now).
template <int JT, bool LN, int TPW, int PER_SM>
__global__ void __launch_bounds__(512 / TPW, PER_SM) rows_prologue_kernel(const PrologueParams p, const GemmPrologueExtra x, const FrontEnd fe,
                                                                   const int log2_c, unsigned int *status) {
    extern __shared__ __align__(128) uint8_t rp_smem[];
    constexpr int r = 8 * JT, kRpThreads = 512 / TPW, W = kRpTokens / TPW;  // W warps: warp w works tokens w (and w + W) of the block
    const int C = 1 << log2_c, token_blocks = (p.M + kRpTokens - 1) / kRpTokens;
    const int cluster = (int)blockIdx.x >> log2_c, rank = (int)blockIdx.x & (C - 1);
    if (cluster >= token_blocks) {
        // the remaining blocks prepare the up-projection's operand (see gemm_prologue_kernel)
        pdl_wait();
        if constexpr (JT > 0) gate_operand(x, r, ((int)blockIdx.x - token_blocks * C) * kRpThreads + (int)threadIdx.x);
        return;
    }
    const int K = p.K, M = p.M, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, t = lane & 3;
    const RpLayout L = rp_layout(K, r, log2_c);
    const int m0 = cluster * kRpTokens, k0 = rank * L.per < K ? rank * L.per : K, cols = K - k0 < L.per ? K - k0 : L.per;
    const int rows = M - m0 < kRpTokens ? M - m0 : kRpTokens;
    const uint32_t s0 = dsmem_u32(rp_smem), bar_x = s0, bar_stat = s0 + 8, bar_amax = s0 + 16, bar_h = s0 + 24, bar_sum = s0 + 32;
    const uint8_t *x_s = rp_smem + L.off_x;

    if (warp == 0) {
        if (lane == 0) {
            for (int i = 0; i < 5; ++i) dmbar_init(s0 + 8 * i, 1);
            asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
            announce(bar_stat, LN ? (uint32_t)(C * kRpTokens * 16) : 0u);
            announce(bar_amax, (uint32_t)(C * kRpTokens * 4));
            announce(bar_h, (uint32_t)(kRpTokens * r * 4));      // C ranks x 16 / C tokens
            announce(bar_sum, (uint32_t)(kRpTokens * 4));
        }
        __syncwarp();
        cluster_arrive_relaxed();
        pdl_wait();  // x, and the workspace this kernel overwrites, belong to earlier work
        if (lane == 0) announce(bar_x, (uint32_t)(rows * cols * 2));
        __syncwarp();
        if (lane < rows && cols > 0)
            bulk_load_announced(s0 + L.off_x + lane * L.pitch, p.x + (size_t)(m0 + lane) * K + k0, (uint32_t)(cols * 2), bar_x);
        __syncwarp();
    } else {
        cluster_arrive_relaxed();
    }
    const int nch = cols >> 5;
    constexpr int JH = JT * kRpParts / W;  // a warp's column tiles of H
    const int part = warp & (kRpParts - 1), j0 = (warp / kRpParts) * 8 * JH;
    const __half *arow = JT > 0 ? p.At + (size_t)(j0 + g) * K + k0 + 8 * t : nullptr;
    uint4 av[JT > 0 ? JH : 1];
    auto load_a = [&](int c) {
        if constexpr (JT > 0)
#pragma unroll
            for (int jt = 0; jt < JH; ++jt) av[jt] = c < nch ? *reinterpret_cast<const uint4 *>(arow + (size_t)8 * jt * K + 32 * c) : make_uint4(0u, 0u, 0u, 0u);
    };
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();  // (the launch that follows finds room only as these blocks leave; let in at the end it came 0.1 to 0.4 us later)
    load_a(part);  // this warp's first chunk of A^T (like every read of this path, after the wait)
    bool ok = warp_wait(bar_x, status, 0x680u);
    cluster_wait_acquire();  // every CTA of the cluster has started

    // ---- statistics --------------------------------------------------------------------------------------------
    const int nu = cols >> 3;  // 16-byte units of a row's slice
    auto has_row = [&](int q) { return warp + W * q < rows; };
    auto unit = [&](int q, int i) { return *reinterpret_cast<const uint4 *>(x_s + (warp + W * q) * L.pitch + 16 * i); };
    float mean[TPW] = {}, rstd[TPW] = {};
    // the normalised values of unit i of the warp's tokens (the weights are read once for all of them)
    auto ln_each = [&](int i, auto &&body) {
        const float4 *w4 = reinterpret_cast<const float4 *>(fe.ln_w + k0 + 8 * i), *b4 = reinterpret_cast<const float4 *>(fe.ln_b + k0 + 8 * i);
        const float4 w0 = w4[0], w1 = w4[1], b0 = b4[0], b1 = b4[1];
        const float w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w}, b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            if (!has_row(q)) continue;
            float f[8], xn[8];
            unpack8(unit(q, i), f);
#pragma unroll
            for (int e = 0; e < 8; ++e) xn[e] = ln_value(f[e], mean[q], rstd[q], w[e], b[e]);
            body(q, xn);
        }
    };
    if constexpr (LN) {
        // Mean and variance in one pass, in double, of x - x[0]: see hgf_decode_small.cu.  A bf16 pattern moved to the top
        // of a double is x 2^-896 (subnormals too), so one fused multiply-add gives x - x[0] without a conversion; infinities and
        // NaNs, which that would miss, make the sum a NaN.
        // (four partial sums each: the additions of one are a chain)
        double first[TPW], sum[TPW][4] = {}, sum2[TPW][4] = {};
        uint32_t top[TPW] = {};
#pragma unroll
        for (int q = 0; q < TPW; ++q) first[q] = has_row(q) ? (double)__bfloat162float(p.x[(size_t)(m0 + warp + W * q) * K]) : 0.0;
        for (int i = lane; i < nu; i += 32)
#pragma unroll
            for (int q = 0; q < TPW; ++q) {
                if (!has_row(q)) continue;
                const uint4 u = unit(q, i);
                top[q] = absmax8_bits(top[q], u);
                const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const uint32_t hi = (e & 1) ? (w[e >> 1] & 0x80000000u) | ((w[e >> 1] & 0x7fff0000u) >> 3)
                                                : ((w[e >> 1] & 0x8000u) << 16) | ((w[e >> 1] & 0x7fffu) << 13);
                    const double d = fma(__hiloint2double((int)hi, 0), 0x1p896, -first[q]);
                    sum[q][e & 3] += d;
                    sum2[q][e & 3] = fma(d, d, sum2[q][e & 3]);
                }
            }
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            double s = (top[q] & 0xffffu) >= 0x7f80u || top[q] >= 0x7f800000u ? __longlong_as_double(0x7ff8000000000000ll)
                                                                                         : (sum[q][0] + sum[q][1]) + (sum[q][2] + sum[q][3]),
                   ss = (sum2[q][0] + sum2[q][1]) + (sum2[q][2] + sum2[q][3]);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                s += __shfl_xor_sync(0xffffffffu, s, o);
                ss += __shfl_xor_sync(0xffffffffu, ss, o);
            }
            if (lane < C) {
                const uint32_t dst = s0 + L.off_stat + (rank * kRpTokens + warp + W * q) * 16;
                st_async_b64(dst, bar_stat, (uint32_t)lane, (uint64_t)__double_as_longlong(s));
                st_async_b64(dst + 8, bar_stat, (uint32_t)lane, (uint64_t)__double_as_longlong(ss));
            }
        }
        ok = warp_wait(bar_stat, status, 0x681u) && ok;
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            double s = 0.0, ss = 0.0;
            for (int k = 0; k < C; ++k) {
                const double2 v = *reinterpret_cast<const double2 *>(rp_smem + L.off_stat + (k * kRpTokens + warp + W * q) * 16);
                s += v.x;
                ss += v.y;
            }
            const double dm = s / (double)K, v0 = ss / (double)K - dm * dm, var = v0 < 0.0 ? 0.0 : v0;  // (NaN stays NaN)
            mean[q] = (float)(first[q] + dm);
            rstd[q] = (float)rsqrt(var + (double)fe.eps);
        }
    }
    uint32_t bits[TPW] = {};
    if constexpr (LN) {
        float a[TPW] = {};
#pragma unroll 2
        for (int i = lane; i < nu; i += 32)
            ln_each(i, [&](int q, const float (&xn)[8]) {
#pragma unroll
                for (int e = 0; e < 8; ++e) a[q] = fmaxf(a[q], fabsf(xn[e]));
            });
#pragma unroll
        for (int q = 0; q < TPW; ++q) bits[q] = __float_as_uint(a[q]);
    } else {
        uint32_t acc[TPW] = {};
        for (int i = lane; i < nu; i += 32)
#pragma unroll
            for (int q = 0; q < TPW; ++q)
                if (has_row(q)) acc[q] = absmax8_bits(acc[q], unit(q, i));
#pragma unroll
        for (int q = 0; q < TPW; ++q) {
            bits[q] = __float_as_uint(absmax_bits_to_float(acc[q]));
            if (bits[q] > 0x7f800000u) bits[q] = 0u;  // a NaN does not count, as in fmaxf
        }
    }
#pragma unroll
    for (int q = 0; q < TPW; ++q) {
        bits[q] = __reduce_max_sync(0xffffffffu, bits[q]);
        if (lane < C) st_async_f32(s0 + L.off_amax + (rank * kRpTokens + warp + W * q) * 4, bar_amax, (uint32_t)lane, __uint_as_float(bits[q]));
    }

    // ---- x A over the slice, while the maxima travel: tokens are the 16-row operand, 8 columns of H the 8-column operand --
    if constexpr (JT > 0) {
        float acc[JH][4];
#pragma unroll
        for (int jt = 0; jt < JH; ++jt)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[jt][c] = 0.0f;
        for (int c = part; c < nch; c += kRpParts) {
            const uint8_t *xr = x_s + g * L.pitch + 64 * c + 16 * t;
            const uint4 x0 = *reinterpret_cast<const uint4 *>(xr), x1 = *reinterpret_cast<const uint4 *>(xr + 8 * L.pitch);
            uint4 a_now[JH];
#pragma unroll
            for (int jt = 0; jt < JH; ++jt) a_now[jt] = av[jt];
            load_a(c + kRpParts);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                // elements 2 i and 2 i + 1 of this lane's eight take the k slots t and t + 4 of MMA i
                const uint32_t w0 = (&x0.x)[i], w1 = (&x1.x)[i];
#pragma unroll
                for (int jt = 0; jt < JH; ++jt) {
                    const float2 bf = __half22float2(*reinterpret_cast<const __half2 *>(&(&a_now[jt].x)[i]));
                    mma_tf32(acc[jt], w0 << 16, w1 << 16, w0 & 0xffff0000u, w1 & 0xffff0000u, __float_as_uint(bf.x), __float_as_uint(bf.y));
                }
            }
        }
        float *sums = reinterpret_cast<float *>(rp_smem + L.off_part) + (size_t)part * kRpTokens * r + j0;
#pragma unroll
        for (int jt = 0; jt < JH; ++jt) {
            *reinterpret_cast<float2 *>(sums + g * r + 8 * jt + 2 * t) = make_float2(acc[jt][0], acc[jt][1]);
            *reinterpret_cast<float2 *>(sums + (g + 8) * r + 8 * jt + 2 * t) = make_float2(acc[jt][2], acc[jt][3]);
        }
        __syncthreads();
        const float *all = reinterpret_cast<const float *>(rp_smem + L.off_part);
        for (int e = tid; e < kRpTokens * r; e += kRpThreads) {  // to the CTA that owns the token, in warp order
            float z = 0.0f;
#pragma unroll
            for (int w = 0; w < kRpParts; ++w) z += all[w * kRpTokens * r + e];
            st_async_f32(s0 + L.off_slots + (rank * kRpTokens * r + e) * 4, bar_h, (uint32_t)((e / r) >> (4 - log2_c)), z);
        }
        __syncwarp();
    }

    // ---- codes ------------------------------------------------------------------------------------------------
    ok = warp_wait(bar_amax, status, 0x682u) && ok;
    float gm[TPW], scale[TPW];
    int sums[TPW] = {};
#pragma unroll
    for (int q = 0; q < TPW; ++q) {
        uint32_t most = 0u;
        for (int k = 0; k < C; ++k) {
            const uint32_t v = *reinterpret_cast<const uint32_t *>(rp_smem + L.off_amax + (k * kRpTokens + warp + W * q) * 4);
            most = v > most ? v : most;
        }
        gm[q] = fmaxf(__uint_as_float(most), 1e-5f);
        scale[q] = __fdiv_rn(127.0f, gm[q]);
    }
    auto store = [&](int q, int i, const uint2 &o) {
        const size_t at = ((size_t)(m0 + warp + W * q) * K + k0) / 8 + i;
        reinterpret_cast<uint2 *>(p.xq)[at] = o;
        if (p.dbg_xq) reinterpret_cast<uint2 *>(p.dbg_xq)[at] = o;
    };
    if (ok) {
        if constexpr (LN) {
#pragma unroll 2
            for (int i = lane; i < nu; i += 32) ln_each(i, [&](int q, const float (&xn)[8]) { store(q, i, ln_codes8(xn, scale[q], sums[q])); });
        } else {
            QuantScale qs[TPW];
#pragma unroll
            for (int q = 0; q < TPW; ++q) qs[q] = make_quant_scale(gm[q]);
            for (int i = lane; i < nu; i += 32)
#pragma unroll
                for (int q = 0; q < TPW; ++q)
                    if (has_row(q)) store(q, i, quant8(unit(q, i), qs[q], sums[q]));
        }
    }
#pragma unroll
    for (int q = 0; q < TPW; ++q) {
        const int ml = warp + W * q, owner = ml >> (4 - log2_c), sum = __reduce_add_sync(0xffffffffu, sums[q]);
        if (lane == 0) st_async_f32(s0 + L.off_sum + (rank * kRpTokens + ml) * 4, bar_sum, (uint32_t)owner, __int_as_float(sum));
        // (the CTA that owns the token writes its values)
        if (lane == 0 && owner == rank && ml < rows && ok) {
            const int m = m0 + ml;
            p.gamma_x[m] = gm[q];
            if (x.tok_sc) x.tok_sc[m] = gm[q] * x.gw_over_127;
            if (p.dbg_gamma_x) p.dbg_gamma_x[m] = gm[q];
            if constexpr (LN) {
                if (fe.dbg_mean) fe.dbg_mean[m] = mean[q];
                if (fe.dbg_rstd) fe.dbg_rstd[m] = rstd[q];
            }
        }
    }

    const int own = kRpTokens >> log2_c, t0 = rank * own;  // this CTA's tokens of the block
    if constexpr (JT > 0) {
        ok = warp_wait(bar_h, status, 0x683u) && ok;
        const float *slots = reinterpret_cast<const float *>(rp_smem + L.off_slots);
        for (int e = tid; e < own * 64; e += kRpThreads) {
            const int ml = t0 + (e >> 6), j = e & 63, m = m0 + ml;
            float h = 0.0f;
            if (j < r) {
                float z = 0.0f;
                for (int k = 0; k < C; ++k) z += slots[(k * kRpTokens + ml) * r + j];
                h = (p.flags & HGF_FLAG_NO_SILU) ? z : silu_f(z);
            }
            if (ml < rows && ok) {
                if (j < r) {
                    p.h[(size_t)m * r + j] = h;
                    if (p.dbg_h) p.dbg_h[(size_t)m * r + j] = h;
                }
                if (p.h16) p.h16[(size_t)m * 64 + j] = __float2half_rn(h);  // (zeros past r)
            }
        }
    }
    ok = warp_wait(bar_sum, status, 0x684u) && ok;
    if (tid < own && t0 + tid < rows && ok && p.row_sum) {
        int sum = 0;
        for (int k = 0; k < C; ++k) sum += *reinterpret_cast<const int *>(rp_smem + L.off_sum + (k * kRpTokens + t0 + tid) * 4);
        p.row_sum[m0 + t0 + tid] = sum;
    }
    if (!ok)  // bounded drain of what is still on its way into this CTA's memory
        for (uint32_t i = 0; i < (1u << 16); ++i) {
            bool all = true;
            for (int b = 0; b < 5; ++b) all = all && dmbar_try_wait(s0 + 8 * b, 0);
            if (all) break;
        }
}

// Where it is used, the cluster size and `least` (bytes of shared memory): see launch_rows_prologue.
template <int JT, bool LN, int TPW, int PER_SM = 0>
static cudaError_t launch_rows_prologue_jt(const PrologueParams &p, const GemmPrologueExtra &x, const FrontEnd &fe, int log2_c, size_t least, cudaStream_t stream) {
    constexpr int kRpThreads = 512 / TPW;
    static std::atomic<unsigned long long> attr_done{0};
    const RpLayout L = rp_layout(p.K, p.r, log2_c);
    cudaError_t e = ensure_dynamic_smem(rows_prologue_kernel<JT, LN, TPW, PER_SM>, kRpSmemLimit, attr_done);
    if (e != cudaSuccess) return e;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    const int C = 1 << log2_c, gate_blocks = (p.r > 0 && x.gb16) ? (x.N * 8 + kRpThreads - 1) / kRpThreads : 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = prologue_cfg(((p.M + kRpTokens - 1) / kRpTokens) * C + (gate_blocks + C - 1) / C * C, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
    cfg.blockDim = dim3(kRpThreads);
    cfg.dynamicSmemBytes = (size_t)L.smem > least ? (size_t)L.smem : least;
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs].val.clusterDim.x = (unsigned)C;
    attr[cfg.numAttrs].val.clusterDim.y = 1;
    attr[cfg.numAttrs].val.clusterDim.z = 1;
    ++cfg.numAttrs;
    e = cudaLaunchKernelEx(&cfg, rows_prologue_kernel<JT, LN, TPW, PER_SM>, p, x, fe, log2_c, status);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <int JT, int W, int TOK>
static cudaError_t launch_gemm_prologue_jt(const PrologueParams &p, const GemmPrologueExtra &x, int blocks, cudaStream_t stream) {
    // Never more than two blocks per SM (the launcher spreads the rows over twice the SM count of
    // blocks, from rank 48 on one): blocks that start as SMs come free at the tail of the preceding launch would otherwise
    // pile up four to an SM on the first SMs free and leave the others idle.
    constexpr int smem = fp_smem_bytes(TOK, 8 * JT) > 80 * 1024 ? fp_smem_bytes(TOK, 8 * JT) : 80 * 1024;
    static std::atomic<unsigned long long> attr_done{0};
    {
        cudaError_t e = ensure_dynamic_smem(gemm_prologue_kernel<JT, W, TOK>, smem, attr_done);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = prologue_cfg(blocks, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
    cfg.blockDim = dim3(32 * W);
    cfg.dynamicSmemBytes = smem;
    cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_prologue_kernel<JT, W, TOK>, p, x);
    return e != cudaSuccess ? e : cudaGetLastError();
}

// The cluster form above where it is the better one; cudaErrorNotSupported where it is not.  Microseconds of the whole layer
// call in a captured chain, the other kernels / this one:
//  - 2048 -> 2048, r = 32: 16.0 / 12.4 at M = 17, 18.4 / 14.8 at M = 512, 25.9 / 24.7 at M = 2000, 38.0 / 40.0 at 4096 (its slices
//    then come in several waves and read A^T more often than 32-token blocks do); K = 512: 9.2 / 9.5 at M = 17;
//  - 5632 -> 2048: 29.6 / 19.1 at M = 17, 34.5 / 23.1 at M = 512; 11008 -> 4096, r = 64: 69 / 32 at M = 17, 94 / 82 at M = 1024,
//    133 / 142 at M = 2000 (eight CTAs a cluster for its size alone: above four CTAs an SM it is left);
//  - rank 16, short rows, K -> 1024: 19.6 / 18.2 at K = 2048 and M = 1200, but 19.9 / 20.7 at M = 1600, 16.0 / 17.1 at K = 1280;
//    32.3 / 25.3 at K = 4096 and M = 1600;
//  - with a LayerNorm, 2048 -> 2048: 23.8 / 14.3 at M = 64, 51.2 / 52.2 at M = 4096; r = 64, 11008 -> 1024: 105 / 26 at M = 64,
//    127 / 123 at M = 2048 (no limit of CTAs there: the other kernels take two launches);
//  - with a LayerNorm and without a correction, 4096 -> 1024: 14.0 / 16.7 at M = 17, 25.2 / 16.7 at M = 64, 82.6 / 62.4 at
//    M = 4096.  Short rows: 512 -> 1024 9.6 / 10.2 at M = 130, 10.6 / 11.1 at 700, 13.3 / 12.3 at 1280, 13.5 / 12.2 at 2000; 512 -> 3040
//    11.1 / 13.9 at M = 500 (96 output tiles), 12.7 / 13.6 at 640 (120), 16.5 / 13.9 at 700 (144); 512 -> 5632 12.5 / 14.2 at M = 300 (132);
//    768 -> 1024 12.9 / 11.7 at M = 700, 15.4 / 18.1 at 1500, 22.9 / 21.4 at 3000; 768 -> 3040 13.0 / 14.3 at M = 500, a quarter less
//    at 700 to 1168.  Long rows in one CTA: K = 3072 72 / 68 at M = 5000, 80.4 / 82.6 at 8192.
// At most two CTAs an SM (by asking for 80 KB) where that many run at once: CTAs start as the SMs come free at the end of the launch before, and
// with room for three the first SMs took three and others none.  As they come / two: 2048 -> 2048, r = 32, LayerNorm 32.0 / 26.7 at M = 2000, without a
// correction 24.1 / 18.0, r = 32 without a LayerNorm 16.6 / 14.9 at M = 1000.  29 clusters of eight and more do need room for three: 4096 -> 2048
// 18.0 / 19.9 at M = 500 (K <= 2048 takes clusters of four there: 1024 -> 2048, r = 16 12.0 / 10.2).
// Sixteen warps a CTA, a token each, or eight with two each, eight / sixteen: r = 32 2048 -> 2048 13.0 / 12.4 at M = 17, 14.9 / 14.7 at 1000, 20.6 / 19.9 at 1184,
// 22.3 / 21.4 at 2300; with a LayerNorm 12.9 / 12.4, 18.5 / 18.4, 25.7 / 26.1, 27.4 / 27.7 (slices of 1024 columns), 4096 -> 4096 31.7 / 32.5 at M = 800 and
// 49.3 / 48.5 at 1184 (of 2048); without a correction 2048 -> 1024 11.8 / 11.4 at M = 200, 17.4 / 17.9 at 1184.  Ranks of 64 leave room for one CTA of
// sixteen warps an SM: 13.3 / 11.6 at M = 200, 13.6 / 15.9 at 440, 23.3 / 21.1 at 1184, 24.1 / 28.4 at 2000; with a LayerNorm 15.0 / 13.6, 17.1 / 19.6, 25.8 / 23.9,
// 30.6 / 33.5; rank 48 11.4 / 10.7 at M = 17, 12.7 / 12.7 at 440, 15.1 / 15.4 at 800.
// Batches: as many blocks of tokens as SMs; the other kernels / this one at M = 2200 26.9 / 21.8 for 2048 -> 2048, 52.5 / 45.5 for 5632 -> 2048, 37.9 / 28.7 with a
// LayerNorm, r = 64 28.3 / 25.0; at M = 3000 31.6 / 32.5, 64.0 / 65.2, 44.4 / 42.5, 35.6 / 38.3; with a LayerNorm 51.2 / 48.5 at 4096, 65.4 / 70.4 at 6000.
// Cluster size: CTAs for every SM, two of them on one if they fit; one step smaller where that many don't run at once: 1024 -> 1024,
// M = 1168, r = 48 16.4 -> 15.0 us, M = 570 15.4 -> 13.9; 8192 -> 1024, M = 525 26.6 -> 28.5.
struct RpForm {
    int c;         // log2 of the CTAs of a cluster
    bool wide;     // sixteen warps a CTA (a token each), or eight
    size_t least;  // bytes of shared memory at least
};
// Whether rows_prologue_kernel takes a batch, and in which form.
static bool rp_form(int M, int K, int N, int r, bool ln, int sms, RpForm *f) {
    const int blocks = (M + kRpTokens - 1) / kRpTokens;
    int c = 0;
    while (c < 3 && (blocks << c) < sms) ++c;
    // (registers: two CTAs an SM at most; 33 clusters of eight or 71 of four run at once on 148 SMs, more take a second round, which
    // only long slices are worth)
    if ((r >= 48 || (ln && r == 32)) && ((c == 3 && K <= 2048 && (blocks << c) > 2 * sms - sms / 4) || (c == 2 && (blocks << c) > 2 * sms - sms / 16))) --c;
    const int crowded = 2 * sms - 2 * sms / 5;  // (29 clusters of eight and more, with the blocks for the up-projection's operand)
    if (r > 0 && r <= 32 && c == 3 && K <= 2048 && (blocks << 3) > crowded) --c;
    while (c < 3 && rp_layout(K, r, c).smem > 110 * 1024) ++c;  // two CTAs on an SM
    if (rp_layout(K, r, c).smem > kRpSmemLimit) return false;
    const int ctas = blocks << c, slice = K >> c;
    bool take;
    if (r == 0) {
        take = M >= 64 && (M <= 7168 || c > 0 || K <= 2048);
        if (K < 896) {  // (by the output tiles of the launch that follows: in one round of them or more)
            const int tiles = ((M + 127) / 128) * ((N + 127) / 128);
            if (M < 640) take = take && tiles > sms;
            else if (2 * blocks < sms) take = take && (K >= 640 || tiles > sms * 5 / 6);
            else take = take && (K <= 512 || M >= 1800 || tiles > sms);
        }
        take = take && ln;
    } else {
        take = (blocks <= sms || (ln && r <= 32 && M <= 4096)) && K >= 1024;
        if (!ln) take = take && ctas <= 4 * sms && (r > 16 || K > 2048 || M <= 1280);
    }
    if (!take) return false;
    const bool three = r > 0 && r <= 32 && c == 3 && ctas > crowded;  // CTAs an SM
    f->c = c;
    if (three) f->wide = false;
    else if (r <= 32) f->wide = !ln || c == 3 || slice <= 512 || (r > 0 && slice >= 2048);
    else if (ln) f->wide = ctas <= sms;
    else if (r == 48) f->wide = c == 3;
    else f->wide = ctas <= (c == 3 ? sms - sms / 6 : (c == 2 ? sms - sms / 10 : sms));
    f->least = !three && ctas <= 2 * sms ? 80 * 1024 : 0;
    return true;
}
// (for the tests; out: log2 of the CTAs of a cluster, sixteen warps, bytes of shared memory at least)
extern "C" int hgf_internal_rows_prologue_form(int32_t M, int32_t K, int32_t N, int32_t r, int32_t ln, int32_t sms, int32_t *out) {
    RpForm f = {};
    if (!rp_form(M, K, N, r, ln != 0, sms, &f)) return 0;
    out[0] = f.c; out[1] = f.wide; out[2] = (int32_t)f.least;
    return 1;
}

static cudaError_t launch_rows_prologue(const PrologueParams &p, const GemmPrologueExtra &x, const FrontEnd *fe, cudaStream_t stream) {
    const int sms = device_sm_count();
    if (!sms) return cudaErrorInvalidDevice;
    RpForm f = {};
    if (!rp_form(p.M, p.K, x.N, p.r, fe != nullptr, sms, &f)) return cudaErrorNotSupported;
    const FrontEnd none = {};
    const int c = f.c;
    const bool wide = f.wide;
    const size_t least = f.least;
    switch (p.r) {
        case 0:
            return wide ? launch_rows_prologue_jt<0, true, 1>(p, x, *fe, c, least, stream) : launch_rows_prologue_jt<0, true, 2>(p, x, *fe, c, least, stream);
        case 16:
            if (fe) return wide ? launch_rows_prologue_jt<2, true, 1>(p, x, *fe, c, least, stream) : launch_rows_prologue_jt<2, true, 2>(p, x, *fe, c, least, stream);
            return wide ? launch_rows_prologue_jt<2, false, 1>(p, x, none, c, least, stream) : launch_rows_prologue_jt<2, false, 2>(p, x, none, c, least, stream);
        case 32:
            if (fe) return wide ? launch_rows_prologue_jt<4, true, 1>(p, x, *fe, c, least, stream) : launch_rows_prologue_jt<4, true, 2>(p, x, *fe, c, least, stream);
            return wide ? launch_rows_prologue_jt<4, false, 1>(p, x, none, c, least, stream) : launch_rows_prologue_jt<4, false, 2>(p, x, none, c, least, stream);
        case 48:
            if (fe) return wide ? launch_rows_prologue_jt<6, true, 1>(p, x, *fe, c, least, stream) : launch_rows_prologue_jt<6, true, 2>(p, x, *fe, c, least, stream);
            return wide ? launch_rows_prologue_jt<6, false, 1>(p, x, none, c, least, stream) : launch_rows_prologue_jt<6, false, 2>(p, x, none, c, least, stream);
        case 64:
            if (!fe) return wide ? launch_rows_prologue_jt<8, false, 1>(p, x, none, c, least, stream) : launch_rows_prologue_jt<8, false, 2>(p, x, none, c, least, stream);
            return wide ? launch_rows_prologue_jt<8, true, 1>(p, x, *fe, c, least, stream) : launch_rows_prologue_jt<8, true, 2, 2>(p, x, *fe, c, least, stream);
        default: return cudaErrorInvalidValue;
    }
}

// Quantisation and (r > 0) LoRA down-projection of the GEMM path, plus gate * B^T for its epilogue.
cudaError_t launch_gemm_prologue(const PrologueParams &p, const GemmPrologueExtra &x, cudaStream_t stream) {
    if (p.xq && p.r > 0) {
        const cudaError_t e = launch_rows_prologue(p, x, nullptr, stream);
        if (e != cudaErrorNotSupported) return e;
    }
    // Tokens per block: as many blocks as are resident at once share the rows evenly; beyond that a
    // block takes its full 32 (rank 48: as many rounds as blocks of 64 need, evenly; see the kernel).
    const int sm_count = device_sm_count();
    if (!sm_count) return cudaErrorInvalidDevice;
    const bool wide = p.r >= 48, big = p.r == 48 && p.M > 32 * sm_count;
    const int per_sm = wide ? 1 : 2, most = big ? 64 : 32;  // blocks that fit an SM (shared memory: 138 KB and more from rank 48 on)
    const int rounds = big ? (p.M + 64 * sm_count - 1) / (64 * sm_count) : 1, shares = per_sm * sm_count * rounds;
    int tpb = (p.M + shares - 1) / shares;
    tpb = (tpb + 3) / 4 * 4;
    tpb = tpb < 8 ? 8 : (tpb > most ? most : tpb);
    GemmPrologueExtra xx = x;
    xx.tokens_per_block = tpb;
    // The rounding pass as a second launch where there is enough of x to pay for a launch: it then runs at twice
    // the occupancy, and the GEMM's set-up overlaps it (measured per layer, M = 8192: 118.8 -> 117.0 us at
    // K = 2048, 141.3 -> 134.3 us at K = 5632; M = 4096: 209.7 -> 205.1 us at K = 11008, unchanged at K = 4096).
    const size_t x_bytes = (size_t)p.M * p.K * 2;
    xx.split_round = (p.xq && p.r > 0 && x_bytes >= ((size_t)8 << 20)) ? 1 : 0;
    const int threads = wide ? 512 : 256;
    const int blocks = (p.M + tpb - 1) / tpb + ((p.r > 0 && x.gb16) ? (x.N * 8 + threads - 1) / threads : 0);
    cudaError_t e;
    switch (p.r) {
        case 0: e = launch_gemm_prologue_jt<0, 8, 32>(p, xx, blocks, stream); break;
        case 16: e = launch_gemm_prologue_jt<2, 8, 32>(p, xx, blocks, stream); break;
        case 32: e = launch_gemm_prologue_jt<4, 8, 32>(p, xx, blocks, stream); break;
        case 48: e = big ? launch_gemm_prologue_jt<6, 16, 64>(p, xx, blocks, stream) : launch_gemm_prologue_jt<6, 16, 32>(p, xx, blocks, stream); break;
        case 64: e = launch_gemm_prologue_jt<8, 16, 32>(p, xx, blocks, stream); break;
        default: return cudaErrorInvalidValue;
    }
    count_launch();
    if (e == cudaSuccess && xx.split_round) {
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = prologue_cfg((p.M + kWarps - 1) / kWarps, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
        e = cudaLaunchKernelEx(&cfg, round_rows_kernel, p);
        count_launch();
        if (e == cudaSuccess) e = cudaGetLastError();
    }
    return e;
}

// Quantisation alone.  Many rows: one warp per row while a row fits its registers, else the GEMM
// path's prologue kernel without its LoRA part; few rows: one block per row.
cudaError_t launch_quant(const PrologueParams &p, const GemmPrologueExtra &x, cudaStream_t stream) {
    const int nv = p.K / 8, row_blocks = (p.M + kWarps - 1) / kWarps;
    if (p.M >= 256 && nv <= 32 * 8) {
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = prologue_cfg(row_blocks, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
        cudaError_t e = cudaLaunchKernelEx(&cfg, quant_rows_kernel<8>, p, x);
        if (e != cudaSuccess) return e;
    } else if (p.M >= 256 && nv <= 32 * 16) {
        cudaLaunchAttribute attr[1];
        cudaLaunchConfig_t cfg = prologue_cfg(row_blocks, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
        cudaError_t e = cudaLaunchKernelEx(&cfg, quant_rows_kernel<16>, p, x);
        if (e != cudaSuccess) return e;
    } else if (p.M >= 64) {
        PrologueParams q = p;
        q.r = 0;
        return launch_gemm_prologue(q, x, stream);
    } else {
        quant_kernel<<<p.M, kThreads, 0, stream>>>(p, x);
    }
    count_launch();
    return cudaGetLastError();
}

cudaLaunchConfig_t prologue_cfg(int blocks, bool pdl, cudaStream_t stream, cudaLaunchAttribute *attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cfg;
}

cudaError_t launch_decode_prologue(const PrologueParams &p, bool pdl, cudaStream_t stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = prologue_cfg(p.M + (p.r / 16) * (p.hpart ? p.nslices : 1), pdl, stream, attr);
    cudaError_t e = cudaLaunchKernelEx(&cfg, decode_prologue_kernel, p);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_decode_prologue_ln(const PrologueParams &p, const FrontEnd &fe, bool pdl, cudaStream_t stream) {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = prologue_cfg(p.M + (p.r / 16) * (p.hpart ? p.nslices : 1), pdl, stream, attr);
    cudaError_t e = cudaLaunchKernelEx(&cfg, decode_prologue_ln_kernel, p, fe);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_gemm_prologue_ln(const PrologueParams &p, const GemmPrologueExtra &x, const FrontEnd &fe, cudaStream_t stream) {
    const cudaError_t whole = launch_rows_prologue(p, x, &fe, stream);
    if (whole != cudaErrorNotSupported) return whole;
    if (p.r) {  // the correction path's part on the raw tokens, its own quantisation switched off
        PrologueParams lora_only = p;
        lora_only.xq = nullptr;
        const cudaError_t e = launch_gemm_prologue(lora_only, x, stream);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchAttribute attr[1];
    const bool by_warp = p.row_sum != nullptr && p.M >= 64;  // many rows: one warp each; few: one block each
    cudaLaunchConfig_t cfg = prologue_cfg(by_warp ? (p.M + kWarps - 1) / kWarps : p.M, !(p.flags & HGF_FLAG_NO_PDL), stream, attr);
    cudaError_t e = by_warp ? cudaLaunchKernelEx(&cfg, ln_quant_rows_kernel, p, x, fe) : cudaLaunchKernelEx(&cfg, ln_quant_kernel, p, x, fe);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// A CTA works one row after the other, eight warps eight rows at a time but each slowly: microseconds of a group's forward, r = 32,
// rows by warps / by CTAs: K = 512 19.4 / 18.6 with 240 rows, 20.3 / 20.7 with 320, 25.0 / 41.3 with 1728; K = 1024 22.9 / 22.3 with 400,
// 23.3 / 24.4 with 448; K = 2048 30.0 / 26.7 with 320, 29.0 / 27.6 with 448, 30.4 / 30.7 with 576, 73 / 85 with 1728; K = 3072
// 37.5 / 36.7 with 576, 41.0 / 41.9 with 720.
bool group_rows_by_cta(const QuantItem *items, int n) {
    const int sms = device_sm_count();
    int K = 0;
    for (int i = 0; i < n; ++i) K = items[i].K > K ? items[i].K : K;
    return 4 * n <= sms * (K >= 3072 ? 18 : (K >= 2048 ? 14 : (K >= 1024 ? 11 : 8)));
}

template <int NT, bool LN_WARPS>
static cudaError_t launch_prologue_group_nt(const QuantItem *d_quant_items, int n_ln, int n_quant, const LoraItem *d_lora_items, int n_lora, bool pdl,
                                            cudaStream_t stream) {
    static std::atomic<unsigned long long> attr_done{0};
    const int sm_count = device_sm_count();
    if (!sm_count) return cudaErrorInvalidDevice;
    constexpr int smem = kPgWarps * (16 / NT) * (1024 + 512 * NT);
    cudaError_t e = ensure_dynamic_smem(decode_prologue_group_kernel<NT, LN_WARPS>, smem, attr_done);
    if (e != cudaSuccess) return e;
    const int most = n_lora > n_quant - n_ln ? n_lora : n_quant - n_ln;
    int blocks = (most + kPgWarps - 1) / kPgWarps + n_ln;  // CTAs of their own for the first n_ln rows
    blocks = blocks < sm_count ? blocks : sm_count;
    if (blocks < 1) blocks = 1;
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg = prologue_cfg(blocks, pdl, stream, attr);
    cfg.blockDim = dim3(kPgThreads);
    cfg.dynamicSmemBytes = smem;
    e = cudaLaunchKernelEx(&cfg, decode_prologue_group_kernel<NT, LN_WARPS>, d_quant_items, n_ln, n_quant, d_lora_items, n_lora);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_decode_prologue_group(const QuantItem *d_quant_items, int n_ln, bool ln_warps, int n_quant, const LoraItem *d_lora_items, int n_lora,
                                         int max_M, bool pdl, cudaStream_t stream) {
    if (max_M <= 8)
        return ln_warps ? launch_prologue_group_nt<1, true>(d_quant_items, n_ln, n_quant, d_lora_items, n_lora, pdl, stream)
                        : launch_prologue_group_nt<1, false>(d_quant_items, n_ln, n_quant, d_lora_items, n_lora, pdl, stream);
    return ln_warps ? launch_prologue_group_nt<2, true>(d_quant_items, n_ln, n_quant, d_lora_items, n_lora, pdl, stream)
                    : launch_prologue_group_nt<2, false>(d_quant_items, n_ln, n_quant, d_lora_items, n_lora, pdl, stream);
}

}  // namespace hgf
