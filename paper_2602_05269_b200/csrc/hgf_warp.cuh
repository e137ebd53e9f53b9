// Warp-level pieces of the decode and prologue kernels: reductions, the quantiser, the LayerNorm arithmetic, warp MMA,
// mbarrier and bulk-copy wrappers (sm_100a).
#pragma once

#include "hgf_common.cuh"

namespace hgf {

constexpr unsigned long long kDecWaitLimitNs = 2000000000ull;  // bounded waits give up after two seconds

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ int warp_sum_i(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Round-to-nearest-even of the exact quotient 127 x / gamma for a bf16 x.
//
// Reference form: 127 x is exact in fp32, the IEEE division is correctly rounded and k + 1/2 is
// representable, so rintf of the rounded quotient equals the rounding of the exact one.
__device__ __forceinline__ int quant1_div(float x, float gamma) {
    float q = rintf(__fdiv_rn(127.0f * x, gamma));
    q = fminf(fmaxf(q, -127.0f), 127.0f);
    return __float2int_rn(q);
}
// Division- and conversion-free form, for gamma = max |x| over bf16 values (so gamma is a bf16 value
// itself, i.e. not the 1e-5 floor).  Adding 1.5 * 2^23 in one fma rounds x * (127 / gamma) to an
// integer (nearest, ties to even) in the low mantissa bits - a candidate that can only be wrong on
// an exact tie of the true quotient.  The residual 127 x - q gamma is exact in one fma (127 x and
// q gamma each have at most 15 significant bits), and the exact quotient is q + residual / gamma:
// off a tie the candidate is always right (checked over every pair of bf16 mantissas and every
// exponent gap in exact arithmetic), so it stands unless 2 |residual| = gamma with q odd: a tie goes
// to the even neighbour, one step towards the residual's sign (2 |residual| > gamma cannot occur).
// No F2I / FRND: those run at an eighth of the FMA rate and bounded the quantisation kernels.
struct QuantScale {
    float gamma, half_gamma, inv127;  // inv127 = 127 / gamma
    bool fast;                        // gamma is a bf16 value
};
__device__ __forceinline__ QuantScale make_quant_scale(float gamma) {
    QuantScale s;
    s.gamma = gamma;
    s.half_gamma = 0.5f * gamma;
    s.inv127 = __fdiv_rn(127.0f, gamma);
    s.fast = (__float_as_uint(gamma) & 0xffffu) == 0u;
    return s;
}
// Largest magnitude of the eight bf16 values of a 16-byte unit, on the bit patterns: without the sign
// bit a bf16 pattern orders like its magnitude, so a packed 16-bit maximum does two values at a time.
__device__ __forceinline__ uint32_t absmax8_bits(uint32_t acc, const uint4 &v) {
    acc = __vmaxu2(acc, v.x & 0x7fff7fffu);
    acc = __vmaxu2(acc, v.y & 0x7fff7fffu);
    acc = __vmaxu2(acc, v.z & 0x7fff7fffu);
    return __vmaxu2(acc, v.w & 0x7fff7fffu);
}
__device__ __forceinline__ float absmax_bits_to_float(uint32_t acc) {
    const uint32_t hi = acc >> 16, lo = acc & 0xffffu;
    return __uint_as_float((hi > lo ? hi : lo) << 16);
}
// The eight values of a 16-byte unit -> eight int8 (two words), their sum added to `sum`.
// The fast form, arranged for throughput: the candidate's low byte is already the low
// byte of the magic-constant sum's bit pattern (its mantissa holds 2^22 + q in two's complement), so
// the bytes are packed straight from those patterns, and the tie test of all eight values is one
// predicate; only a unit that holds an exact tie (rare) goes back over its values to move the odd
// candidates to their even neighbours.
// PAIRS: two values an instruction (f32x2), each rounded as by itself, the same bytes: for the kernels that are bound by the number of
// instructions (layer calls, one at a time / pairs: 4096 -> 4096 without a correction at M = 4000 75.4 / 74.2 us, 2048 -> 2048 at M = 100 11.05 / 10.8,
// 6144 -> 1024, r = 64 at M = 6000 121.1 / 119.2, 2048 -> 5632 at M = 8192 equal, at the power limit).  Where a warp has one unit and waits for
// the result the pairs' latency shows (32 decode launches in a row 217 / 222 us), and rows_prologue_kernel's registers would no longer leave room for
// three CTAs an SM (5632 -> 2048 at M = 512 20.1 / 22.6): those take one value at a time.
template <bool PAIRS = false>
__device__ __forceinline__ uint2 quant8(const uint4 &v, const QuantScale &s, int &sum) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    uint32_t b[8];
    if (s.fast) {
        constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
        float res[8];
        bool tie = false;
        if constexpr (PAIRS) {
            const uint64_t magic = pack_f32x2(kMagic, kMagic), inv = pack_f32x2(s.inv127, s.inv127), gamma = pack_f32x2(s.gamma, s.gamma);
#pragma unroll
            for (int e = 0; e < 8; e += 2) {
                const uint64_t x = pack_f32x2(bf16lo_to_float(w[e >> 1]), bf16hi_to_float(w[e >> 1])), tm = fma_f32x2(x, inv, magic);
                float t0, t1;
                unpack_f32x2(tm, t0, t1);
                b[e] = __float_as_uint(t0);
                b[e + 1] = __float_as_uint(t1);
                // 127 x - q gamma, exact (magic - tm = -q is, too)
                unpack_f32x2(fma_f32x2(fma_f32x2(tm, pack_f32x2(-1.0f, -1.0f), magic), gamma, mul_f32x2(x, pack_f32x2(127.0f, 127.0f))), res[e], res[e + 1]);
                tie = tie || fabsf(res[e]) == s.half_gamma || fabsf(res[e + 1]) == s.half_gamma;
            }
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float x = (e & 1) ? bf16hi_to_float(w[e >> 1]) : bf16lo_to_float(w[e >> 1]);
                const float tm = fmaf(x, s.inv127, kMagic);
                res[e] = fmaf(kMagic - tm, s.gamma, 127.0f * x);  // 127 x - q gamma, exact
                tie = tie || fabsf(res[e]) == s.half_gamma;
                b[e] = __float_as_uint(tm);
            }
        }
        if (tie) {
#pragma unroll
            for (int e = 0; e < 8; ++e)
                if (fabsf(res[e]) == s.half_gamma && (b[e] & 1u)) b[e] += res[e] > 0.0f ? 1u : 0xffffffffu;
        }
    } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
            b[e] = (uint32_t)quant1_div((e & 1) ? bf16hi_to_float(w[e >> 1]) : bf16lo_to_float(w[e >> 1]), s.gamma);
    }
    uint32_t o[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t p01 = __byte_perm(b[4 * h], b[4 * h + 1], 0x0040), p23 = __byte_perm(b[4 * h + 2], b[4 * h + 3], 0x0040);
        o[h] = __byte_perm(p01, p23, 0x5410);
        sum = __dp4a((int)o[h], 0x01010101, sum);
    }
    return make_uint2(o[0], o[1]);
}

// ---- LayerNorm front end ---------------------------------------------------------------------------
// One binary32 operation each, in this order: the rounded value decides the int8 code.
__device__ __forceinline__ float ln_value(float x, float mean, float rstd, float w, float b) {
    return __fadd_rn(__fmul_rn(__fmul_rn(__fsub_rn(x, mean), rstd), w), b);
}
__device__ __forceinline__ void unpack8(const uint4 &v, float (&f)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 8; ++e) f[e] = (e & 1) ? bf16hi_to_float(w[e >> 1]) : bf16lo_to_float(w[e >> 1]);
}

// Codes of eight normalised values, rint(xn * scale) clipped to +-127, as eight int8; their sum is added to `sum`.  Clipped first
// (the bounds are integers, so that is the same; a NaN gives -127), then rounded to nearest even by adding 1.5 * 2^23, whose low mantissa
// byte is the code: FRND and F2I run at an eighth of the FMA rate.
__device__ __forceinline__ uint2 ln_codes8(const float (&xn)[8], float scale, int &sum) {
    uint32_t c[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) c[e] = __float_as_uint(__fadd_rn(fminf(fmaxf(__fmul_rn(xn[e], scale), -127.0f), 127.0f), 12582912.0f));
    uint32_t o[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const uint32_t p01 = __byte_perm(c[4 * h], c[4 * h + 1], 0x0040), p23 = __byte_perm(c[4 * h + 2], c[4 * h + 3], 0x0040);
        o[h] = __byte_perm(p01, p23, 0x5410);
        sum = __dp4a((int)o[h], 0x01010101, sum);
    }
    return make_uint2(o[0], o[1]);
}

// ---- PTX wrappers -------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t dsmem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mma_u8s8(int (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+r"(d[0]), "+r"(d[1]), "+r"(d[2]), "+r"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                        uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void dmbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ bool dmbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p;\n"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// One bulk copy global -> shared of `bytes` (a multiple of 16; both addresses 16-byte aligned),
// completing on the mbarrier.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void mma_tf32(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                         uint32_t a3, uint32_t b0, uint32_t b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ unsigned long long dec_timer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
    return t;
}
// Programmatic dependent launch: both are no-ops when the launch carries no such attribute.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }

// ---- clusters, distributed shared memory ------------------------------------------------------------
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_release() { asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory"); }
// Stores v at the same shared-memory address of another CTA of the cluster; its bytes count towards that CTA's barrier.
__device__ __forceinline__ void st_async_f32(uint32_t addr, uint32_t bar, uint32_t rank, float v) {
    asm volatile("{\n.reg .b32 ra, rb;\nmapa.shared::cluster.u32 ra, %0, %2;\nmapa.shared::cluster.u32 rb, %1, %2;\n"
                 "st.async.shared::cluster.mbarrier::complete_tx::bytes.f32 [ra], %3, [rb];\n}\n" ::"r"(addr), "r"(bar), "r"(rank), "f"(v)
                 : "memory");
}
__device__ __forceinline__ void st_async_b64(uint32_t addr, uint32_t bar, uint32_t rank, uint64_t v) {
    asm volatile("{\n.reg .b32 ra, rb;\nmapa.shared::cluster.u32 ra, %0, %2;\nmapa.shared::cluster.u32 rb, %1, %2;\n"
                 "st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [ra], %3, [rb];\n}\n" ::"r"(addr), "r"(bar), "r"(rank), "l"(v)
                 : "memory");
}
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, uint32_t rank, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("{\n.reg .b32 ra, rb;\nmapa.shared::cluster.u32 ra, %0, %2;\nmapa.shared::cluster.u32 rb, %1, %2;\n"
                 "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [ra], {%3, %4, %5, %6}, [rb];\n}\n"
                 ::"r"(addr), "r"(bar), "r"(rank), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}
__device__ __forceinline__ void bar_sync(int id, int threads) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id, int threads) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void prefetch_l2(const void *ptr) { asm volatile("prefetch.global.L2 [%0];\n" ::"l"(ptr)); }
__device__ __forceinline__ void announce(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// Bulk copy whose bytes were announced to the barrier already.
__device__ __forceinline__ void bulk_load_announced(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
// A warp waits (bounded) until the barrier's first phase is complete.
__device__ __forceinline__ bool warp_wait(uint32_t bar, unsigned int *status, unsigned int code) {
    bool got = dmbar_try_wait(bar, 0);
    if (__all_sync(0xffffffffu, got)) return true;  // the warp goes on together
    const unsigned long long t0 = dec_timer_ns();
    for (uint32_t polls = 1; !got && !(got = dmbar_try_wait(bar, 0)); ++polls)
        if ((polls & 255u) == 0 && dec_timer_ns() - t0 > kDecWaitLimitNs) break;
    if (!got) atomicExch(status, code);
    return __all_sync(0xffffffffu, got);
}

}  // namespace hgf
