// Decode groups on the 5th-generation tensor cores (M <= 16 tokens): the contraction of Algorithm 1, step 3, with the
// epilogue of steps 4, 7 and 8.  It takes groups on base-3 weights and those of more than eight tokens where it is the faster kernel
// (decode_tc_pays in hgf_api.cu: the rule and its figures); the others stay on the warp MMA of hgf_decode.cu.
//
// In hgf_decode.cu every warp carries codes, activations and accumulators through its own registers: 155 instructions a 1 KiB
// weight tile for two sets of eight tokens (counted over a launch), and the issue slots bound it.  Here 128 output rows go
// through one instruction: a thread owns one row, turns the row's packed bytes into int8 operands and puts them into tensor
// memory (tcgen05.st), and tcgen05.mma.kind::i8 contracts them with the tokens, which lie in shared memory in the operand's
// order: the expansion of a tile is 43 instructions for any number of tokens (150 on base-3 weights), all roles with their waits 132.
//
// One persistent CTA per SM:
//   warp 0 and one of the last two: producers, in turns; a stage is two column tiles of eight row tiles (128 rows), one bulk
//                copy a row tile
//   warp 1       allocates tensor memory, issues the MMAs of the weights (converged, elect.sync)
//   the last     issues those of the correction
//   warps 2-5    epilogue: a thread owns an output channel; they also fetch the rows of B^T of the row tiles to come
//   warps 6-     expansion, four warps an operand stage in tensor memory (three stages, two on base-3 weights)
//   then four or eight warps that stage a problem's activations (one problem ahead where shared memory has the room), H and scales
// What bounds it is the chain of the MMA issuer.  Stamped on one B200, 36 blocks of 2048, 16 tokens: of 241 thousand clocks in the middle
// CTA the issuer waits 13 for the first x~, 10 for x~ at changes of problem, 46 for operands and 33 for accumulators that the epilogue
// still reads; the rest is 360 clocks for the 8 MMAs of a column tile, their commits and loops, where HBM alone would take 330.  8 blocks of
// 4096 on base-3 weights, one token: 199 thousand, 9 for x~, 50 for operands, 7 for accumulators, 490 a column tile of 10 MMAs.
// A run costs whole blocks of eight row tiles, so the shares are cut by them (plan_decode_tc): cut by row tiles the CTAs ended 123 to 143 us
// after the first one's start, the busiest with 418 column tiles for an even 381, and the groups took 155.4 -> 151.9 and 133.2 -> 121.7 us.
// Against the warp MMA, one launch with its prologue, 2048-wide blocks with r = 32: 16 tokens, 36 blocks 167 -> 152 us, 2 blocks
// 31.2 -> 26.2; base-3 weights, 4096-wide, r = 64, one token, 8 blocks 153.5 -> 122; 2048-wide, 8 tokens, 36 blocks 212 -> 165.
//
// Two-bit codes: masked in place they are codes times 1, 4, 16 (the fourth position is shifted down by two: 64 times a code
// would not fit a signed byte), and each scale has an accumulator; the scaled sums are exact multiples.  The order of K
// inside a column tile is free, so the eight registers of an MMA's operand are the eight words of half a row masked alike, and
// the activations are laid out to match.
//
// Base-3 bytes b = c0 + 3 c1 + 9 c2 + 27 c3 + 81 c4: with Q_e = floor(b / 3^e), c_e = Q_e - 3 Q_{e+1}, so
//     sum_e c_e x_e = Q_0 x_0 + sum_{e >= 1} (Q_e x_e - 3 Q_e x_{e-1}):
// the operand is the quotients, not the digits, and the second operand carries x_e and x_{e-1} as two sets of columns (the
// planes x_4 .. x_0 lie one after the other, so the rows of x_{e-1} follow those of x_e).  Q_0 is the byte itself (less 128: a
// signed byte), the others are a 16-bit multiplication for two bytes each, exact for all 256 values (a byte above 242, which no packed
// matrix holds, has a fifth digit of 3: weight 2).  18 operations give 20 weights.
//
// Bank conflicts: a row tile's 64-byte rows would put the eight threads of a phase on two bank groups.  Row tiles are placed
// 16 bytes past a multiple of 128 apart and a warp's lanes run over four row tiles, so the eight threads meet all eight groups.
//
// Every wait is bounded; on a time-out the roles leave, copies in flight are drained, tensor memory is freed.
#include "hgf_tc.cuh"
#include "hgf_warp.cuh"

namespace hgf {

constexpr int kDtStageTiles = 2;                       // column tiles per ring stage
constexpr int kDtRowTilePitch = kDtStageTiles * 1024 + 16, kDtStageBytes = 8 * kDtRowTilePitch;
constexpr int kDtAhead = 4;                                                  // row-tile blocks
constexpr int kDtMaxSegs = 32, kDtMaxStages = 10, kDtMinStages = 4;

// shared memory (offsets from a 1 KiB boundary)
constexpr int kDtOffBT = 0;                                                  // two of 128 rows of B^T, 128 bytes each, swizzled
constexpr int kDtOffH = kDtOffBT + 2 * 128 * 128;                            // [side][value, residual][16 rows of 128 bytes]
constexpr int kDtOffTok = kDtOffH + 2 * 2 * 2048;                            // [side]: scale[16], row sum[16]
constexpr int kDtOffSegs = kDtOffTok + 2 * 128;
constexpr int kDtOffBar = kDtOffSegs + kDtMaxSegs * (int)sizeof(DecodeTcSeg);
constexpr int kDtOffX = (kDtOffBar + 512 + 1023) / 1024 * 1024;              // activations, then the ring
constexpr int kDtSmemLimit = 227 * 1024 - 1024;

template <bool B3, int NT>
struct DtCfg {
    static constexpr int TOK = 8 * NT, TILE_K = B3 ? 320 : 256, A_COLS = TILE_K / 4;
    static constexpr int TILE_X = NT * 8 * TILE_K;                           // bytes of a column tile's activations
    // Accumulators of W columns (the first of 16): two-bit one a scale, base-3 plane 0, plane 1, planes 2 and 3, plane 4 (all
    // but plane 0 with both sets of tokens); then the correction's, which for M <= 8 takes H's fp16 value and its residual
    // side by side.
    static constexpr int W = B3 ? 16 * NT : 16;
    static constexpr int C1 = 16, C2 = C1 + W, C3 = C2 + W, CORR = B3 ? C3 + W : C3, ACC_COLS = CORR + 16;
    static constexpr int H_LO = NT * 1024;                                   // the residual's image behind the value's
    static constexpr int ACCS = B3 && NT == 2 ? 1 : 2;                       // accumulators in turns
    static constexpr int A_COL = ACCS * ACC_COLS, A_STAGES = (512 - A_COL) / (kDtStageTiles * A_COLS);  // operand stages
    static constexpr int W_EXPAND = 6, W_STAGE = W_EXPAND + 4 * A_STAGES, STAGERS = NT == 2 ? 8 : 4, W_PROD2 = W_STAGE + STAGERS, W_LORA = W_PROD2 + 1, WARPS = W_LORA + 1;
    static constexpr int BAR_PFULL = 0, BAR_PEMPTY = kDtMaxStages, BAR_AFULL = 2 * kDtMaxStages, BAR_AEMPTY = BAR_AFULL + A_STAGES,
                         BAR_ACCFULL = BAR_AEMPTY + A_STAGES, BAR_CORRFULL = BAR_ACCFULL + 2, BAR_ACCEMPTY = BAR_CORRFULL + 2, BAR_XFULL = BAR_ACCEMPTY + 2,
                         BAR_XEMPTY = BAR_XFULL + 2, BAR_HFULL = BAR_XEMPTY + 2, BAR_HEMPTY = BAR_HFULL + 2, BAR_BTFULL = BAR_HEMPTY + 2,
                         BAR_COUNT = BAR_BTFULL + 1;
    static_assert(BAR_COUNT * 8 + 8 <= 512 && A_STAGES >= 2, "barriers and tensor memory");
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n"
                 ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
                 : "memory");
}
// A few suspended tries, in as few instructions as that takes: a stage passes six hand-overs, and each is on some role's
// path.  What is not there by then is waited for out of line, with the bounds.
__device__ __forceinline__ bool mbar_wait_some(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n.reg .pred p, q;\n.reg .u32 n;\nmov.u32 n, 64;\n"
        "AGAIN:\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n@p bra DONE;\n"
        "sub.u32 n, n, 1;\nsetp.ne.u32 q, n, 0;\n@q bra AGAIN;\n"
        "DONE:\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
__device__ __noinline__ bool wait_long(uint32_t bar, uint32_t parity, volatile int *abort_flag, unsigned int *status, unsigned int code) {
    return mbar_wait_poll(bar, parity, abort_flag, status, code);
}
// A value that all lanes hold, by an instruction whose result is uniform to the compiler too: loop bounds and operands of the
// MMA issuer then live in uniform registers.
__device__ __forceinline__ uint32_t warp_uniform(uint32_t v) { return __reduce_or_sync(0xffffffffu, v); }
// Row (0..127) of an operand of 128-byte rows, 16-byte unit u: its place under the 128-byte swizzle.
__device__ __forceinline__ uint32_t sw128_at(int row, int u) { return (uint32_t)((row >> 3) * 1024 + (row & 7) * 128 + ((u ^ (row & 7)) << 4)); }
__device__ __forceinline__ void sts_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};\n" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 lds_v4(uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}

// The MMAs of a column tile, from a converged warp (see warp_mma_i8_ts): one elect.sync for all of them.
template <int NT>
__device__ __forceinline__ void issue_tile(uint32_t acc, uint32_t a, uint64_t x, uint32_t idesc, uint32_t more) {
    asm volatile("{\n.reg .pred p, e, t;\n.reg .b32 d1, d2, a1, a2, a3, a4, a5, a6, a7;\n.reg .b64 x1, x2, x3, y0, y1, y2, y3;\n"
                 "elect.sync _|e, 0xffffffff;\nsetp.ne.b32 p, %4, 0;\nsetp.eq.b32 t, 0, 0;\n"
                 "add.u32 d1, %0, 16;\nadd.u32 d2, %0, 32;\n"
                 "add.u32 a1, %1, 8;\nadd.u32 a2, %1, 16;\nadd.u32 a3, %1, 24;\nadd.u32 a4, %1, 32;\nadd.u32 a5, %1, 40;\nadd.u32 a6, %1, 48;\nadd.u32 a7, %1, 56;\n"
                 "add.u64 x1, %2, 2;\nadd.u64 x2, %2, 4;\nadd.u64 x3, %2, 6;\nadd.u64 y0, %2, %5;\nadd.u64 y1, y0, 2;\nadd.u64 y2, y0, 4;\nadd.u64 y3, y0, 6;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], %2, %3, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d1], [a1], x1, %3, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a2], x2, %3, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a3], x3, %3, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], [a4], y0, %3, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d1], [a5], y1, %3, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a6], y2, %3, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a7], y3, %3, t;\n}\n"
                 ::"r"(acc), "r"(a), "l"(x), "r"(idesc), "r"(more), "n"(NT * 1024 >> 4)
                 : "memory");
}
// Base-3: plane e of the tile's activations at (4 - e) NT 512 bytes, rows of 64 bytes; planes 1 to 4 with both sets of tokens.
template <int NT>
__device__ __forceinline__ void issue_b3_tile(uint32_t acc, uint32_t a, uint64_t x, uint32_t idesc0, uint32_t idesc, uint32_t more) {
    constexpr int P = NT * 512 >> 4, W = 16 * NT, C1 = 16;
    asm volatile("{\n.reg .pred p, e, t;\n.reg .b32 d1, d2, d3, a1, a2, a3, a4, a5, a6, a7, a8, a9;\n.reg .b64 x0, x1, x2, x3, y0, y1, y2, y3, y4;\n"
                 "elect.sync _|e, 0xffffffff;\nsetp.ne.b32 p, %5, 0;\nsetp.eq.b32 t, 0, 0;\n"
                 "add.u32 d1, %0, %6;\nadd.u32 d2, d1, %7;\nadd.u32 d3, d2, %7;\n"
                 "add.u32 a1, %1, 8;\nadd.u32 a2, %1, 16;\nadd.u32 a3, %1, 24;\nadd.u32 a4, %1, 32;\nadd.u32 a5, %1, 40;\nadd.u32 a6, %1, 48;\nadd.u32 a7, %1, 56;\n"
                 "add.u32 a8, %1, 64;\nadd.u32 a9, %1, 72;\n"
                 "add.u64 x3, %2, %8;\nadd.u64 x2, x3, %8;\nadd.u64 x1, x2, %8;\nadd.u64 x0, x1, %8;\n"
                 "add.u64 y0, x0, 2;\nadd.u64 y1, x1, 2;\nadd.u64 y2, x2, 2;\nadd.u64 y3, x3, 2;\nadd.u64 y4, %2, 2;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], x0, %3, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d1], [a2], x1, %4, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a4], x2, %4, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a6], x3, %4, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d3], [a8], %2, %4, p;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [%0], [a1], y0, %3, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d1], [a3], y1, %4, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a5], y2, %4, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d2], [a7], y3, %4, t;\n"
                 "@e tcgen05.mma.cta_group::1.kind::i8 [d3], [a9], y4, %4, t;\n}\n"
                 ::"r"(acc), "r"(a), "l"(x), "r"(idesc0), "r"(idesc), "r"(more), "n"(C1), "n"(W), "n"(P)
                 : "memory");
}

template <bool B3, int NT>
__global__ void __launch_bounds__(DtCfg<B3, NT>::WARPS * 32, 1) decode_tc_kernel(const DecodeTcLaunch L, unsigned int *status) {
    using C = DtCfg<B3, NT>;
    extern __shared__ uint8_t dt_smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)dt_smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem), bar0 = sbase + kDtOffBar;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + kDtOffBar + C::BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + kDtOffBar + C::BAR_COUNT * 8 + 4);
    const DecodeTcSeg *segs = reinterpret_cast<const DecodeTcSeg *>(smem + kDtOffSegs);

    pdl_launch_dependents();
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int2 mine = L.cta[blockIdx.x];  // (written when the group was made)
    const int nseg = (int)warp_uniform(mine.y), stages = L.stages;
    const uint32_t ring = sbase + kDtOffX + L.x_bytes;
    for (int i = tid; i < nseg * (int)(sizeof(DecodeTcSeg) / 16); i += C::WARPS * 32)
        reinterpret_cast<uint4 *>(smem + kDtOffSegs)[i] = reinterpret_cast<const uint4 *>(L.segs + mine.x)[i];
    if (tid == 0) {
        for (int s = 0; s < stages; ++s) {
            mbar_init(bar(C::BAR_PFULL + s), 1);
            mbar_init(bar(C::BAR_PEMPTY + s), 4);
        }
        for (int s = 0; s < C::A_STAGES; ++s) {
            mbar_init(bar(C::BAR_AFULL + s), 4);
            mbar_init(bar(C::BAR_AEMPTY + s), 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(C::BAR_ACCFULL + b), 1);
            mbar_init(bar(C::BAR_CORRFULL + b), 1);
            mbar_init(bar(C::BAR_ACCEMPTY + b), 4);
            mbar_init(bar(C::BAR_XFULL + b), C::STAGERS);
            mbar_init(bar(C::BAR_XEMPTY + b), 1);
            mbar_init(bar(C::BAR_HFULL + b), C::STAGERS);
            mbar_init(bar(C::BAR_HEMPTY + b), 4);
        }
        mbar_init(bar(C::BAR_BTFULL), 4);
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
    const uint32_t tmem_base = warp_uniform(*tmem_slot);
    auto wait = [&](int i, uint32_t par, unsigned int code) {
        if (__all_sync(0xffffffffu, mbar_wait_some(bar(i), par))) return true;
        return __all_sync(0xffffffffu, wait_long(bar(i), par, abort_flag, status, code)) != 0;
    };
    // where segment i's activations lie: even ones at the start of their region, odd ones at its end
    auto x_size = [&](int i) { return segs[i].steps * C::TILE_X; };
    auto x_at = [&](int i) { return sbase + kDtOffX + ((i & 1) ? (uint32_t)((L.x_bytes - x_size(i)) & ~1023) : 0u); };

    if (warp == 0 || warp == C::W_PROD2) {
        // ------------------------------------------------------------------ producers of the packed weights, stages in turns
        const int turn = warp ? 1 : 0;
        bool ok = true;
        int ps = 0;
        uint32_t issued = 0;
        uint32_t ph = 1;
        for (int i = 0; ok && i < nseg; ++i) {
            const int steps = segs[i].steps, n = segs[i].n;
            const uint8_t *packed = segs[i].packed;
            for (int t0 = 0; ok && t0 < n; t0 += 8) {
                const int rows = n - t0 < 8 ? n - t0 : 8;
                const uint8_t *src = packed + (size_t)(t0 + (lane < rows ? lane : 0)) * steps * 1024;
                for (int ct = 0; ct < steps; ct += kDtStageTiles) {
                    const uint32_t bytes = (steps - ct < kDtStageTiles ? steps - ct : kDtStageTiles) * 1024u;
                    if ((int)(issued & 1u) == turn) {
                        if (!(ok = wait(C::BAR_PEMPTY + ps, ph, 0xb00u + ps))) break;
                        if (lane == 0) mbar_arrive_expect_tx(bar(C::BAR_PFULL + ps), rows * bytes);
                        __syncwarp();
                        if (lane < rows) bulk_load_1d(ring + ps * kDtStageBytes + lane * kDtRowTilePitch, src + (size_t)ct * 1024, bytes, bar(C::BAR_PFULL + ps));
                    }
                    ++issued;  // (by both; the ring is even, so a stage has one producer)
                    if (++ps == stages) { ps = 0; ph ^= 1u; }
                }
            }
        }
        for (uint32_t q = 0; q < (uint32_t)stages; ++q) {  // never leave with a copy in flight
            const uint32_t rounds = (issued + stages - 1 - q) / stages;
            if (rounds && (int)(q & 1u) == turn)
                for (uint32_t k = 0; k < kSpinLimit && !mbar_try_wait(bar(C::BAR_PFULL + q), (rounds - 1u) & 1u); ++k) {}
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        constexpr uint32_t I8 = (2u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
        constexpr uint32_t I8_16 = I8 | (2u << 17), I8_W = I8 | ((uint32_t)(C::W >> 3) << 17);
        bool ok = true;
        int as = 0, b = 0;
        uint32_t aph = 0, bph = 1;
        for (int i = 0; ok && i < nseg; ++i) {
            const int steps = (int)warp_uniform(segs[i].steps), n = (int)warp_uniform(segs[i].n), side = i & 1;
            const uint32_t x_begin = x_at(i);
            if (!(ok = wait(C::BAR_XFULL + side, (uint32_t)(i >> 1) & 1u, 0xb10u + side))) break;
            for (int t0 = 0; ok && t0 < n; t0 += 8) {
                const uint32_t acc = warp_uniform(tmem_base + b * C::ACC_COLS);
                if (!(ok = wait(C::BAR_ACCEMPTY + b, bph, 0xb12u))) break;
                uint32_t xaddr = x_begin;
                for (int ct = 0; ct < steps; ct += kDtStageTiles, xaddr += kDtStageTiles * C::TILE_X) {
                    // (operands the compiler knows to be uniform: from general registers an MMA takes 35 to 50 clocks to issue)
                    const uint32_t a = warp_uniform(tmem_base + C::A_COL + as * kDtStageTiles * C::A_COLS), x = warp_uniform(xaddr), more = ct ? 1u : 0u;
                    if (!(ok = wait(C::BAR_AFULL + as, aph, 0xb14u))) break;
                    tc_fence_after();
                    if constexpr (B3) {
                        issue_b3_tile<NT>(acc, a, make_sw64_desc(x), I8_16, I8_W, more);
                        if (ct + 1 < steps) issue_b3_tile<NT>(acc, a + C::A_COLS, make_sw64_desc(x + C::TILE_X), I8_16, I8_W, 1u);
                    } else {
                        issue_tile<NT>(acc, a, make_sw128_desc(x), I8_16, more);
                        if (ct + 1 < steps) issue_tile<NT>(acc, a + C::A_COLS, make_sw128_desc(x + C::TILE_X), I8_16, 1u);
                    }
                    warp_commit(bar(C::BAR_AEMPTY + as));
                    if (++as == C::A_STAGES) { as = 0; aph ^= 1u; }
                }
                if (!ok) break;
                warp_commit(bar(C::BAR_ACCFULL + b));
                if (t0 + 8 >= n) warp_commit(bar(C::BAR_XEMPTY + side));
                if (++b == C::ACCS) { b = 0; bph ^= 1u; }
            }
        }
    } else if (warp == C::W_LORA) {
        // ------------------------------------------------------------------ the correction's MMAs
        // (B^T rows) x (H, its fp16 value and residual), an accumulator of their own: issued by a warp of its own, since at the end of a
        // row-tile block they and their waits cost the other issuer 1000 clocks.
        constexpr uint32_t F16 = (1u << 4) | (2u << 17) | (8u << 24);
        const uint64_t bt_desc = make_sw128_desc(sbase + kDtOffBT), h_desc = make_sw128_desc(sbase + kDtOffH);
        bool ok = true;
        int b = 0, tb = 0;
        uint32_t bph = 1, btph = 0;
        for (int i = 0; ok && i < nseg; ++i) {
            const int n = segs[i].n, r = (int)warp_uniform(segs[i].r), side = i & 1;
            if (!(ok = wait(C::BAR_HFULL + side, (uint32_t)(i >> 1) & 1u, 0xb16u))) break;
            for (int t0 = 0; t0 < n; t0 += 8) {
                if (r) {
                    if (!(ok = wait(C::BAR_BTFULL, btph, 0xb17u))) break;
                    btph ^= 1u;
                }
                if (!(ok = wait(C::BAR_ACCEMPTY + b, bph, 0xb18u))) break;
                tc_fence_after();
                for (int kk = 0; kk < r / 16; ++kk) {
                    const uint64_t h = h_desc + (uint64_t)(side * (4096 >> 4) + 2 * kk), bt = bt_desc + (uint64_t)(tb * (128 * 128 >> 4) + 2 * kk);
                    warp_mma_f16(tmem_base + b * C::ACC_COLS + C::CORR, bt, h, F16, kk ? 1u : 0u);  // (M <= 8: the residual's columns too)
                    if (NT == 2) warp_mma_f16(tmem_base + b * C::ACC_COLS + C::CORR, bt, h + (C::H_LO >> 4), F16, 1u);
                }
                warp_commit(bar(C::BAR_CORRFULL + b));
                tb ^= 1;
                if (++b == C::ACCS) { b = 0; bph ^= 1u; }
            }
        }
    } else if (warp < 6) {
        // ------------------------------------------------------------------ epilogue, and the rows of B^T
        // Thread m = 32 q + lane owns the MMA's row m: row 8 (q & 1) + lane / 4 of row tile 4 (q >> 1) + lane % 4.
        const int q = warp & 3, row_tile = 4 * (q >> 1) + (lane & 3), row = 8 * (q & 1) + (lane >> 2), m_row = 32 * q + lane;
        const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16);
        pdl_wait();  // the gate may be an output of earlier work; y is written
        float gate = 0.0f;
        auto fetch = [&](int i, int t0, int b) {  // the thread's row of B^T (into buffer b) and its gate, for a row-tile block to come
            const DecodeTcSeg &S = segs[i];
            const int nb = 16 * (S.lo + t0 + row_tile) + row, n = nb < S.N ? nb : S.N - 1, units = S.r >> 3;
            const __half *src = S.Bt + (size_t)n * S.r;
            const uint32_t dst = sbase + kDtOffBT + b * (128 * 128);
            for (int u = 0; u < units; ++u)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(dst + sw128_at(m_row, u)), "l"(src + 8 * u) : "memory");
            asm volatile("cp.async.commit_group;\n" ::: "memory");
            return S.r ? __ldg(S.gate + (S.gate_group > 1 ? n / S.gate_group : n)) : 0.0f;
        };
        // The same rows and gates into L2, kDtAhead blocks before they are fetched.
        auto ahead = [&](int i, int t) {
            for (; i < nseg; t -= (segs[i].n + 7) & ~7, ++i) {
                const DecodeTcSeg &S = segs[i];
                if (t >= S.n) continue;
                const int nb = 16 * (S.lo + t + row_tile) + row, n = nb < S.N ? nb : S.N - 1;
                if (S.r) {
                    prefetch_l2(S.Bt + (size_t)n * S.r);
                    prefetch_l2(S.gate + (S.gate_group > 1 ? n / S.gate_group : n));
                }
                return;
            }
        };
        auto put = [&](int i) {
            if (!segs[i].r) return;
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_BTFULL));
        };
        bool ok = true;
        int b = 0, tb = 0;
        uint32_t bph = 0;
        if (nseg > 0) {
            for (int k = 1; k < kDtAhead; ++k) ahead(0, 8 * k);
            gate = fetch(0, 0, 0);
            put(0);
        }
        for (int i = 0; ok && i < nseg; ++i) {
            const DecodeTcSeg &S = segs[i];
            const int n_tiles = S.n, M = S.M, N = S.N, r = S.r, side = i & 1;
            const bool out_bf16 = (S.flags & HGF_FLAG_OUT_BF16) != 0;
            int32_t *dbg_y_int = *S.dbg_y_int_at;
            void *y_out = S.y;
            if (!(ok = wait(C::BAR_HFULL + side, (uint32_t)(i >> 1) & 1u, 0xb20u))) break;
            const float *tok_sc = reinterpret_cast<const float *>(smem + kDtOffTok + side * 128);
            const int *tok_rs = reinterpret_cast<const int *>(tok_sc + 16);
            for (int t0 = 0; t0 < n_tiles; t0 += 8) {
                const int n = 16 * (S.lo + t0 + row_tile) + row;
                const bool row_ok = t0 + row_tile < n_tiles && n < N;
                const float g = gate;
                const bool last = t0 + 8 >= n_tiles, next = !last || i + 1 < nseg;
                const int ni = last ? i + 1 : i;
                ahead(i, t0 + 8 * kDtAhead);
                if (next) gate = fetch(ni, last ? 0 : t0 + 8, tb ^ 1);  // (its last readers, MMAs of the block before, are complete)
                if (!(ok = wait(C::BAR_CORRFULL + b, bph, 0xb24u) && wait(C::BAR_ACCFULL + b, bph, 0xb22u))) break;
                tc_fence_after();
                const uint32_t acc = lane_base + b * C::ACC_COLS;
#pragma unroll
                for (int half = 0; half < NT; ++half) {
                    uint32_t s[8], corr[8], res[8];
                    if (half && M <= 8) break;
                    tmem_ld8(acc + 8 * half, s);
                    if (r) {
                        tmem_ld8(acc + C::CORR + 8 * half, corr);
                        if (NT == 1) tmem_ld8(acc + C::CORR + 8, res);
                    }
                    if constexpr (B3) {  // c_e x_e = Q_e x_e - 3 Q_e x_{e-1}; planes 2 and 3 hold twice Q, plane 4 thirty-two times
                        constexpr int at[3] = {C::C1, C::C2, C::C3}, shift[3] = {0, 1, 5};
#pragma unroll
                        for (int e = 0; e < 3; ++e) {
                            uint32_t v[8], u[8];
                            tmem_ld8(acc + at[e] + 8 * half, v);
                            tmem_ld8(acc + at[e] + C::TOK + 8 * half, u);
                            tmem_ld_wait();
#pragma unroll
                            for (int c = 0; c < 8; ++c) s[c] += (uint32_t)(((int)v[c] - 3 * (int)u[c]) >> shift[e]);
                        }
                    } else {
                        uint32_t v[8], w[8];
                        tmem_ld8(acc + C::C1 + 8 * half, v);
                        tmem_ld8(acc + C::C2 + 8 * half, w);
                        tmem_ld_wait();
#pragma unroll
                        for (int c = 0; c < 8; ++c) s[c] += (uint32_t)(((int)v[c] >> 2) + ((int)w[c] >> 4));
                    }
#pragma unroll
                    for (int c = 0; c < 8; ++c) {
                        const int m = 8 * half + c;
                        if (m < M && row_ok) {
                            const int y_int = (int)s[c] - tok_rs[m];
                            const float base = (float)y_int * tok_sc[m];
                            const float y = r ? fmaf(g, NT == 1 ? __uint_as_float(corr[c]) + __uint_as_float(res[c]) : __uint_as_float(corr[c]), base) : base;
                            const size_t o = (size_t)m * N + n;
                            if (out_bf16) reinterpret_cast<__nv_bfloat16 *>(y_out)[o] = __float2bfloat16_rn(y);
                            else reinterpret_cast<float *>(y_out)[o] = y;
                            if (dbg_y_int) dbg_y_int[o] = y_int;
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(bar(C::BAR_ACCEMPTY + b));
                    if (last) mbar_arrive(bar(C::BAR_HEMPTY + side));
                }
                if (next) put(ni);
                tb ^= 1;
                if (++b == C::ACCS) { b = 0; bph ^= 1u; }
            }
        }
    } else if (warp < C::W_STAGE) {
        // ------------------------------------------------------------------ expansion into tensor memory
        // Four warps an operand stage, which takes a ring stage (two column tiles) at a time, in turns with the others.
        const int q = warp & 3, as = (warp - C::W_EXPAND) >> 2;
        const uint32_t row_off = (uint32_t)((4 * (q >> 1) + (lane & 3)) * kDtRowTilePitch + (8 * (q & 1) + (lane >> 2)) * 64);
        const uint32_t dst0 = tmem_base + ((uint32_t)(32 * q) << 16) + C::A_COL + as * kDtStageTiles * C::A_COLS;
        bool ok = true;
        int ps = as, at = as;  // ring stage; place of the stage in its row-tile block
        uint32_t ph = 0, aph = 1;
        for (int i = 0; ok && i < nseg; ++i) {
            const int steps = segs[i].steps, pairs = (steps + 1) >> 1, all = pairs * ((segs[i].n + 7) >> 3);
            int in_block = at % pairs;
            for (; at < all; at += C::A_STAGES) {
                // The operand stage first: its MMAs, three stages back, are behind all earlier copies, so the ring's barrier cannot be
                // a phase behind.
                if (!(ok = wait(C::BAR_AEMPTY + as, aph, 0xb32u) && wait(C::BAR_PFULL + ps, ph, 0xb30u))) break;
                tc_fence_after();
                const uint32_t src0 = ring + ps * kDtStageBytes + row_off;
                const int tiles = steps - 2 * in_block < 2 ? 1 : 2;
#pragma unroll
                for (int tile = 0; tile < kDtStageTiles; ++tile) {
                    if (tile >= tiles) break;
                    const uint32_t src = src0 + tile * 1024, dst = dst0 + tile * C::A_COLS;
                    uint32_t w[16];
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        const uint4 v = lds_v4(src + 16 * c);
                        w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
                    }
                    if constexpr (B3) {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t p0[8], p1[8], p2[8], p3[8], p4[8];
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                const uint32_t b4 = w[8 * h + k], e = b4 & 0x00ff00ffu, o = __byte_perm(b4, 0u, 0x4341);
                                p0[k] = b4 ^ 0x80808080u;                                                          // b - 128
                                p1[k] = __byte_perm(e * 85u + 0x00550055u, o * 85u + 0x00550055u, 0x7351);         // floor(b / 3)
                                p2[k] = __byte_perm(e * 57u, o * 57u, 0x7351) & 0xfefefefeu;                       // 2 floor(b / 9)
                                p3[k] = __byte_perm(e * 19u, o * 19u, 0x7351) & 0xfefefefeu;                       // 2 floor(b / 27)
                                p4[k] = __byte_perm(e * 101u + 0x00210021u, o * 101u + 0x00210021u, 0x7351) & 0x60606060u;  // 32 floor(b / 81)
                            }
                            tmem_st8(dst + 8 * h, p0);
                            tmem_st8(dst + 16 + 8 * h, p1);
                            tmem_st8(dst + 32 + 8 * h, p2);
                            tmem_st8(dst + 48 + 8 * h, p3);
                            tmem_st8(dst + 64 + 8 * h, p4);
                        }
                    } else {
#pragma unroll
                        for (int h = 0; h < 2; ++h) {
                            uint32_t a[32];
#pragma unroll
                            for (int k = 0; k < 8; ++k) {
                                a[k] = w[8 * h + k] & 0x03030303u;
                                a[8 + k] = w[8 * h + k] & 0x0c0c0c0cu;
                                a[16 + k] = w[8 * h + k] & 0x30303030u;
                                a[24 + k] = (w[8 * h + k] >> 2) & 0x30303030u;
                            }
                            tmem_st32(dst + 32 * h, a);
                        }
                    }
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane < 2) mbar_arrive(bar(lane ? C::BAR_AFULL + as : C::BAR_PEMPTY + ps));
                aph ^= 1u;
                ps += C::A_STAGES;
                if (ps >= stages) { ps -= stages; ph ^= 1u; }
                in_block += C::A_STAGES;
                while (in_block >= pairs) in_block -= pairs;
            }
            at -= all;  // (the first of this warp's stages in the next segment)
        }
    } else {
        // ------------------------------------------------------------------ activations, H and per-token values of the problems
        constexpr int TH = C::STAGERS * 32;
        const int tid4 = tid - C::W_STAGE * 32;
        pdl_wait();  // all of it comes from the prologue launch
        bool ok = true;
        for (int i = 0; ok && i < nseg; ++i) {
            const DecodeTcSeg &S = segs[i];
            const int side = i & 1, M = S.M, K = S.K, steps = S.steps, r = S.r;
            const uint32_t free_par = (uint32_t)((i >> 1) - 1) & 1u;
            if (i >= 2 && !(ok = wait(C::BAR_XEMPTY + side, free_par, 0xb40u))) break;
            // the other side's problem (the one before) may need some of this one's room
            if (i >= 1 && x_size(i - 1) + x_size(i) > ((i & 1) ? x_at(i) - sbase - kDtOffX + x_size(i) : x_at(i - 1) - sbase - kDtOffX + x_size(i - 1)) &&
                !(ok = wait(C::BAR_XEMPTY + (side ^ 1), (uint32_t)((i - 1) >> 1) & 1u, 0xb42u)))
                break;
            const uint32_t xb = x_at(i);
            const int8_t *xq = S.xq;
            if constexpr (B3) {
                // item: token m, column tile ct, u: the 64 columns 64 u .. of it and the 16 columns 256 + 16 u ..
                for (int v = tid4; v < M * steps * 4; v += TH) {
                    const int m = v % M, cu = v / M, ct = cu >> 2, u = cu & 3, k = ct * 320 + 64 * u, k4 = ct * 320 + 256 + 16 * u;
                    const int8_t *row = xq + (size_t)m * K;
                    uint4 x[5];
#pragma unroll
                    for (int b = 0; b < 4; ++b) x[b] = k < K ? __ldcg(reinterpret_cast<const uint4 *>(row + k + 16 * b)) : make_uint4(0u, 0u, 0u, 0u);
                    x[4] = k4 < K ? __ldcg(reinterpret_cast<const uint4 *>(row + k4)) : make_uint4(0u, 0u, 0u, 0u);
                    const uint32_t xw[5][4] = {{x[0].x, x[0].y, x[0].z, x[0].w}, {x[1].x, x[1].y, x[1].z, x[1].w}, {x[2].x, x[2].y, x[2].z, x[2].w},
                                               {x[3].x, x[3].y, x[3].z, x[3].w}, {x[4].x, x[4].y, x[4].z, x[4].w}};
                    // plane e, word 4 t + u of the token's 64 bytes: digit e's columns 64 u + 16 b + 4 t + e, b = 0..3 (e < 4),
                    // 256 + 16 u + 4 t + b (e = 4)
                    const uint32_t tok = xb + ct * C::TILE_X + (m >> 3) * 512 + (m & 7) * 64 + 4 * u;
#pragma unroll
                    for (int t = 0; t < 4; ++t) {
                        const uint32_t at = tok + ((t ^ ((m & 7) >> 1)) << 4);
                        const uint32_t p01 = __byte_perm(xw[0][t], xw[1][t], 0x5140), q01 = __byte_perm(xw[0][t], xw[1][t], 0x7362);
                        const uint32_t p23 = __byte_perm(xw[2][t], xw[3][t], 0x5140), q23 = __byte_perm(xw[2][t], xw[3][t], 0x7362);
                        const uint32_t pl[5] = {__byte_perm(p01, p23, 0x5410), __byte_perm(p01, p23, 0x7632), __byte_perm(q01, q23, 0x5410),
                                                __byte_perm(q01, q23, 0x7632), xw[4][t]};
#pragma unroll
                        for (int e = 0; e < 5; ++e)
                            asm volatile("st.shared.u32 [%0], %1;\n" ::"r"(at + (4 - e) * NT * 512), "r"(pl[e]) : "memory");
                    }
                }
            } else {
                // item: token m, 64 columns: word j of 16-byte unit c goes to row bytes 32 j + 4 (c % 8) of 128-column block c / 8.
                // Two items' loads in flight.
                for (int v0 = tid4; v0 < M * steps * 4; v0 += 2 * TH) {
                    uint4 x[2][4];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int v = v0 + e * TH, m = v % M, k = 64 * (v / M);
                        const bool in = v < M * steps * 4 && k < K;
#pragma unroll
                        for (int b = 0; b < 4; ++b) x[e][b] = in ? __ldcg(reinterpret_cast<const uint4 *>(xq + (size_t)m * K + k + 16 * b)) : make_uint4(0u, 0u, 0u, 0u);
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int v = v0 + e * TH, m = v % M, c4 = v / M;
                        if (v >= M * steps * 4) break;
                        const uint32_t blk = xb + (c4 >> 1) * NT * 1024 + (m >> 3) * 1024 + (m & 7) * 128;
                        const int odd = c4 & 1, mr = m & 7;
                        sts_v4(blk + (((0 + odd) ^ mr) << 4), x[e][0].x, x[e][1].x, x[e][2].x, x[e][3].x);
                        sts_v4(blk + (((2 + odd) ^ mr) << 4), x[e][0].y, x[e][1].y, x[e][2].y, x[e][3].y);
                        sts_v4(blk + (((4 + odd) ^ mr) << 4), x[e][0].z, x[e][1].z, x[e][2].z, x[e][3].z);
                        sts_v4(blk + (((6 + odd) ^ mr) << 4), x[e][0].w, x[e][1].w, x[e][2].w, x[e][3].w);
                    }
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_XFULL + side));

            if (i >= 2 && !(ok = wait(C::BAR_HEMPTY + side, free_par, 0xb44u))) break;
            float *tok_sc = reinterpret_cast<float *>(smem + kDtOffTok + side * 128);
            int *tok_rs = reinterpret_cast<int *>(tok_sc + 16);
            if constexpr (B3) {
                // sum_k c x~ - sum_k x~, and plane 0 enters as b - 128: 128 times the sum over its columns comes back.  A warp
                // adds up a token's plane-0 values (x~ of columns 4 n of the first 256 of a tile).
                for (int m = tid4 >> 5; m < M; m += C::STAGERS) {
                    int s0 = 0;
                    const int8_t *row = xq + (size_t)m * K;
                    for (int k = 16 * lane; k < K; k += 512) {
                        if (k % 320 < 256) {
                            const uint4 x = __ldcg(reinterpret_cast<const uint4 *>(row + k));
                            s0 += (int)(int8_t)x.x + (int)(int8_t)x.y + (int)(int8_t)x.z + (int)(int8_t)x.w;
                        }
                    }
                    s0 = warp_sum_i(s0);
                    if (lane == 0) tok_rs[m] = __ldcg(S.row_sum + m) - 128 * s0;
                }
                if (tid4 < M) tok_sc[tid4] = __ldcg(S.gamma_x + tid4) * S.gw_over_127;
            } else if (tid4 < M) {
                tok_sc[tid4] = __ldcg(S.gamma_x + tid4) * S.gw_over_127;
                tok_rs[tid4] = __ldcg(S.row_sum + tid4);
            }
            // H = act(sum over K slices of the parked partial sums of x A), slices in order.  The partial sums sit in the warp
            // MMA's accumulator layout: column 16 jt + jl and token m are register 4 (m / 8) + 2 (jl / 8) + m % 2 of lane
            // 4 (jl % 8) + (m % 8) / 2.  A thread takes four of them at a time, four slices each in flight.
            const int ns = S.nslices, units = (r >> 4) * NT * 128;
            const bool no_silu = (S.flags & HGF_FLAG_NO_SILU) != 0;
            const uint32_t himg = sbase + kDtOffH + side * 4096;
            for (int v0 = tid4; v0 < units; v0 += 4 * TH) {
                float z[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                const float *src[4];
                int tok[4], col[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int v = v0 + TH * e, jt = v / (NT * 128), idx = (v >> 5) % (NT * 4), ln = v & 31, c = idx & 3;
                    tok[e] = v < units ? 8 * (idx >> 2) + 2 * (ln & 3) + (c & 1) : 16;
                    col[e] = 16 * jt + (ln >> 2) + 8 * (c >> 1);
                    src[e] = S.hpart + ((size_t)jt * ns * 8 + idx) * 32 + ln;
                }
                for (int sl = 0; sl < ns; sl += 4) {
                    float p[4][4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int k = 0; k < 4; ++k) p[e][k] = tok[e] < M && sl + k < ns ? __ldcg(src[e] + (size_t)(sl + k) * 256) : 0.0f;
#pragma unroll
                    for (int e = 0; e < 4; ++e)
#pragma unroll
                        for (int k = 0; k < 4; ++k) z[e] += p[e][k];
                }
#pragma unroll
                for (int e = 0; e < 4; ++e)
                    if (tok[e] < M) {
                        const float h = no_silu ? z[e] : silu_f(z[e]);
                        const __half hi = __float2half_rn(h), lo = __float2half_rn(h - __half2float(hi));
                        const uint32_t at = himg + sw128_at(tok[e], col[e] >> 3) + 2 * (col[e] & 7);
                        asm volatile("st.shared.u16 [%0], %1;\n" ::"r"(at), "h"(__half_as_ushort(hi)) : "memory");
                        asm volatile("st.shared.u16 [%0], %1;\n" ::"r"(at + C::H_LO), "h"(__half_as_ushort(lo)) : "memory");
                    }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(C::BAR_HFULL + side));
        }
    }

    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(512) : "memory");
    }
}

// ---- host side -----------------------------------------------------------------------------------------
// Shared memory of a launch: the activations' region (two problems side by side where they fit beside a ring of six stages,
// else what six stages leave, else the largest problem) and the ring.  False: the largest problem leaves fewer than four stages.
static bool dt_layout(int max_image, int *x_bytes, int *stages) {
    const int room = kDtSmemLimit - kDtOffX;
    max_image = (max_image + 1023) & ~1023;
    int x = (room - 6 * kDtStageBytes) & ~1023;  // (down: rounded up it cost the sixth stage, and with it the fifth)
    x = x < max_image ? max_image : (x > 2 * max_image ? 2 * max_image : x);
    *x_bytes = x;
    *stages = (room - x) / kDtStageBytes;
    if (*stages > kDtMaxStages) *stages = kDtMaxStages;
    *stages &= ~1;  // (even: a stage always has the same producer)
    return *stages >= kDtMinStages;
}

int decode_tc_image_bytes(int max_M, int K, uint32_t flags) {
    return (flags & HGF_FLAG_BASE3) ? (max_M <= 8 ? 8 : 16) * weight_steps(K, flags) * 320 : 16 * weight_steps(K, flags) * 256;
}
bool decode_tc_fits(int max_image, int max_segs) {
    int x, s;
    return max_segs <= kDtMaxSegs && dt_layout(max_image, &x, &s);
}
// (for the tests: the layout for activations of that size; out: their region, ring stages, bytes of a stage, shared memory for both)
extern "C" int hgf_internal_decode_tc_layout(int32_t max_image, int32_t *out) {
    out[2] = kDtStageBytes;
    out[3] = kDtSmemLimit - kDtOffX;
    return dt_layout(max_image, &out[0], &out[1]) ? 1 : 0;
}

template <bool B3, int NT>
static cudaError_t launch_decode_tc_variant(const DecodeTcLaunch &L, int grid, bool pdl, cudaStream_t stream) {
    static std::atomic<unsigned long long> attr_done{0};
    cudaError_t e = ensure_dynamic_smem(decode_tc_kernel<B3, NT>, kDtSmemLimit + 1024, attr_done);
    if (e != cudaSuccess) return e;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(DtCfg<B3, NT>::WARPS * 32);
    cfg.dynamicSmemBytes = (size_t)(1024 + kDtOffX + L.x_bytes + L.stages * kDtStageBytes);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    e = cudaLaunchKernelEx(&cfg, decode_tc_kernel<B3, NT>, L, status);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

cudaError_t launch_decode_tc(const DecodeTcSeg *segs, const int2 *cta, int grid, int max_image, int max_M, uint32_t flags, bool pdl, cudaStream_t stream) {
    DecodeTcLaunch L = {};
    L.segs = segs;
    L.cta = cta;
    if (!dt_layout(max_image, &L.x_bytes, &L.stages)) return cudaErrorInvalidValue;
    if (flags & HGF_FLAG_BASE3)
        return max_M <= 8 ? launch_decode_tc_variant<true, 1>(L, grid, pdl, stream) : launch_decode_tc_variant<true, 2>(L, grid, pdl, stream);
    return launch_decode_tc_variant<false, 2>(L, grid, pdl, stream);  // (two-bit groups of up to eight tokens do not come here)
}

}  // namespace hgf
