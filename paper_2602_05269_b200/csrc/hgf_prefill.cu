// GEMM path (M > 16 tokens): Y_int = X~ x T^T on the 5th-generation tensor cores
// (tcgen05.mma kind::i8, int32 accumulator in tensor memory), with the dequantisation, the LoRA
// up-projection (a small tcgen05.mma kind::f16 on top of the dequantised accumulator, with the gate
// folded into B) and the gated fusion in the epilogue.  Algorithm 1, steps 3, 4, 7, 8.
//
// The ternary weights are the MMA's first operand and are read from TENSOR MEMORY: the tensor core
// cannot read 2-bit codes, and expanding them to int8 in shared memory costs four times their bytes
// in shared-memory writes plus the same again when the MMA reads them - more than the port has.
// Here four warps expand a packed 128 x 256 tile straight from its 8 KiB in shared memory into
// registers (one 128-channel row per thread: a shift and a mask per register) and store it with two
// tcgen05.st into the operand's place in tensor memory, so shared memory carries only the int8
// activation tile (TMA in, MMA out) and the packed codes.  The output tile is therefore
// 128 output channels (tensor-memory lanes, MMA M) x 128 tokens (columns, MMA N); two accumulators
// alternate, so the epilogue of a tile runs under the main loop of the next.  A pipeline stage is
// 256 input columns (eight MMAs): every hand-over between the roles costs a shared-memory round
// trip.
//
// One persistent CTA per SM, 15 warps with fixed roles:
//   warp 0      producer (all lanes): per stage the int8 activation tile as two 128 tokens x 128 B
//               boxes (128-byte swizzle); per tile what its epilogue needs: row sums, scales, the H
//               tile and the (g B)^T tile
//   warp 1      allocates tensor memory; issues the MMAs and commits to mbarriers
//   warps 2-5, 11-14  epilogue, two warps per tensor-memory lane quarter (32 channels), one for each
//               half of the tile's tokens: dequantise the accumulator in place (tcgen05.ld /
//               tcgen05.st), wait for the correction MMA, read the result, transpose it through shared
//               memory and store y with TMA
//   warps 6-9   expand the packed tile into tensor memory
//   warp 10     producer of the packed codes (1 KiB tiles of eight consecutive row tiles of the tiled weight
//               layout per stage, with one TMA copy), in a ring that runs ahead of the activations'
// Codes are c = t + 1 (both operands are declared signed 8-bit; 0, 1, 2 read the same either way);
// sum_k t x~ = sum_k c x~ - sum_k x~ is restored in the epilogue from the row sums.
//
// Every wait is bounded: when one gives up, the CTA records it in the device status word, all
// roles leave their loops, in-flight bulk copies are drained, tensor memory is freed and the
// kernel returns.
#include "hgf_tc.cuh"
#include "hgf_warp.cuh"

namespace hgf {

constexpr int TILE_C = 128;   // output channels per tile (MMA M, tensor-memory lanes)
constexpr int TILE_T = 128;   // tokens per tile (MMA N, accumulator columns) at most: see prefill_tile_tokens
constexpr int KBLK = 256;      // input columns per pipeline stage: one column tile of the packed layout
constexpr int X_HALF_BYTES = TILE_T * 128;       // 16 KiB: 128 tokens x 128 columns, one 128-byte-swizzled operand tile
constexpr int X_TILE_BYTES = 2 * X_HALF_BYTES;   // 32 KiB per stage
constexpr int P_TILE_BYTES = TILE_C * KBLK / 4;  // 8 KiB: 8 weight tiles of 16 rows x 256 columns
constexpr int TOKV_BYTES = TILE_T * 8;           // row sums and scales of the tile's tokens
constexpr int STORE_BUF_BYTES = 2048;            // per epilogue warp: 32 channels x 32 tokens (bf16) or x 16 tokens (fp32)
constexpr int GEMM_THREADS = 480;  // 15 warps
// tensor memory: two accumulators of 128 columns, then one weight operand of 64 columns (= 256 int8 per lane) per stage
constexpr int TMEM_COLS = 512, ACC_COLS = TILE_T, A_COL = 2 * ACC_COLS, A_STAGE_COLS = KBLK / 4;

// Shared-memory map and barrier slots of a kernel variant.  NS = pipeline stages (activation tile +
// packed codes in shared memory, weight operand in tensor memory).  OPSB = bytes per row of the
// correction's two operand tiles: 128 (64 fp16, any rank), or 64 when r <= 32 - which leaves room
// for a fourth stage.
template <int NS, int OPSB>
struct Cfg {
    static constexpr int STAGES = NS;
    static constexpr int PSTAGES = NS + 1;  // the packed codes run one stage further ahead than the activations
    static constexpr int LORA_H_BYTES = TILE_T * OPSB, LORA_B_BYTES = TILE_C * OPSB;
    static constexpr int OFF_X = 0;
    static constexpr int OFF_LH = OFF_X + NS * X_TILE_BYTES;
    static constexpr int OFF_LB = OFF_LH + 2 * LORA_H_BYTES;  // the epilogue's operands are double-buffered like the accumulators
    static constexpr int OFF_P = OFF_LB + 2 * LORA_B_BYTES;
    static constexpr int OFF_TOKV = OFF_P + PSTAGES * P_TILE_BYTES;
    static constexpr int OFF_ST = OFF_TOKV + 2 * TOKV_BYTES;
    static constexpr int OFF_BAR = OFF_ST + 8 * STORE_BUF_BYTES;
    static constexpr int SMEM_BYTES = OFF_BAR + 512 + 1024;  // + slack for the 1024-byte alignment of the base
    // barrier slots (8 bytes each) inside the OFF_BAR block
    static constexpr int BAR_FULL = 0, BAR_EMPTY = BAR_FULL + NS, BAR_PFULL = BAR_EMPTY + NS, BAR_PEMPTY = BAR_PFULL + PSTAGES,
                         BAR_ACCFULL = BAR_PEMPTY + PSTAGES,
                         BAR_ACCEMPTY = BAR_ACCFULL + 2, BAR_LORAREADY = BAR_ACCEMPTY + 2, BAR_LORADONE = BAR_LORAREADY + 2,
                         BAR_OPSFULL = BAR_LORADONE + 2, BAR_OPSEMPTY = BAR_OPSFULL + 2, 
                         BAR_SPLIT = BAR_OPSEMPTY + 2, BAR_COUNT = BAR_SPLIT + 1;
    static_assert(SMEM_BYTES <= 227 * 1024, "shared memory budget");
    static_assert(BAR_COUNT * 8 + 16 <= 512, "barrier block too small");
    static_assert(A_COL + NS * A_STAGE_COLS <= TMEM_COLS, "tensor memory budget");
};

// Instruction descriptor: D format (bits 4-5), A format (7-9), B format (10-12), K-major A and B,
// N >> 3 (17-22), M >> 4 (24-28).
constexpr uint32_t IDESC_I8 = (2u << 4) /*s32*/ | (1u << 7) /*A s8*/ | (1u << 10) /*B s8*/ | ((uint32_t)(TILE_C >> 4) << 24);  // (N: the launch's)
constexpr uint32_t IDESC_F16 = (1u << 4) /*f32*/ | (0u << 7) /*A f16*/ | (0u << 10) /*B f16*/ | ((uint32_t)(TILE_C >> 4) << 24);

// SPLIT: a layer with fewer tiles than half the SMs has each tile's K divided over a cluster of 2, 4 or 8 CTAs (one tile a
// cluster, the tile loops below run once).  The CTAs keep their int32 sums in tensor memory, hand each other
// the token chunks the others own through distributed shared memory (st.async into the spent operand ring, counted
// by the receiver's mbarrier), and each finishes its own 128 / S tokens; the sums are exact in any order.
template <bool OUT_BF16, int NS, int OPSB, bool SPLIT>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
prefill_gemm_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_h,
                    const __grid_constant__ CUtensorMap tmap_gb, const __grid_constant__ CUtensorMap tmap_y,
                    const __grid_constant__ CUtensorMap tmap_w, const GemmParams p, unsigned int *status) {
    using C = Cfg<NS, OPSB>;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *smem = reinterpret_cast<uint8_t *>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const uint32_t sbase = smem_u32(smem);
    const uint32_t bar0 = sbase + C::OFF_BAR;
    auto bar = [&](int i) { return bar0 + 8u * i; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem + C::OFF_BAR + C::BAR_COUNT * 8);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(smem + C::OFF_BAR + C::BAR_COUNT * 8 + 4);
    static_assert(TILE_T == 128, "a tile has 128 tokens or 64: the epilogue's warps take half of them each, in steps of 32 or 16");

    // the next launch in the stream, if it asks for it, may be set up while this one runs (it waits
    // for this grid's completion before it touches memory)
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int S = SPLIT ? 1 << p.split_log2 : 1, rank = SPLIT ? (int)blockIdx.x & (S - 1) : 0;
    const int tile_first = SPLIT ? (int)blockIdx.x >> p.split_log2 : (int)blockIdx.x, tile_step = SPLIT ? (int)gridDim.x >> p.split_log2 : (int)gridDim.x;
    bool arrived = false, waited = false;  // (SPLIT) the cluster barrier that frees the operand rings
    const int T = SPLIT ? TILE_T : p.tile_t;  // tokens of a tile
    const int tiles_t = (p.M + T - 1) / T, tiles_c = (p.N + TILE_C - 1) / TILE_C;
    const int num_tiles = tiles_t * tiles_c;
    const int kblocks = (p.K + KBLK - 1) / KBLK, kb0 = SPLIT ? rank * kblocks / S : 0, kb1 = SPLIT ? (rank + 1) * kblocks / S : kblocks;
    const bool has_lora = p.r > 0;

    if (tid == 0) {
        for (int s = 0; s < C::STAGES; ++s) {
            // FULL: the stage's activation tile has landed (producer's arrival + bytes) and the four unpack
            // warps have put the weight operand into tensor memory, so the MMA warp waits on this one
            // barrier only (every barrier operation costs it a shared-memory round trip).  EMPTY: the MMAs that read the stage are complete (one commit; the producer
            // and the unpack warps both wait on it).
            mbar_init(bar(C::BAR_FULL + s), 1 + 4);
            mbar_init(bar(C::BAR_EMPTY + s), 1);
        }
        for (int j = 0; j < C::PSTAGES; ++j) {
            // the packed codes have a ring of their own, filled ahead of the activations: the expansion into
            // tensor memory then starts the moment a stage's MMAs are complete, in parallel with the reload
            // of the activation tile, instead of after it
            mbar_init(bar(C::BAR_PFULL + j), 1);
            mbar_init(bar(C::BAR_PEMPTY + j), 4);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(bar(C::BAR_ACCFULL + b), 1);
            mbar_init(bar(C::BAR_ACCEMPTY + b), 8);
            mbar_init(bar(C::BAR_LORAREADY + b), 8);
            mbar_init(bar(C::BAR_LORADONE + b), 1);
            mbar_init(bar(C::BAR_OPSFULL + b), 1);
            mbar_init(bar(C::BAR_OPSEMPTY + b), 8);
        }
        if (SPLIT) {
            mbar_init(bar(C::BAR_SPLIT), 1);
            mbar_arrive_expect_tx(bar(C::BAR_SPLIT), (uint32_t)((S - 1) * (8 / S) * TILE_C * 16 * 4));
        }
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
        fence_proxy_async();
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);  // (warp-uniform)
    // Everything above touches only this CTA's own shared and tensor memory; what follows reads what
    // the prologue launch wrote (a no-op unless the launch carries the programmatic-dependency attribute).
    // The packed codes it does not write: where their producer and the expansion may start at once (early_weights), the first stages'
    // operands are in tensor memory by the time the prologue is complete.  Microseconds of a layer call, all warps waiting / this:
    // 2048 -> 2048 13.6 / 12.2 at M = 64, with a LayerNorm 28.7 / 27.7 at M = 2000; 5632 -> 2048 21.4 / 21.1 at M = 512; 2048 -> 5632
    // 124.1 / 122.4 at M = 8192.
    if (!(p.early_weights && warp >= 6 && warp < 11)) asm volatile("griddepcontrol.wait;\n" ::: "memory");

    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        // The whole warp walks the loop: every lane polls the barriers, lane 0 posts the byte counts and issues the copies, two a
        // stage (the activation tile's halves) and up to four a tile (the epilogue's operands).
        {
            int s = 0;
            uint32_t ph = 0;
            uint32_t issued[C::STAGES] = {}, ops_issued[2] = {};
            int pit = 0;
            bool ok = true;
            for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step) {
                const int t0 = (tile % tiles_t) * T, c0 = (tile / tiles_t) * TILE_C;
                {
                    // what the tile's epilogue needs, into the buffer of the tile's accumulator: row sums and
                    // scales of the T tokens, and with a correction the H tile and the (g B)^T tile
                    const int b = pit & 1;
                    ok = mbar_wait(bar(C::BAR_OPSEMPTY + b), ((uint32_t)(pit >> 1) & 1u) ^ 1u, abort_flag, status, 0x120u + b);
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                    if (lane == 0) {
                        mbar_arrive_expect_tx(bar(C::BAR_OPSFULL + b), 2u * T * 4u + (has_lora ? T * OPSB + C::LORA_B_BYTES : 0));
                        bulk_load_1d(sbase + C::OFF_TOKV + b * TOKV_BYTES, p.row_sum + t0, T * 4u, bar(C::BAR_OPSFULL + b));
                        bulk_load_1d(sbase + C::OFF_TOKV + b * TOKV_BYTES + TILE_T * 4, p.tok_sc + t0, T * 4u, bar(C::BAR_OPSFULL + b));
                        if (has_lora) {
                            tma_load_2d(sbase + C::OFF_LH + b * C::LORA_H_BYTES, &tmap_h, 0, t0, bar(C::BAR_OPSFULL + b));
                            tma_load_2d(sbase + C::OFF_LB + b * C::LORA_B_BYTES, &tmap_gb, 0, c0, bar(C::BAR_OPSFULL + b));
                        }
                    }
                    ++ops_issued[b];
                    ++pit;
                }
                for (int kb = kb0; kb < kb1; ++kb) {
                    ok = mbar_wait(bar(C::BAR_EMPTY + s), ph ^ 1u, abort_flag, status, 0x100u + s);
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                    if (lane == 0) {
                        // 256 columns of T tokens as two 128-byte-swizzled tiles (columns past K read as zeros)
                        mbar_arrive_expect_tx(bar(C::BAR_FULL + s), 2u * 128u * T);
                        tma_load_2d(sbase + C::OFF_X + s * X_TILE_BYTES, &tmap_x, kb * KBLK, t0, bar(C::BAR_FULL + s));
                        tma_load_2d(sbase + C::OFF_X + s * X_TILE_BYTES + X_HALF_BYTES, &tmap_x, kb * KBLK + 128, t0, bar(C::BAR_FULL + s));
                    }
                    ++issued[s];
                    if (++s == C::STAGES) { s = 0; ph ^= 1u; }
                }
            }
            // drain: wait (bounded) until every copy this warp issued has landed, so that the CTA
            // never exits with a bulk copy in flight (immediate when the consumers ran to the end)
            for (int q = 0; q < C::STAGES; ++q)
                if (issued[q]) {
                    const uint32_t par = (issued[q] - 1u) & 1u;
                    for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_FULL + q), par); ++i) {}
                }
            for (int q = 0; q < 2; ++q)
                if (ops_issued[q]) {
                    const uint32_t par = (ops_issued[q] - 1u) & 1u;
                    for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_OPSFULL + q), par); ++i) {}
                }
        }
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        // Tile `it` accumulates into accumulator it % 2, so the epilogue of one tile runs under the main
        // loop of the next.  With a correction, the epilogue first rewrites the accumulator as fp32
        // (dequantised), then this warp adds (g B) H^T onto it with one more MMA, slipped in between
        // the k blocks of the tile in progress as soon as the epilogue is ready for it.
        //
        // The whole warp walks the loop and elect.sync picks the lane that issues, so the descriptors live in
        // uniform registers: eight MMAs take 230 clocks to issue, a stage 750 with its two barriers.  (One thread in a
        // divergent branch needed 1100, two such threads taking stages in turns 890.)  Large layers are then held by
        // the power limit: 1.75 GHz at 985 W, 8192 x 2048 x 5632 in 122.4 us against 126.1, 4096 x 4096 x 11008 in 201.5
        // against 209.8 (with the swizzled weight tiles of launch_prefill_gemm 118.6 and 194); two issuing warps, or asking for the next stage ahead of time, change neither.
        {
            auto wait = [&](int i, uint32_t par, unsigned int code) { return __all_sync(0xffffffffu, mbar_wait_poll(bar(i), par, abort_flag, status, code)) != 0; };
            bool ok = true;
            int it = 0, pend = -1;  // pend: tile whose correction MMA is still to be issued
            int gs = 0;             // stage number, counted through all tiles of this CTA
            const uint64_t xdesc0 = make_sw128_desc(sbase + C::OFF_X);
            const uint32_t idesc_i8 = IDESC_I8 | ((uint32_t)(T >> 3) << 17), idesc_f16 = IDESC_F16 | ((uint32_t)(T >> 3) << 17);
            auto issue_lora = [&](int t) {
                const int b = t & 1;
                tc_fence_after();
                const uint32_t la = sbase + C::OFF_LB + b * C::LORA_B_BYTES, lh = sbase + C::OFF_LH + b * C::LORA_H_BYTES;
                const uint64_t adesc = OPSB == 128 ? make_sw128_desc(la) : make_sw64_desc(la);
                const uint64_t bdesc = OPSB == 128 ? make_sw128_desc(lh) : make_sw64_desc(lh);
#pragma unroll
                for (int kk = 0; kk < OPSB / 32; ++kk)  // K = 16 fp16 (32 bytes of a row) per MMA, on top of the fp32 values
                    warp_mma_f16(tmem_base + b * ACC_COLS, adesc + 2u * kk, bdesc + 2u * kk, idesc_f16, 1u);
                warp_commit(bar(C::BAR_LORADONE + b));
            };
            for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step, ++it) {
                const int b = it & 1;
                const uint32_t acc = tmem_base + b * ACC_COLS;
                if (it >= 2 && !(ok = wait(C::BAR_ACCEMPTY + b, (uint32_t)((it >> 1) - 1) & 1u, 0x200u))) break;
                for (int kb = kb0; kb < kb1; ++kb, ++gs) {
                    if (pend >= 0 && __all_sync(0xffffffffu, mbar_test_wait(bar(C::BAR_LORAREADY + (pend & 1)), (uint32_t)(pend >> 1) & 1u))) {
                        issue_lora(pend);
                        pend = -1;
                    }
                    const int s = gs % C::STAGES;
                    const uint32_t ph = (uint32_t)(gs / C::STAGES) & 1u;
                    if (!(ok = wait(C::BAR_FULL + s, ph, 0x210u + s))) break;
                    tc_fence_after();
                    const uint64_t bdesc = xdesc0 + (uint64_t)(s * (X_TILE_BYTES >> 4));
                    const uint32_t a_tmem = tmem_base + A_COL + s * A_STAGE_COLS;
                    warp_mma_i8_ts(acc, a_tmem, bdesc, idesc_i8, kb > kb0 ? 1u : 0u);
                    warp_mma_i8_ts(acc, a_tmem + 8u, bdesc + 2u, idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 16u, bdesc + 4u, idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 24u, bdesc + 6u, idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 32u, bdesc + (X_HALF_BYTES >> 4), idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 40u, bdesc + (X_HALF_BYTES >> 4) + 2u, idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 48u, bdesc + (X_HALF_BYTES >> 4) + 4u, idesc_i8, 1u);
                    warp_mma_i8_ts(acc, a_tmem + 56u, bdesc + (X_HALF_BYTES >> 4) + 6u, idesc_i8, 1u);
                    warp_commit(bar(C::BAR_EMPTY + s));
                }
                if (!ok) break;
                warp_commit(bar(C::BAR_ACCFULL + b));
                if (SPLIT) { cluster_arrive_release(); arrived = true; }
                if (pend >= 0) {  // the previous tile's correction has to be out before its accumulator's next turn
                    if (!(ok = wait(C::BAR_LORAREADY + (pend & 1), (uint32_t)(pend >> 1) & 1u, 0x230u)))
                        break;
                    issue_lora(pend);
                    pend = -1;
                }
                if (has_lora) pend = it;
            }
            if (ok && pend >= 0 && wait(C::BAR_LORAREADY + (pend & 1), (uint32_t)(pend >> 1) & 1u, 0x231u)) issue_lora(pend);
        }
    } else if (warp < 6 || warp >= 11) {
        // ------------------------------------------------------------------ epilogue warps
        // Eight of them: the warp pair of a tensor-memory lane quarter (32 output channels) shares the
        // tile's 128 tokens, 64 each, so a tile's epilogue takes half as long as with one warp per
        // quarter: the main loop of a short-K tile is over sooner than that.
        const int e2 = warp < 6 ? 0 : 1;                  // which half of the tile's tokens
        const int q = warp & 3;                           // tensor-memory lane quarter this warp may access
        const int half_t = T / 2;
        constexpr int W = OUT_BF16 ? 32 : 16;             // tokens per staging step (2 KiB of staging either way)
        uint8_t *buf = smem + C::OFF_ST + (4 * e2 + q) * STORE_BUF_BYTES;
        bool ok = true;
        int it = 0;
        for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step, ++it) {
            const int t0 = (tile % tiles_t) * T, c0 = (tile / tiles_t) * TILE_C;
            const int b = it & 1;
            const uint32_t par = (uint32_t)(it >> 1) & 1u;
            // the tile's row sums and scales (and the correction's operands) were fetched by the producer
            const int *tok_rs = reinterpret_cast<const int *>(smem + C::OFF_TOKV + b * TOKV_BYTES);
            const float *tok_sc = reinterpret_cast<const float *>(tok_rs + TILE_T);
            ok = mbar_wait(bar(C::BAR_OPSFULL + b), par, abort_flag, status, 0x320u + b);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;

            const int n = c0 + 32 * q + lane;  // this thread's output channel = its tensor-memory lane
            const bool n_ok = n < p.N;

            ok = mbar_wait(bar(C::BAR_ACCFULL + b), par, abort_flag, status, 0x300u);
            if (!(ok = __all_sync(0xffffffffu, ok))) break;  // the whole warp leaves together
            tc_fence_after();
            const uint32_t lane_base = tmem_base + ((uint32_t)(32 * q) << 16) + b * ACC_COLS;

            // int32 sums -> fp32 (Y_int - row sum) * scale, for the WN tokens from cc on
            // (the per-token values are read as vectors ahead of the arithmetic: a shared-memory load per
            // element in the dependent chain costs its full latency every time)
            auto dequant_chunk = [&](int cc, auto &ai) {
                constexpr int WN = (int)(sizeof(ai) / sizeof(uint32_t));
                if (p.dbg_y_int && n_ok) {
#pragma unroll
                    for (int j = 0; j < WN; ++j)
                        if (t0 + cc + j < p.M) p.dbg_y_int[(size_t)(t0 + cc + j) * p.N + n] = (int)ai[j] - tok_rs[cc + j];
                }
#pragma unroll
                for (int v = 0; v < WN / 4; ++v) {
                    const int4 rs4 = *reinterpret_cast<const int4 *>(tok_rs + cc + 4 * v);
                    const float4 sc4 = *reinterpret_cast<const float4 *>(tok_sc + cc + 4 * v);
                    ai[4 * v + 0] = __float_as_uint((float)((int)ai[4 * v + 0] - rs4.x) * sc4.x);
                    ai[4 * v + 1] = __float_as_uint((float)((int)ai[4 * v + 1] - rs4.y) * sc4.y);
                    ai[4 * v + 2] = __float_as_uint((float)((int)ai[4 * v + 2] - rs4.z) * sc4.z);
                    ai[4 * v + 3] = __float_as_uint((float)((int)ai[4 * v + 3] - rs4.w) * sc4.w);
                }
            };
            if constexpr (SPLIT) {
                // chunks of 16 tokens: chunk c belongs to CTA c / (8 / S); this warp works those of its parity
                cluster_arrive_release();
                arrived = waited = true;
                cluster_wait_acquire();  // every CTA's MMAs are complete: the operand rings are free
                const int per = 8 / S;
                for (int c = e2; c < 8; c += 2) {
                    const int owner = c / per;
                    if (owner == rank) continue;
                    uint32_t ai[16];
                    tmem_ld16(lane_base + 16 * c, ai);
                    tmem_ld_wait();
                    const uint32_t dst = sbase + C::OFF_X + ((rank * per + c % per) * 4 + q) * 2048 + 16 * lane;
#pragma unroll
                    for (int v = 0; v < 4; ++v)
                        st_async_v4(dst + 512 * v, bar(C::BAR_SPLIT), (uint32_t)owner, ai[4 * v], ai[4 * v + 1], ai[4 * v + 2], ai[4 * v + 3]);
                }
                ok = mbar_wait_poll(bar(C::BAR_SPLIT), 0u, abort_flag, status, 0x330u);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                for (int c = rank * per; c < (rank + 1) * per; ++c) {
                    if ((c & 1) != e2) continue;
                    uint32_t ai[16];
                    tmem_ld16(lane_base + 16 * c, ai);
                    tmem_ld_wait();
                    for (int o = 0; o < S; ++o) {
                        if (o == rank) continue;
                        const uint8_t *src = smem + C::OFF_X + ((o * per + c % per) * 4 + q) * 2048 + 16 * lane;
#pragma unroll
                        for (int v = 0; v < 4; ++v) {
                            const uint4 a = *reinterpret_cast<const uint4 *>(src + 512 * v);
                            ai[4 * v] += a.x; ai[4 * v + 1] += a.y; ai[4 * v + 2] += a.z; ai[4 * v + 3] += a.w;
                        }
                    }
                    dequant_chunk(16 * c, ai);
                    tmem_st16(lane_base + 16 * c, ai);
                }
                tmem_st_wait();
                if (has_lora) {
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbar_arrive(bar(C::BAR_LORAREADY + b));
                    ok = mbar_wait_poll(bar(C::BAR_LORADONE + b), par, abort_flag, status, 0x310u);
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                    tc_fence_after();
                }
                for (int c = rank * per; c < (rank + 1) * per; ++c) {
                    if ((c & 1) != e2) continue;
                    uint32_t ai[16];
                    tmem_ld16(lane_base + 16 * c, ai);
                    tmem_ld_wait();
                    if (lane == 0) bulk_wait_read<0>();
                    __syncwarp();
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        if (OUT_BF16) reinterpret_cast<__nv_bfloat16 *>(buf)[j * 32 + lane] = __float2bfloat16_rn(__uint_as_float(ai[j]));
                        else reinterpret_cast<uint32_t *>(buf)[j * 32 + lane] = ai[j];
                    }
                    fence_proxy_async();
                    __syncwarp();
                    if (lane == 0) {
                        tma_store_2d(&tmap_y, c0 + 32 * q, t0 + 16 * c, smem_u32(buf));
                        bulk_commit();
                    }
                }
                break;  // one tile a cluster
            }
            if (has_lora) {
                // first pass: dequantise in place (int32 -> fp32), then let the MMA warp add the correction
                for (int cc = half_t * e2; cc < half_t * (e2 + 1); cc += 32) {
                    uint32_t ai[32];
                    tmem_ld32(lane_base + cc, ai);
                    tmem_ld_wait();
                    dequant_chunk(cc, ai);
                    tmem_st32(lane_base + cc, ai);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(bar(C::BAR_LORAREADY + b));
                ok = mbar_wait(bar(C::BAR_LORADONE + b), par, abort_flag, status, 0x310u);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                tc_fence_after();
            }

            // read the result, transpose it through shared memory (a thread holds one channel of W
            // tokens; y wants the channels of a token next to each other) and store with TMA
            for (int cc = half_t * e2; cc < half_t * (e2 + 1); cc += W) {
                uint32_t ai[W];
                if constexpr (W == 32) tmem_ld32(lane_base + cc, ai); else tmem_ld16(lane_base + cc, ai);
                tmem_ld_wait();
                if (!has_lora) dequant_chunk(cc, ai);
                // the buffer was handed to a TMA store one chunk ago: wait until it was read
                if (lane == 0) bulk_wait_read<0>();
                __syncwarp();
                if (OUT_BF16) {
#pragma unroll
                    for (int j = 0; j < W; ++j)
                        reinterpret_cast<__nv_bfloat16 *>(buf)[j * 32 + lane] = __float2bfloat16_rn(__uint_as_float(ai[j]));
                } else {
#pragma unroll
                    for (int j = 0; j < W; ++j) reinterpret_cast<uint32_t *>(buf)[j * 32 + lane] = ai[j];
                }
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) {
                    tma_store_2d(&tmap_y, c0 + 32 * q, t0 + cc, smem_u32(buf));
                    bulk_commit();
                }
            }
            // all tensor-memory reads of this tile are done: hand the accumulator back to the MMA warps
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bar(C::BAR_ACCEMPTY + b));
                mbar_arrive(bar(C::BAR_OPSEMPTY + b));
            }
        }
        if (lane == 0) bulk_wait_read<0>();
        __syncwarp();
    } else if (warp == 10) {
        // ------------------------------------------------------------------ packed-code producer
        // Its own warp and ring: the codes run ahead of the activations, so the expansion into tensor
        // memory starts the moment a stage's MMAs are complete, in parallel with the reload of the
        // activation tile.  Per stage the 1 KiB tiles (16 rows x 256 columns) of 8 consecutive row tiles with one
        // copy (row tiles past the matrix are zeros); as eight bulk copies 512 tokens of 5632 -> 2048 took 21.0 us in place
        // of 20.7, 64 of 2048 -> 2048 11.15 in place of 11.0.
        int pj = 0;
        uint32_t pph = 0;
        uint32_t pissued[C::PSTAGES] = {};
        bool ok = true;
        for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step) {
            const int rt0 = ((tile / tiles_t) * TILE_C) >> 4;
            for (int kb = kb0; kb < kb1; ++kb) {
                ok = mbar_wait(bar(C::BAR_PEMPTY + pj), pph ^ 1u, abort_flag, status, 0x110u + pj);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;
                if (lane == 0) {
                    mbar_arrive_expect_tx(bar(C::BAR_PFULL + pj), P_TILE_BYTES);
                    tma_load_4d(sbase + C::OFF_P + pj * P_TILE_BYTES, &tmap_w, 0, 0, kb, rt0, bar(C::BAR_PFULL + pj));
                }
                ++pissued[pj];
                if (++pj == C::PSTAGES) { pj = 0; pph ^= 1u; }
            }
        }
        for (int q = 0; q < C::PSTAGES; ++q)
            if (pissued[q]) {
                const uint32_t par = (pissued[q] - 1u) & 1u;
                for (uint32_t i = 0; i < kSpinLimit && !mbar_try_wait(bar(C::BAR_PFULL + q), par); ++i) {}
            }
    } else {
        // ------------------------------------------------------------------ unpack warps
        const int q = warp & 3;              // tensor-memory lane quarter this warp may access
        const int row = 32 * q + lane;       // this thread's channel row of the tile = its tensor-memory lane
        const int swizzle = (row >> 1) & 3;  // (of the 16-byte units of its codes: see the tensor map)
        int s = 0, pj = 0;
        uint32_t ph = 0, pph = 0;
        bool ok = true;
        for (int tile = tile_first; ok && tile < num_tiles; tile += tile_step) {
            for (int kb = kb0; kb < kb1; ++kb) {
                // the stage's packed codes have landed, and the MMAs that read this stage's previous operand
                // are complete
                ok = mbar_wait(bar(C::BAR_PFULL + pj), pph, abort_flag, status, 0x400u + pj) &&
                     mbar_wait(bar(C::BAR_EMPTY + s), ph ^ 1u, abort_flag, status, 0x410u + s);
                if (!(ok = __all_sync(0xffffffffu, ok))) break;  // the whole warp leaves together
                // this row's 64 bytes hold the stage's 256 columns; register 4 i + j of a half = columns
                // 16 i + 4 j .. + 3, one code per byte
                const uint8_t *prow = smem + C::OFF_P + pj * P_TILE_BYTES + row * 64;
                const uint32_t taddr = tmem_base + ((uint32_t)(32 * q) << 16) + A_COL + s * A_STAGE_COLS;
#pragma unroll
                for (int half = 0; half < 2; ++half) {
                    const uint4 lo = *reinterpret_cast<const uint4 *>(prow + ((2 * half) ^ swizzle) * 16);
                    const uint4 hi = *reinterpret_cast<const uint4 *>(prow + ((2 * half + 1) ^ swizzle) * 16);
                    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
                    uint32_t a[32];
#pragma unroll
                    for (int i = 0; i < 8; ++i)
#pragma unroll
                        for (int j = 0; j < 4; ++j) a[4 * i + j] = (w[i] >> (2 * j)) & 0x03030303u;
                    tmem_st32(taddr + 32 * half, a);
                }
                tmem_st_wait();
                tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(bar(C::BAR_FULL + s));
                    mbar_arrive(bar(C::BAR_PEMPTY + pj));
                }
                if (++pj == C::PSTAGES) { pj = 0; pph ^= 1u; }
                if (++s == C::STAGES) { s = 0; ph ^= 1u; }
            }
        }
    }

    if constexpr (SPLIT) {
        // every thread arrives once, whatever happened above; then no CTA leaves while another may still write into it
        __syncwarp();
        if (!arrived) cluster_arrive_release();
        if (!waited) cluster_wait_acquire();
        cluster_arrive_release();
        cluster_wait_acquire();
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
    }
}

// The bounded wait on a barrier that nothing completes: it gives up after `limit_ns`, records that
// in the status word and the kernel returns (the error path of every role above, exercised alone).
__global__ void wait_timeout_selftest_kernel(unsigned long long limit_ns, unsigned int *status) {
    __shared__ __align__(8) unsigned long long bar_mem;
    __shared__ int abort_mem;
    const uint32_t bar = smem_u32(&bar_mem);
    if (threadIdx.x == 0) {
        mbar_init(bar, 1);
        abort_mem = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) mbar_wait(bar, 0u, &abort_mem, status, 0x700u, limit_ns);
}

cudaError_t launch_wait_timeout_selftest(unsigned long long limit_ns, cudaStream_t stream) {
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    wait_timeout_selftest_kernel<<<1, 32, 0, stream>>>(limit_ns, status);
    count_launch();
    return cudaGetLastError();
}

// ---- host side: tensor maps and launch -----------------------------------------------------------
template <bool OUT_BF16, int NS, int OPSB, bool SPLIT>
static cudaError_t launch_split(const CUtensorMap &mx, const CUtensorMap &mh, const CUtensorMap &mgb, const CUtensorMap &my, const CUtensorMap &mw,
                                  const GemmParams &p, int grid, unsigned int *status, cudaStream_t stream) {
    static std::atomic<unsigned long long> attr_done{0};
    constexpr int smem = Cfg<NS, OPSB>::SMEM_BYTES;
    {
        cudaError_t e = ensure_dynamic_smem(prefill_gemm_kernel<OUT_BF16, NS, OPSB, SPLIT>, smem, attr_done);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3(GEMM_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = (p.flags & HGF_FLAG_NO_PDL) ? 0 : 1;  // set-up (barriers, tensor memory) may overlap the prologue's tail
    if (SPLIT) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
        attr[cfg.numAttrs].val.clusterDim.x = 1u << p.split_log2;
        attr[cfg.numAttrs].val.clusterDim.y = 1;
        attr[cfg.numAttrs].val.clusterDim.z = 1;
        ++cfg.numAttrs;
    }
    cudaError_t e = cudaLaunchKernelEx(&cfg, prefill_gemm_kernel<OUT_BF16, NS, OPSB, SPLIT>, mx, mh, mgb, my, mw, p, status);
    return e != cudaSuccess ? e : cudaGetLastError();
}

template <bool OUT_BF16, int NS, int OPSB>
static cudaError_t launch_variant(const CUtensorMap &mx, const CUtensorMap &mh, const CUtensorMap &mgb, const CUtensorMap &my, const CUtensorMap &mw,
                                  const GemmParams &p, int grid, unsigned int *status, cudaStream_t stream) {
    return p.split_log2 ? launch_split<OUT_BF16, NS, OPSB, true>(mx, mh, mgb, my, mw, p, grid, status, stream)
                        : launch_split<OUT_BF16, NS, OPSB, false>(mx, mh, mgb, my, mw, p, grid, status, stream);
}

// Tokens of a tile: 64 where that many tiles still run in one round (or there are no more), else 128.  A tile of 64 halves the products, the
// copies of x~ and the epilogue of a CTA, but not the expansion of its weights, so more rounds than one cost more than they save.
// Microseconds of a layer call in a captured chain, tiles of 128 / 112 / 96 / 80 / 64 / 48: 1024 -> 1024 9.7 / 9.7 / 9.1 / 9.1 / 8.5 / 8.4 at M = 100
// (16 tiles of 64), 13.5 / 14.0 / 12.6 / 12.6 / 11.4 / 12.6 at M = 512 (64), 11.9 / 11.9 / 11.5 / 11.4 / 10.9 / 12.0 at M = 1000 (128), 13.0 / 13.0 / 12.7 /
// 14.0 / 13.1 / 13.9 at M = 1500 (192); 2048 -> 5632 11.7 / 11.5 / 11.1 / 11.0 / 10.5 / 11.6 at M = 100 (88), 12.5 / 12.4 / 12.8 / 12.7 / 14.5 / 14.6 at
// M = 200 (176); 2048 -> 2048 14.6 / 15.6 / 15.1 / 14.7 / 14.3 / 17.5 at M = 512 (128), 19.9 / 20.9 / 20.4 / 22.6 / 23.0 / 26.3 at M = 1500.
static int prefill_tile_tokens(int M, int N, int sms) {
    const long long tiles = (long long)((M + 63) / 64) * ((N + TILE_C - 1) / TILE_C);
    return M <= 64 || tiles <= sms ? 64 : TILE_T;
}

cudaError_t launch_prefill_gemm(const GemmParams &p_in, cudaStream_t stream) {
    GemmParams p = p_in;
    const int sm_count = device_sm_count();
    if (!sm_count) return cudaErrorInvalidDevice;
    const bool bf16 = (p.flags & HGF_FLAG_OUT_BF16) != 0;
    const bool narrow = p.r <= 32;  // 64-byte operand rows for the correction, and room for a fourth stage
    const int tiles = ((p.M + TILE_T - 1) / TILE_T) * ((p.N + TILE_C - 1) / TILE_C), kblocks = (p.K + KBLK - 1) / KBLK;
    // K divided over a cluster where tiles leave SMs idle and K is long (at least 16 blocks of 256, four a CTA).  Microseconds of the
    // layer call in a captured chain, whole / over 2 / 4 / 8 CTAs: 5632 -> 2048 23.1 / 20.3 at M = 512 (64 tiles), 18.9 / 16.1 /
    // 14.4 at M = 64 (16 tiles); 11008 -> 1024 35.6 / 28.8 / 24.6 / 23.1 at M = 17 (8 tiles); 2048 -> 2048 12.0 / 11.7 / 11.3 at M = 64,
    // 15.6 / 15.3 / 17.5 at M = 256.  Clusters of four or eight do not fill the chip (an SM count that is no multiple of their
    // size in every part of it: 128 CTAs by eights took two rounds, 22.2 for 14.4), so they stop at half of it, except fours
    // with a very long K: 11008 -> 4096 32.6 / 28.6 / 25.8 at M = 128 (32 tiles).
    auto may_split = [&](int log2) {
        return kblocks >= (log2 == 1 ? 16 : 4 << log2) && (tiles << log2) <= (log2 == 1 || (log2 == 2 && kblocks >= 32) ? sm_count : sm_count / 2);
    };
    for (int log2 = 1; log2 <= 3; ++log2)
        if (may_split(log2)) p.split_log2 = log2;
    p.tile_t = p.split_log2 ? TILE_T : prefill_tile_tokens(p.M, p.N, sm_count);
    const uint32_t T = (uint32_t)p.tile_t;
    CUtensorMap mx, mh, mgb, my, mw;
    if (!make_map_2d(&mx, CU_TENSOR_MAP_DATA_TYPE_UINT8, p.xq, (uint64_t)p.K, (uint64_t)p.M, (uint64_t)p.K, 128, T,
                     CU_TENSOR_MAP_SWIZZLE_128B))
        return cudaErrorInvalidValue;
    if (p.r > 0) {  // H [M][64] and (g B)^T [N][64] fp16: tiles of 128 rows; the first 32 or all 64 columns
        const uint32_t cols = narrow ? 32 : 64;
        const CUtensorMapSwizzle sw = narrow ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
        if (!make_map_2d(&mh, CU_TENSOR_MAP_DATA_TYPE_UINT16, p.h16, 64, (uint64_t)p.M, 128, cols, T, sw)) return cudaErrorInvalidValue;
        if (!make_map_2d(&mgb, CU_TENSOR_MAP_DATA_TYPE_UINT16, p.gb16, 64, (uint64_t)p.N, 128, cols, TILE_C, sw)) return cudaErrorInvalidValue;
    } else {
        mh = mx;
        mgb = mx;
    }
    if (!make_map_2d(&my, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, p.y, (uint64_t)p.N,
                     (uint64_t)p.M, (uint64_t)p.N * (bf16 ? 2 : 4), 32, bf16 && !p.split_log2 ? 32 : 16, CU_TENSOR_MAP_SWIZZLE_NONE))
        return cudaErrorInvalidValue;
    const int work = ((p.M + p.tile_t - 1) / p.tile_t) * ((p.N + TILE_C - 1) / TILE_C);
    const int grid = p.split_log2 ? tiles << p.split_log2 : (work < sm_count ? work : sm_count);
    // the packed codes: [row tile][column tile][row][64 bytes].  The 64-byte swizzle puts the 16-byte units of neighbouring rows on different
    // banks for the expansion, whose threads read a row each: unswizzled, four rows of every eight met on the same banks, and the
    // shared-memory pipe, which also carries the tiles in and the activations to the tensor cores, was what a stage waited for.
    // 4096 -> 11008 at M = 4096 200.5 -> 194.9 us, 4096 -> 4096 at M = 4000 79.4 -> 74.7, at M = 1000 28.3 -> 26.8, 2048 -> 5632 at M = 8192
    // 120.9 -> 119.1, 5632 -> 2048 at M = 512 20.5 -> 20.1.
    const uint64_t w_dims[4] = {64, 16, (uint64_t)kblocks, (uint64_t)((p.N + 15) / 16)}, w_strides[3] = {64, 1024, (uint64_t)kblocks * 1024};
    const uint32_t w_box[4] = {64, 16, 1, TILE_C / 16};
    if (!make_map_4d(&mw, CU_TENSOR_MAP_DATA_TYPE_UINT8, p.packed, w_dims, w_strides, w_box, CU_TENSOR_MAP_SWIZZLE_64B)) return cudaErrorInvalidValue;
    unsigned int *status = device_status_word();
    if (!status) return cudaErrorMemoryAllocation;
    cudaError_t e;
    if (narrow)
        e = bf16 ? launch_variant<true, 4, 64>(mx, mh, mgb, my, mw, p, grid, status, stream)
                 : launch_variant<false, 4, 64>(mx, mh, mgb, my, mw, p, grid, status, stream);
    else
        e = bf16 ? launch_variant<true, 3, 128>(mx, mh, mgb, my, mw, p, grid, status, stream)
                 : launch_variant<false, 3, 128>(mx, mh, mgb, my, mw, p, grid, status, stream);
    count_launch();
    return e;
}

}  // namespace hgf
