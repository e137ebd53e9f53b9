// Offline weight preparation: absmean scale, ternary codes, 2-bit packing (and its inverse).
// Paper: Section 2.2, Definition "Absmax Quantization" (the scale is the mean of |W|).
#include "hgf_warp.cuh"

namespace hgf {

constexpr int kAbsBlocks = 1024;
constexpr int kAbsThreads = 256;

// Scratch of one scale computation: the blocks' partial sums, the scale, and the count of blocks that are done
// (zero between calls: the last block puts it back).
struct AbsScratch {
    double partials[kAbsBlocks];
    float gamma;
    unsigned int done;
    unsigned char pad[248];
};

// mean |W| into s->gamma.  Per-block sums in double (fixed grid-stride order, fixed tree), then the block that
// finishes last adds the partials with one warp (lane-strided, then a fixed shuffle tree) and rounds the mean
// once to fp32: the same order every time, whichever block is last.  As long as the sums and their addition took as two launches;
// what a packing call gained came from its scratch (below).  Four 16-byte loads in flight per thread, added in index order.
// What is beyond the bytes (5632 x 2048: 13.7 us where HBM needs 7) is the chain at either end: a thread's last loads, the partial sums
// of the last block and the start of the packing kernel were each waited for in turn.  Asked for together, and the packing kernel let in
// when the weights are read: whole calls, host to host, 5632 x 2048 51.3 -> 44.8 us, 1000 x 2048 40.4 -> 37.6, 333 x 1088 40.3 -> 32.7, 11008 x 4096
// 93.7 -> 91.8; 2048 x 2048 and 4096 x 4096, with no last loads, as before.  A training step of 64 x 512 -> 512 71.5 -> 64.7, 512 x 2048 -> 2048 112.6 -> 107.
__global__ void __launch_bounds__(kAbsThreads) abs_mean_kernel(const float4 *W4, size_t n4, double count, AbsScratch *s) {
    double acc = 0.0;
    const size_t stride = (size_t)gridDim.x * kAbsThreads;
    auto add = [&](const float4 &v) { acc += (double)fabsf(v.x) + (double)fabsf(v.y) + (double)fabsf(v.z) + (double)fabsf(v.w); };
    size_t i = (size_t)blockIdx.x * kAbsThreads + threadIdx.x;
    for (; i + 3 * stride < n4; i += 4 * stride) {
        const float4 v0 = W4[i], v1 = W4[i + stride], v2 = W4[i + 2 * stride], v3 = W4[i + 3 * stride];
        add(v0); add(v1); add(v2); add(v3);
    }
    float4 rest[3];  // (fewer than four left: asked for together, too)
#pragma unroll
    for (int u = 0; u < 3; ++u) rest[u] = i + u * stride < n4 ? W4[i + u * stride] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int u = 0; u < 3; ++u)
        if (i + u * stride < n4) add(rest[u]);
    pdl_launch_dependents();  // the packing kernel may ask for its weights
    __shared__ double red[kAbsBlocks];
    __shared__ bool last;
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int k = kAbsThreads / 2; k > 0; k >>= 1) {
        if (threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        s->partials[blockIdx.x] = red[0];
        __threadfence();
        last = atomicAdd(&s->done, 1u) + 1u == gridDim.x;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < kAbsBlocks; k += kAbsThreads) red[k + threadIdx.x] = __ldcg(&s->partials[k + threadIdx.x]);
    __syncthreads();
    if (threadIdx.x >= 32) return;
    double sum = 0.0;
#pragma unroll 8
    for (int k = threadIdx.x; k < kAbsBlocks; k += 32) sum += red[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (threadIdx.x == 0) {
        s->gamma = (float)(sum / count);
        s->done = 0u;
    }
}

// Decomposition of a packed word index into its place in the matrix.  Words are numbered in storage
// order: 16 per row segment, 16 row segments per tile, column tiles fastest, then row tiles.
struct WordPos {
    int64_t n, k0;  // output row and first of the 16 input columns the word covers
};
__device__ __forceinline__ WordPos word_pos(size_t w, int64_t steps) {
    const int64_t kw = (int64_t)(w & 15), r = (int64_t)((w >> 4) & 15);
    const int64_t tile = (int64_t)(w >> 8);
    WordPos p;
    p.n = (tile / steps) * 16 + r;
    p.k0 = (tile % steps) * 256 + kw * 16;
    return p;
}

// Sixteen lanes a row of a tile, 16 words of 16 weights.  Weight k0 + 4 j + b goes to bits
// 8 b + 2 j of the word; code = t + 1; t = sign(w) * [|w| > gamma/2].  Padding words hold code 1.
// Lane l asks for the 16 bytes l, l + 16, l + 32, l + 48 of the row, neighbours next to each other, before it waits for the scale;
// four lanes have the quarters of a word.  (A word a lane, 64 bytes apart, left the reading to the L1's tag look-ups.)
__global__ void __launch_bounds__(256) ternarise_pack_kernel(const float *W, int64_t N, int64_t K, int64_t steps,
                                                             const float *gamma, uint32_t *packed) {
    const size_t w = (size_t)blockIdx.x * 256 + threadIdx.x;  // (a block is a tile)
    const int l = threadIdx.x & 15;
    const WordPos p = word_pos(w - l, steps);
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const int64_t k = p.k0 + 64 * i + 4 * l;
        v[i] = p.n < N && k < K ? *reinterpret_cast<const float4 *>(W + p.n * K + k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);  // (0: code 1)
    }
    pdl_wait();
    const float half = 0.5f * __ldcg(gamma);  // exact
    uint32_t mine = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float e[4] = {v[i].x, v[i].y, v[i].z, v[i].w};
        uint32_t word = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) word |= (e[b] > half ? 2u : (e[b] < -half ? 0u : 1u)) << (8 * b);
        word <<= 2 * (l & 3);
        word |= __shfl_xor_sync(0xffffffffu, word, 1);
        word |= __shfl_xor_sync(0xffffffffu, word, 2);
        if ((l & 3) == i) mine = word;
    }
    packed[w - l + 4 * (l & 3) + (l >> 2)] = mine;
}

__global__ void __launch_bounds__(256) unpack_kernel(const uint32_t *packed, int64_t N, int64_t K, int64_t steps,
                                                     size_t n_words, int8_t *T) {
    size_t w = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (w >= n_words) return;
    const WordPos p = word_pos(w, steps);
    if (p.n >= N || p.k0 >= K) return;
    uint32_t word = packed[w];
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t e = (word >> (2 * j)) & 0x03030303u;  // codes 0..3 per byte
        uint32_t r = 0;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            int c = (e >> (8 * b)) & 0xff;
            int t = c == 3 ? 0 : c - 1;
            r |= (uint32_t)(t & 0xff) << (8 * b);
        }
        o[j] = r;
    }
    *reinterpret_cast<uint4 *>(T + p.n * K + p.k0) = make_uint4(o[0], o[1], o[2], o[3]);
}

// ---- base-3 layout: five codes per byte ---------------------------------------------------------
// Tiles of 16 rows x 320 columns, 64 bytes per row.  Byte q = 16 t + j of a row holds, as digits of a
// base-3 number, the codes of tile columns col(j, t) + 0..3 (digits 0..3) and col(16 + j / 4, t) + j % 4
// (digit 4), col(p, t) = 32 (p / 2) + 16 (p % 2) + 4 t: lane t of the decode kernel's warp MMA then
// finds the operand registers of its ten MMAs in its own 16 bytes of the row.
__host__ __device__ inline int b3_col(int p, int t) { return 32 * (p >> 1) + 16 * (p & 1) + 4 * t; }

// One thread per packed byte.
__global__ void __launch_bounds__(256) ternarise_pack_b3_kernel(const float *W, int64_t N, int64_t K, int64_t steps,
                                                                size_t n_bytes, const float *gamma, uint8_t *packed) {
    size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n_bytes) return;
    const int q = (int)(i & 63), row = (int)((i >> 6) & 15);
    const int64_t tile = (int64_t)(i >> 10);
    const int64_t n = (tile / steps) * 16 + row, k_tile = (tile % steps) * 320;
    const int t = q >> 4, j = q & 15;
    const float half = 0.5f * *gamma;  // exact
    int cols[5];
#pragma unroll
    for (int e = 0; e < 4; ++e) cols[e] = b3_col(j, t) + e;
    cols[4] = b3_col(16 + (j >> 2), t) + (j & 3);
    int v = 0, power = 1;
#pragma unroll
    for (int e = 0; e < 5; ++e) {
        const int64_t k = k_tile + cols[e];
        int c = 1;  // padding: weight 0
        if (n < N && k < K) {
            const float w = W[n * K + k];
            c = w > half ? 2 : (w < -half ? 0 : 1);
        }
        v += c * power;
        power *= 3;
    }
    packed[i] = (uint8_t)v;
}

// One thread per weight.
__global__ void __launch_bounds__(256) unpack_b3_kernel(const uint8_t *packed, int64_t N, int64_t K, int64_t steps, int8_t *T) {
    const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
    if (idx >= N * K) return;
    const int64_t n = idx / K, k = idx % K;
    const int col = (int)(k % 320), p = 2 * (col / 32) + (col % 32) / 16, t = (col % 16) / 4, e = col % 4;
    const int j = p < 16 ? p : 4 * (p - 16) + e;
    const int digit = p < 16 ? e : 4;
    const size_t off = (size_t)((n / 16) * steps + k / 320) * 1024 + (size_t)(n % 16) * 64 + 16 * t + j;
    int v = packed[off];
    int c = 1;
    if (v <= 242) {
        for (int d = 0; d < digit; ++d) v /= 3;
        c = v % 3;
    }
    T[idx] = (int8_t)(c - 1);
}

// Base-3 bytes -> two-bit tiles (the GEMM path reads only those).  A thread takes a row of a base-3 tile: its 64 bytes as four vectors,
// every byte through a table of its five digits, and its 320 columns out as five vectors of four words.  Bytes 16 t + j of the row hold
// columns 16 j + 4 t .. + 3 (digits 0..3) and 16 (16 + j / 4) + 4 t + j % 4 (digit 4), so a two-bit word - columns 4 t + e of a group of
// 16 at bits 8 e + 2 t - is one byte of each of the four vectors, or the fifth digits of four bytes of each.
// Bound by the launch at these sizes (4 + 4 MB for 4096 x 4096): a layer call of 128 tokens there 63.5 -> 23.1 us, 17 tokens of 8192 x 8192 192.6 -> 35.2 against a thread per
// two-bit word, which divided its way through up to sixteen bytes one after the other.
__global__ void __launch_bounds__(256) repack_b3_kernel(const uint8_t *packed_b3, int64_t N, int64_t K, int64_t steps2, int64_t steps3, int64_t tiles,
                                                        size_t n_items, uint32_t *packed2) {
    __shared__ uint32_t digits[256];  // digit e < 4 of the byte in byte e, digit 4 in bits 4 and 5
    {
        const uint32_t v = threadIdx.x;
        digits[v] = v <= 242 ? v % 3 | v / 3 % 3 << 8 | v / 9 % 3 << 16 | v / 27 % 3 << 24 | v / 81 << 4 : 0x01010111u;
    }
    __syncthreads();
    pdl_wait();
    pdl_launch_dependents();
    const size_t i = (size_t)blockIdx.x * 256 + threadIdx.x;
    if (i >= n_items) return;
    const int r = (int)(i & 15);
    const int64_t tile = (int64_t)(i >> 4) % tiles, row_tile = (int64_t)(i >> 4) / tiles, left = K - tile * 320;  // columns of the matrix from the tile on
    const bool inside = row_tile * 16 + r < N && left > 0;
    uint32_t word[20];
#pragma unroll
    for (int g = 0; g < 20; ++g) word[g] = inside ? 0u : 0x55555555u;
    if (inside) {
        const uint4 *src = reinterpret_cast<const uint4 *>(packed_b3 + (size_t)(row_tile * steps3 + tile) * 1024 + r * 64);
        uint4 v[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) v[t] = src[t];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            const uint32_t w[4] = {v[t].x, v[t].y, v[t].z, v[t].w};
#pragma unroll
            for (int j = 0; j < 16; ++j) {
                const uint32_t d = digits[w[j >> 2] >> 8 * (j & 3) & 0xffu];
                word[j] |= (d & 0x03030303u) << 2 * t;
                word[16 + (j >> 2)] |= (d >> 4 & 3u) << (8 * (j & 3) + 2 * t);
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        const int64_t c = tile * 320 + 64 * u;
        if (c >= steps2 * 256) break;
        const bool in = 64 * u < left;  // (K is a multiple of 64)
        *reinterpret_cast<uint4 *>(packed2 + (size_t)(row_tile * steps2 + (c >> 8)) * 256 + r * 16 + ((c & 255) >> 4)) =
            make_uint4(in ? word[4 * u] : 0x55555555u, in ? word[4 * u + 1] : 0x55555555u, in ? word[4 * u + 2] : 0x55555555u, in ? word[4 * u + 3] : 0x55555555u);
    }
}

cudaError_t launch_repack_b3(const void *packed_b3, int64_t d_out, int64_t d_in, void *packed2, bool pdl, cudaStream_t stream) {
    const int64_t steps2 = padded_k(d_in) / 256, steps3 = padded_k_b3(d_in) / 320, tiles = (steps2 * 256 + 319) / 320;
    const size_t n_items = (size_t)row_tiles(d_out) * tiles * 16;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((n_items + 255) / 256));
    cfg.blockDim = dim3(256);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, repack_b3_kernel, (const uint8_t *)packed_b3, d_out, d_in, steps2, steps3, tiles, n_items, (uint32_t *)packed2);
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

// ---- scratch of the packing calls -----------------------------------------------------------------
// Part of the library image (one copy per device that loads it), a slot per call in flight: a call synchronises
// its stream before it returns, so its slot is free again then.  cudaMalloc and cudaFree took their place here:
// cudaFree waits for the whole device and cost 0.1 to 3 ms a call, depending on what else the process had allocated.
// More calls at a time than slots (from that many threads) allocate theirs.
constexpr int kPackSlots = 16;
static __device__ __align__(256) AbsScratch g_pack_scratch[kPackSlots];

struct PackScratch {
    AbsScratch *p = nullptr;
    explicit PackScratch(cudaStream_t stream) {
        dev = current_device();
        if (dev >= 0 && dev < kMaxDevices) {
            AbsScratch *base = slots();
            uint32_t used = busy[dev].load(std::memory_order_relaxed);
            while (base && slot < 0 && used != (1u << kPackSlots) - 1u) {
                const int free_slot = __builtin_ctz(~used);
                if (busy[dev].compare_exchange_weak(used, used | (1u << free_slot), std::memory_order_acquire)) slot = free_slot;
            }
            if (slot >= 0) p = base + slot;
        }
        if (!p) {
            void *mem = nullptr;
            if (cudaMalloc(&mem, sizeof(AbsScratch)) != cudaSuccess) return;
            p = (AbsScratch *)mem;
            if (cudaMemsetAsync(&p->done, 0, sizeof(unsigned int), stream) != cudaSuccess) { cudaFree(mem); p = nullptr; }
        }
    }
    ~PackScratch() {
        if (slot >= 0) busy[dev].fetch_and(~(1u << slot), std::memory_order_release);
        else if (p) cudaFree(p);
    }
    PackScratch(const PackScratch &) = delete;
    PackScratch &operator=(const PackScratch &) = delete;

private:
    int dev = -1, slot = -1;
    static std::atomic<uint32_t> busy[kMaxDevices];
    AbsScratch *slots() const {
        static std::atomic<AbsScratch *> cache[kMaxDevices];
        AbsScratch *ptr = cache[dev].load(std::memory_order_acquire);
        if (!ptr) {
            if (cudaGetSymbolAddress((void **)&ptr, g_pack_scratch) != cudaSuccess) return nullptr;
            cache[dev].store(ptr, std::memory_order_release);
        }
        return ptr;
    }
};
std::atomic<uint32_t> PackScratch::busy[kMaxDevices];

// Both layouts: the scale, then `pack` (which enqueues the layout's kernel with the scale's device address), then
// the scale to the host.
template <typename Pack>
static hgf_status pack_with_scale(const float *W, int64_t d_out, int64_t d_in, float *gamma_out, cudaStream_t stream, Pack pack) {
    PackScratch scratch(stream);
    if (!scratch.p) return HGF_ERR_CUDA;
    const size_t n = (size_t)d_out * (size_t)d_in;
    abs_mean_kernel<<<kAbsBlocks, kAbsThreads, 0, stream>>>((const float4 *)W, n / 4, (double)n, scratch.p);
    const cudaError_t e0 = pack(&scratch.p->gamma);
    count_launch(2);
    cudaError_t e = cudaMemcpyAsync(gamma_out, &scratch.p->gamma, sizeof(float), cudaMemcpyDeviceToHost, stream);
    const cudaError_t e1 = cudaStreamSynchronize(stream);  // also after a failed copy: the slot must be idle
    const cudaError_t e2 = cudaGetLastError();
    return (e0 == cudaSuccess && e == cudaSuccess && e1 == cudaSuccess && e2 == cudaSuccess) ? HGF_OK : HGF_ERR_CUDA;
}

}  // namespace hgf

using namespace hgf;

extern "C" size_t hgf_packed_bytes_b3(int64_t d_out, int64_t d_in) {
    if (d_out <= 0 || d_in <= 0 || d_in % 64 != 0) return 0;
    return (size_t)row_tiles(d_out) * 16 * (size_t)padded_k_b3(d_in) / 5;
}

extern "C" hgf_status hgf_pack_ternary_b3(const float *W, int64_t d_out, int64_t d_in, void *packed, float *gamma_out,
                                          void *stream_) {
    if (!W || !packed || !gamma_out || d_out <= 0 || d_in <= 0) return HGF_ERR_INVALID_ARG;
    if (d_in % 64 != 0) return HGF_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)W | (uintptr_t)packed) & 15) return HGF_ERR_MISALIGNED;
    cudaStream_t stream = (cudaStream_t)stream_;
    const int64_t steps = padded_k_b3(d_in) / 320;
    const size_t n_bytes = (size_t)row_tiles(d_out) * (size_t)steps * 1024;
    return pack_with_scale(W, d_out, d_in, gamma_out, stream, [&](const float *gamma) {
        ternarise_pack_b3_kernel<<<(unsigned)((n_bytes + 255) / 256), 256, 0, stream>>>(W, d_out, d_in, steps, n_bytes, gamma,
                                                                                        (uint8_t *)packed);
        return cudaGetLastError();
    });
}

extern "C" hgf_status hgf_unpack_ternary_b3(const void *packed, int64_t d_out, int64_t d_in, int8_t *T, void *stream_) {
    if (!packed || !T || d_out <= 0 || d_in <= 0) return HGF_ERR_INVALID_ARG;
    if (d_in % 64 != 0 || d_out * d_in > ((int64_t)1 << 40)) return HGF_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)T | (uintptr_t)packed) & 15) return HGF_ERR_MISALIGNED;
    const int64_t steps = padded_k_b3(d_in) / 320, n = d_out * d_in;
    unpack_b3_kernel<<<(unsigned)((n + 255) / 256), 256, 0, (cudaStream_t)stream_>>>((const uint8_t *)packed, d_out, d_in, steps, T);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? HGF_OK : HGF_ERR_CUDA;
}

extern "C" size_t hgf_packed_bytes(int64_t d_out, int64_t d_in) {
    if (d_out <= 0 || d_in <= 0 || d_in % 64 != 0) return 0;
    return (size_t)row_tiles(d_out) * 16 * (size_t)padded_k(d_in) / 4;
}

extern "C" hgf_status hgf_pack_ternary(const float *W, int64_t d_out, int64_t d_in, void *packed,
                                       float *gamma_out, void *stream_) {
    if (!W || !packed || !gamma_out || d_out <= 0 || d_in <= 0) return HGF_ERR_INVALID_ARG;
    if (d_in % 64 != 0) return HGF_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)W | (uintptr_t)packed) & 15) return HGF_ERR_MISALIGNED;
    cudaStream_t stream = (cudaStream_t)stream_;
    const int64_t steps = padded_k(d_in) / 256;
    const size_t n_words = (size_t)row_tiles(d_out) * (size_t)steps * 256;
    return pack_with_scale(W, d_out, d_in, gamma_out, stream, [&](const float *gamma) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // (after the scale's kernel alone, which starts when all work before it is done)
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)(n_words / 256));
        cfg.blockDim = dim3(256);
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, ternarise_pack_kernel, W, d_out, d_in, steps, gamma, (uint32_t *)packed);
    });
}

extern "C" hgf_status hgf_unpack_ternary(const void *packed, int64_t d_out, int64_t d_in, int8_t *T,
                                         void *stream_) {
    if (!packed || !T || d_out <= 0 || d_in <= 0) return HGF_ERR_INVALID_ARG;
    if (d_in % 64 != 0) return HGF_ERR_UNSUPPORTED_SHAPE;
    if (((uintptr_t)T | (uintptr_t)packed) & 15) return HGF_ERR_MISALIGNED;
    const int64_t steps = padded_k(d_in) / 256;
    size_t n_words = (size_t)row_tiles(d_out) * (size_t)steps * 256;
    unpack_kernel<<<(unsigned)((n_words + 255) / 256), 256, 0, (cudaStream_t)stream_>>>((const uint32_t *)packed, d_out, d_in,
                                                                                        steps, n_words, T);
    count_launch(1);
    return cudaGetLastError() == cudaSuccess ? HGF_OK : HGF_ERR_CUDA;
}
