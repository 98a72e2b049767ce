// Codec variant: one bit per element with error feedback (the 1-bit scheme of the paper's
// related-work section).  Per element v = g + e with e the worker's residual of the last
// iteration; the code is the sign of v (a zero counts as non-negative); a bucket's two
// reconstruction values are the means of its two classes, sent as (neg, pos) in the (min, max)
// variant's wire format so that the ordinary K = 1 receiver decodes them; the new residual is
// v minus the value that receiver will reconstruct: neg for code 0, fl(fl(pos - neg) + neg) for
// code 1, and neg for every element of a bucket whose spread fl(pos - neg) is below 2^-96 (its
// codes are cleared).  The class sums have a fixed order - inside a row of 32 elements a
// left-to-right chain over the members of the class, then the balanced tree over the bucket's
// rows - and the counts are exact, so the results are reproducible bit for bit.
//
// One pass: a CTA stages a tile of whole buckets (up to 256 rows) of g and of e in shared memory
// with 16-byte asynchronous copies (the whole tile in flight at once, nothing through registers),
// every thread owns a row, and the new residual leaves through e's tile with coalesced stores.
// 12 + 1/8 bytes per element of traffic for almost no arithmetic.
#include <atomic>

#include "mqg_quantize_tile.cuh"
#include "mqg_tree.cuh"

namespace mqg {

namespace {

struct OneBitArgs {
    const void* grad;
    float* residual;
    uint32_t* codes;
    float* ranges;
    uint64_t n, nrows, nbuckets, ncode_words, bucket_len;   // bucket_len = min(bucket, n)
    uint32_t rows_per_bucket, tile_rows, buckets_per_tile;
};

// tile_g <- g, tile_e <- e for `rows` rows starting at element e0 (a multiple of 32, so 16-byte aligned in
// every buffer); elements at or beyond n are staged as zeros.  Whole 16-byte chunks travel as asynchronous
// copies, so a CTA has its entire tile in flight at once; bf16 gradients are staged as they are (read_row_swizzled
// widens them): 18.8 us at n = 9 M, bucket 2048, against 26.5 us widened through registers on the way in.
template <int DTYPE, int THREADS>
__device__ __forceinline__ void stage_tiles(uint8_t* tile_g, float4* tile_e, const OneBitArgs& a, uint64_t e0, int rows)
{
    const uint64_t valid = a.n - e0;
    auto stage_f32 = [&](float4* tile, const float* src) {
        for (int idx = threadIdx.x; idx < rows * 8; idx += THREADS) {
            const uint64_t e = 4ull * idx;
            float4* dst = &tile[swz(idx >> 3, idx & 7)];
            if (e + 4 <= valid) { cp_async16(dst, src + e0 + e); continue; }
            float r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) r[k] = e + k < valid ? __ldcs(src + e0 + e + k) : 0.0f;
            *dst = make_float4(r[0], r[1], r[2], r[3]);
        }
    };
    stage_f32(tile_e, a.residual);
    if constexpr (DTYPE == 0) {
        stage_f32(reinterpret_cast<float4*>(tile_g), static_cast<const float*>(a.grad));
    } else {
        const uint16_t* src = static_cast<const uint16_t*>(a.grad) + e0;
        for (int idx = threadIdx.x; idx < rows * 4; idx += THREADS) {
            const uint64_t e = 8ull * idx;
            const int row = idx >> 2;
            uint16_t* dst = reinterpret_cast<uint16_t*>(tile_g) + (row * 4 + ((idx & 3) ^ ((row >> 1) & 3))) * 8;
            if (e + 8 <= valid) { cp_async16(dst, src + e); continue; }
#pragma unroll
            for (int k = 0; k < 8; ++k) dst[k] = e + k < valid ? src[e + k] : (uint16_t)0;
        }
    }
    cp_async_wait_all();
}

template <int DTYPE, int THREADS>
constexpr size_t onebit_smem_bytes() { return THREADS * (DTYPE == 0 ? 256 : 192) + 3 * THREADS * sizeof(float) + 1024; }

template <int DTYPE, int THREADS>
__global__ void __launch_bounds__(THREADS, 768 / THREADS)
onebit_ef_kernel(const __grid_constant__ OneBitArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    uint8_t* base = smem_raw + ((1024u - ((uint32_t)__cvta_generic_to_shared(smem_raw) & 1023u)) & 1023u);
    float4* tile = reinterpret_cast<float4*>(base);      // the residual's tile, rewritten in place
    uint8_t* tile_g = base + THREADS * 128;
    float* s_part = reinterpret_cast<float*>(tile_g + THREADS * (DTYPE == 0 ? 128 : 64));

    const uint32_t t = threadIdx.x;
    const uint64_t row0 = (uint64_t)blockIdx.x * a.tile_rows;
    const uint64_t rows_left = a.nrows - row0;
    const int rows = (int)(rows_left < a.tile_rows ? rows_left : a.tile_rows);
    grid_dependency_wait();
    stage_tiles<DTYPE, THREADS>(tile_g, tile, a, row0 * 32, rows);
    __syncthreads();

    const bool active = t < (uint32_t)rows;
    const uint64_t row = row0 + t;
    float v[32];
    uint32_t mask = 0u;                          // the row's elements that exist
    if (active) {
        float g[32];
        read_row_swizzled<DTYPE>(tile_g, (int)t, g);
        read_row(tile, (int)t, v);
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __fadd_rn(g[j], v[j]);      // v = g + e, one rounding
        const uint64_t left = a.n - row * 32;
        mask = left >= 32 ? 0xFFFFFFFFu : ((1u << (uint32_t)left) - 1u);
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0.0f;
    }
    // sign bits and the two class sums of the row, left to right (a non-member adds +0: exact)
    uint32_t word = 0u;
    float pos = 0.0f, neg = 0.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const bool nn = v[j] >= 0.0f;
        word |= (nn ? 1u : 0u) << j;
        pos = __fadd_rn(pos, nn ? v[j] : 0.0f);
        neg = __fadd_rn(neg, nn ? 0.0f : v[j]);
    }
    word &= mask;                                // padding is staged as +0, which is no member
    float sums[3] = {pos, neg, (float)__popc(word)};          // the count is exact: <= 8192
    bucket_tree_sums<THREADS, 3>(sums, a.rows_per_bucket, s_part);
    const float S1 = sums[0], S0 = sums[1], c1 = sums[2];

    const uint32_t local_bucket = t / a.rows_per_bucket;
    const uint64_t bucket = (uint64_t)blockIdx.x * a.buckets_per_tile + local_bucket;
    float e_new[32];
    if (active) {
        const uint64_t start = bucket * a.bucket_len;
        const uint64_t len = a.n - start < a.bucket_len ? a.n - start : a.bucket_len;
        const float c0 = (float)len - c1;
        const float mean0 = __fadd_rn(c0 > 0.0f ? __fdiv_rn(S0, c0) : 0.0f, 0.0f);   // -0 -> +0
        const float mean1 = __fadd_rn(c1 > 0.0f ? __fdiv_rn(S1, c1) : 0.0f, 0.0f);
        if (t % a.rows_per_bucket == 0)
            reinterpret_cast<float2*>(a.ranges)[bucket] = make_float2(mean0, mean1);
        const float r = __fsub_rn(mean1, mean0);
        const bool constant = r < flush_limit();
        const float top = __fadd_rn(r, mean0);          // what the receiver makes of code 1
        if (constant) word = 0u;
#pragma unroll
        for (int j = 0; j < 32; ++j)
            e_new[j] = __fsub_rn(v[j], ((word >> j) & 1u) ? top : mean0);
        write_row(tile, (int)t, e_new);                 // own row only: no other thread reads it
        if (row < a.ncode_words) a.codes[row] = word;   // one bit per element: one word per row
    }
    __syncthreads();
    store_tile_f32<THREADS>(tile, a.residual + row0 * 32, a.n - row0 * 32, rows);
}

template <int DTYPE, int THREADS>
cudaError_t launch_onebit_inst(OneBitArgs& a, cudaStream_t stream)
{
    a.buckets_per_tile = (uint32_t)THREADS / a.rows_per_bucket;
    a.tile_rows = a.buckets_per_tile * a.rows_per_bucket;
    const uint64_t ntiles = (a.nrows + a.tile_rows - 1) / a.tile_rows;
    if (ntiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    auto kernel = onebit_ef_kernel<DTYPE, THREADS>;
    static std::atomic<bool> ready[64];                 // per device (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev].load(std::memory_order_relaxed)) {
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)onebit_smem_bytes<DTYPE, THREADS>());
        if (err != cudaSuccess) return err;
        ready[dev].store(true, std::memory_order_relaxed);
    }
    return launch_pdl_smem(kernel, (unsigned)ntiles, THREADS, onebit_smem_bytes<DTYPE, THREADS>(), stream, a);
}

}  // namespace

cudaError_t launch_quantize_onebit_ef(const void* grad, float* residual, uint64_t n, uint64_t bucket,
                                      uint32_t* codes, float* ranges, int dtype, cudaStream_t stream)
{
    OneBitArgs a;
    a.grad = grad; a.residual = residual; a.codes = codes; a.ranges = ranges;
    a.n = n;
    a.nrows = (n + 31) / 32;
    a.nbuckets = (n + bucket - 1) / bucket;
    a.ncode_words = a.nrows;
    a.bucket_len = bucket < n ? bucket : n;
    // bucket % 32 == 0 and bucket <= 8192, or a single bucket of at most 8192 elements
    const uint64_t rpb = (bucket >= n) ? a.nrows : bucket / 32;
    a.rows_per_bucket = (uint32_t)rpb;
    // the CTA whose rows the buckets fill best, the smaller of two: more CTAs per SM in more different phases
    // (20.6 us at n = 9 M, bucket 2048, against 22.5 us with 256 rows)
    uint32_t threads = 256, used = (256 / (uint32_t)rpb) * (uint32_t)rpb;
    for (uint32_t th = 128; th >= 64 && th >= rpb; th /= 2) {
        const uint32_t u = (th / (uint32_t)rpb) * (uint32_t)rpb;
        if (u * threads >= used * th) { threads = th; used = u; }
    }
#define MQG_ONEBIT(T) return dtype == 0 ? launch_onebit_inst<0, T>(a, stream) : launch_onebit_inst<1, T>(a, stream)
    if (threads == 64) MQG_ONEBIT(64);
    if (threads == 128) MQG_ONEBIT(128);
    MQG_ONEBIT(256);
#undef MQG_ONEBIT
}

}  // namespace mqg
