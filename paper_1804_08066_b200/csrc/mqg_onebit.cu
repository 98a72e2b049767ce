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
// One pass: a CTA stages a tile of whole buckets of g and of e in shared memory, every thread owns a row, and the new
// residual leaves through e's tile.  12 + 1/8 bytes per element of traffic for almost no arithmetic.  Two kernels: persistent
// CTAs fed by bulk copies (onebit_tma_kernel), and a CTA per tile of up to 256 rows, staged with 16-byte asynchronous copies
// (the whole tile in flight at once, nothing through registers), for buckets of more than 128 rows, very short and very long
// gradients.
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

// A row's sign word and its bucket's two means (written by the bucket's first row); v[] <- the row's new residual.  Every
// thread of the CTA calls it; `mask` = the row's elements that exist.
template <int THREADS>
__device__ __forceinline__ uint32_t encode_row(const OneBitArgs& a, float (&v)[32], uint32_t mask, bool active,
                                               uint64_t bucket, float* s_part)
{
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
    if (active) {
        const uint64_t start = bucket * a.bucket_len;
        const uint64_t len = a.n - start < a.bucket_len ? a.n - start : a.bucket_len;
        const float c0 = (float)len - c1;
        const float mean0 = __fadd_rn(c0 > 0.0f ? __fdiv_rn(S0, c0) : 0.0f, 0.0f);   // -0 -> +0
        const float mean1 = __fadd_rn(c1 > 0.0f ? __fdiv_rn(S1, c1) : 0.0f, 0.0f);
        if (threadIdx.x % a.rows_per_bucket == 0)
            reinterpret_cast<float2*>(a.ranges)[bucket] = make_float2(mean0, mean1);
        const float r = __fsub_rn(mean1, mean0);
        const bool constant = r < flush_limit();
        const float top = __fadd_rn(r, mean0);          // what the receiver makes of code 1
        if (constant) word = 0u;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __fsub_rn(v[j], ((word >> j) & 1u) ? top : mean0);
    }
    return word;
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
    const uint64_t bucket = (uint64_t)blockIdx.x * a.buckets_per_tile + t / a.rows_per_bucket;
    const uint32_t word = encode_row<THREADS>(a, v, mask, active, bucket, s_part);
    if (active) {
        write_row(tile, (int)t, v);                     // own row only: no other thread reads it
        if (row < a.ncode_words) a.codes[row] = word;   // one bit per element: one word per row
    }
    __syncthreads();
    store_tile_f32<THREADS>(tile, a.residual + row0 * 32, a.n - row0 * 32, rows);
}

// ---- the same fed and drained by TMA -------------------------------------------------------------------
// Persistent CTAs of 128 rows, two stages of both tiles: bulk copies fetch the next tile while this one is worked on, the new
// residual leaves from the stage by a bulk store, and the stage is refilled half a turn later, when that store has long
// read it.  What bounds it is memory: 12 bytes per element, in and out.  Against a CTA per tile, whose waves of loads and of
// stores follow one another: 2.6 against 3.1 us at n = 131,072, 12.7 against 14.3 us at 9 M (from L2; four workers from DRAM
// and the step 91 against 100 us), bf16 11.3 against 13.2 us, 47 us either way at 25 M.
constexpr int kTmaThreads = 128;

struct OneBitTmaArgs {
    OneBitArgs b;
    uint64_t nrows_full;         // floor(n / 32): rows the tensor maps cover
    uint32_t ntiles;
    uint32_t poll_limit, arm_only;       // as in QuantizeArgs
};

template <int DTYPE>
struct OneBitShared {
    static constexpr uint32_t kGradRow = DTYPE == 0 ? 128 : 64;
    struct Stage {
        alignas(1024) float4 e[kTmaThreads * 8];
        alignas(1024) uint8_t g[kTmaThreads * kGradRow];
    } stage[2];
    float part[3 * kTmaThreads];
    alignas(16) uint8_t ragged[2][kTmaThreads / 32][128];      // a last row of fewer than 32 elements: of g, of e
    alignas(8) uint64_t bar[2];
};

template <int DTYPE>
__global__ void __launch_bounds__(kTmaThreads, DTYPE == 0 ? 3 : 4)
onebit_tma_kernel(const __grid_constant__ CUtensorMap map_g, const __grid_constant__ CUtensorMap map_e,
                  const __grid_constant__ OneBitTmaArgs ta, unsigned int* __restrict__ timeouts)
{
    using Shared = OneBitShared<DTYPE>;
    extern __shared__ uint8_t smem_raw[];
    Shared& sh = *reinterpret_cast<Shared*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    const OneBitArgs& a = ta.b;
    const uint32_t t = threadIdx.x, stride = gridDim.x;
    const uint32_t bytes = a.tile_rows * (128u + Shared::kGradRow);
    if (t == 0) {
        for (int s = 0; s < 2; ++s) mbar_init(smem_u32(&sh.bar[s]), 1);
        fence_barrier_init();
        prefetch_tensormap(&map_g);
        prefetch_tensormap(&map_e);
    }
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory

    auto load = [&](uint32_t tile, uint32_t s) {               // thread 0 only
        const uint32_t bar = smem_u32(&sh.bar[s]);
        mbar_expect_tx(bar, bytes);
        if (ta.arm_only) return;
        tma_load_2d(smem_u32(sh.stage[s].e), &map_e, 0, (int)(tile * a.tile_rows), bar);
        tma_load_2d(smem_u32(sh.stage[s].g), &map_g, 0, (int)(tile * a.tile_rows), bar);
    };
    uint32_t tile = blockIdx.x;
    if (t == 0) {
        if (tile < ta.ntiles) load(tile, 0);
        if (tile + stride < ta.ntiles) load(tile + stride, 1);
    }
    const uint32_t local_bucket = t / a.rows_per_bucket;
    bool ok = true;
    uint32_t k = 0;
#pragma unroll 1
    for (; tile < ta.ntiles; tile += stride, ++k) {
        const uint32_t s = k & 1;
        typename Shared::Stage& stage = sh.stage[s];
        const uint32_t row0 = tile * a.tile_rows, row = row0 + t, bar = smem_u32(&sh.bar[s]);
        const bool active = t < a.tile_rows && row < (uint32_t)a.nrows;
        const bool ragged_warp = a.nrows > ta.nrows_full && tile + 1 == ta.ntiles && warp_has_row(ta.nrows_full, row - (t & 31u));
        const bool ragged = ragged_warp && active && row >= (uint32_t)ta.nrows_full;
        if (ragged_warp) {
            fetch_ragged_row(smem_u32(sh.ragged[0][t >> 5]), static_cast<const uint8_t*>(a.grad), ta.nrows_full,
                             a.n * (DTYPE == 0 ? 4 : 2), Shared::kGradRow);
            fetch_ragged_row(smem_u32(sh.ragged[1][t >> 5]), reinterpret_cast<const uint8_t*>(a.residual), ta.nrows_full,
                             a.n * 4, 128);
        }
        ok = mbar_try_wait(bar, (k >> 1) & 1);
        if (!ok) ok = mbar_wait(bar, (k >> 1) & 1, ta.poll_limit);
        if (ragged_warp) { cp_async_wait_all(); __syncwarp(); }

        float v[32];
        uint32_t mask = 0u;                          // the row's elements that exist
        if (active) {
            float g[32];
            read_row_swizzled<DTYPE>(ragged ? sh.ragged[0][t >> 5] : stage.g, ragged ? 0 : (int)t, g);
            read_row(ragged ? reinterpret_cast<const float4*>(sh.ragged[1][t >> 5]) : stage.e, ragged ? 0 : (int)t, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = __fadd_rn(g[j], v[j]);      // v = g + e, one rounding
            mask = ragged ? (1u << (uint32_t)(a.n - (uint64_t)row * 32)) - 1u : 0xFFFFFFFFu;
        } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = 0.0f;
        }
        // every thread has read its row, or the CTA gives up before it has written anything
        if (__syncthreads_or(!ok)) { ok = false; break; }
        if (t == 0 && k != 0 && tile + stride < ta.ntiles) {
            bulk_wait_read<0>();                     // the store of the tile before has read the other stage
            load(tile + stride, s ^ 1);
        }
        const uint32_t word = encode_row<kTmaThreads>(a, v, mask, active, (uint64_t)tile * a.buckets_per_tile + local_bucket,
                                                      sh.part);
        if (active) {
            if (ragged) {
                float* to = a.residual + (uint64_t)row * 32;
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if ((mask >> j) & 1u) to[j] = v[j];
            } else {
                write_row(stage.e, (int)t, v);       // own row only: no other thread reads it
            }
            a.codes[row] = word;                     // one bit per element: one word per row
        }
        fence_proxy_async();                         // the bulk store must see these writes
        __syncthreads();
        if (t == 0) {
            // rows beyond the last complete one are clipped by the tensor's bounds
            if (row0 < (uint32_t)ta.nrows_full) tma_store_2d(&map_e, 0, (int)row0, smem_u32(stage.e));
            bulk_commit();
        }
    }
    if (t == 0) {
        if (!ok) {
            // A tile never landed: record it, then give the copies in flight a last bounded chance before the shared
            // memory can be handed to another CTA.
            atomicAdd(timeouts, 1u);
            for (uint32_t j = k; j < k + 2 && tile < ta.ntiles && (j == k || k == 0); ++j, tile += stride)
                mbar_wait(smem_u32(&sh.bar[j & 1]), (j >> 1) & 1, ta.poll_limit);
        }
        bulk_wait_all<0>();                          // stores done before the stages go away
    }
}

template <int DTYPE>
cudaError_t launch_onebit_tma(OneBitTmaArgs& ta, cudaStream_t stream)
{
    OneBitArgs& a = ta.b;
    auto kernel = onebit_tma_kernel<DTYPE>;
    constexpr size_t kSmem = sizeof(OneBitShared<DTYPE>) + 1024;         // + slack to round the base up
    static std::atomic<int> grid_cap[64];                // per device; 0 = not yet set up (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kTmaThreads, kSmem);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    a.buckets_per_tile = (uint32_t)kTmaThreads / a.rows_per_bucket;
    a.tile_rows = a.buckets_per_tile * a.rows_per_bucket;
    ta.nrows_full = a.n / 32;
    ta.ntiles = (uint32_t)((a.nrows + a.tile_rows - 1) / a.tile_rows);
    const WaitPolicy policy = wait_policy();
    ta.poll_limit = policy.poll_limit;
    ta.arm_only = policy.arm_only;
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    CUtensorMap map_g, map_e;
    const char* why = nullptr;
    if (!encode_rows_map(&map_g, a.grad, ta.nrows_full, DTYPE == 0 ? 4 : 2, 32, a.tile_rows, &why) ||
        !encode_rows_map(&map_e, a.residual, ta.nrows_full, 4, 32, a.tile_rows, &why))
        return cudaErrorNotSupported;
    const unsigned grid = (unsigned)cap < ta.ntiles ? (unsigned)cap : ta.ntiles;
    return launch_pdl_smem(kernel, grid, kTmaThreads, kSmem, stream, map_g, map_e, ta, timeouts);
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

// Up to 32 M elements (bf16 28 M): the CTAs of a longer launch drift apart and with them their requests for a DRAM page, where
// a CTA per tile keeps the order of the blocks: 66.7 against 66.4 us at n = 36 M, 119 against 107 us at 60 M, bf16 69 against
// 62 us at 40 M.
bool onebit_tma_applies(uint64_t n, uint64_t rpb, int dtype)
{
    return n >= 2048 && n < (dtype == 0 ? 32ull << 20 : 28ull << 20) && rpb <= (uint64_t)kTmaThreads;
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
    if (onebit_tma_applies(n, rpb, dtype)) {
        OneBitTmaArgs ta;
        ta.b = a;
        return dtype == 0 ? launch_onebit_tma<0>(ta, stream) : launch_onebit_tma<1>(ta, stream);
    }
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
