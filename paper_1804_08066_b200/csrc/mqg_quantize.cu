// Worker side: per-bucket max-abs scale, stochastic-rounding encode and bit packing in one
// pass over the gradient (Quantize(g, K) of Algorithm 1, WorkerIterate).
//
// Work decomposition: the gradient is cut into rows of 32 elements; a CTA takes a tile of
// up to 256 rows that holds whole buckets, stages it in shared memory with coalesced 128-bit
// loads, and each thread then owns one row: it reads its 32 values from shared memory,
// takes part in the bucket's max reduction, draws its 32 sixteen-bit random numbers from
// four Philox blocks, encodes, packs into K words and stores them.  The gradient is read
// from HBM exactly once.
#include <string.h>

#include <atomic>

#include "mqg_quantize_tile.cuh"

namespace mqg {

// Max over the rows of each bucket of the tile.  `m` is this thread's row max (bit pattern of
// a non-negative float, so unsigned order = float order).  Returns the bucket's max.
__device__ __forceinline__ uint32_t bucket_max(uint32_t m, uint32_t rpb, uint32_t local_bucket,
                                               bool active, uint32_t* s_bucket)
{
    if ((rpb & (rpb - 1)) == 0 && rpb <= 32) {
        // a bucket is an aligned group of rpb lanes: butterfly inside the group
        for (uint32_t d = rpb >> 1; d > 0; d >>= 1)
            m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
        return m;
    }
    if (rpb % 32 == 0) {
        // a warp lies inside one bucket: one shared-memory atomic per warp
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if ((threadIdx.x & 31) == 0 && active) atomicMax(&s_bucket[local_bucket], m);
    } else if (active) {
        atomicMax(&s_bucket[local_bucket], m);
    }
    __syncthreads();
    return active ? s_bucket[local_bucket] : 0u;
}

template <int BITS, int DTYPE, bool ALIGNED_DRAWS>
__global__ void __launch_bounds__(kMaxTileRows)
quantize_pack_kernel(const __grid_constant__ QuantizeArgs a)
{
    __shared__ __align__(1024) float4 tile[kMaxTileRows * 8];
    __shared__ uint32_t s_bucket[kMaxTileRows];

    const uint32_t t = threadIdx.x;
    const uint64_t row0 = (uint64_t)blockIdx.x * a.tile_rows;
    const uint64_t rows_left = a.nrows - row0;
    const int rows = (int)(rows_left < a.tile_rows ? rows_left : a.tile_rows);

    if (t < a.buckets_per_tile) s_bucket[t] = 0u;
    grid_dependency_wait();
    if constexpr (DTYPE == 0)
        load_tile_f32<kMaxTileRows>(tile, static_cast<const float*>(a.grad) + row0 * 32,
                                    a.n - row0 * 32, rows);
    else
        load_tile_bf16<kMaxTileRows>(tile, static_cast<const uint16_t*>(a.grad) + row0 * 32,
                                     a.n - row0 * 32, rows);
    __syncthreads();

    const bool active = t < (uint32_t)rows;
    float x[32];
    if (active) read_row(tile, (int)t, x);
    else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = 0.0f;
    }

    const float mx = row_abs_max(x);

    const uint32_t local_bucket = t / a.rows_per_bucket;
    const uint32_t mbits = bucket_max(__float_as_uint(mx), a.rows_per_bucket, local_bucket, active,
                                      s_bucket);
    if (!active) return;

    float s = __uint_as_float(mbits);
    if (s < flush_limit()) s = 0.0f;
    const uint64_t bucket = (uint64_t)blockIdx.x * a.buckets_per_tile + local_bucket;
    if (t % a.rows_per_bucket == 0 && bucket < a.nbuckets) a.scales[bucket] = s;

    const EncodeScale es = encode_scale<BITS>(s);
    const uint64_t row = row0 + t;
    uint32_t h[16];
    if constexpr (ALIGNED_DRAWS) draw_row_aligned(a.elem_offset + row * 32, make_round_keys(a.key), h);
    else draw_row_any(a.elem_offset + row * 32, a.key.worker, make_round_keys(a.key), h);

    uint32_t w[BITS];
    encode_pack_row<BITS>(x, es, h, w);

    const uint64_t word0 = row * BITS;
    const uint64_t e0 = row * 32;
    if (e0 + 32 <= a.n) {
        store_row_words<BITS>(a.codes, word0, w);
    } else {
        // ragged last row: pad bits are zero, words beyond the stream are not written
        mask_row_words<BITS>(w, (int)(a.n - e0) * BITS);
#pragma unroll
        for (int k = 0; k < BITS; ++k)
            if (word0 + k < a.ncode_words) a.codes[word0 + k] = w[k];
    }
}



template <int BITS, int DTYPE, int THREADS, int RED, int MODE, bool RAGGED, int STAGES>
__global__ void __launch_bounds__(THREADS, quantize_min_ctas<DTYPE, THREADS>())
quantize_tma_kernel(const __grid_constant__ CUtensorMap tmap, const __grid_constant__ QuantizeArgs a,
                    const __grid_constant__ TmaQuantizeConsts c, unsigned int* __restrict__ timeouts)
{
    using Shared = TmaQuantizeShared<DTYPE, THREADS, STAGES>;
    constexpr int kQuantStages = Shared::kStages;
    Shared& sh = tile_shared<Shared>();
    constexpr bool kHalves = THREADS == 512;       // more rows than the box of a copy

    const uint32_t t = threadIdx.x;
    const uint32_t stride = gridDim.x;
    const uint32_t box_bytes = a.tile_rows * Shared::kRowBytes;
    if (t == 0) {
        for (int s = 0; s < kQuantStages; ++s) mbar_init(smem_u32(&sh.bar[s]), 1);
        fence_barrier_init();
    }
    init_slots<DTYPE, THREADS>(sh);
    if (t == 0) prefetch_tensormap(&tmap);
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory
    uint32_t tile = blockIdx.x;
    if (t == 0) {
        for (uint32_t s = 0; s < (uint32_t)kQuantStages && tile + s * stride < a.ntiles; ++s) {
            mbar_expect_tx(smem_u32(&sh.bar[s]), box_bytes);
            if (!a.arm_only)
                load_tile_rows(smem_u32(sh.stage[s]), &tmap, (tile + s * stride) * a.tile_rows, a.tile_rows, Shared::kRowBytes,
                               kHalves, smem_u32(&sh.bar[s]));
        }
    }
    const uint32_t local_bucket = t / a.rows_per_bucket;
    const bool scale_writer = (t % a.rows_per_bucket) == 0;
    const uint32_t ahead = kQuantStages * stride;       // distance to the tile that refills a stage
    const WorkerView wv = {&tmap, a.grad, a.codes, a.scales, c.head, c.blk0_lo};

    uint32_t k = 0, rot = 0;
    bool ok = true;
#pragma unroll 1
    for (; ok && tile < a.ntiles; tile += stride, ++k, rot = (rot == 2 ? 0 : rot + 1)) {
        auto refill = [&](uint32_t stage, uint32_t bar) {
            const uint32_t next_tile = tile + ahead;
            if (next_tile < a.ntiles) {
                mbar_expect_tx(bar, box_bytes);
                if (!a.arm_only)
                    load_tile_rows(stage, &tmap, next_tile * a.tile_rows, a.tile_rows, Shared::kRowBytes, kHalves, bar);
            }
        };
        ok = tile < c.full_tiles
            ? mode_tile<BITS, DTYPE, THREADS, true, RED, MODE, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket,
                                                                       scale_writer)
            : mode_tile<BITS, DTYPE, THREADS, false, RED, MODE, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket,
                                                                        scale_writer);
    }
    if (!ok) {
        // A copy never landed: record it, then give the copies still in flight (the one that was
        // being waited for and those issued after it) a last bounded chance to finish before the
        // CTA's shared memory can be handed to another CTA.  The loop's update ran once after the
        // failing tile, so that tile is k - 1 / tile - stride.
        if (t == 0) {
            atomicAdd(timeouts, 1u);
            uint32_t j = k - 1, tl = tile - stride;
            for (int s = 0; s < kQuantStages && tl < a.ntiles; ++s, ++j, tl += stride)
                mbar_wait(smem_u32(&sh.bar[j % kQuantStages]), (j / kQuantStages) & 1, a.poll_limit);
        }
        __syncthreads();
    }
}

template <int BITS>
static cudaError_t launch_bits(const QuantizeArgs& a, int dtype, bool aligned, unsigned grid,
                               cudaStream_t stream)
{
    if (dtype == 0)
        return aligned ? launch_pdl(quantize_pack_kernel<BITS, 0, true>, grid, kMaxTileRows, stream, a)
                       : launch_pdl(quantize_pack_kernel<BITS, 0, false>, grid, kMaxTileRows, stream, a);
    return aligned ? launch_pdl(quantize_pack_kernel<BITS, 1, true>, grid, kMaxTileRows, stream, a)
                   : launch_pdl(quantize_pack_kernel<BITS, 1, false>, grid, kMaxTileRows, stream, a);
}

template <int BITS, int DTYPE, int THREADS, int RED, int MODE, bool RAGGED, int STAGES>
static cudaError_t launch_tma_inst(const CUtensorMap& map, const QuantizeArgs& a,
                                   const TmaQuantizeConsts& c, unsigned int* timeouts,
                                   cudaStream_t stream)
{
    auto kernel = quantize_tma_kernel<BITS, DTYPE, THREADS, RED, MODE, RAGGED, STAGES>;
    constexpr size_t kSmem = dynamic_bytes<TmaQuantizeShared<DTYPE, THREADS, STAGES>>();
    static std::atomic<int> grid_cap[64];                  // per device; 0 = not yet queried (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        if (kSmem != 0) err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, THREADS, kSmem);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    unsigned grid = (unsigned)cap;
    if (grid > a.ntiles) grid = a.ntiles;
    return launch_pdl_smem(kernel, grid, THREADS, kSmem, stream, map, a, c, timeouts);
}

template <int BITS, int DTYPE, int MODE>
static cudaError_t launch_tma_shape(const CUtensorMap& map, const QuantizeArgs& a, const TmaQuantizeConsts& c, int threads,
                                    unsigned int* timeouts, cudaStream_t stream)
{
    auto launch = [&](auto cta, auto reduction) {
        constexpr int kThreads = decltype(cta)::value, kRed = decltype(reduction)::value;
        constexpr bool kKeeps = keeps_ragged_code<DTYPE, kThreads, kRed, MODE>();
        auto rows = [&](auto stages) {
            constexpr int kStages = decltype(stages)::value;
            if (a.nrows > a.nrows_full)
                return launch_tma_inst<BITS, DTYPE, kThreads, kRed, MODE, true, kStages>(map, a, c, timeouts, stream);
            return launch_tma_inst<BITS, DTYPE, kThreads, kRed, MODE, kKeeps, kStages>(map, a, c, timeouts, stream);
        };
        if constexpr (DTYPE == 0 && kThreads == 256)
            if (one_stage((uint64_t)a.ntiles * a.tile_rows)) return rows(Int<1>());
        return rows(Int<2>());
    };
    const int red = reduction_of(a.rows_per_bucket);
    if (threads == 256) return launch(Int<256>(), Int<kByWarps>());
    if constexpr (DTYPE != kBf16Wide && MODE != kNorm)       // 256 rows of 64 hold every bucket; no norm of longer ones
        if (threads == 512) return launch(Int<512>(), Int<kByWarps>());
    if (threads != 128) return cudaErrorInvalidValue;
    if (red == kByShuffle) return launch(Int<128>(), Int<kByShuffle>());
    if (red == kByRows) return launch(Int<128>(), Int<kByRows>());
    return launch(Int<128>(), Int<kByWarps>());
}

// One worker on the TMA kernel (tma_path_applies() holds).
template <int MODE>
static cudaError_t launch_tma(QuantizeArgs& a, uint64_t rpb, int bits, int dtype, cudaStream_t stream)
{
    TmaQuantizeConsts c;
    const int threads = fill_tma_args(a, c, rpb);
    if (threads == 0) return cudaErrorInvalidValue;
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    CUtensorMap map;
    const char* why = nullptr;
    if (!encode_rows_map(&map, a.grad, a.nrows_full, dtype == 0 ? 4 : 2, a.row_elems, box_rows(a), &why))
        return cudaErrorNotSupported;        // the driver cannot encode a tensor map: no silent detour
    switch (bits) {
#define MQG_TMA_CASE(B) \
        case B: \
            if constexpr (MODE == kMaxAbs) \
                if (a.row_elems == 64) return launch_tma_shape<B, kBf16Wide, MODE>(map, a, c, threads, timeouts, stream); \
            return dtype == 0 ? launch_tma_shape<B, 0, MODE>(map, a, c, threads, timeouts, stream) \
                              : launch_tma_shape<B, 1, MODE>(map, a, c, threads, timeouts, stream)
        MQG_TMA_CASE(1); MQG_TMA_CASE(2); MQG_TMA_CASE(3); MQG_TMA_CASE(4);
        MQG_TMA_CASE(5); MQG_TMA_CASE(6); MQG_TMA_CASE(7); MQG_TMA_CASE(8);
#undef MQG_TMA_CASE
    }
    return cudaErrorInvalidValue;
}

// The Philox blocks of the launch (four per row, from block elem_offset / 8 on) all have the same
// high half of the 64-bit block index, so that the part of a block that depends on it is a launch
// constant (PhiloxHead) and a row's block numbers need no carry.  Fails only for a gradient that
// straddles a multiple of 2^35 elements of the flat model; that one takes the general kernels.
static bool blocks_share_high_half(uint64_t n, uint64_t elem_offset)
{
    const uint64_t first = elem_offset >> 3, last = first + 4 * ((n + 31) / 32) - 1;
    return (first >> 32) == (last >> 32);
}

// TMA path: enough rows exist and the draws are block-aligned.  Buckets of more than 128 rows have a CTA of 256 or
// (above 256 rows, main codec and range) 512 threads each and must be whole warps.
bool tma_path_applies(uint64_t n, uint64_t rpb, uint64_t elem_offset)
{
    if (n < 32 * 64 || (elem_offset & 7u) != 0 || rpb == 0 || rpb > (uint64_t)kMaxTmaBucket / 32) return false;
    if (n / 32 > 0x7FFFFFFFull) return false;
    if (!blocks_share_high_half(n, elem_offset)) return false;
    return reduction_of(rpb) != kByRows || rpb <= 128;
}

// Rows of 64 halve the number of tiles, so a short launch is longer with them: us narrow / wide at one worker, K = 4,
// n = 2^21 / 2^23 / 2^24 / 2^25: 3.2 / 4.4, 7.1 / 7.6, 11.6 / 11.3, 22.0 / 20.0 (four workers of a quarter of
// that the same).  Long launches, held at the power limit: 30.6 -> 27.2 us per 50 M elements at K = 1, 29.8 -> 27.8 at
// K = 4, 33.4 -> 32.6 at K = 8.
bool bf16_wide_applies(uint64_t n, uint64_t total, uint64_t bucket, int dtype)
{
    const uint64_t rows = bucket >= n ? (n + 63) / 64 : bucket / 64;          // of a bucket: above 128, whole warps
    return dtype == 1 && total >= (20ull << 20) && n >= 64 * 64 && (bucket >= n || bucket % 64 == 0) &&
           (rows <= 128 || rows % 32 == 0);
}

// Fills the arguments every fused kernel shares.  Returns rows per bucket.
uint64_t fill_args(QuantizeArgs& a, const void* grad, uint64_t n, int bits, uint64_t bucket,
                          uint64_t seed, uint32_t* codes, float* scales, uint32_t worker, uint32_t step,
                          uint64_t elem_offset, uint32_t row_elems)
{
    a.grad = grad; a.codes = codes; a.scales = scales;
    a.n = n;
    a.row_elems = row_elems;
    a.nrows = (n + row_elems - 1) / row_elems;
    a.nbuckets = (n + bucket - 1) / bucket;
    a.ncode_words = (n * (uint64_t)bits + 31) / 32;
    a.elem_offset = elem_offset;
    // bucket % 32 == 0 and bucket <= kMaxTmaBucket (the norm kMaxFusedBucket), or a single bucket of at most that many elements
    const uint64_t rpb = (bucket >= n) ? a.nrows : bucket / row_elems;
    a.rows_per_bucket = (uint32_t)rpb;
    a.buckets_per_tile = (uint32_t)(kMaxTileRows / rpb);
    a.tile_rows = a.buckets_per_tile * a.rows_per_bucket;
    a.key.seed_lo = (uint32_t)seed; a.key.seed_hi = (uint32_t)(seed >> 32);
    a.key.worker = worker; a.key.step = step;
    a.nrows_full = n / row_elems;
    const WaitPolicy policy = wait_policy();
    a.poll_limit = policy.poll_limit;
    a.arm_only = policy.arm_only;
    return rpb;
}

// Tile shape and constants of the TMA kernels (tma_path_applies() holds).  Returns the CTA size,
// or 0 if the tile count does not fit.
int fill_tma_args(QuantizeArgs& a, TmaQuantizeConsts& c, uint64_t rpb)
{
    const int threads = rpb <= 128 ? 128 : rpb <= 256 ? 256 : 512;
    a.buckets_per_tile = (uint32_t)(threads / rpb);
    a.tile_rows = a.buckets_per_tile * a.rows_per_bucket;
    const uint64_t nt = (a.nrows + a.tile_rows - 1) / a.tile_rows;
    if (nt > 0x7FFFFFFFull) return 0;
    a.ntiles = (uint32_t)nt;
    uint32_t k0 = a.key.seed_lo, k1 = a.key.seed_hi;
    for (int r = 0; r < 10; ++r) {
        c.rk.k0[r] = k0; c.rk.k1[r] = k1;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    c.rk.worker = a.key.worker; c.rk.step = a.key.step;
    c.ragged_tile = a.nrows > a.nrows_full ? a.ntiles - 1 : 0xFFFFFFFFu;
    c.full_tiles = a.tile_rows == (uint32_t)threads ? (uint32_t)(a.nrows_full / a.tile_rows) : 0u;
    c.blk0_lo = (uint32_t)(a.elem_offset >> 3); c.blk0_hi = (uint32_t)(a.elem_offset >> 35);
    c.head = philox_head(c.blk0_hi, c.rk.worker, c.rk.k0[0]);
    return threads;
}

cudaError_t launch_quantize_fused(const void* grad, uint64_t n, int bits, uint64_t bucket,
                                  uint64_t seed, uint32_t* codes, float* scales, int dtype,
                                  uint32_t worker, uint32_t step, uint64_t elem_offset,
                                  cudaStream_t stream)
{
    QuantizeArgs a;
    const uint64_t rpb = fill_args(a, grad, n, bits, bucket, seed, codes, scales, worker, step, elem_offset);
    if (tma_path_applies(n, rpb, elem_offset)) {
        if (!bf16_wide_applies(n, n, bucket, dtype)) return launch_tma<kMaxAbs>(a, rpb, bits, dtype, stream);
        const uint64_t wide = fill_args(a, grad, n, bits, bucket, seed, codes, scales, worker, step, elem_offset, 64);
        return launch_tma<kMaxAbs>(a, wide, bits, dtype, stream);
    }
    a.buckets_per_tile = (uint32_t)(kMaxTileRows / rpb);
    a.tile_rows = a.buckets_per_tile * a.rows_per_bucket;
    const uint64_t ntiles = (a.nrows + a.tile_rows - 1) / a.tile_rows;
    if (ntiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    a.ntiles = (uint32_t)ntiles;
    const bool aligned = (elem_offset & 7u) == 0;
    switch (bits) {
        case 1: return launch_bits<1>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 2: return launch_bits<2>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 3: return launch_bits<3>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 4: return launch_bits<4>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 5: return launch_bits<5>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 6: return launch_bits<6>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 7: return launch_bits<7>(a, dtype, aligned, (unsigned)ntiles, stream);
        case 8: return launch_bits<8>(a, dtype, aligned, (unsigned)ntiles, stream);
    }
    return cudaErrorInvalidValue;
}

bool quantize_long_fused_applies(uint64_t n, uint64_t bucket, uint64_t elem_offset)
{
    return tma_path_applies(n, bucket >= n ? (n + 31) / 32 : bucket / 32, elem_offset);
}

// ---- (min, max) nearest-rounding variant on the TMA kernel ----
bool quantize_range_fused_applies(uint64_t n, uint64_t bucket)
{
    if (n == 0) return false;
    return tma_path_applies(n, bucket >= n ? (n + 31) / 32 : bucket / 32, 0);
}

cudaError_t launch_quantize_range_fused(const void* grad, uint64_t n, int bits, uint64_t bucket,
                                        uint32_t* codes, float* ranges, int dtype, cudaStream_t stream)
{
    QuantizeArgs a;
    const uint64_t rpb = fill_args(a, grad, n, bits, bucket, 0, codes, ranges, 0, 0, 0);
    return launch_tma<kRange>(a, rpb, bits, dtype, stream);
}

// ---- L2-norm scale variant on the TMA kernel (block-aligned draws) ----
bool quantize_norm_fused_applies(uint64_t n, uint64_t bucket, uint64_t elem_offset)
{
    if (n == 0 || (bucket < n ? bucket : n) > (uint64_t)kMaxFusedBucket) return false;
    return tma_path_applies(n, bucket >= n ? (n + 31) / 32 : bucket / 32, elem_offset);
}

cudaError_t launch_quantize_norm_fused(const void* grad, uint64_t n, int bits, uint64_t bucket, uint64_t seed,
                                       uint32_t* codes, float* scales, int dtype, uint32_t worker,
                                       uint32_t step, uint64_t elem_offset, cudaStream_t stream)
{
    QuantizeArgs a;
    const uint64_t rpb = fill_args(a, grad, n, bits, bucket, seed, codes, scales, worker, step, elem_offset);
    return launch_tma<kNorm>(a, rpb, bits, dtype, stream);
}

// ---- encode against a given scale (mqg_segments_workers.cu): whole rows, block-aligned draws, bulk copies ----
bool quantize_given_scale_applies(const void* grad, uint64_t n, uint64_t elem_offset)
{
    return n >= 32 * 64 && n / 32 <= 0x7FFFFFFFull && (elem_offset & 7u) == 0 &&
           blocks_share_high_half(n, elem_offset) &&
           (reinterpret_cast<uintptr_t>(grad) & 15u) == 0;
}

}  // namespace mqg
