// The one-pass quantizers for several workers' gradients of one shape in one launch (see mqg_quantize.cu).
#include <string.h>

#include <atomic>

#include "mqg_quantize_tile.cuh"

namespace mqg {

// ---------------------------------------------------------------------------------------
// Several workers' gradients in ONE launch (the server-side simulation of P workers, or a host
// with several model replicas on one device).  The launch's fixed costs - scheduling the grid,
// the first tiles' DRAM latency, the last tiles' drain - are paid once instead of once per
// worker.  The tiles of all workers form one sequence v = worker * ntiles + tile, walked exactly
// like the one-worker kernel walks its tiles; every tile is encoded by the same code, so worker
// w's outputs are bit-identical to a one-worker launch with worker id first_worker + w.
// ---------------------------------------------------------------------------------------
struct WorkerTable {
    CUtensorMap map[kMaxWorkers];
    const void* grad[kMaxWorkers];
    uint32_t* codes[kMaxWorkers];
    float* scales[kMaxWorkers];
    PhiloxHead head[kMaxWorkers];
};

template <int BITS, int DTYPE, int THREADS, int RED, int MODE, bool RAGGED, int STAGES>
__global__ void __launch_bounds__(THREADS, quantize_min_ctas<DTYPE, THREADS>())
quantize_workers_kernel(const __grid_constant__ WorkerTable tab, const __grid_constant__ QuantizeArgs a,
                        const __grid_constant__ TmaQuantizeConsts c, uint32_t total_tiles,
                        unsigned int* __restrict__ timeouts)
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
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory

    // Position in the sequence of all workers' tiles, as (worker, tile of the worker), advanced by
    // `stride` tiles at a time without a division.
    struct Pos { uint32_t w, tile; };
    auto advance = [&](Pos& p, uint32_t by) {
        p.tile += by;
        while (p.tile >= a.ntiles) { p.tile -= a.ntiles; ++p.w; }
    };
    auto load_tile = [&](const Pos& p, uint32_t stage, uint32_t bar) {     // thread 0 only
        mbar_expect_tx(bar, box_bytes);
        if (!a.arm_only)
            load_tile_rows(stage, &tab.map[p.w], p.tile * a.tile_rows, a.tile_rows, Shared::kRowBytes, kHalves, bar);
    };
    uint32_t v = blockIdx.x;
    Pos cur = {0u, 0u}, fill = {0u, 0u};   // the tile in work and the one kQuantStages turns ahead of it
    advance(cur, v);
    advance(fill, v);
    uint32_t vfill = v;
    for (uint32_t s = 0; s < (uint32_t)kQuantStages; ++s) {
        if (t == 0 && vfill < total_tiles) load_tile(fill, smem_u32(sh.stage[s]), smem_u32(&sh.bar[s]));
        vfill += stride;
        if (vfill < total_tiles) advance(fill, stride);
    }
    const uint32_t local_bucket = t / a.rows_per_bucket;
    const bool scale_writer = (t % a.rows_per_bucket) == 0;

    uint32_t k = 0, rot = 0;
    bool ok = true;
    uint32_t w = cur.w, tile = cur.tile;
    // Outer loop: the workers this CTA's walk passes through; inner loop: its tiles of that worker.  The
    // worker's table entries (pointers, Philox head) are fetched once per worker, not once per tile:
    // indexed loads from the kernel's parameter block are long-latency loads the tile would wait for.
#pragma unroll 1
    while (ok && v < total_tiles) {
        const WorkerView wv = {&tab.map[w], tab.grad[w], tab.codes[w], tab.scales[w], tab.head[w], c.blk0_lo};
#pragma unroll 1
        for (; ok && tile < a.ntiles && v < total_tiles;
             tile += stride, v += stride, ++k, rot = (rot == 2 ? 0 : rot + 1)) {
            auto refill = [&](uint32_t stage, uint32_t bar) {
                if (vfill < total_tiles) load_tile(fill, stage, bar);
            };
            ok = tile < c.full_tiles
                ? mode_tile<BITS, DTYPE, THREADS, true, RED, MODE, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket,
                                                                           scale_writer)
                : mode_tile<BITS, DTYPE, THREADS, false, RED, MODE, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket,
                                                                            scale_writer);
            vfill += stride;
            if (vfill < total_tiles) advance(fill, stride);
        }
        while (tile >= a.ntiles) { tile -= a.ntiles; ++w; }     // into the next worker (if the walk goes on)
    }
    if (!ok) {                         // as in the one-worker kernel
        if (t == 0) {
            atomicAdd(timeouts, 1u);
            uint32_t j = k - 1, vl = v - stride;
            for (int s = 0; s < kQuantStages && vl < total_tiles; ++s, ++j, vl += stride)
                mbar_wait(smem_u32(&sh.bar[j % kQuantStages]), (j / kQuantStages) & 1, a.poll_limit);
        }
        __syncthreads();
    }
}

template <int BITS, int DTYPE, int THREADS, int RED, int MODE, bool RAGGED, int STAGES>
static cudaError_t launch_workers_inst(const WorkerTable& tab, const QuantizeArgs& a,
                                       const TmaQuantizeConsts& c, uint32_t total_tiles,
                                       unsigned int* timeouts, cudaStream_t stream)
{
    auto kernel = quantize_workers_kernel<BITS, DTYPE, THREADS, RED, MODE, RAGGED, STAGES>;
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
    if (grid > total_tiles) grid = total_tiles;
    return launch_pdl_smem(kernel, grid, THREADS, kSmem, stream, tab, a, c, total_tiles, timeouts);
}

template <int BITS, int DTYPE, int MODE>
static cudaError_t launch_workers_shape(const WorkerTable& tab, const QuantizeArgs& a, const TmaQuantizeConsts& c,
                                        uint32_t total_tiles, int threads, unsigned int* timeouts, cudaStream_t stream)
{
    auto launch = [&](auto cta, auto reduction) {
        constexpr int kThreads = decltype(cta)::value, kRed = decltype(reduction)::value;
        constexpr bool kKeeps = keeps_ragged_code<DTYPE, kThreads, kRed, MODE>();
        auto rows = [&](auto stages) {
            constexpr int kStages = decltype(stages)::value;
            if (a.nrows > a.nrows_full)
                return launch_workers_inst<BITS, DTYPE, kThreads, kRed, MODE, true, kStages>(tab, a, c, total_tiles, timeouts, stream);
            return launch_workers_inst<BITS, DTYPE, kThreads, kRed, MODE, kKeeps, kStages>(tab, a, c, total_tiles, timeouts, stream);
        };
        if constexpr (DTYPE == 0 && kThreads == 256)
            if (one_stage((uint64_t)total_tiles * a.tile_rows)) return rows(Int<1>());
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

template <int BITS>
static cudaError_t launch_workers_bits(const WorkerTable& tab, const QuantizeArgs& a, const TmaQuantizeConsts& c,
                                       uint32_t total_tiles, int threads, int dtype, int mode, unsigned int* timeouts,
                                       cudaStream_t stream)
{
#define MQG_WORKERS_MODE(M) \
    return dtype == 0 ? launch_workers_shape<BITS, 0, M>(tab, a, c, total_tiles, threads, timeouts, stream) \
                      : launch_workers_shape<BITS, 1, M>(tab, a, c, total_tiles, threads, timeouts, stream)
    if (mode == kNorm) MQG_WORKERS_MODE(kNorm);
    if (mode == kRange) MQG_WORKERS_MODE(kRange);
    if (a.row_elems == 64) return launch_workers_shape<BITS, kBf16Wide, kMaxAbs>(tab, a, c, total_tiles, threads, timeouts, stream);
    MQG_WORKERS_MODE(kMaxAbs);
#undef MQG_WORKERS_MODE
}

bool quantize_workers_applies(int W, uint64_t n, uint64_t bucket, uint64_t elem_offset, int mode)
{
    if (W < 2 || W > kMaxWorkers || n == 0) return false;
    const uint64_t nrows = (n + 31) / 32;
    const uint64_t rpb = (bucket >= n) ? nrows : bucket / 32;
    if ((bucket < n ? bucket : n) > (uint64_t)(mode == kNorm ? kMaxFusedBucket : kMaxTmaBucket)) return false;
    if (!tma_path_applies(n, rpb, elem_offset)) return false;
    const uint64_t tile_rows = rpb <= 128 ? (128 / rpb) * rpb : rpb;
    const uint64_t nt = (nrows + tile_rows - 1) / tile_rows;
    return nt * (uint64_t)W <= 0x7FFFFFFFull;
}

cudaError_t launch_quantize_workers(const void* const* grads, int W, uint64_t n, int bits,
                                    uint64_t bucket, uint64_t seed, uint32_t* const* codes,
                                    float* const* scales, int dtype, uint32_t first_worker,
                                    uint32_t step, uint64_t elem_offset, int mode, cudaStream_t stream)
{
    QuantizeArgs a;
    const bool wide = mode == kMaxAbs && bf16_wide_applies(n, n * (uint64_t)W, bucket, dtype);
    const uint64_t rpb = fill_args(a, grads[0], n, bits, bucket, seed, codes[0], scales[0], first_worker,
                                   step, elem_offset, wide ? 64 : 32);
    TmaQuantizeConsts c;
    const int threads = fill_tma_args(a, c, rpb);
    if (threads == 0) return cudaErrorInvalidValue;
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    WorkerTable tab;
    memset(&tab, 0, sizeof(tab));
    for (int w = 0; w < W; ++w) {
        const char* why = nullptr;
        if (!encode_rows_map(&tab.map[w], grads[w], a.nrows_full, dtype == 0 ? 4 : 2, a.row_elems, box_rows(a), &why))
            return cudaErrorNotSupported;
        tab.grad[w] = grads[w]; tab.codes[w] = codes[w]; tab.scales[w] = scales[w];
        tab.head[w] = philox_head(c.blk0_hi, first_worker + (uint32_t)w, c.rk.k0[0]);
    }
    const uint32_t total_tiles = a.ntiles * (uint32_t)W;
    switch (bits) {
#define MQG_WORKERS_CASE(B) \
        case B: return launch_workers_bits<B>(tab, a, c, total_tiles, threads, dtype, mode, timeouts, stream)
        MQG_WORKERS_CASE(1); MQG_WORKERS_CASE(2); MQG_WORKERS_CASE(3); MQG_WORKERS_CASE(4);
        MQG_WORKERS_CASE(5); MQG_WORKERS_CASE(6); MQG_WORKERS_CASE(7); MQG_WORKERS_CASE(8);
#undef MQG_WORKERS_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace mqg
