// Worker side with one scale per segment (per-layer scale) or with buckets longer than the tiles of the
// one-pass kernels.  Two ways:
//   * span_kernel - a span is a segment or a bucket that fits one CTA's shared memory: the CTA stages all of it,
//     finds the scale and encodes from there, so the gradient is read once and every span of every worker
//     is one launch's work (spans_absmax_kernel: the same beside a max pass);
//   * absmax_table_kernel, encode_table_kernel - longer ones: a max pass that folds every tile's maximum into
//     scales[] with an atomic max on the float's bit pattern, then an encode pass.
// Worker w of W is blockIdx.y in all of them; its results do not depend on W or on the way taken.
#include <string.h>

#include <atomic>
#include <type_traits>

#include "mqg_segments.cuh"
#include "mqg_tma.cuh"
#include "mqg_tree.cuh"

namespace mqg {

// The encode of one row: elements `left` (>= 1) long at flat position g0, words word0 .. of a stream that ends at
// words_end.  VEC: the row's words start where store_row_words may use its widest access.
template <int BITS, bool RANGE, typename Scale>
__device__ __forceinline__ void encode_store_row(const float (&x)[32], const Scale& es, const TableArgs& a, uint32_t w,
                                                 uint64_t g0, uint64_t left, uint64_t word0, uint64_t words_end, bool vec)
{
    uint32_t cw[BITS];
    if constexpr (RANGE) {
        range_encode_pack_row<BITS>(x, es, cw);
    } else {
        uint32_t h[16];
        if ((g0 & 7u) == 0) {
            const uint64_t blk = g0 >> 3;
            draw_row_blocks((uint32_t)blk, (uint32_t)(blk >> 32), a.first_worker + w, a.rk, h);
        } else {
            draw_row_any(g0, a.first_worker + w, a.rk, h);
        }
        encode_pack_row_best<BITS>(x, es, h, cw);
    }
    if (vec && left >= 32) {
        store_row_words<BITS>(a.codes[w], word0, cw);
    } else {
        if (left < 32) mask_row_words<BITS>(cw, (int)left * BITS);
#pragma unroll
        for (int k = 0; k < BITS; ++k)
            if (word0 + k < words_end) a.codes[w][word0 + k] = cw[k];
    }
}

// ---- spans ---------------------------------------------------------------------------------------
// What bounds it: a short launch its latency (one staging copy, one reduction, one encode), a long one the
// encode's instructions; CTAs on an SM are in different phases, which overlaps the copies with the encode.
// Up to 512 rows: 256 threads (one or two rows each) and the registers of three CTAs per SM; longer spans: 512
// threads, one CTA per SM.
//
// JOINED: a long span is the work of several CTAs of a cluster, kJoinedChunk elements and one row to a thread each; their
// maxima (sums: aligned subtrees of the span's tree) meet through distributed shared memory.  A cluster has the CTAs of as many
// such spans as fit in it, or of spans that are one CTA's.  (A cluster to a span, all as large as the longest one wants: 8
// workers' 63 tensors of 9,000 elements and one of 60,000 37.0 against 10.5 us, eight CTAs of ten then without an element.)
__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t rank;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    return rank;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// The word of CTA `rank` of the cluster that lies where `word` lies in this one.
__device__ __forceinline__ uint32_t cluster_load(const uint32_t* word, uint32_t rank)
{
    uint32_t at, v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"(smem_u32(word)), "r"(rank));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(at) : "memory");
    return v;
}

template <int BITS, int DTYPE, int MODE, int THREADS, bool JOINED = false>
__device__ __forceinline__ void quantize_span(const TableArgs& a, const SpanTable& tab, const JoinedTable* places = nullptr)
{
    static_assert(!JOINED || MODE != kSpanRange, "one word per CTA meets");
    extern __shared__ uint8_t smem_raw[];
    float4* tile = reinterpret_cast<float4*>(smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    constexpr int kWarps = THREADS / 32;
    __shared__ uint32_t s_a[kMaxSpanRows / 32], s_b[kWarps];   // kSpanNorm: a sum per 32 rows, else a word per warp
    __shared__ uint32_t s_cta;                                 // JOINED: this CTA's maximum or sum
    const uint32_t t = threadIdx.x, lane = t & 31u, wid = t >> 5, w = blockIdx.y;
    uint64_t elem0, len, code0, scale_idx;
    uint32_t part = 0, parts = 1;                              // JOINED: this CTA's part of the span
    if constexpr (!JOINED) grid_dependency_wait();
    if constexpr (JOINED) {
        const uint32_t place = places->cta[blockIdx.x], j = place & 255u;
        if (place == kNoPart) return;                          // the others' barriers do not wait for it
        part = place >> 8;
        parts = places->parts[j];
        grid_dependency_wait();
        const uint64_t all = tab.len[j], done = part * kJoinedChunk;
        elem0 = tab.elem0[j] + done;
        len = parts > 1 && all - done > kJoinedChunk ? kJoinedChunk : all - done;
        code0 = tab.code0[j] + done / 32 * BITS;
        scale_idx = tab.scale_idx[j];
    } else if (tab.bucket != 0) {
        scale_idx = blockIdx.x;
        elem0 = scale_idx * tab.bucket;
        len = tab.n - elem0 < tab.bucket ? tab.n - elem0 : tab.bucket;
        code0 = elem0 / 32 * BITS;
    } else {
        if (blockIdx.x == 0 && t < (uint32_t)kMaxSegmentsPerLaunch && ((tab.clear[t >> 5] >> (t & 31u)) & 1u))
            a.scales[w][tab.first + t] = 0.0f;
        if (blockIdx.x >= (uint32_t)tab.nspan) return;
        elem0 = tab.elem0[blockIdx.x];
        len = tab.len[blockIdx.x];
        code0 = tab.code0[blockIdx.x];
        scale_idx = tab.scale_idx[blockIdx.x];
    }
    const uint64_t words_end = code0 + (len * BITS + 31) / 32;
    const int rows = (int)((len + 31) / 32);
    if constexpr (DTYPE == 0) load_tile_f32<THREADS>(tile, static_cast<const float*>(a.grad[w]) + elem0, len, rows);
    else load_tile_bf16<THREADS>(tile, static_cast<const uint16_t*>(a.grad[w]) + elem0, len, rows);
    __syncthreads();

    const int turns = (rows + THREADS - 1) / THREADS;
    float x[32];
    uint32_t lo = kOrderedMinIdentity, hi = MODE == kSpanRange ? kOrderedMaxIdentity : 0u;
    for (int k = 0; k < turns; ++k) {
        const int r = k * THREADS + (int)t;
        const bool active = r < rows;
        if (active) read_row(tile, r, x);                     // elements beyond the span were staged as zeros
        if constexpr (MODE == kSpanNorm) {
            const float s = warp_tree(active ? row_sum_squares(x) : 0.0f, 32);
            if (lane == 0) s_a[k * kWarps + wid] = __float_as_uint(s);
        } else if (active) {
            if constexpr (MODE == kSpanRange) {
                const uint64_t left = len - 32ull * r;        // the elements a ragged row lacks repeat its first one
#pragma unroll
                for (int j = 1; j < 32; ++j) x[j] = (uint64_t)j < left ? x[j] : x[0];
                float l, h;
                row_min_max(x, l, h);
                lo = min(lo, ordered_bits(l));
                hi = max(hi, ordered_bits(h));
            } else {
                hi = max(hi, __float_as_uint(row_abs_max(x)));
            }
        }
    }
    // Every part's word to lane `part` of every warp, 0 to the lanes beyond.  The shared memory stays until the second wait.
    auto meet = [&](uint32_t word) -> uint32_t {
        if (t == 0) s_cta = word;
        cluster_arrive();
        cluster_wait();
        const uint32_t v = lane < parts ? cluster_load(&s_cta, cluster_rank() - part + lane) : 0u;
        cluster_arrive();
        return v;
    };
    float scale = 0.0f;
    RangeEncodeScale range = {0.0f, 0.0f};
    if constexpr (MODE == kSpanNorm) {
        __syncthreads();
        // the tree over the sums of 32 rows: lane l on leaves 2l, 2l + 1 of 64, zeros beyond the last
        const uint32_t n32 = (uint32_t)(turns * kWarps);
        const float p = 2 * lane < n32 ? __uint_as_float(s_a[2 * lane]) : 0.0f;
        const float q = 2 * lane + 1 < n32 ? __uint_as_float(s_a[2 * lane + 1]) : 0.0f;
        float S = warp_tree(__fadd_rn(p, q), 32);
        if (JOINED && parts > 1)                      // eight leaves, on lanes 0 .. 7
            S = __shfl_sync(0xFFFFFFFFu, warp_tree(__uint_as_float(meet(__float_as_uint(S))), 8), 0);
        scale = S < flush_limit() ? 0.0f : __fsqrt_rn(S);
        if (t == 0 && part == 0) a.scales[w][scale_idx] = scale;
    } else {
        hi = __reduce_max_sync(0xFFFFFFFFu, hi);
        if (MODE == kSpanRange) lo = __reduce_min_sync(0xFFFFFFFFu, lo);
        if (lane == 0) { s_a[wid] = hi; s_b[wid] = lo; }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kWarps; ++i) { hi = max(hi, s_a[i]); lo = min(lo, s_b[i]); }
        if (JOINED && parts > 1) hi = __reduce_max_sync(0xFFFFFFFFu, meet(hi));
        if constexpr (MODE == kSpanRange) {
            // a zero of either sign is stored as +0
            const float l = __fadd_rn(from_ordered_bits(lo), 0.0f), h = __fadd_rn(from_ordered_bits(hi), 0.0f);
            if (t == 0) reinterpret_cast<float2*>(a.scales[w])[scale_idx] = make_float2(l, h);
            range = range_encode_scale<BITS>(l, h);
        } else {
            scale = __uint_as_float(hi);
            if (scale < flush_limit()) scale = 0.0f;
            if (t == 0 && part == 0) a.scales[w][scale_idx] = scale;
        }
    }
    const EncodeScale es = encode_scale<BITS>(scale);
    const bool vec = (reinterpret_cast<uintptr_t>(a.codes[w] + code0) & 15u) == 0;
    for (int r = (int)t; r < rows; r += THREADS) {
        read_row(tile, r, x);
        const uint64_t g0 = a.elem_offset + elem0 + 32ull * r, left = len - 32ull * r, word0 = code0 + (uint64_t)r * BITS;
        if constexpr (MODE == kSpanRange) encode_store_row<BITS, true>(x, range, a, w, g0, left, word0, words_end, vec);
        else encode_store_row<BITS, false>(x, es, a, w, g0, left, word0, words_end, vec);
    }
    if (JOINED && parts > 1) cluster_wait();          // no CTA's shared memory goes before the others have read it
}

template <int BITS, int DTYPE, int MODE, int THREADS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 3 : 1)
span_kernel(const __grid_constant__ TableArgs a, const __grid_constant__ SpanTable tab)
{
    quantize_span<BITS, DTYPE, MODE, THREADS>(a, tab);
}

template <int BITS, int DTYPE, int MODE>
__global__ void __launch_bounds__(kMaxTileRows, 3)
joined_span_kernel(const __grid_constant__ TableArgs a, const __grid_constant__ JoinedTable tab)
{
    quantize_span<BITS, DTYPE, MODE, kMaxTileRows, true>(a, tab.spans, &tab);
}

// ---- two passes over tiles of 256 rows ---------------------------------------------------------------
// Tile `tile` of the table, whose first segment has the scale a.scales[w][first].
template <int DTYPE>
__device__ __forceinline__ void absmax_tile(const TableArgs& a, const SegmentTable& tab, uint32_t tile, uint32_t first)
{
    constexpr int THREADS = kMaxTileRows;
    __shared__ uint32_t s_warp[THREADS / 32];
    const TileGeom g = locate_tile<1>(tab, tile);
    const uint64_t count = g.valid < (uint64_t)(kMaxTileRows * 32) ? g.valid : (uint64_t)(kMaxTileRows * 32);
    grid_dependency_wait();

    using T = typename std::conditional<DTYPE == 0, float, uint16_t>::type;
    const T* src = static_cast<const T*>(a.grad[blockIdx.y]) + g.elem0;
    auto value = [&](uint64_t i) {
        if constexpr (DTYPE == 0) return fabsf(__ldcg(src + i));
        else return fabsf(bf16_lo(__ldcg(src + i)));
    };
    // 16-byte accesses from the tile's first 16-byte boundary on
    constexpr uint64_t kPer = 16 / sizeof(T);
    const uint64_t to_align = (kPer - (reinterpret_cast<uintptr_t>(src) / sizeof(T)) % kPer) % kPer;
    const uint64_t head = to_align < count ? to_align : count, nvec = (count - head) / kPer;
    const uint4* v4 = reinterpret_cast<const uint4*>(src + head);
    float m = 0.0f;
    auto take = [&](const uint4& v) {
        const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int k = 0; k < 4; k += DTYPE == 0 ? 2 : 1) {
            if constexpr (DTYPE == 0) m = max3_abs(m, __uint_as_float(u[k]), __uint_as_float(u[k + 1]));
            else m = max3_abs(m, bf16_lo(u[k]), bf16_hi(u[k]));
        }
    };
    constexpr int kFull = kMaxTileRows * 32 / kPer / THREADS;          // accesses per thread of a whole tile
    // A tile off the boundary takes its successor's first elements instead of its own, where the segment goes on that far: a
    // maximum may see them twice.  (23 M elements off the boundary, two workers, with the encode: 66 against 73 us, bf16 51
    // against 56 us.)
    if (g.valid >= to_align + kMaxTileRows * 32) {
        if (g.tile_local == 0 && threadIdx.x < to_align) m = value(threadIdx.x);
        uint4 v[kFull];
#pragma unroll
        for (int k = 0; k < kFull; ++k) v[k] = __ldcg(v4 + k * THREADS + threadIdx.x);
#pragma unroll
        for (int k = 0; k < kFull; ++k) take(v[k]);
    } else {
        if (threadIdx.x < head) m = value(threadIdx.x);
#pragma unroll 4
        for (uint64_t i = threadIdx.x; i < nvec; i += THREADS) take(__ldcg(v4 + i));
        const uint64_t tail = head + nvec * kPer + threadIdx.x;
        if (tail < count) m = fmaxf(m, value(tail));
    }
    uint32_t r = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(m));
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = r;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 1; i < THREADS / 32; ++i) r = max(r, s_warp[i]);
        // a tile's maximum below the flush limit does not count: a segment whose every tile stays below it
        // keeps the scale 0 the pass started from, so the scale that stands after the pass is final
        if (r >= __float_as_uint(flush_limit()))
            atomicMax(reinterpret_cast<unsigned int*>(a.scales[blockIdx.y]) + first + g.seg, r);
    }
}

template <int DTYPE>
__global__ void __launch_bounds__(kMaxTileRows)
absmax_table_kernel(const __grid_constant__ TableArgs a, const __grid_constant__ SegmentTable tab)
{
    absmax_tile<DTYPE>(a, tab, blockIdx.x, 0);
}

// The spans of a table and the max pass over its longer segments, whose scales are clear, in one launch: a span is a
// chain of a staging copy, a reduction and an encode, 3 us beside which the max pass reads.
template <int BITS, int DTYPE>
__global__ void __launch_bounds__(kMaxTileRows, 3)
spans_absmax_kernel(const __grid_constant__ TableArgs a, const __grid_constant__ SpanTable spans,
                    const __grid_constant__ SegmentTable longs)
{
    if (blockIdx.x < (uint32_t)spans.nspan) quantize_span<BITS, DTYPE, kSpanMaxAbs, kMaxTileRows>(a, spans);
    else absmax_tile<DTYPE>(a, longs, blockIdx.x - (uint32_t)spans.nspan, (uint32_t)spans.first);
}

__global__ void __launch_bounds__(kMaxTileRows)
clear_scales_kernel(const __grid_constant__ TableArgs a, int nseg)
{
    grid_dependency_wait();
    for (int j = (int)threadIdx.x; j < nseg; j += kMaxTileRows) a.scales[blockIdx.x][j] = 0.0f;
}

// A 256-row tile of the table is two CTAs' work.
constexpr int kEncodeThreads = 128;
template <int BITS, int DTYPE>
__global__ void __launch_bounds__(kEncodeThreads)
encode_table_kernel(const __grid_constant__ TableArgs a, const __grid_constant__ SegmentTable tab)
{
    __shared__ __align__(1024) float4 tile[kEncodeThreads * 8];
    const TileGeom g = locate_tile<BITS>(tab, blockIdx.x >> 1);
    const int r0 = (int)(blockIdx.x & 1u) * kEncodeThreads, t = (int)threadIdx.x;
    const uint32_t w = blockIdx.y;
    grid_dependency_wait();
    if (r0 >= g.rows) return;
    const uint64_t elem0 = g.elem0 + 32ull * r0, valid = g.valid - 32ull * r0;
    const int rows = min(kEncodeThreads, g.rows - r0);
    if constexpr (DTYPE == 0) load_tile_f32<kEncodeThreads>(tile, static_cast<const float*>(a.grad[w]) + elem0, valid, rows);
    else load_tile_bf16<kEncodeThreads>(tile, static_cast<const uint16_t*>(a.grad[w]) + elem0, valid, rows);
    const EncodeScale es = encode_scale<BITS>(__ldcg(a.scales[w] + g.seg));   // final: the max pass applied the flush
    __syncthreads();
    if (t >= rows) return;
    float x[32];
    read_row(tile, t, x);
    const uint64_t word0 = g.word0 + (uint64_t)(r0 + t) * BITS;
    const bool vec = (reinterpret_cast<uintptr_t>(a.codes[w] + g.word0) & 15u) == 0;
    encode_store_row<BITS, false>(x, es, a, w, a.elem_offset + elem0 + 32ull * t, valid - 32ull * t, word0, g.words_end, vec);
}

// ---- host side -------------------------------------------------------------------------------------
TableArgs make_table_args(const void* const* grads, int W, uint32_t* const* codes, float* const* scales, uint64_t seed,
                          uint32_t first_worker, uint32_t step, uint64_t elem_offset)
{
    TableArgs a;
    memset(&a, 0, sizeof(a));
    for (int w = 0; w < W; ++w) { a.grad[w] = grads[w]; a.codes[w] = codes[w]; a.scales[w] = scales[w]; }
    a.elem_offset = elem_offset;
    a.first_worker = first_worker;
    a.W = W;
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        a.rk.k0[r] = k0; a.rk.k1[r] = k1;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    a.rk.worker = first_worker; a.rk.step = step;
    return a;
}

// Shared memory of a launch whose longest span has `most` elements (with slack to round the base up), and the attribute
// that allows a kernel the most of it.
static size_t span_smem(uint64_t most) { return (size_t)((most + 31) / 32) * 128 + 1024; }
template <typename Kernel>
static cudaError_t allow_span_smem(Kernel kernel, std::atomic<bool> (&ready)[64], int threads)
{
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    if (!ready[dev].load(std::memory_order_relaxed)) {
        const int most = (threads == 256 ? 512 : kMaxSpanRows) * 128 + 1024;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (err == cudaSuccess) ready[dev].store(true, std::memory_order_relaxed);
    }
    return err;
}

template <int BITS, int DTYPE, int MODE, int THREADS>
static cudaError_t launch_span_inst(const TableArgs& a, const SpanTable& tab, unsigned nspan, uint64_t most,
                                    cudaStream_t stream)
{
    static std::atomic<bool> ready[64];                                // per device (zero-initialised)
    const cudaError_t err = allow_span_smem(span_kernel<BITS, DTYPE, MODE, THREADS>, ready, THREADS);
    if (err != cudaSuccess) return err;
    return launch_pdl_grid(span_kernel<BITS, DTYPE, MODE, THREADS>, dim3(nspan, (unsigned)a.W), THREADS, span_smem(most),
                           stream, a, tab);
}

template <int MODE>
static cudaError_t launch_span_mode(const TableArgs& a, const SpanTable& tab, unsigned nspan, uint64_t most, int bits,
                                    int dtype, cudaStream_t stream)
{
    const bool wide = most > 512 * 32;
    switch (bits) {
#define MQG_SPAN_CASE(B) \
        case B: return dtype == 0 ? (wide ? launch_span_inst<B, 0, MODE, 512>(a, tab, nspan, most, stream)  \
                                          : launch_span_inst<B, 0, MODE, 256>(a, tab, nspan, most, stream)) \
                                  : (wide ? launch_span_inst<B, 1, MODE, 512>(a, tab, nspan, most, stream)  \
                                          : launch_span_inst<B, 1, MODE, 256>(a, tab, nspan, most, stream))
        MQG_SPAN_CASE(1); MQG_SPAN_CASE(2); MQG_SPAN_CASE(3); MQG_SPAN_CASE(4);
        MQG_SPAN_CASE(5); MQG_SPAN_CASE(6); MQG_SPAN_CASE(7); MQG_SPAN_CASE(8);
#undef MQG_SPAN_CASE
    }
    return cudaErrorInvalidValue;
}

template <int BITS, int DTYPE, int MODE>
static cudaError_t launch_joined_inst(const TableArgs& a, const JoinedTable& tab, unsigned ctas, unsigned cluster, uint64_t most,
                                      cudaStream_t stream)
{
    static std::atomic<bool> ready[64];                                // per device (zero-initialised)
    const cudaError_t err = allow_span_smem(joined_span_kernel<BITS, DTYPE, MODE>, ready, kMaxTileRows);
    if (err != cudaSuccess) return err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas, (unsigned)a.W);
    cfg.blockDim = dim3(kMaxTileRows);
    cfg.dynamicSmemBytes = span_smem(most);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, joined_span_kernel<BITS, DTYPE, MODE>, a, tab);
}

// The CTAs of the spans' parts, a cluster of as many as the longest span has: the longest span that still fits into a cluster
// is placed in it, until none of several parts is left.  Returns the launch's CTAs.
unsigned place_joined_spans(const SpanTable& spans, uint64_t alone, JoinedTable& tab, unsigned& cluster)
{
    int first[kMaxCluster + 1], next[kMaxSegmentsPerLaunch];           // lists of the spans of so many parts
    for (unsigned p = 0; p <= kMaxCluster; ++p) first[p] = -1;
    cluster = 1;
    for (int j = spans.nspan - 1; j >= 0; --j) {
        const unsigned parts = spans.len[j] <= alone ? 1u : (unsigned)((spans.len[j] + kJoinedChunk - 1) / kJoinedChunk);
        tab.parts[j] = (uint8_t)parts;
        next[j] = first[parts];
        first[parts] = j;
        if (parts > cluster) cluster = parts;
    }
    unsigned cta = 0;
    auto place = [&](unsigned parts) {
        const int j = first[parts];
        first[parts] = next[j];
        for (unsigned p = 0; p < parts; ++p) tab.cta[cta++] = (uint16_t)(j + 256 * p);
    };
    auto fill_up = [&] {
        while (cta % cluster != 0) tab.cta[cta++] = kNoPart;
    };
    unsigned room = cluster, most = cluster;                           // CTAs left of the cluster; of the longest span left
    for (;;) {
        while (most > 1 && first[most] < 0) --most;
        if (most == 1) break;
        unsigned p = most < room ? most : room;
        while (p > 1 && first[p] < 0) --p;
        if (p > 1) {
            place(p);
            room -= p;
        } else {
            fill_up();
            room = cluster;
        }
    }
    fill_up();                                 // no span of one CTA beside some whose CTAs wait for one another
    while (first[1] >= 0) place(1);
    fill_up();
    return cta;
}

cudaError_t launch_joined_spans(const TableArgs& a, const SpanTable& spans, uint64_t alone, int mode, int bits, int dtype,
                                cudaStream_t stream)
{
    uint64_t most = 0;                                                 // of a CTA
    for (int j = 0; j < spans.nspan; ++j) {
        if (spans.len[j] > kMaxJoinedElems) return cudaErrorInvalidValue;
        const uint64_t part = spans.len[j] <= alone ? spans.len[j] : kJoinedChunk;
        if (part > most) most = part;
    }
    JoinedTable tab;
    tab.spans = spans;
    unsigned cluster;
    const unsigned ctas = place_joined_spans(spans, alone, tab, cluster);
    switch (bits) {
#define MQG_JOINED(B, D) \
        (mode == kSpanNorm ? launch_joined_inst<B, D, kSpanNorm>(a, tab, ctas, cluster, most, stream) \
                           : launch_joined_inst<B, D, kSpanMaxAbs>(a, tab, ctas, cluster, most, stream))
#define MQG_JOINED_CASE(B) case B: return dtype == 0 ? MQG_JOINED(B, 0) : MQG_JOINED(B, 1)
        MQG_JOINED_CASE(1); MQG_JOINED_CASE(2); MQG_JOINED_CASE(3); MQG_JOINED_CASE(4);
        MQG_JOINED_CASE(5); MQG_JOINED_CASE(6); MQG_JOINED_CASE(7); MQG_JOINED_CASE(8);
#undef MQG_JOINED_CASE
#undef MQG_JOINED
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_spans(const TableArgs& a, const SpanTable& tab, unsigned nspan, uint64_t most, int mode, int bits,
                         int dtype, cudaStream_t stream)
{
    if (most > (uint64_t)kMaxSpanRows * 32) return cudaErrorInvalidValue;
    if (mode == kSpanRange) return launch_span_mode<kSpanRange>(a, tab, nspan, most, bits, dtype, stream);
    if (mode == kSpanNorm) return launch_span_mode<kSpanNorm>(a, tab, nspan, most, bits, dtype, stream);
    return launch_span_mode<kSpanMaxAbs>(a, tab, nspan, most, bits, dtype, stream);
}

bool bucket_spans_apply(uint64_t n, uint64_t bucket)
{
    const uint64_t b = bucket < n ? bucket : n;
    return b <= (uint64_t)kMaxSpanRows * 32 && (n + b - 1) / b <= 0x7FFFFFFFull;
}

cudaError_t launch_bucket_spans(const void* const* grads, int W, uint64_t n, int bits, uint64_t bucket, uint64_t seed,
                                uint32_t* const* codes, float* const* scales, int mode, int dtype, uint32_t first_worker,
                                uint32_t step, uint64_t elem_offset, cudaStream_t stream)
{
    const TableArgs a = make_table_args(grads, W, codes, scales, seed, first_worker, step, elem_offset);
    SpanTable tab;
    tab.bucket = bucket < n ? bucket : n;
    tab.n = n;
    tab.nspan = 0;
    return launch_spans(a, tab, (unsigned)((n + tab.bucket - 1) / tab.bucket), tab.bucket, mode, bits, dtype, stream);
}

cudaError_t launch_absmax_table(const TableArgs& a, const SegmentTable& tab, int dtype, cudaStream_t stream)
{
    const uint32_t tiles = tab_tiles(tab);
    if (tiles == 0) return cudaSuccess;
    const dim3 grid(tiles, (unsigned)a.W);
    return dtype == 0 ? launch_pdl_grid(absmax_table_kernel<0>, grid, kMaxTileRows, 0, stream, a, tab)
                      : launch_pdl_grid(absmax_table_kernel<1>, grid, kMaxTileRows, 0, stream, a, tab);
}

cudaError_t launch_clear_scales(const TableArgs& a, int nseg, cudaStream_t stream)
{
    return launch_pdl(clear_scales_kernel, (unsigned)a.W, kMaxTileRows, stream, a, nseg);
}

template <int BITS, int DTYPE>
static cudaError_t launch_spans_absmax_inst(const TableArgs& a, const SpanTable& spans, uint64_t most,
                                            const SegmentTable& longs, cudaStream_t stream)
{
    static std::atomic<bool> ready[64];                                // per device (zero-initialised)
    const cudaError_t err = allow_span_smem(spans_absmax_kernel<BITS, DTYPE>, ready, kMaxTileRows);
    if (err != cudaSuccess) return err;
    return launch_pdl_grid(spans_absmax_kernel<BITS, DTYPE>, dim3((unsigned)spans.nspan + tab_tiles(longs), (unsigned)a.W),
                           kMaxTileRows, span_smem(most), stream, a, spans, longs);
}

cudaError_t launch_spans_absmax(const TableArgs& a, const SpanTable& spans, uint64_t most, const SegmentTable& longs,
                                int bits, int dtype, cudaStream_t stream)
{
    switch (bits) {
#define MQG_FUSED_CASE(B) \
        case B: return dtype == 0 ? launch_spans_absmax_inst<B, 0>(a, spans, most, longs, stream) \
                                  : launch_spans_absmax_inst<B, 1>(a, spans, most, longs, stream)
        MQG_FUSED_CASE(1); MQG_FUSED_CASE(2); MQG_FUSED_CASE(3); MQG_FUSED_CASE(4);
        MQG_FUSED_CASE(5); MQG_FUSED_CASE(6); MQG_FUSED_CASE(7); MQG_FUSED_CASE(8);
#undef MQG_FUSED_CASE
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_encode_table(const TableArgs& a, const SegmentTable& tab, int bits, int dtype, cudaStream_t stream)
{
    const uint32_t tiles = tab_tiles(tab);
    if (tiles == 0) return cudaSuccess;
    if (tiles > 0x3FFFFFFFu) return cudaErrorInvalidValue;
    const dim3 grid(2 * tiles, (unsigned)a.W);
    switch (bits) {
#define MQG_TAB_CASE(B) \
        case B: return dtype == 0 ? launch_pdl_grid(encode_table_kernel<B, 0>, grid, kEncodeThreads, 0, stream, a, tab) \
                                  : launch_pdl_grid(encode_table_kernel<B, 1>, grid, kEncodeThreads, 0, stream, a, tab)
        MQG_TAB_CASE(1); MQG_TAB_CASE(2); MQG_TAB_CASE(3); MQG_TAB_CASE(4);
        MQG_TAB_CASE(5); MQG_TAB_CASE(6); MQG_TAB_CASE(7); MQG_TAB_CASE(8);
#undef MQG_TAB_CASE
    }
    return cudaErrorInvalidValue;
}

// Buckets longer than a span: two passes per worker.
cudaError_t launch_quantize_big_buckets(const void* grad, uint64_t n, int bits, uint64_t bucket,
                                        uint64_t seed, uint32_t* codes, float* scales, int dtype,
                                        uint32_t worker, uint32_t step, uint64_t elem_offset,
                                        cudaStream_t stream)
{
    const TableArgs a = make_table_args(&grad, 1, &codes, &scales, seed, worker, step, elem_offset);
    SegmentTable tab;
    memset(&tab, 0, sizeof(tab));
    const uint64_t b = bucket < n ? bucket : n;          // a single bucket is n long
    tab.uniform_bucket = b;
    tab.n_total = n;
    const uint64_t tile_elems = (uint64_t)kMaxTileRows * 32;
    const uint64_t tpb = (b + tile_elems - 1) / tile_elems;
    if (tpb > 0xFFFFFFFFull) return cudaErrorInvalidValue;
    tab.tiles_per_bucket = (uint32_t)tpb;
    const uint64_t nb = (n + b - 1) / b;
    const uint64_t full = n / b;                          // full buckets have tpb tiles each
    uint64_t ntiles = full * tpb;
    // the grid enumerates tiles_per_bucket tiles for every bucket; the last (shorter) bucket
    // has fewer real tiles, so its tail tiles are simply not launched
    if (nb > full) ntiles += ((n - full * b) + tile_elems - 1) / tile_elems;
    if (ntiles > 0x3FFFFFFFull) return cudaErrorInvalidValue;
    tab.tile_start[0] = (uint32_t)ntiles;                 // nseg = 0: the grid's tiles
    cudaError_t err = cudaMemsetAsync(scales, 0, nb * sizeof(float), stream);
    if (err == cudaSuccess) err = launch_absmax_table(a, tab, dtype, stream);
    if (err == cudaSuccess) err = launch_encode_table(a, tab, bits, dtype, stream);
    return err;
}

}  // namespace mqg
