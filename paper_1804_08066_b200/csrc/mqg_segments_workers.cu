// Per-layer quantization (one scale per segment; Section 4.1 quantizes whole layers) of one or several
// workers' gradients that share a segment table (Algorithm 1, WorkerIterate line 3, for every worker of the
// simulation), in up to three launches whatever the number of workers and segments:
//   1. span_kernel (mqg_segments.cu) - every segment of at most kSegmentSpanElems elements, scale and codes;
//      the launch also clears the scales of the longer ones;
//   2. absmax_table_kernel - the max pass over the longer segments;
//   3. encode_entries_kernel - their encode.  Every (worker, segment) pair is an entry with a tensor map of its
//      own; the persistent CTAs walk the 128-row tiles of all entries as one sequence, fed by tiled bulk copies
//      exactly like quantize_workers_kernel (tile code of mqg_quantize_tile.cuh, given-scale mode).  Segments
//      that start where bulk copies cannot go through encode_table_kernel instead.
// Worker w's outputs are the same whichever way a segment goes and however many workers there are.
#include <string.h>

#include <atomic>
#include <vector>

#include "mqg_quantize_tile.cuh"
#include "mqg_segments.cuh"

namespace mqg {

// Entries per launch: the table is a kernel parameter, copied at every launch, so calls with few entries take
// the small one (paper-sized calls of two segments: 3 against 13 KB of parameters).
constexpr int kFewEntries = 16, kMaxEntries = 64;

// Longest segment that one CTA handles alone: two rows per thread, 2 to 3 us.
constexpr uint64_t kSegmentSpanElems = 512 * 32;

struct SegEntry {
    const void* grad;        // the segment's first element (for its ragged last row)
    uint32_t* codes;         // the segment's first code word
    float* scale;            // its scale, final when the encode pass starts
    uint64_t n;              // elements
    uint32_t ntiles;         // tiles of 128 rows
    uint32_t full_tiles;     // leading tiles whose 128 rows are all complete
    uint32_t blk0_lo;        // low half of the Philox block index of the segment's first element
    PhiloxHead head;         // launch-wide part of its blocks (worker, high half of the block index)
};

template <int CAP>
struct SegEntryTable {
    CUtensorMap map[CAP];
    SegEntry e[CAP];
    int nent;
};

// total_tiles = tiles of all entries.
template <int BITS, int DTYPE, int CAP>
__global__ void __launch_bounds__(128, 5)
encode_entries_kernel(const __grid_constant__ SegEntryTable<CAP> ent, const __grid_constant__ QuantizeArgs a,
                      const __grid_constant__ TmaQuantizeConsts c, uint32_t total_tiles,
                      unsigned int* __restrict__ timeouts)
{
    constexpr int THREADS = 128;
    using Shared = TmaQuantizeShared<DTYPE, THREADS>;
    constexpr int kQuantStages = Shared::kStages;
    __shared__ Shared sh;

    const uint32_t t = threadIdx.x;
    const uint32_t stride = gridDim.x;
    const uint32_t box_bytes = THREADS * Shared::kRowBytes;
    if (t == 0) {
        for (int s = 0; s < kQuantStages; ++s) mbar_init(smem_u32(&sh.bar[s]), 1);
        fence_barrier_init();
    }
    grid_dependency_release();
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory

    // ---- the tiles of the entries, one sequence walked like quantize_workers_kernel walks its workers
    struct Pos { uint32_t e, tile; };
    auto advance = [&](Pos& p, uint32_t by) {
        p.tile += by;
        while (p.tile >= ent.e[p.e].ntiles) { p.tile -= ent.e[p.e].ntiles; ++p.e; }
    };
    auto load_tile = [&](const Pos& p, uint32_t stage, uint32_t bar) {     // thread 0 only
        mbar_expect_tx(bar, box_bytes);
        if (!a.arm_only) tma_load_2d(stage, &ent.map[p.e], 0, (int)(p.tile * THREADS), bar);
    };
    uint32_t v = blockIdx.x;
    Pos cur = {0u, 0u}, fill = {0u, 0u};
    if (v < total_tiles) { advance(cur, v); advance(fill, v); }
    uint32_t vfill = v;
    for (uint32_t s = 0; s < (uint32_t)kQuantStages; ++s) {
        if (t == 0 && vfill < total_tiles) load_tile(fill, smem_u32(sh.stage[s]), smem_u32(&sh.bar[s]));
        vfill += stride;
        if (vfill < total_tiles) advance(fill, stride);
    }

    uint32_t k = 0, rot = 0;
    bool ok = true;
#pragma unroll 1
    for (; ok && v < total_tiles; v += stride, ++k, rot = (rot == 2 ? 0 : rot + 1)) {
        const SegEntry& e = ent.e[cur.e];
        const uint32_t tile = cur.tile;
        const WorkerView wv = {&ent.map[cur.e], e.grad, e.codes, e.scale, e.head, e.blk0_lo,
                               (reinterpret_cast<uintptr_t>(e.codes) & 15u) != 0};
        auto refill = [&](uint32_t stage, uint32_t bar) {
            if (vfill < total_tiles) load_tile(fill, stage, bar);
        };
        if (tile < e.full_tiles) {
            ok = quantize_tile<BITS, DTYPE, THREADS, true, kByWarps, false, true>(sh, wv, a, c, k, rot, tile, refill,
                                                                                0u, false);
        } else {
            QuantizeArgs ae = a;           // the bounds of this entry, needed by its last tile only
            ae.n = e.n;
            ae.nrows = (e.n + 31) / 32;
            ae.nrows_full = e.n / 32;
            ae.ncode_words = (e.n * BITS + 31) / 32;
            ok = quantize_tile<BITS, DTYPE, THREADS, false, kByWarps, false, true>(sh, wv, ae, c, k, rot, tile, refill,
                                                                                 0u, false);
        }
        if (v + stride < total_tiles) advance(cur, stride);
        vfill += stride;
        if (vfill < total_tiles) advance(fill, stride);
    }
    if (!ok) {                         // as in quantize_workers_kernel
        if (t == 0) {
            atomicAdd(timeouts, 1u);
            uint32_t j = k - 1, vl = v - stride;
            for (int s = 0; s < kQuantStages && vl < total_tiles; ++s, ++j, vl += stride)
                mbar_wait(smem_u32(&sh.bar[j % kQuantStages]), (j / kQuantStages) & 1, a.poll_limit);
        }
        __syncthreads();
    }
}

// ---- host side --------------------------------------------------------------------------------
namespace {

struct EntryHost {
    const void* grad;
    uint32_t* codes;
    float* scale;
    uint64_t n, elem_offset;
    uint32_t worker;
};

template <int BITS, int DTYPE, int CAP>
cudaError_t launch_entries_inst(const SegEntryTable<CAP>& ent, const QuantizeArgs& a, const TmaQuantizeConsts& c,
                                uint32_t total_tiles, unsigned int* timeouts, cudaStream_t stream)
{
    auto kernel = encode_entries_kernel<BITS, DTYPE, CAP>;
    static std::atomic<int> grid_cap[64];          // per device; 0 = not yet queried (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 128, 0);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    unsigned grid = (unsigned)cap;
    if (grid > total_tiles) grid = total_tiles;
    return launch_pdl(kernel, grid, 128, stream, ent, a, c, total_tiles, timeouts);
}

template <int CAP>
cudaError_t launch_entries(const EntryHost* entries, int nent, int bits, const RoundKeys& rk, int dtype,
                           cudaStream_t stream)
{
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    QuantizeArgs a;
    memset(&a, 0, sizeof(a));
    a.tile_rows = 128; a.rows_per_bucket = 128; a.buckets_per_tile = 1; a.nbuckets = 1;
    const WaitPolicy policy = wait_policy();
    a.poll_limit = policy.poll_limit;
    a.arm_only = policy.arm_only;
    TmaQuantizeConsts c;
    memset(&c, 0, sizeof(c));
    c.rk = rk;
    SegEntryTable<CAP> ent;
    ent.nent = nent;
    uint64_t total = 0;
    for (int i = 0; i < nent; ++i) {
        const EntryHost& h = entries[i];
        SegEntry& e = ent.e[i];
        const uint64_t nrows = (h.n + 31) / 32, nrows_full = h.n / 32;
        const char* why = nullptr;
        if (!encode_rows_map(&ent.map[i], h.grad, nrows_full, dtype == 0 ? 4 : 2, 32, 128, &why))
            return cudaErrorNotSupported;
        e.grad = h.grad; e.codes = h.codes; e.scale = h.scale; e.n = h.n;
        e.ntiles = (uint32_t)((nrows + 127) / 128);
        e.full_tiles = (uint32_t)(nrows_full / 128);
        const uint64_t blk0 = h.elem_offset >> 3;
        e.blk0_lo = (uint32_t)blk0;
        e.head = philox_head((uint32_t)(blk0 >> 32), h.worker, rk.k0[0]);
        total += e.ntiles;
    }
    if (total > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    switch (bits) {
#define MQG_ENT_CASE(B) \
        case B: return dtype == 0 ? launch_entries_inst<B, 0, CAP>(ent, a, c, (uint32_t)total, timeouts, stream) \
                                  : launch_entries_inst<B, 1, CAP>(ent, a, c, (uint32_t)total, timeouts, stream)
        MQG_ENT_CASE(1); MQG_ENT_CASE(2); MQG_ENT_CASE(3); MQG_ENT_CASE(4);
        MQG_ENT_CASE(5); MQG_ENT_CASE(6); MQG_ENT_CASE(7); MQG_ENT_CASE(8);
#undef MQG_ENT_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_quantize_segments(const void* const* grads, int W, int nseg, const uint64_t* seg_off,
                                     const uint64_t* code_off, int bits, uint64_t seed, uint32_t* const* codes,
                                     float* const* scales, int dtype, uint32_t first_worker, uint32_t step,
                                     uint64_t elem_offset, float* workspace, cudaStream_t stream)
{
    const size_t esz = dtype == 0 ? 4 : 2;
    const TableArgs a = make_table_args(grads, W, codes, scales, seed, first_worker, step, elem_offset);
    auto bulk = [&](int j) {                          // every worker's gradient is aligned for bulk copies
        for (int w = 0; w < W; ++w)
            if (!quantize_given_scale_applies(static_cast<const char*>(grads[w]) + seg_off[j] * esz,
                                              seg_off[j + 1] - seg_off[j], elem_offset + seg_off[j]))
                return false;
        return true;
    };
    std::vector<EntryHost> entries;
    cudaError_t err = cudaSuccess;
    uint64_t sums = 0;                                // partial sums of the tables already launched
    for (int first = 0; first < nseg; first += kMaxSegmentsPerLaunch) {
        const int count = nseg - first < kMaxSegmentsPerLaunch ? nseg - first : kMaxSegmentsPerLaunch;
        SpanTable spans;
        SegmentTable longs, plain;                    // the segments that are no spans; those the table encode takes
        memset(&spans, 0, sizeof(spans));
        memset(&longs, 0, sizeof(longs));
        spans.first = first;
        longs.nseg = count;
        uint64_t most = 0, tiles = 0, plain_tiles = 0;
        plain = longs;
        for (int i = 0; i < count; ++i) {
            const int j = first + i;
            const uint64_t len = seg_off[j + 1] - seg_off[j];
            longs.tile_start[i] = (uint32_t)tiles;
            plain.tile_start[i] = (uint32_t)plain_tiles;
            longs.seg_off[i] = plain.seg_off[i] = seg_off[j];
            longs.code_off[i] = plain.code_off[i] = code_off[j];
            if (len <= kSegmentSpanElems) {
                const int k = spans.nspan++;
                spans.elem0[k] = seg_off[j]; spans.len[k] = len; spans.code0[k] = code_off[j];
                spans.scale_idx[k] = (uint32_t)j;
                if (len > most) most = len;
            } else {
                if (!workspace) spans.clear[i >> 5] |= 1u << (i & 31);
                const uint64_t nt = (len + kMaxTileRows * 32 - 1) / (kMaxTileRows * 32);
                tiles += nt;
                if (bulk(j)) {
                    for (int w = 0; w < W; ++w)
                        entries.push_back({static_cast<const char*>(grads[w]) + seg_off[j] * esz, codes[w] + code_off[j],
                                           scales[w] + j, len, elem_offset + seg_off[j], first_worker + (uint32_t)w});
                } else {
                    plain_tiles += nt;
                }
            }
            if (tiles > 0x3FFFFFFFull) return cudaErrorInvalidValue;
        }
        longs.tile_start[count] = (uint32_t)tiles;
        plain.tile_start[count] = (uint32_t)plain_tiles;
        longs.seg_off[count] = plain.seg_off[count] = seg_off[first + count];
        if (spans.nspan != 0 || (tiles != 0 && !workspace)) {
            err = launch_spans(a, spans, spans.nspan != 0 ? (unsigned)spans.nspan : 1u, most,
                               workspace ? kSpanNorm : kSpanMaxAbs, bits, dtype, stream);
            if (err != cudaSuccess) return err;
        }
        if (tiles == 0) continue;
        TableArgs t = a;                              // a table numbers its segments from 0
        for (int w = 0; w < W; ++w) t.scales[w] += first;
        err = workspace ? launch_segments_l2_scales(grads[0], longs, t.scales[0], dtype, workspace + sums, stream)
                        : launch_absmax_table(t, longs, dtype, stream);
        sums += tiles;
        if (err == cudaSuccess) err = launch_encode_table(t, plain, bits, dtype, stream);
        if (err != cudaSuccess) return err;
    }
    const size_t total = entries.size();
    for (size_t from = 0; from < total && err == cudaSuccess; from += (size_t)kMaxEntries) {
        const int n = (int)(total - from < (size_t)kMaxEntries ? total - from : (size_t)kMaxEntries);
        err = n <= kFewEntries ? launch_entries<kFewEntries>(entries.data() + from, n, bits, a.rk, dtype, stream)
                               : launch_entries<kMaxEntries>(entries.data() + from, n, bits, a.rk, dtype, stream);
    }
    return err;
}

}  // namespace mqg
