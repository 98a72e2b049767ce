// Tile lookup for the kernels that work on segments (per-layer scale) or on buckets larger
// than one CTA tile.
#pragma once

#include "mqg_common.cuh"
#include "mqg_internal.h"

namespace mqg {

// The gradients of the workers that share a table, and the keys of their draws.
struct TableArgs {
    const void* grad[kMaxWorkers];
    uint32_t* codes[kMaxWorkers];
    float* scales[kMaxWorkers];     // scale of the table's segment j at scales[w][j]
    uint64_t elem_offset;
    uint32_t first_worker;
    int W;
    RoundKeys rk;
};
TableArgs make_table_args(const void* const* grads, int W, uint32_t* const* codes, float* const* scales, uint64_t seed,
                          uint32_t first_worker, uint32_t step, uint64_t elem_offset);

// The two passes over the tiles a table lists, for every worker (scales zeroed before the first).
inline uint32_t tab_tiles(const SegmentTable& tab) { return tab.tile_start[tab.nseg]; }
cudaError_t launch_absmax_table(const TableArgs& a, const SegmentTable& tab, int dtype, cudaStream_t stream);
cudaError_t launch_encode_table(const TableArgs& a, const SegmentTable& tab, int bits, int dtype, cudaStream_t stream);

// Spans: what one CTA quantizes as a whole.  bucket != 0: span j is bucket j of a gradient of n elements;
// otherwise the lists, and the launch also clears the scales first + i for which bit i of clear[] is set.
constexpr int kMaxSpanRows = 1536;      // 192 KB of shared memory
enum : int { kSpanMaxAbs = 0, kSpanRange = 1, kSpanNorm = 2 };
struct SpanTable {
    uint64_t bucket, n;
    int nspan, first;
    uint32_t clear[kMaxSegmentsPerLaunch / 32];
    uint32_t scale_idx[kMaxSegmentsPerLaunch];
    uint64_t elem0[kMaxSegmentsPerLaunch], len[kMaxSegmentsPerLaunch], code0[kMaxSegmentsPerLaunch];
};
// `nspan` CTAs per worker; `most` = elements of the longest span.
cudaError_t launch_spans(const TableArgs& a, const SpanTable& tab, unsigned nspan, uint64_t most, int mode, int bits,
                         int dtype, cudaStream_t stream);

// Spans of a list (no clears) of up to kMaxJoinedElems elements, kSpanMaxAbs or kSpanNorm: those of more than `alone`
// elements (kJoinedChunk .. 16384) are several CTAs' of a cluster, one for every kJoinedChunk elements.
constexpr unsigned kMaxCluster = 8;                                  // CTAs, the portable limit
constexpr uint64_t kJoinedChunk = (uint64_t)kMaxTileRows * 32;       // elements per CTA, a power of two of rows
constexpr uint64_t kMaxJoinedElems = kMaxCluster * kJoinedChunk;
constexpr uint32_t kNoPart = 0xFFFF;
struct JoinedTable {
    SpanTable spans;
    uint16_t cta[kMaxCluster * kMaxSegmentsPerLaunch];       // span of a CTA + 256 times its part; kNoPart: fills a cluster up
    uint8_t parts[kMaxSegmentsPerLaunch];                    // CTAs of a span
};
cudaError_t launch_joined_spans(const TableArgs& a, const SpanTable& tab, uint64_t alone, int mode, int bits, int dtype,
                                cudaStream_t stream);

// The same in the main codec together with the max pass over `longs`, whose scales launch_clear_scales has cleared.
cudaError_t launch_clear_scales(const TableArgs& a, int nseg, cudaStream_t stream);
cudaError_t launch_spans_absmax(const TableArgs& a, const SpanTable& spans, uint64_t most, const SegmentTable& longs,
                                int bits, int dtype, cudaStream_t stream);

struct TileGeom {
    uint64_t elem0;       // flat index of the tile's first element
    uint64_t valid;       // elements from elem0 to the end of the segment
    uint64_t word0;       // code word of the tile's first row
    uint64_t words_end;   // one past the segment's last code word
    uint64_t seg;         // segment index (= index of its scale)
    uint32_t tile_local;  // tile index inside the segment
    int rows;             // rows of this tile that exist
};

template <int BITS>
__device__ __forceinline__ TileGeom locate_tile(const SegmentTable& tab, uint32_t tile)
{
    TileGeom g;
    uint64_t seg_start, seg_len, code0;
    if (tab.uniform_bucket != 0) {
        g.seg = tile / tab.tiles_per_bucket;
        g.tile_local = tile % tab.tiles_per_bucket;
        seg_start = g.seg * tab.uniform_bucket;
        const uint64_t left = tab.n_total - seg_start;
        seg_len = left < tab.uniform_bucket ? left : tab.uniform_bucket;
        code0 = seg_start / 32 * BITS;
    } else {
        int lo = 0, hi = tab.nseg - 1;              // last j with tile_start[j] <= tile
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (tab.tile_start[mid] <= tile) lo = mid; else hi = mid - 1;
        }
        g.seg = (uint64_t)lo;
        g.tile_local = tile - tab.tile_start[lo];
        seg_start = tab.seg_off[lo];
        seg_len = tab.seg_off[lo + 1] - seg_start;
        code0 = tab.code_off[lo];
    }
    const uint64_t done = (uint64_t)g.tile_local * (kMaxTileRows * 32);
    g.elem0 = seg_start + done;
    g.valid = seg_len - done;
    g.word0 = code0 + (uint64_t)g.tile_local * kMaxTileRows * BITS;
    g.words_end = code0 + (seg_len * BITS + 31) / 32;
    const uint64_t rows = (g.valid + 31) / 32;
    g.rows = (int)(rows < (uint64_t)kMaxTileRows ? rows : (uint64_t)kMaxTileRows);
    return g;
}

}  // namespace mqg
