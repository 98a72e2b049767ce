// Per-layer quantization (one scale per segment; Section 4.1 quantizes whole layers) of one or several
// workers' gradients that share a segment table (Algorithm 1, WorkerIterate line 3, for every worker of the
// simulation), in three launches for up to 64 segments and 64 (worker, long segment) pairs:
//   1. clear_scales_kernel (mqg_segments.cu);
//   2. spans_absmax_kernel - every segment of at most kSegmentSpanElems elements, scale and codes by one CTA, and beside
//      them the max pass over the longer segments; a launch for every 64 segments;
//   3. encode_entries_kernel - the longer ones' encode.  Every (worker, segment) pair is an entry with a tensor map of its
//      own; the persistent CTAs walk the 128-row tiles of all entries as one sequence, fed by tiled bulk copies; a launch
//      for every 64 entries.  Segments that start where bulk copies cannot: encode_flat_kernel, by rows of the whole gradient
//      (encode_table_kernel where that cannot either).
// Where these two do not go together (spans_join_max_pass), span_kernel also clears the scales and absmax_table_kernel
// follows it.
// Worker w's outputs are the same whichever way a segment goes and however many workers there are.
#include <string.h>

#include <atomic>

#include "mqg_quantize_tile.cuh"
#include "mqg_segments.cuh"

namespace mqg {

// Entries per launch: the table is a kernel parameter, copied at every launch, so calls with few entries take
// the small one (paper-sized calls of two segments: 3 against 13 KB of parameters).
constexpr int kFewEntries = 16, kMaxEntries = 64;

// Longest segment that one CTA handles alone: two rows per thread, 2 to 3 us.
constexpr uint64_t kSegmentSpanElems = 512 * 32;

// Whether the spans and the max pass share a launch (`tiles` of 256 rows in the max pass).  Spans on their own are 3 us
// during which a few CTAs are at work; the launch before then only clears the scales, 1.2 us.  The other side is the spans'
// registers and shared memory, with which three CTAs share an SM: the max pass reads hardly slower in fp32 (32 KB requested
// by every CTA: an AlexNet-shaped gradient 80.4 against 83.0 us, four 303 against 305 us, eight with the server's step 763
// against 759 us), but in bf16 (16 KB: eight 463 against 409 us) or where segments start off a 16-byte boundary (100 against
// 93 us for 31 M elements in 16 tensors).  bf16 gradients of 41 M elements in 100 tensors 65 against 70 us, fp32 74 against 81 us; 10 M off
// the boundary in 20 tensors 28 against 30 us.
static bool spans_join_max_pass(uint64_t tiles, int dtype, bool aligned)
{
    return tiles <= (!aligned ? 2048u : dtype == 0 ? 32768u : 8192u);
}

struct SegEntry {
    const void* grad;        // the segment's first element (for its ragged last row)
    uint32_t* codes;         // the segment's first code word
    float* scale;            // its scale, final when the encode pass starts
    uint64_t n;              // elements
    uint32_t tile0;          // its first tile's number in the launch's sequence
    uint32_t blk0_lo;        // low half of the Philox block index of the segment's first element
    PhiloxHead head;         // launch-wide part of its blocks (worker, high half of the block index)
};

template <int CAP>
struct SegEntryTable {
    CUtensorMap map[CAP];
    SegEntry e[CAP];
    uint32_t tile_end[CAP];              // one past each entry's last tile; 2^32 - 1 beyond the last entry
    uint32_t tiles;
    uint32_t poll_limit, arm_only;       // as in QuantizeArgs
    RoundKeys rk;
};

// The scale is given, so no warp needs another: the four warps of a CTA share the tiles' copies (16 KB: 128 rows of
// 32 fp32 or 64 bf16 elements; a copy per warp's 4 KB took 635 against 622 us for eight AlexNet-shaped gradients) and
// nothing else.  There is no CTA barrier: the last warp to have read a stage refills it.  What an entry's tiles share -
// pointers, Philox head, the encode's constants with their division - is fetched when the entry changes.  The draws
// come before the wait for the data, at the price of the fifth CTA per SM: 604 against 620 us for that call, 413
// against 440 us in bf16 (622 and 437 us with a CTA barrier per tile and the tile code of the one-pass kernels).
template <int BITS, int DTYPE, int CAP>
__global__ void __launch_bounds__(128, 4)
encode_entries_kernel(const __grid_constant__ SegEntryTable<CAP> T, unsigned int* __restrict__ timeouts)
{
    constexpr uint32_t kWarps = 4, kStages = 2, kRows = 32 * kWarps, kTileBytes = kRows * 128;
    constexpr int kHalves = DTYPE == 0 ? 1 : 2, kElems = 32 * kHalves, kWords = BITS * kHalves;
    struct Shared {
        alignas(1024) uint8_t stage[kStages][kTileBytes];
        alignas(8) uint64_t bar[kStages];
        uint32_t read[kStages];        // warps that have read the stage, over all its uses
    };
    __shared__ Shared sh;
    const uint32_t t = threadIdx.x, lane = t & 31u;
    const uint32_t step = gridDim.x;
    if (t == 0) {
        for (uint32_t s = 0; s < kStages; ++s) { mbar_init(smem_u32(&sh.bar[s]), 1); sh.read[s] = 0u; }
        fence_barrier_init();
    }
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory

    uint32_t u = blockIdx.x, fill = u;             // the tile in work, the next one to fetch
    uint32_t fe = 0;                               // the entry of `fill`: searched once, then only moved forward
#pragma unroll
    for (uint32_t half = CAP / 2; half > 0; half >>= 1)
        if (u >= T.tile_end[fe + half - 1]) fe += half;
    if (u >= T.tiles) fe = 0;
    uint32_t e = fe;
    auto fetch = [&](uint32_t s, bool mine) {
        if (fill < T.tiles) {
            while (fill >= T.tile_end[fe]) ++fe;
            if (mine) {
                const uint32_t bar = smem_u32(&sh.bar[s]);
                mbar_expect_tx(bar, kTileBytes);
                if (!T.arm_only)
                    tma_load_2d(smem_u32(sh.stage[s]), &T.map[fe], 0, (int)((fill - T.e[fe].tile0) * kRows), bar);
            }
        }
        fill += step;
    };
    for (uint32_t s = 0; s < kStages; ++s) fetch(s, t == 0);

    uint32_t k = 0, end = 0, tile0 = 0, blk0 = 0, rows = 0, rows_full = 0;
    uint32_t* codes = nullptr;
    bool vec = false, ok = true;
    PhiloxHead head = {};
    EncodeScale es = {0.0f, 0.0f};
#pragma unroll 1
    for (; u < T.tiles; u += step, ++k) {
        if (u >= end) {
            while (u >= T.tile_end[e]) ++e;
            const SegEntry& x = T.e[e];
            end = T.tile_end[e]; tile0 = x.tile0; blk0 = x.blk0_lo; head = x.head; codes = x.codes;
            rows = (uint32_t)((x.n + kElems - 1) / kElems); rows_full = (uint32_t)(x.n / kElems);
            vec = (reinterpret_cast<uintptr_t>(codes) & 15u) == 0;
            es = encode_scale<BITS>(__ldcg(x.scale));
        }
        const uint32_t s = k % kStages, row = (u - tile0) * kRows + t;
        uint8_t* stage = sh.stage[s];
        const uint32_t bar = smem_u32(&sh.bar[s]);
        uint32_t h[16];
        draw_row_blocks_head(blk0 + 4u * kHalves * row, head, T.rk, h);
        const bool active = row < rows;
        ok = mbar_try_wait(bar, (k / kStages) & 1);
        if (!ok) ok = mbar_wait(bar, (k / kStages) & 1, T.poll_limit);
        if (!__all_sync(0xFFFFFFFFu, ok)) { ok = false; break; }
        if (active && row >= rows_full)    // a last row that the copy does not cover
            stage_ragged_row(stage, t, static_cast<const uint8_t*>(T.e[e].grad), row, T.e[e].n * (DTYPE == 0 ? 4 : 2));

        uint4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = reinterpret_cast<const uint4*>(stage)[swz((int)t, i)];
        __syncwarp();                      // every lane has read the stage
        bool last = false;
        if (lane == 0) {
            __threadfence_block();
            last = (atomicAdd(&sh.read[s], 1u) & (kWarps - 1)) == kWarps - 1;
            if (last) __threadfence_block();
        }
        fetch(s, last);

        const uint32_t* raw = reinterpret_cast<const uint32_t*>(v);
        uint32_t w[kWords];
#pragma unroll
        for (int half = 0; half < kHalves; ++half) {
            float x[32];
            if constexpr (DTYPE == 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j] = __uint_as_float(raw[j]);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) { x[2 * j] = bf16_lo(raw[16 * half + j]); x[2 * j + 1] = bf16_hi(raw[16 * half + j]); }
            }
            if (half != 0) draw_row_blocks_head(blk0 + 4u * (kHalves * row + half), head, T.rk, h);
            uint32_t wh[BITS];
            encode_pack_row_best<BITS>(x, es, h, wh);
#pragma unroll
            for (int j = 0; j < BITS; ++j) w[half * BITS + j] = wh[j];
        }
        const uint64_t word0 = (uint64_t)row * kWords;
        if (row < rows_full) {
            if (vec) {
                store_row_words<kWords>(codes, word0, w);
            } else {
#pragma unroll
                for (int j = 0; j < kWords; ++j) codes[word0 + j] = w[j];
            }
        } else if (active) {
            const uint64_t n = T.e[e].n, words = (n * BITS + 31) / 32;
            mask_row_words<kWords>(w, (int)(n - (uint64_t)row * kElems) * BITS);
#pragma unroll
            for (int j = 0; j < kWords; ++j)
                if (word0 + j < words) codes[word0 + j] = w[j];
        }
    }
    if (!ok && lane == 0) {
        // A copy never landed: record it, then give the copies still in flight (the one that was being waited for and
        // the one after it) a last bounded chance before the shared memory can be handed to another CTA.
        atomicAdd(timeouts, 1u);
        for (uint32_t j = k; j < k + kStages && u < T.tiles; ++j, u += step)
            mbar_wait(smem_u32(&sh.bar[j % kStages]), (j / kStages) & 1, T.poll_limit);
    }
}

// The encode of segments that start off a 16-byte boundary (a layered gradient whose tensors are not padded).  A row here is
// a row of the worker's whole gradient, 128 aligned bytes that belong to one or two segments, so that bulk copies fetch the
// tiles and the draws come in whole blocks; what is shifted is the bit stream.  A row's packed words go to shared memory, where
// a warp's 32 rows are one stretch of the gradient's stream, and the warp writes the segment's words from there, each
// from two neighbouring ones by a shift that is the segment's.  A word may need the row after the warp's last, so a warp
// writes 31 rows' words from the 32 it encodes.  Bound by the encode, like the entries'.  23 M elements off the boundary, two
// workers, four bits, max pass and encode 66 us (61 on it), bf16 51 (49), against 100 and 97 us with encode_table_kernel, which
// copies four and two bytes at a time and draws a fifth block per row.
struct FlatEntry {
    const void* base;        // the gradient's row in which the segment starts
    uint32_t* codes;         // the segment's first code word
    float* scale;            // its scale, final when the encode pass starts
    uint64_t n;              // elements
    uint64_t bytes;          // from `base` to the gradient's end
    uint32_t pad;            // elements of that row before the segment
    uint32_t rows;           // rows the segment touches
    uint32_t tile0;          // its first tile's number in the launch's sequence
    uint32_t blk0_lo;        // low half of the Philox block index of the row's first element
    PhiloxHead head;         // launch-wide part of its blocks (worker, high half of the block index)
};

template <int CAP>
struct FlatTable {
    CUtensorMap map[CAP];
    FlatEntry e[CAP];
    uint32_t tile_end[CAP];              // one past each entry's last tile; 2^32 - 1 beyond the last entry
    uint32_t tiles;
    uint32_t poll_limit, arm_only;       // as in QuantizeArgs
    RoundKeys rk;
};
constexpr uint32_t kFlatWarps = 4, kFlatWarpRows = 31, kFlatTileRows = kFlatWarps * kFlatWarpRows;

template <int BITS, int DTYPE, int CAP>
__global__ void __launch_bounds__(32 * kFlatWarps, 4)
encode_flat_kernel(const __grid_constant__ FlatTable<CAP> T, unsigned int* __restrict__ timeouts)
{
    constexpr uint32_t kStages = 2, kBoxRows = 128, kTileBytes = kBoxRows * 128;
    constexpr int kHalves = DTYPE == 0 ? 1 : 2, kElems = 32 * kHalves, kWords = BITS * kHalves;
    struct Shared {
        alignas(1024) uint8_t stage[kStages][kTileBytes];
        alignas(16) uint32_t out[kFlatWarps][32 * kWords];
        alignas(8) uint64_t bar[kStages];
        uint32_t read[kStages];        // warps that have read the stage, over all its uses
    };
    __shared__ Shared sh;
    const uint32_t t = threadIdx.x, lane = t & 31u, wid = t >> 5;
    const uint32_t step = gridDim.x;
    if (t == 0) {
        for (uint32_t s = 0; s < kStages; ++s) { mbar_init(smem_u32(&sh.bar[s]), 1); sh.read[s] = 0u; }
        fence_barrier_init();
    }
    __syncthreads();
    grid_dependency_wait();            // nothing above touches global memory

    uint32_t u = blockIdx.x, fill = u;             // the tile in work, the next one to fetch
    uint32_t fe = 0;                               // the entry of `fill`: searched once, then only moved forward
#pragma unroll
    for (uint32_t half = CAP / 2; half > 0; half >>= 1)
        if (u >= T.tile_end[fe + half - 1]) fe += half;
    if (u >= T.tiles) fe = 0;
    uint32_t e = fe;
    auto fetch = [&](uint32_t s, bool mine) {
        if (fill < T.tiles) {
            while (fill >= T.tile_end[fe]) ++fe;
            if (mine) {
                const uint32_t bar = smem_u32(&sh.bar[s]);
                mbar_expect_tx(bar, kTileBytes);
                if (!T.arm_only)
                    tma_load_2d(smem_u32(sh.stage[s]), &T.map[fe], 0, (int)((fill - T.e[fe].tile0) * kFlatTileRows), bar);
            }
        }
        fill += step;
    };
    for (uint32_t s = 0; s < kStages; ++s) fetch(s, t == 0);

    uint32_t k = 0, end = 0, tile0 = 0, blk0 = 0, rows = 0, rows_full = 0, pad = 0, off = 0, shift = 0;
    uint64_t words = 0, last = 0;                  // the segment's words; one past its last element, from `base`
    uint32_t* codes = nullptr;
    bool ok = true;
    PhiloxHead head = {};
    EncodeScale es = {0.0f, 0.0f};
#pragma unroll 1
    for (; u < T.tiles; u += step, ++k) {
        if (u >= end) {
            while (u >= T.tile_end[e]) ++e;
            const FlatEntry& x = T.e[e];
            end = T.tile_end[e]; tile0 = x.tile0; blk0 = x.blk0_lo; head = x.head; codes = x.codes;
            rows = x.rows; rows_full = (uint32_t)(x.bytes >> 7 < rows ? x.bytes >> 7 : rows); pad = x.pad;
            off = (pad * BITS) >> 5; shift = (pad * BITS) & 31u;
            words = (x.n * BITS + 31) / 32; last = pad + x.n;
            es = encode_scale<BITS>(__ldcg(x.scale));
        }
        const uint32_t s = k % kStages, at = wid * kFlatWarpRows + lane;         // the row's place in the stage
        const uint32_t row0 = (u - tile0) * kFlatTileRows + wid * kFlatWarpRows, row = row0 + lane;
        uint8_t* stage = sh.stage[s];
        const uint32_t bar = smem_u32(&sh.bar[s]);
        uint32_t h[16];
        draw_row_blocks_head(blk0 + 4u * kHalves * row, head, T.rk, h);
        ok = mbar_try_wait(bar, (k / kStages) & 1);
        if (!ok) ok = mbar_wait(bar, (k / kStages) & 1, T.poll_limit);
        if (!__all_sync(0xFFFFFFFFu, ok)) { ok = false; break; }
        if (row < rows && row >= rows_full)        // as in encode_entries_kernel (two warps may share it: both put the same there)
            stage_ragged_row(stage, at, static_cast<const uint8_t*>(T.e[e].base), row, T.e[e].bytes);

        uint4 v[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] = reinterpret_cast<const uint4*>(stage)[swz((int)at, i)];
        __syncwarp();                      // every lane has read the stage
        bool refill = false;
        if (lane == 0) {
            __threadfence_block();
            refill = (atomicAdd(&sh.read[s], 1u) & (kFlatWarps - 1)) == kFlatWarps - 1;
            if (refill) __threadfence_block();
        }
        fetch(s, refill);

        // what lies beside the segment in its first and last row is another's, and no value of this scale
        const uint32_t* raw = reinterpret_cast<const uint32_t*>(v);
        const uint64_t first_elem = (uint64_t)row * kElems;
        const bool edge = row == 0 || row + 1 >= rows;
        uint32_t w[kWords];
#pragma unroll
        for (int half = 0; half < kHalves; ++half) {
            float x[32];
            if constexpr (DTYPE == 0) {
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j] = __uint_as_float(raw[j]);
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j) { x[2 * j] = bf16_lo(raw[16 * half + j]); x[2 * j + 1] = bf16_hi(raw[16 * half + j]); }
            }
            if (edge) {
#pragma unroll
                for (int j = 0; j < 32; ++j) {
                    const uint64_t i = first_elem + 32 * half + j;
                    x[j] = i >= pad && i < last ? x[j] : 0.0f;
                }
            }
            if (half != 0) draw_row_blocks_head(blk0 + 4u * (kHalves * row + half), head, T.rk, h);
            uint32_t wh[BITS];
            encode_pack_row_best<BITS>(x, es, h, wh);
#pragma unroll
            for (int j = 0; j < BITS; ++j) w[half * BITS + j] = wh[j];
        }
        if (row + 1 >= rows) {             // nothing beyond the segment's last code
            const uint64_t left = last > first_elem ? last - first_elem : 0;
            mask_row_words<kWords>(w, (int)(left < (uint64_t)kElems ? left : (uint64_t)kElems) * BITS);
        }
        uint32_t* out = sh.out[wid];
        store_row_words<kWords>(out, lane * kWords, w);
        __syncwarp();
#pragma unroll
        for (int i0 = 0; i0 < kWords; ++i0) {
            const uint32_t i = 32u * i0 + lane;
            const int64_t m = (int64_t)((uint64_t)row0 * kWords + i) - off;
            if (i < kFlatWarpRows * kWords && m >= 0 && m < (int64_t)words) codes[m] = __funnelshift_r(out[i], out[i + 1], shift);
        }
        __syncwarp();                      // every lane has read the words
    }
    if (!ok && lane == 0) {                // as in encode_entries_kernel
        atomicAdd(timeouts, 1u);
        for (uint32_t j = k; j < k + kStages && u < T.tiles; ++j, u += step)
            mbar_wait(smem_u32(&sh.bar[j % kStages]), (j / kStages) & 1, T.poll_limit);
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
    uint32_t pad;            // flat entries: elements of `grad`'s row before the segment,
    uint64_t bytes;          // and bytes from `grad` to the gradient's end
};

template <int BITS, int DTYPE, int CAP>
auto entries_kernel(const SegEntryTable<CAP>&) { return encode_entries_kernel<BITS, DTYPE, CAP>; }
template <int BITS, int DTYPE, int CAP>
auto entries_kernel(const FlatTable<CAP>&) { return encode_flat_kernel<BITS, DTYPE, CAP>; }

template <int BITS, int DTYPE, int CAP, template <int> class Table>
cudaError_t launch_entries_inst(const Table<CAP>& tab, unsigned int* timeouts, cudaStream_t stream)
{
    auto kernel = entries_kernel<BITS, DTYPE, CAP>(tab);
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
    if (grid > tab.tiles) grid = tab.tiles;
    return launch_pdl(kernel, grid, 128, stream, tab, timeouts);
}

template <int CAP, template <int> class Table>
cudaError_t launch_table(Table<CAP>& tab, int nent, uint64_t tiles, int bits, const RoundKeys& rk, int dtype,
                         cudaStream_t stream)
{
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    const WaitPolicy policy = wait_policy();
    tab.poll_limit = policy.poll_limit;
    tab.arm_only = policy.arm_only;
    tab.rk = rk;
    for (int i = nent; i < CAP; ++i) tab.tile_end[i] = 0xFFFFFFFFu;
    tab.tiles = (uint32_t)tiles;
    switch (bits) {
#define MQG_ENT_CASE(B) \
        case B: return dtype == 0 ? launch_entries_inst<B, 0>(tab, timeouts, stream) \
                                  : launch_entries_inst<B, kBf16Wide>(tab, timeouts, stream)
        MQG_ENT_CASE(1); MQG_ENT_CASE(2); MQG_ENT_CASE(3); MQG_ENT_CASE(4);
        MQG_ENT_CASE(5); MQG_ENT_CASE(6); MQG_ENT_CASE(7); MQG_ENT_CASE(8);
#undef MQG_ENT_CASE
    }
    return cudaErrorInvalidValue;
}

template <int CAP>
cudaError_t launch_entries(const EntryHost* entries, int nent, int bits, const RoundKeys& rk, int dtype,
                           cudaStream_t stream)
{
    SegEntryTable<CAP> tab;
    const uint32_t row_elems = dtype == 0 ? 32 : 64;
    uint64_t tiles = 0;
    for (int i = 0; i < nent; ++i) {
        const EntryHost& h = entries[i];
        SegEntry& e = tab.e[i];
        const char* why = nullptr;
        if (!encode_rows_map(&tab.map[i], h.grad, h.n / row_elems, dtype == 0 ? 4 : 2, row_elems, 128, &why))
            return cudaErrorNotSupported;
        e.grad = h.grad; e.codes = h.codes; e.scale = h.scale; e.n = h.n;
        e.tile0 = (uint32_t)tiles;
        tiles += (h.n + 128 * row_elems - 1) / (128 * row_elems);
        if (tiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
        tab.tile_end[i] = (uint32_t)tiles;
        const uint64_t blk0 = h.elem_offset >> 3;
        e.blk0_lo = (uint32_t)blk0;
        e.head = philox_head((uint32_t)(blk0 >> 32), h.worker, rk.k0[0]);
    }
    return launch_table(tab, nent, tiles, bits, rk, dtype, stream);
}

template <int CAP>
cudaError_t launch_flat(const EntryHost* entries, int nent, int bits, const RoundKeys& rk, int dtype, cudaStream_t stream)
{
    FlatTable<CAP> tab;
    const uint32_t row_elems = dtype == 0 ? 32 : 64;
    uint64_t tiles = 0;
    for (int i = 0; i < nent; ++i) {
        const EntryHost& h = entries[i];
        FlatEntry& e = tab.e[i];
        const uint64_t rows = (h.pad + h.n + row_elems - 1) / row_elems, whole = h.bytes / 128;
        const char* why = nullptr;
        if (!encode_rows_map(&tab.map[i], h.grad, rows < whole ? rows : whole, dtype == 0 ? 4 : 2, row_elems, 128, &why))
            return cudaErrorNotSupported;
        e.base = h.grad; e.codes = h.codes; e.scale = h.scale; e.n = h.n; e.bytes = h.bytes; e.pad = h.pad;
        e.rows = (uint32_t)rows;
        e.tile0 = (uint32_t)tiles;
        tiles += (rows + kFlatTileRows - 1) / kFlatTileRows;
        if (tiles > 0x7FFFFFFFull / kFlatTileRows) return cudaErrorInvalidValue;
        tab.tile_end[i] = (uint32_t)tiles;
        const uint64_t blk0 = h.elem_offset >> 3;
        e.blk0_lo = (uint32_t)blk0;
        e.head = philox_head((uint32_t)(blk0 >> 32), h.worker, rk.k0[0]);
    }
    return launch_table(tab, nent, tiles, bits, rk, dtype, stream);
}

// Whether the segments of a call may be encoded by rows of the whole gradient: rows that start on 16-byte boundaries and on
// blocks of draws, nothing read before the first segment, and one high half of the blocks' indexes.
bool flat_applies(const void* const* grads, int W, uint64_t begin, uint64_t end, uint64_t elem_offset)
{
    for (int w = 0; w < W; ++w)
        if ((reinterpret_cast<uintptr_t>(grads[w]) & 15u) != 0) return false;
    const uint64_t first = elem_offset >> 3, last = (elem_offset + end + 63) >> 3;
    return begin % 64 == 0 && elem_offset % 8 == 0 && first >> 32 == last >> 32 && (end + 31) / 32 <= 0x7FFFFFFFull;
}

// Whether a call's segments, none longer than a cluster's, are quantized by launch_joined_spans and not by a launch that clears
// the scales, the max pass with the short segments beside it, and the encode; per worker: elements, those in segments of several
// CTAs and those in segments of more than five.
bool joined_spans_pay(int W, uint64_t elements, uint64_t in_joined, uint64_t in_long_joined, int dtype)
{
    const uint64_t all = elements * (uint64_t)W;
    // A long launch with next to nothing that joins gains nothing from it and loses where clusters do not fill the SMs: 63 tensors of
    // 9,000 and one of 60,000, 32 workers, 30.6 against 28.9 us (8 workers 10.5 / 13.9).
    if (all > (16u << 20) && 8 * in_joined < elements) return false;
    // bf16, whose two passes read half as much: short launches, and those of segments of up to five CTAs.  Against the three
    // launches, us: 8 of 65,000, 4 / 8 / 32 workers 5.7 / 10.6 / 29.7 against 7.2 / 8.4 / 24.0; 20 of 41,000, 4 / 8 / 32
    // workers 9.7 / 15.0 / 50.1 against 9.8 / 14.7 / 47.6; 20 of 33,000, 4 / 8 / 32 workers 6.3 / 11.2 / 39.1 against 9.6 / 14.2 /
    // 44.9; 63 of 17,000 and one of 60,000, 8 workers 23.9 against 30.7.
    // fp32: 40 of 60,000, 1 / 8 / 32 workers 6.0 / 33.3 / 132 against 8.5 / 41.4 / 181; 20 of 33,000, 1 / 8 / 32 workers 4.0 / 10.5 /
    // 38.3 against 5.6 / 13.8 / 47.4.  (Parts of 512 and 1024 rows, for tensors of up to 262,144 elements, one worker: 4.9 and 6.8
    // against 5.1 for 100,000 and 200,000.)
    return dtype == 0 || all <= (3u << 20) || 3 * in_long_joined <= elements;
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
    uint64_t long_tiles = 0, longest = 0;             // tiles of 256 rows
    uint64_t in_joined = 0, in_long_joined = 0;       // elements of the segments of several CTAs, of more than five
    bool any_span = false, aligned = true;            // aligned: the long segments, as the gradients are
    for (int j = 0; j < nseg; ++j) {
        const uint64_t len = seg_off[j + 1] - seg_off[j];
        if (len > longest) longest = len;
        if (len <= kSegmentSpanElems) { any_span = true; continue; }
        in_joined += len;
        if (len > 5 * kJoinedChunk) in_long_joined += len;
        long_tiles += (len + kMaxTileRows * 32 - 1) / (kMaxTileRows * 32);
        aligned = aligned && (seg_off[j] * esz) % 16 == 0;
    }
    // Nothing longer than a cluster's: one launch for every 64 segments instead of three launches, where that pays.
    if (longest > kSegmentSpanElems && longest <= kMaxJoinedElems &&
        (workspace || joined_spans_pay(W, seg_off[nseg] - seg_off[0], in_joined, in_long_joined, dtype))) {
        for (int first = 0; first < nseg; first += kMaxSegmentsPerLaunch) {
            SpanTable spans;
            memset(&spans, 0, sizeof(spans));
            spans.first = first;
            uint64_t parts = 0;
            for (int j = first; j < nseg && j < first + kMaxSegmentsPerLaunch; ++j) {
                const int k = spans.nspan++;
                spans.elem0[k] = seg_off[j]; spans.len[k] = seg_off[j + 1] - seg_off[j]; spans.code0[k] = code_off[j];
                spans.scale_idx[k] = (uint32_t)j;
                parts += (spans.len[k] + kJoinedChunk - 1) / kJoinedChunk;
            }
            // A CTA of two rows per thread for those it holds (20 tensors of 12,000 and one of 20,000, 16 workers 6.6 against 9.7
            // us), unless the launch has at most two CTAs of one row per thread per SM (8,192 to 16,384 elements, 40 of 16,000, one
            // worker 3.9 against 4.3 us; 32 of 9,000 and 32 of 33,000 5.0 against 6.0).
            const cudaError_t err = launch_joined_spans(a, spans, parts * (uint64_t)W <= 2 * 148 ? kJoinedChunk : kSegmentSpanElems,
                                                        workspace ? kSpanNorm : kSpanMaxAbs, bits, dtype, stream);
            if (err != cudaSuccess) return err;
        }
        return cudaSuccess;
    }
    const bool together = !workspace && any_span && long_tiles != 0 &&
                          spans_join_max_pass(long_tiles * (uint64_t)W, dtype, aligned);
    cudaError_t err = together ? launch_clear_scales(a, nseg, stream) : cudaSuccess;
    if (err != cudaSuccess) return err;
    const bool flat = flat_applies(grads, W, seg_off[0], seg_off[nseg], elem_offset);
    bool any_entries = false, any_flat = false;
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
                if (!workspace && !together) spans.clear[i >> 5] |= 1u << (i & 31);
                const uint64_t nt = (len + kMaxTileRows * 32 - 1) / (kMaxTileRows * 32);
                tiles += nt;
                if (bulk(j)) any_entries = true;
                else if (flat) any_flat = true;
                else plain_tiles += nt;
            }
            if (tiles > 0x3FFFFFFFull) return cudaErrorInvalidValue;
        }
        longs.tile_start[count] = (uint32_t)tiles;
        plain.tile_start[count] = (uint32_t)plain_tiles;
        longs.seg_off[count] = plain.seg_off[count] = seg_off[first + count];
        const bool one_launch = together && spans.nspan != 0 && tiles != 0;
        if (one_launch) {
            err = launch_spans_absmax(a, spans, most, longs, bits, dtype, stream);
            if (err != cudaSuccess) return err;
        } else if (spans.nspan != 0 || (tiles != 0 && !workspace && !together)) {
            err = launch_spans(a, spans, spans.nspan != 0 ? (unsigned)spans.nspan : 1u, most,
                               workspace ? kSpanNorm : kSpanMaxAbs, bits, dtype, stream);
            if (err != cudaSuccess) return err;
        }
        if (tiles == 0) continue;
        TableArgs t = a;                              // a table numbers its segments from 0
        for (int w = 0; w < W; ++w) t.scales[w] += first;
        err = workspace ? launch_segments_l2_scales(grads[0], longs, t.scales[0], dtype, workspace + sums, stream)
            : one_launch ? cudaSuccess : launch_absmax_table(t, longs, dtype, stream);
        sums += tiles;
        if (err == cudaSuccess) err = launch_encode_table(t, plain, bits, dtype, stream);
        if (err != cudaSuccess) return err;
    }
    // no heap here: the C ABI throws nothing
    EntryHost batch[kMaxEntries];
    for (int pass = any_entries ? 0 : 1; pass < (any_flat ? 2 : 1) && err == cudaSuccess; ++pass) {
        int n = 0;
        auto launch = [&] {
            if (pass == 0)
                err = n <= kFewEntries ? launch_entries<kFewEntries>(batch, n, bits, a.rk, dtype, stream)
                                       : launch_entries<kMaxEntries>(batch, n, bits, a.rk, dtype, stream);
            else
                err = n <= kFewEntries ? launch_flat<kFewEntries>(batch, n, bits, a.rk, dtype, stream)
                                       : launch_flat<kMaxEntries>(batch, n, bits, a.rk, dtype, stream);
            n = 0;
        };
        for (int j = 0; j < nseg && err == cudaSuccess; ++j) {
            const uint64_t len = seg_off[j + 1] - seg_off[j];
            if (len <= kSegmentSpanElems || bulk(j) != (pass == 0)) continue;
            const uint32_t pad = pass == 0 ? 0u : (uint32_t)(seg_off[j] % (dtype == 0 ? 32 : 64));
            const uint64_t from = seg_off[j] - pad;
            for (int w = 0; w < W && err == cudaSuccess; ++w) {
                batch[n++] = {static_cast<const char*>(grads[w]) + from * esz, codes[w] + code_off[j], scales[w] + j, len,
                              elem_offset + from, first_worker + (uint32_t)w, pad, (seg_off[nseg] - from) * esz};
                if (n == kMaxEntries) launch();
            }
        }
        if (n != 0 && err == cudaSuccess) launch();
    }
    return err;
}

}  // namespace mqg
