// Fused server pass (the fast path of mqg_server_step for uniform buckets of at least 1024 elements,
// of 512, 768, 896, 960 or 992, and - for few workers - of 32 to 256): every WARP is an independent
// pipeline over a contiguous range of 32-row tiles.  Nothing is loaded through registers:
//   * a tile's 32 x 32 parameters arrive by a tiled bulk copy (TMA) into the warp's own swizzled
//     shared-memory stage while the tile's workers are being summed, are updated in place and leave
//     by a tiled bulk store;
//   * the code words of the tile (32 rows x K words per worker, contiguous in each worker's
//     stream) arrive by 16-byte asynchronous copies, one instruction of the warp per worker (two
//     above four bits), into a two-deep ring of code stages, a group of workers per stage, issued
//     two stages ahead of their use.  (One linear bulk copy per worker, completing on an mbarrier,
//     cost about a dozen instructions of the warp per copy - the operands of a bulk copy travel
//     through the uniform datapath - and with eight of them per tile a third of the kernel's
//     instructions were overhead: 40.1 executed instructions per parameter at four bits and eight
//     workers against 31.4 without it, before sums in units of 2^40.)
// A warp therefore never waits for DRAM latency in steady state and there is no CTA-wide barrier
// anywhere.  Per-(worker, bucket) de-quantization constants are computed once per tile into the
// warp's small shared table, one tile ahead.
#include <string.h>

#include <atomic>
#include <type_traits>

#include "mqg_segments.cuh"
#include "mqg_tma.cuh"

namespace mqg {

constexpr int kSrvWarps = 4;                      // warps per CTA, each with its own pipeline
constexpr int kSrvThreads = 32 * kSrvWarps;
constexpr int kSrvTileRows = 32;                  // rows per tile = lanes per warp
constexpr uint32_t kSrvTileBytes = kSrvTileRows * 128;
constexpr int kCodeDepth = 2;                     // code stages per warp

// Workers whose code words share one code stage: at most 4 KB per stage, so that a CTA's shared
// memory (13 KB per warp) lets four CTAs = 16 warps share an SM, and a power of two, so that the
// usual worker counts fill whole stages.
template <int BITS>
struct ServerGroup { static constexpr int value = BITS <= 4 ? 8 : 4; };

// Barrier ID (1 .. 15; 0 is the one of __syncthreads) among `threads` threads of a CTA (a multiple of 32:
// whole warps); every thread that takes part names the same count.
template <int ID>
__device__ __forceinline__ void named_barrier(uint32_t threads)
{
    asm volatile("bar.sync %0, %1;" ::"n"(ID), "r"(threads) : "memory");
}

struct ServerTmaArgs {
    WorkerPtrs ptrs;
    float* params;
    uint64_t n, ncode_words;
    uint32_t nrows;              // ceil(n / 32)
    uint32_t nrows_full;         // floor(n / 32): rows the tensor map and the code copies cover
    uint32_t ntiles;             // ceil(nrows_full / 32)
    uint32_t nbuckets;
    uint32_t rows_per_bucket;    // such that a tile touches at most 1 << nbt_shift buckets
    int rpb_shift;               // log2(rows_per_bucket) if a power of two, else -1
    int nbt_shift;               // log2 of the buckets a tile can touch: 1 (two buckets), or 2..5 for
                                 // buckets of 8, 4, 2, 1 rows; W << nbt_shift <= 2 * kMaxWorkers
    int W;
    float neg_lr;
    float unit_factor;           // what a sum in units of 2^40 is multiplied with: 2^40 times -lr (MODE 1), 1 or the mean's factor
    uint32_t one;                // 1, as a run-time constant
    uint32_t bias_bits;          // 0x4B000000 (2^23), a run-time constant for the byte permutes
    uint32_t poll_limit;         // polls of one barrier wait before the warp gives up
    uint32_t arm_only;           // test hook: 1 = arm the barriers but issue no parameter copy
};

// SEGS: the launch covers several gradients ("segments" of a per-layer step, each ONE bucket with a
// scale of its own) instead of one gradient with uniform buckets.  The tiles of all segments form
// one sequence that is split over the warps as usual; a tile's segment is found with a cursor that
// only moves forward.
constexpr int kMaxSrvSegs = kMaxServerSegsPerLaunch;
struct ServerSegEntry {
    uint32_t tile_start;     // number of the segment's first tile in the launch's sequence
    uint32_t nrows_full;     // floor(n / 32): rows its tensor map and code copies cover
    uint32_t scale_idx;      // index of its scale in every worker's scale array
    uint32_t ragged;         // elements of its last, incomplete row (0 = none)
    uint32_t head, shift;    // FLAT: elements before its first row, bit of code_word0 at which that row's codes start
    uint64_t code_word0;     // word offset of its first row's codes in every worker's code buffer
    uint64_t words0, words_end;          // its bit stream there
    uint64_t elem0;          // offset of its first element in a.params
};
struct ServerSegTable {
    CUtensorMap map[kMaxSrvSegs];
    ServerSegEntry e[kMaxSrvSegs + 1];     // e[nseg].tile_start = tiles of the launch
    int nseg;
};

// Where a tile lives: the tensor map of its gradient, its first row there, the rows the map covers,
// the word offset of the gradient's bit stream and (SEGS) the index of its scale.
struct TileLoc {
    const CUtensorMap* map;
    uint32_t row0, nrows_full, scale_idx;
    uint32_t shift;                              // FLAT, and the end of the bit stream
    uint64_t code_word0, words_end;
};

template <bool SEGS>
__device__ __forceinline__ TileLoc locate_srv_tile(const CUtensorMap* map_full, const ServerTmaArgs& a,
                                                   const ServerSegTable* segs, uint32_t tile, uint32_t& cursor)
{
    TileLoc t;
    if constexpr (SEGS) {
        while (tile >= segs->e[cursor + 1].tile_start) ++cursor;
        const ServerSegEntry& e = segs->e[cursor];
        t.map = &segs->map[cursor];
        t.row0 = (tile - e.tile_start) * kSrvTileRows;
        t.nrows_full = e.nrows_full;
        t.scale_idx = e.scale_idx;
        t.shift = e.shift;
        t.code_word0 = e.code_word0;
        t.words_end = e.words_end;
    } else {
        t.map = map_full;
        t.row0 = tile * kSrvTileRows;
        t.nrows_full = a.nrows_full;
        t.scale_idx = t.shift = 0;
        t.code_word0 = t.words_end = 0;
    }
    return t;
}

// FLAT: the segments of the launch may start anywhere.  Their rows are rows of the whole parameter buffer, so the
// parameters travel as ever; a row's codes then start at any bit, the same one for all rows of a segment.  A tile's
// words are copied one by one, each worker's and the one behind them, so that they lie in the stage as ever, and a lane shifts
// its K + 1 words into place.
template <int BITS, bool FLAT>
__host__ __device__ constexpr uint32_t stage_words() { return kSrvTileRows * BITS + (FLAT ? 4 : 0); }      // of one worker

// Dynamic shared memory of one CTA (base rounded up to 1024 bytes for the 128-byte swizzle).
template <int BITS, bool FLAT>
struct ServerSmem {
    alignas(1024) uint8_t stage[kSrvWarps][kSrvTileBytes];      // one parameter tile per warp
    alignas(16) uint32_t code[kSrvWarps][kCodeDepth][ServerGroup<BITS>::value][stage_words<BITS, FLAT>()];
    float4 table[kSrvWarps][2 * kMaxWorkers];     // (2h, 2h, -h, -h) per (worker, bucket of the tile): entry
                                                  // (worker << nbt_shift) + bucket-of-tile
    uint64_t bar[kSrvWarps];                      // parameter tile landed
};

__device__ __forceinline__ uint32_t bucket_of_row(const ServerTmaArgs& a, uint32_t row)
{
    return a.rpb_shift >= 0 ? row >> a.rpb_shift : row / a.rows_per_bucket;
}

// Scales of the (worker, bucket) pairs of the tile that starts at row0: lane l holds pair l and,
// when there are more than 32 pairs (`wide`), pair l + 32 (pair = (worker << nbt_shift) +
// bucket-of-tile).  RANGE: the pair's (lo, hi) instead of its scale (the `scales` pointers then
// address arrays of two floats per bucket).
template <bool RANGE, bool SEGS>
__device__ __forceinline__ void load_tile_scales(const ServerTmaArgs& a, const TileLoc& loc, uint32_t lane,
                                                 bool wide, float2 (&s)[2])
{
    // SEGS: the tile lies in one bucket, the segment's (nbt_shift = 0: pair = worker)
    const uint32_t first = SEGS ? loc.scale_idx : bucket_of_row(a, loc.row0);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !wide) break;
        const uint32_t pair = lane + 32u * h, w = pair >> a.nbt_shift;
        const uint32_t b = first + (pair & ((1u << a.nbt_shift) - 1u));
        const bool have = w < (uint32_t)a.W && (SEGS || b < a.nbuckets);
        if (RANGE) s[h] = have ? __ldg(reinterpret_cast<const float2*>(a.ptrs.scales[w]) + b) : make_float2(0.0f, 0.0f);
        else s[h] = make_float2(have ? __ldg(a.ptrs.scales[w] + b) : 0.0f, 0.0f);
    }
}

// Returns (for the whole warp) whether the entries are those of a sum in units of 2^40 (UNIT: where such a sum may be).
template <int BITS, bool RANGE, bool UNIT>
__device__ __forceinline__ bool store_tile_scales(const ServerTmaArgs& a, float4* table, uint32_t lane,
                                                  bool wide, const float2 (&s)[2])
{
    if constexpr (!UNIT) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h == 1 && !wide) break;
            const uint32_t pair = lane + 32u * h, w = pair >> a.nbt_shift;
            if (w < (uint32_t)a.W) {
                const DecodeScale d = RANGE ? range_decode_scale<BITS>(s[h].x, s[h].y) : decode_scale<BITS>(s[h].x);
                table[pair] = make_float4(d.two_h, d.two_h, d.minus_h, d.minus_h);
            }
        }
        return false;
    }
    DecodeScale d[2];
    bool fits = true;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !wide) break;
        // a pair beyond the last worker has the scale 0 and is not stored
        d[h] = RANGE ? range_decode_scale<BITS>(s[h].x, s[h].y) : decode_scale<BITS>(s[h].x);
        fits = fits && unit_decode_applies(d[h], RANGE);
    }
    fits = __all_sync(0xFFFFFFFFu, fits);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        if (h == 1 && !wide) break;
        const uint32_t pair = lane + 32u * h, w = pair >> a.nbt_shift;
        if (w < (uint32_t)a.W)
            table[pair] = fits ? unit_decode_entry<BITS, RANGE>(d[h])
                                       : make_float4(d[h].two_h, d[h].two_h, d[h].minus_h, d[h].minus_h);
    }
    return fits;
}

// A lane's K words of one worker from a code stage, with the widest shared-memory access the
// lane's offset (lane * K words) allows.
template <int BITS>
__device__ __forceinline__ void read_stage_words(const uint32_t* __restrict__ stage_row, uint32_t (&w)[BITS])
{
    if constexpr (BITS % 4 == 0) {
        const uint4* p = reinterpret_cast<const uint4*>(stage_row);
#pragma unroll
        for (int k = 0; k < BITS / 4; ++k) {
            const uint4 v = p[k];
            w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
        }
    } else if constexpr (BITS % 2 == 0) {
        const uint2* p = reinterpret_cast<const uint2*>(stage_row);
#pragma unroll
        for (int k = 0; k < BITS / 2; ++k) {
            const uint2 v = p[k];
            w[2 * k] = v.x; w[2 * k + 1] = v.y;
        }
    } else {
#pragma unroll
        for (int k = 0; k < BITS; ++k) w[k] = stage_row[k];
    }
}

// 16-byte asynchronous copy that reads only the first `src_bytes` bytes of the source and fills the
// rest of the 16 bytes with zeros.
__device__ __forceinline__ void cp_async16_partial(uint32_t smem_dst, const void* gmem_src, uint32_t src_bytes)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gmem_src), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async16_to(uint32_t smem_dst, const void* gmem_src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait_group() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// Starts the copies of one code stage: the words of rows [row0, row0 + 32) (fewer in the last tile
// of the gradient) of workers g0 .. g0 + group - 1 (those that exist).  A worker's words of these
// rows are contiguous in its stream and start on a 16-byte boundary (row0 is a multiple of 32):
// (and so does the bit stream of a segment that takes part in a SEGS launch): the warp copies them in 16-byte pieces, lane l the l-th piece (and the (l + 32)-th for more than
// four bits), asynchronously and without passing through registers.  The piece that holds the end
// of a short last tile is copied up to that end and zero-filled.  `lane_off` = 16 * lane.
// TO_END: the gradient's last, ragged row takes part too; its words end where the stream does.
template <int BITS, bool TO_END = false>
__device__ __forceinline__ void fill_code_stage(const ServerTmaArgs& a, uint32_t stage, const TileLoc& loc, int g0,
                                                uint32_t lane_off)
{
    constexpr int kGroup = ServerGroup<BITS>::value;
    constexpr uint32_t kWorkerBytes = kSrvTileRows * BITS * 4;
    constexpr int kPieces = (int)((kWorkerBytes / 16 + 31) / 32);       // pieces per lane: 1 or 2
    const uint32_t rows_here = TO_END && loc.row0 >= loc.nrows_full ? 0u
                                                                    : min((uint32_t)kSrvTileRows, loc.nrows_full - loc.row0);
    const uint64_t byte0 = (loc.code_word0 + (uint64_t)loc.row0 * BITS) * 4 + lane_off;
    if (rows_here == (uint32_t)kSrvTileRows && g0 + kGroup <= a.W) {
#pragma unroll
        for (int pc = 0; pc < kPieces; ++pc) {
            if (lane_off + 512u * pc < kWorkerBytes) {
#pragma unroll
                for (int i = 0; i < kGroup; ++i)
                    cp_async16_to(stage + i * kWorkerBytes + lane_off + 512u * pc,
                                  reinterpret_cast<const uint8_t*>(a.ptrs.codes[g0 + i]) + byte0 + 512u * pc);
            }
        }
    } else {
        uint32_t bytes_here = rows_here * BITS * 4;
        if (TO_END && rows_here < (uint32_t)kSrvTileRows)
            bytes_here = (uint32_t)(a.ncode_words - (uint64_t)loc.row0 * BITS) * 4;
        const int nwk = min(kGroup, a.W - g0);
#pragma unroll
        for (int pc = 0; pc < kPieces; ++pc) {
            const uint32_t off = lane_off + 512u * pc;
            if (off < bytes_here) {
                const uint32_t nb = min(16u, bytes_here - off);
                for (int i = 0; i < nwk; ++i)
                    cp_async16_partial(stage + i * kWorkerBytes + off,
                                       reinterpret_cast<const uint8_t*>(a.ptrs.codes[g0 + i]) + byte0 + 512u * pc, nb);
            }
        }
    }
}

template <int BITS>
__device__ __forceinline__ void fill_code_stage_flat(const ServerTmaArgs& a, uint32_t stage, const TileLoc& loc, int g0,
                                                     uint32_t lane)
{
    constexpr int kGroup = ServerGroup<BITS>::value;
    constexpr uint32_t kBytes = stage_words<BITS, true>() * 4, kWords = kSrvTileRows * BITS;
    const uint64_t word0 = loc.code_word0 + (uint64_t)loc.row0 * BITS;
    const int nwk = min(kGroup, a.W - g0);
    auto copy = [&](uint32_t to, const uint32_t* from, bool in) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to), "l"(from), "r"(in ? 4u : 0u) : "memory");
    };
    if (word0 + kWords + 1 <= loc.words_end && nwk == kGroup) {
#pragma unroll
        for (int i = 0; i < kGroup; ++i) {
            const uint32_t* from = a.ptrs.codes[g0 + i] + word0 + lane;
#pragma unroll
            for (int k = 0; k < BITS; ++k) copy(stage + i * kBytes + (32 * k + lane) * 4, from + 32 * k, true);
            if (lane == 0) copy(stage + i * kBytes + kWords * 4, from + kWords, true);
        }
    } else {
        for (int i = 0; i < nwk; ++i)
            for (uint32_t k = lane; k < kWords + 1; k += 32) {       // words past the stream's end are zeros
                const bool in = word0 + k < loc.words_end;
                copy(stage + i * kBytes + k * 4, a.ptrs.codes[g0 + i] + (in ? word0 + k : 0), in);
            }
    }
}

// CTAs per SM the register budget is set for (what the shared memory allows at three bits and more;
// five CTAs of 96 registers at one and two bits measured 0.3 us slower per launch than four).
template <int BITS>
constexpr int server_min_ctas() { return 4; }

// The one row of a gradient that has fewer than 32 elements (row `row`, the last one): a warp, lane j on
// element j, with plain loads and stores.  What bounds it is one round trip to memory and the chain of the sum: the code
// words of eight workers are requested at a time, and lane w divides for worker w (at most 32).  131,073 parameters, 1 / 8 / 16
// workers: 2.4 / 3.2 / 4.2 us, against 3.1 / 4.7 / 7.0 us with a division per worker and element, after the warp's tile.
// `params` is the row's first parameter, `count` its length; its codes start at bit `bit0` of word `word0` of every worker's
// buffer, and their stream ends before word `words_end`; `bucket` is the index of the row's scale.
// MODE and RANGE as in server_tma_body.  SEGS: every lane divides for every worker.  (With the shuffles in a function that a grid over segments calls, its main loop
// is compiled to something 2.5 % slower at four bits and eight workers.)
template <int BITS, int MODE, bool RANGE, bool SEGS>
__device__ __noinline__ void server_ragged_row(const ServerTmaArgs& a, float* params, uint32_t count, uint64_t word0,
                                               uint32_t bit0, uint64_t words_end, uint32_t bucket, uint32_t lane)
{
    static_assert(kMaxWorkers <= 32, "a lane per worker");
    const bool in = lane < count;                // the others keep going: the shuffles need them
    if (SEGS && !in) return;
    const uint32_t bit = bit0 + lane * BITS, shift = bit & 31u;
    const uint64_t at = word0 + (bit >> 5), word = at < words_end ? at : words_end - 1;
    const bool two = shift + BITS > 32 && word + 1 < words_end;
    const float old = MODE != 0 && in ? params[lane] : 0.0f;
    auto load_scale = [&](int w) {
        return RANGE ? __ldg(reinterpret_cast<const float2*>(a.ptrs.scales[w]) + bucket)
                     : make_float2(__ldg(a.ptrs.scales[w] + bucket), 0.0f);
    };
    auto constants = [](float2 s) { return RANGE ? range_decode_scale<BITS>(s.x, s.y) : decode_scale<BITS>(s.x); };
    DecodeScale mine = {0.0f, 0.0f};
    float2 v = make_float2(MODE == 2 ? sum_start<BITS, RANGE>(old) : 0.0f, 0.0f);
    constexpr int kBatch = 8;
#pragma unroll 1
    for (int w0 = 0; w0 < a.W; w0 += kBatch) {
        uint32_t lo[kBatch], hi[kBatch];
        float2 sc[SEGS ? kBatch : 1];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (w0 + i >= a.W) break;
            lo[i] = __ldg(a.ptrs.codes[w0 + i] + word);
            hi[i] = two ? __ldg(a.ptrs.codes[w0 + i] + word + 1) : 0u;
            if (SEGS) sc[SEGS ? i : 0] = load_scale(w0 + i);
        }
        if (!SEGS && w0 == 0) mine = constants(load_scale(min((int)lane, a.W - 1)));
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (w0 + i >= a.W) break;
            DecodeScale d;
            if (SEGS) {
                d = constants(sc[SEGS ? i : 0]);
            } else {
                d.two_h = __shfl_sync(0xFFFFFFFFu, mine.two_h, w0 + i);
                d.minus_h = __shfl_sync(0xFFFFFFFFu, mine.minus_h, w0 + i);
            }
            const uint32_t q = __funnelshift_r(lo[i], hi[i], shift) & ((1u << BITS) - 1u);
            if constexpr (BITS == 1 && !RANGE)
                v.x = __fadd_rn(v.x, one_bit_value(d.minus_h, q << 31));
            else
                v = accumulate2<BITS, RANGE>(v, make_float2(__uint_as_float(q | 0x4B000000u), 8388608.0f),
                                             make_float2(d.two_h, d.two_h), make_float2(d.minus_h, d.minus_h));
        }
    }
    if (in) params[lane] = MODE == 1 ? __fmaf_rn(a.neg_lr, v.x, old) : v.x;
}

// MODE 1: dst = params, dst <- fma(-lr, sum, dst).  MODE 0: dst = acc, dst <- sum.
// MODE 2: dst = acc, the sum continues from the value already there.
// RANGE: the (min, max) nearest-rounding variant (x^ = fma(q, step, lo)).
template <int BITS, int MODE, bool RANGE, bool SEGS, bool kUnit, bool FLAT = false>
__device__ __forceinline__ void server_tma_body(const CUtensorMap* map_full, const ServerTmaArgs& a,
                                                const ServerSegTable* segs, unsigned int* __restrict__ timeouts)
{
    extern __shared__ uint8_t smem_raw[];
    ServerSmem<BITS, FLAT>& sm = *reinterpret_cast<ServerSmem<BITS, FLAT>*>(
        smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u));
    constexpr int kGroup = ServerGroup<BITS>::value;
    constexpr uint32_t kWorkerWords = stage_words<BITS, FLAT>();
    const uint32_t lane = threadIdx.x & 31u;
    // the warp's number, taken from lane 0 so that the compiler knows it is the same in every lane
    const uint32_t wid = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
    uint8_t* stage = sm.stage[wid];
    float4* table = sm.table[wid];
    const uint32_t bar = smem_u32(&sm.bar[wid]);
    const uint32_t code_base = smem_u32(&sm.code[wid][0][0][0]);
    constexpr uint32_t kCodeStageBytes = kGroup * kWorkerWords * 4;

    if (lane == 0) {
        mbar_init(bar, 1);
        fence_barrier_init();
        if (!SEGS) prefetch_tensormap(map_full);
    }
    __syncwarp();
    grid_dependency_wait();            // nothing above touches global memory

    // This warp's tiles: gwarp, gwarp + nwarps, gwarp + 2 nwarps, ...  At any moment the grid then works
    // on one window of consecutive tiles, and the four warps of a CTA on four consecutive ones: their
    // requests for a worker's code words (32 K bytes per tile) fall into the same DRAM pages at about the
    // same time.  Against a contiguous range of tiles per warp, per launch at eight workers: 37.5 against
    // 39.7 us at one bit, 44.5 against 47.6 at three, 61.0 against 63.0 at eight (n = 25 M); 89 against 94,
    // 115 against 123, 143 against 147 us at n = 61 M.
    const uint32_t gwarp = blockIdx.x * kSrvWarps + wid, nwarps = gridDim.x * kSrvWarps;
    const uint32_t base = a.ntiles / nwarps, extra = a.ntiles % nwarps;
    const uint32_t t_begin = gwarp, t_step = nwarps;
    const uint32_t ntiles = base + (gwarp < extra ? 1u : 0u);
    // Three and four bits: the warps of a CTA start every tile together (a CTA barrier per tile, for the
    // `base` tiles that every warp of the grid has), which keeps those requests together for the whole
    // launch: 106 against 116 us at three bits, 121 against 127 us at four (n = 61 M; 44.3 and 46.9 against
    // 44.3 and 48.0 us at n = 25 M); no gain at one and two bits, a loss of 1 to 2 % from five bits on.
    constexpr bool kCtaSync = BITS == 3 || BITS == 4;
    const uint32_t sync_tiles = base;
    const uint32_t last_row = a.nrows_full - 1;    // nrows_full >= 1 on this path (not used by SEGS)
    uint32_t cur_e = 0, next_e = 0, fill_e = 0;    // SEGS: segment cursors of the tile in work, the next
                                                   // tile (its scales) and the tile whose codes are fetched
    const uint32_t groups = ((uint32_t)a.W + kGroup - 1) / kGroup;      // code stages per tile
    const uint32_t nunits = ntiles * groups;
    const bool wide = ((uint32_t)a.W << a.nbt_shift) > 32u;             // more than 32 table entries
    const uint32_t lane_off = lane * 16u;
    // MODE 1: the tile's parameters are requested before this worker of the tile is summed (see
    // load_params below); measured best of 1 .. 4 at eight workers, per launch of n = 25 M: 55.8 us
    // against 57.7 us at five bits, 65.2 against 68.0 us at eight, no difference up to four bits
    constexpr int kIssueAt = 4;
    const int issue_at = min(kIssueAt, a.W - 1);

    // (a long launch gains nothing from it and loses 1 % at two bits, 45.6 against 46.1 us: the parameter tiles
    // of all warps then stand in front of the codes of all warps)
    const bool params_first = ntiles < 4;

    const UnitBits<BITS, RANGE> unit_bits(a.one);
    bool unit = false;                             // the tile in work is summed in units of 2^40

    auto fill = [&](uint32_t to, const TileLoc& loc, int g0) {
        if constexpr (FLAT) fill_code_stage_flat<BITS>(a, to, loc, g0, lane);
        else fill_code_stage<BITS>(a, to, loc, g0, lane_off);
    };

    bool failed = false;
    uint32_t k = 0, u = 0;                         // tile and code stage in use
    if (ntiles > 0) {
        // with a few tiles per warp, everything the first tile needs is requested before any of it is waited for
        const TileLoc first = locate_srv_tile<SEGS>(map_full, a, segs, t_begin, next_e);
        if ((MODE == 2 || (MODE == 1 && params_first)) && lane == 0) {
            mbar_expect_tx(bar, kSrvTileBytes);
            if (!a.arm_only) tma_load_2d(smem_u32(stage), first.map, 0, (int)first.row0, bar);
        }
        float2 s0[2];
        load_tile_scales<RANGE, SEGS>(a, first, lane, wide, s0);
        // the first kCodeDepth code stages (u2 = stage number, tile u2 / groups, group u2 % groups);
        // one copy group per stage, empty when there is no such stage
#pragma unroll
        for (uint32_t u2 = 0; u2 < (uint32_t)kCodeDepth; ++u2) {
            if (u2 < nunits)
                fill(code_base + u2 * kCodeStageBytes,
                     locate_srv_tile<SEGS>(map_full, a, segs, t_begin + (u2 / groups) * t_step, fill_e),
                     (int)(u2 % groups) * kGroup);
            cp_async_commit();
        }
        unit = store_tile_scales<BITS, RANGE, kUnit>(a, table, lane, wide, s0);
        __syncwarp();
    }
    // position of the code stage kCodeDepth ahead of the one in use, kept incrementally
    uint32_t fill_tile = kCodeDepth / groups, fill_group = kCodeDepth % groups;

#pragma unroll 1
    for (; k < ntiles; ++k) {
        if constexpr (kCtaSync) {
            if (k < sync_tiles) named_barrier<1>(kSrvThreads);
        }
        const uint32_t parity = k & 1;
        const TileLoc loc = locate_srv_tile<SEGS>(map_full, a, segs, t_begin + k * t_step, cur_e);
        const uint32_t row0 = loc.row0;
        const bool have_next = k + 1 < ntiles;
        float2 s_next[2];
        TileLoc loc_next = loc;
        if (have_next) {
            loc_next = locate_srv_tile<SEGS>(map_full, a, segs, t_begin + (k + 1) * t_step, next_e);
            load_tile_scales<RANGE, SEGS>(a, loc_next, lane, wide, s_next);
        }

        // Sum of the W de-quantized rows, in worker order.  Lanes past the end of the gradient
        // (only in the very last tile) decode whatever their slot of the stage holds; they are
        // never stored.
        const uint32_t row = min(row0 + lane, last_row);
        const uint32_t lb = SEGS ? 0u : bucket_of_row(a, row) - bucket_of_row(a, row0);
        const float4* my_table = table + lb;
        float2 v2[16];
        bool ok = true;
        if constexpr (MODE == 2) {
            // the sum continues from the accumulator: its tile is needed before the first worker
            ok = mbar_try_wait(bar, parity);
            if (!ok) ok = mbar_wait(bar, parity, a.poll_limit);
            if (!__all_sync(0xFFFFFFFFu, ok)) { failed = true; break; }
            const float4* tl = reinterpret_cast<const float4*>(stage);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const float4 p = tl[swz((int)lane, c)];
                v2[2 * c] = make_float2(sum_start<BITS, RANGE>(p.x), sum_start<BITS, RANGE>(p.y));
                v2[2 * c + 1] = make_float2(sum_start<BITS, RANGE>(p.z), sum_start<BITS, RANGE>(p.w));
            }
        } else {
#pragma unroll
            for (int p = 0; p < 16; ++p) v2[p] = make_float2(0.0f, 0.0f);
        }

#pragma unroll 1
        for (uint32_t g = 0; g < groups; ++g, ++u) {
            const uint32_t cs = u % kCodeDepth;
            const uint32_t cstage_addr = code_base + cs * kCodeStageBytes;
            const uint32_t* cstage = &sm.code[wid][cs][0][0] + lane * BITS;
            cp_async_wait_group<kCodeDepth - 1>();     // this lane's pieces of the stage have landed
            __syncwarp();                              // ... and so have the other lanes'
            const int g0 = (int)g * kGroup;
            auto decode_worker = [&](int i, auto in_units) {
                uint32_t w[BITS];
                read_stage_words<BITS>(cstage + i * kWorkerWords, w);
                if constexpr (FLAT) {
                    const uint32_t behind = cstage[i * kWorkerWords + BITS];
#pragma unroll
                    for (int q = 0; q < BITS; ++q) w[q] = __funnelshift_r(w[q], q + 1 < BITS ? w[q + 1 < BITS ? q + 1 : 0] : behind, loc.shift);
                }
                const float4 e = my_table[(uint32_t)(g0 + i) << a.nbt_shift];
                if constexpr (decltype(in_units)::value) {
                    add_decoded_row_unit<BITS, RANGE>(w, e, unit_bits, v2);
                } else {
                    DecodeScale2 d;
                    d.two_h = make_float2(e.x, e.y); d.minus_h = make_float2(e.z, e.w);
                    add_decoded_row<BITS, RANGE>(w, d, v2, a.bias_bits);
                }
            };
            const std::integral_constant<bool, kUnit> units;
            // MODE 1: the parameter stage held tile k-1, whose store was committed at the end of the last
            // iteration: once that store has read its source the stage takes tile k, which is not
            // needed before the last worker is summed.  The load starts when half of eight workers are
            // summed, by when the store has long read the stage.  The gradient's last tile may be short: the
            // box is clipped by the tensor's bounds and the rows beyond arrive as zeros, still counted
            // in the bytes.
            auto load_params = [&]() {
                if (lane == 0 && (k != 0 || !params_first)) {
                    bulk_wait_read<0>();
                    mbar_expect_tx(bar, kSrvTileBytes);
                    if (!a.arm_only) tma_load_2d(smem_u32(stage), loc.map, 0, (int)row0, bar);
                }
            };
            static_assert(kIssueAt == 4 && kGroup % 4 == 0, "the parameter load is issued between blocks of four workers");
            const bool in_units = !kUnit || __builtin_expect(unit, 1);
            if (in_units && g0 + kGroup <= a.W) {  // a whole stage: blocks of four workers in straight-line code
#pragma unroll 1
                for (int i0 = 0; i0 < kGroup; i0 += 4) {
                    // (the positions a whole stage can hold issue_at at: worker 4 when W >= 5, else the
                    // stage's last worker when W == group size)
                    if (MODE == 1 && g0 + i0 == issue_at) load_params();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        if (MODE == 1 && i == 3 && i0 + i == kGroup - 1 && g0 + i0 + i == issue_at) load_params();
                        decode_worker(i0 + i, units);
                    }
                }
            } else if (in_units) {
#pragma unroll 1
                for (int i = 0; g0 + i < a.W; ++i) {
                    if (MODE == 1 && g0 + i == issue_at) load_params();
                    decode_worker(i, units);
                }
            } else {                               // a tile with a scale outside the range: one worker after another
#pragma unroll 1
                for (int i = 0; i < kGroup && g0 + i < a.W; ++i) {
                    if (MODE == 1 && g0 + i == issue_at) load_params();
                    decode_worker(i, std::false_type());
                }
            }
            __syncwarp();                          // every lane has read the stage: refill it
            if (u + kCodeDepth < nunits)
                fill(cstage_addr, locate_srv_tile<SEGS>(map_full, a, segs, t_begin + fill_tile * t_step, fill_e),
                     (int)fill_group * kGroup);
            cp_async_commit();
            if (++fill_group == groups) { fill_group = 0; ++fill_tile; }
        }

        if constexpr (MODE == 1) {
            ok = mbar_try_wait(bar, parity);
            if (!ok) ok = mbar_wait(bar, parity, a.poll_limit);
            if (!__all_sync(0xFFFFFFFFu, ok)) { failed = true; break; }
        }
        if constexpr (MODE == 0) {
            // nothing is loaded: the stage is only written by this warp, once the store of the tile
            // before has read it
            if (lane == 0) bulk_wait_read<0>();
            __syncwarp();
        }

        {
            float4* tl = reinterpret_cast<float4*>(stage);
            const float factor = kUnit && unit ? a.unit_factor : MODE == 1 ? a.neg_lr : 1.0f;
            const float2 nlr = make_float2(factor, factor);
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const int idx = swz((int)lane, c);
                float2 lo = v2[2 * c], hi = v2[2 * c + 1];
                if constexpr (MODE == 0 && kUnit) {
                    lo = __fmul2_rn(nlr, lo);
                    hi = __fmul2_rn(nlr, hi);
                }
                if constexpr (MODE == 1) {          // params <- fma(-lr, sum, params), in place
                    const float4 p = tl[idx];
                    lo = __ffma2_rn(nlr, lo, make_float2(p.x, p.y));
                    hi = __ffma2_rn(nlr, hi, make_float2(p.z, p.w));
                }
                tl[idx] = make_float4(lo.x, lo.y, hi.x, hi.y);
            }
        }
        fence_proxy_async();                                   // the bulk store must see these writes
        if (have_next) {
            // constants of the next tile; the table was last read before the group loop's last
            // __syncwarp
            unit = store_tile_scales<BITS, RANGE, kUnit>(a, table, lane, wide, s_next);
        }
        __syncwarp();
        if (lane == 0) {
            // a short last tile is clipped by the tensor's bounds
            tma_store_2d(loc.map, 0, (int)row0, smem_u32(stage));
            bulk_commit();
            if (MODE == 2 && have_next) {
                bulk_wait_read<0>();
                mbar_expect_tx(bar, kSrvTileBytes);
                if (!a.arm_only) tma_load_2d(smem_u32(stage), loc_next.map, 0, (int)loc_next.row0, bar);
            }
        }
    }
    if constexpr (kCtaSync) {
        if (failed)                     // a warp that gave up still arrives at the barriers the others expect
            for (uint32_t kk = k + 1; kk < sync_tiles; ++kk) named_barrier<1>(kSrvThreads);
    }
    cp_async_wait_group<0>();                                  // no code copy outlives the warp
    if (lane == 0) {
        if (failed) {
            // The tile's copy did not land within the poll limit: count it and give it one more
            // bounded chance before the shared memory can be handed to another CTA.
            atomicAdd(timeouts, 1u);
            mbar_wait(bar, k & 1, a.poll_limit);
        }
        bulk_wait_all<0>();                                    // stores done before the stage goes away
    }

    // A last row of fewer than 32 elements is not covered by the tensor map: the grid's last warp takes it, which has no
    // tile unless the grid is as large as it may be.  (SEGS: the segments that have such a row go to the grid's last warps
    // in turn.)
    const uint32_t from_end = nwarps - 1 - gwarp;
    if constexpr (SEGS) {
        for (uint32_t j = from_end; j < (uint32_t)segs->nseg * (FLAT ? 2u : 1u); j += nwarps) {
            const bool first = FLAT && j >= (uint32_t)segs->nseg;              // the elements before the first row
            const ServerSegEntry& e = segs->e[first ? j - (uint32_t)segs->nseg : j];
            const uint32_t count = first ? e.head : e.ragged;
            if (count == 0) continue;
            const uint64_t done = first ? 0 : (uint64_t)(FLAT ? e.head : 0u) + 32ull * e.nrows_full;
            server_ragged_row<BITS, MODE, RANGE, SEGS>(a, a.params + e.elem0 + done, count, e.words0 + (done * BITS >> 5),
                                                       (uint32_t)(done * BITS) & 31u, e.words_end, e.scale_idx, lane);
        }
    } else if (a.nrows > a.nrows_full && from_end == 0) {
        server_ragged_row<BITS, MODE, RANGE, SEGS>(a, a.params + (uint64_t)a.nrows_full * 32, (uint32_t)(a.n & 31u),
                                                   (uint64_t)a.nrows_full * BITS, 0u, a.ncode_words,
                                                   bucket_of_row(a, a.nrows_full), lane);
    }
}

// One gradient with uniform buckets.  UNIT: tiles whose scales allow it are summed in units of 2^40.
template <int BITS, int MODE, bool RANGE, bool UNIT>
__global__ void __launch_bounds__(kSrvThreads, server_min_ctas<BITS>())
server_tma_kernel(const __grid_constant__ CUtensorMap map_full, const __grid_constant__ ServerTmaArgs a,
                  unsigned int* __restrict__ timeouts)
{
    server_tma_body<BITS, MODE, RANGE, false, UNIT>(&map_full, a, nullptr, timeouts);
}

// The short segments of a per-layer step (those that are not entries of the segment table): their
// tiles come from the table-driven layout of mqg_segments.cuh, cut into pieces of 32 rows, one per warp
// turn.  A lane owns a row: plain loads of its code words, four workers requested at a time, and of its
// 32 parameters.  A few per cent of a layered gradient; folded into the launch of the long segments so
// that the step is one launch.
struct ServerShortSegs {
    SegmentTable tab;
    int scale_first;             // index of the table's first segment in every worker's scale array
    uint32_t pieces;             // 8 x tiles of the table
};

template <int BITS>
__device__ __noinline__ void server_short_piece(const ServerTmaArgs& a, const ServerShortSegs& ss, uint32_t piece,
                                                uint32_t lane)
{
    const TileGeom g = locate_tile<BITS>(ss.tab, piece >> 3);
    const uint32_t r = (piece & 7u) * 32u + lane;
    if (r >= (uint32_t)g.rows) return;
    const uint64_t e0 = g.elem0 + 32ull * r;
    const uint64_t left = g.valid - 32ull * r;            // elements from this row to the segment's end
    const uint64_t word0 = g.word0 + (uint64_t)r * BITS;
    const uint64_t scale_idx = (uint64_t)ss.scale_first + g.seg;
    float2 v2[16];
#pragma unroll
    for (int p = 0; p < 16; ++p) v2[p] = make_float2(0.0f, 0.0f);
    constexpr int kBatch = 4;
    for (int w0 = 0; w0 < a.W; w0 += kBatch) {
        uint32_t cw[kBatch][BITS];
        float sc[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const int wk = min(w0 + i, a.W - 1);          // a worker past the last one repeats it (not summed)
#pragma unroll
            for (int k = 0; k < BITS; ++k)
                cw[i][k] = (word0 + k < g.words_end) ? __ldg(a.ptrs.codes[wk] + word0 + k) : 0u;
            sc[i] = __ldg(a.ptrs.scales[wk] + scale_idx);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
            if (w0 + i < a.W) add_decoded_row<BITS>(cw[i], widen(decode_scale<BITS>(sc[i])), v2);
    }
    float* p = a.params + e0;
    if (left >= 32 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
        const float2 nlr = make_float2(a.neg_lr, a.neg_lr);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
            const float4 q = reinterpret_cast<const float4*>(p)[c];
            const float2 lo = __ffma2_rn(nlr, v2[2 * c], make_float2(q.x, q.y));
            const float2 hi = __ffma2_rn(nlr, v2[2 * c + 1], make_float2(q.z, q.w));
            reinterpret_cast<float4*>(p)[c] = make_float4(lo.x, lo.y, hi.x, hi.y);
        }
    } else {
        float v[32];
        floats_from_pairs(v2, v);
#pragma unroll
        for (int j = 0; j < 32; ++j)
            if ((uint64_t)j < left) p[j] = __fmaf_rn(a.neg_lr, v[j], p[j]);
    }
}

// Several long segments of a per-layer step (fused update only), then the step's short segments.
template <int BITS, bool UNIT, bool FLAT>
__global__ void __launch_bounds__(kSrvThreads, server_min_ctas<BITS>())
server_tma_segments_kernel(const __grid_constant__ ServerSegTable segs, const __grid_constant__ ServerShortSegs ss,
                           const __grid_constant__ ServerTmaArgs a, unsigned int* __restrict__ timeouts)
{
    server_tma_body<BITS, 1, false, true, UNIT, FLAT>(nullptr, a, &segs, timeouts);
    const uint32_t wid = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
    const uint32_t nwarps = gridDim.x * kSrvWarps, from_end = nwarps - 1 - (blockIdx.x * kSrvWarps + wid);
    // the warps that finished their share of the long segments first are the last ones of the grid; the very last ones may
    // have a segment's last row
    const uint32_t skip = (uint32_t)segs.nseg * (FLAT ? 2u : 1u) % nwarps;
    for (uint32_t piece = from_end >= skip ? from_end - skip : from_end + nwarps - skip; piece < ss.pieces; piece += nwarps)
        server_short_piece<BITS>(a, ss, piece, threadIdx.x & 31u);
}

// Whether a launch sums in units of 2^40, and its arguments for that; `factor`: what the sum is multiplied with.  From a
// whole code stage of workers on: with fewer, what it saves is less than what the second form of the decode costs a launch
// (three workers, four bits: 7.9 against 7.5 us for 5 M parameters, 2.85 against 2.7 us for 131,072; four to seven workers at
// two to four bits stay with those: not measured).
template <int BITS>
static bool sum_in_units(ServerTmaArgs& a, float factor)
{
    a.unit_factor = factor * kSumUnit;
    a.one = 1u;
    return a.W >= ServerGroup<BITS>::value && fits_sum_unit(factor);
}

template <int BITS, int MODE, bool RANGE, bool UNIT>
static cudaError_t launch_server_tma_inst(const void* params, ServerTmaArgs& a, unsigned int* timeouts,
                                          cudaStream_t stream)
{
    auto kernel = server_tma_kernel<BITS, MODE, RANGE, UNIT>;
    constexpr size_t kSmemBytes = sizeof(ServerSmem<BITS, false>) + 1024;   // + slack to round the base up
    static std::atomic<int> grid_cap[64];                 // per device; 0 = not yet set up (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kSrvThreads, kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    // The tiles are split evenly over the warps of the grid, down to one tile per warp: a warp's tiles follow one
    // another, so a short gradient is done soonest when it is spread as thin as it goes.  Per step at two bits
    // against at least four tiles per warp (and the parameter tile, the scales and the codes of a warp's first
    // tile requested in turn): 3.4 against 7.4 us at n = 2^20, W = 4, 5.4 against 12.5 us at W = 16, 6.7 against
    // 8.8 us at n = 2^22, W = 4.
    // A last row of fewer than 32 elements is a warp's of its own.
    const uint64_t warps = (uint64_t)a.ntiles + (a.nrows > a.nrows_full ? 1 : 0);
    uint64_t grid = (uint64_t)cap;
    if (grid * kSrvWarps > warps) grid = (warps + kSrvWarps - 1) / kSrvWarps;
    CUtensorMap map_full;
    const char* why = nullptr;
    if (!encode_rows_map(&map_full, params, a.nrows_full, 4, 32, kSrvTileRows, &why)) return cudaErrorNotSupported;
    // Launched as a programmatic dependent of the kernel before it (2.2 us per launch at every bit width, eight
    // launches back to back).
    return launch_pdl_smem(kernel, (unsigned)grid, kSrvThreads, kSmemBytes, stream, map_full, a, timeouts);
}

template <int BITS, bool RANGE>
static cudaError_t launch_server_tma_bits(const void* dst, ServerTmaArgs& a, int mode, unsigned int* timeouts,
                                          cudaStream_t stream)
{
    // a sum that continues from an accumulator is not kept in other units: the accumulator need not fit them
    if (mode == 2) return launch_server_tma_inst<BITS, 2, RANGE, false>(dst, a, timeouts, stream);
    if constexpr (UnitDecode<BITS, RANGE>::kExists) {
        if (sum_in_units<BITS>(a, mode == 1 ? a.neg_lr : 1.0f))
            return mode == 1 ? launch_server_tma_inst<BITS, 1, RANGE, true>(dst, a, timeouts, stream)
                             : launch_server_tma_inst<BITS, 0, RANGE, true>(dst, a, timeouts, stream);
    }
    return mode == 1 ? launch_server_tma_inst<BITS, 1, RANGE, false>(dst, a, timeouts, stream)
                     : launch_server_tma_inst<BITS, 0, RANGE, false>(dst, a, timeouts, stream);
}

bool server_tma_applies(uint64_t n, uint64_t bucket)
{
    const uint64_t nrows = (n + 31) / 32;
    const uint64_t rpb = bucket >= n ? nrows : bucket / 32;
    if (n / 32 < 4 * (uint64_t)kSrvTileRows || nrows > 0x7FFFFFFFull) return false;
    if (rpb >= (uint64_t)kSrvTileRows) return true;
    // Shorter buckets qualify when no 32-row tile (tiles start at multiples of 32 rows) can hold two
    // bucket boundaries, i.e. touch three buckets: the boundaries' offsets inside a tile are multiples
    // of g = gcd(rows per bucket, 32), so the first one lies at least g rows in and the next one
    // rows-per-bucket further: beyond the tile iff g + rpb >= 32 (buckets of 16, 24, 28, 30, 31 rows).
    if (rpb < 16) return false;
    uint64_t g = rpb, r = 32;
    while (r != 0) { const uint64_t t = g % r; g = r; r = t; }
    return g + rpb >= 32;
}

// log2 of the buckets a tile can touch, or -1 if the kernel does not take the shape: 1 for the shapes
// above; buckets of 8, 4, 2 or 1 rows (256 .. 32 elements) divide a tile into 4 .. 32 buckets, which
// the warp's table of 2 * kMaxWorkers entries holds for up to 16, 8, 4, 2 workers.
static int server_tma_nbt_shift(uint64_t n, uint64_t bucket, int W)
{
    if (server_tma_applies(n, bucket)) return 1;
    const uint64_t nrows = (n + 31) / 32;
    if (n / 32 < 4 * (uint64_t)kSrvTileRows || nrows > 0x7FFFFFFFull || bucket >= n) return -1;
    const uint64_t rpb = bucket / 32;
    for (int sft = 2; sft <= 5; ++sft)
        if (rpb == (32u >> sft)) return ((uint64_t)W << sft) <= 2 * (uint64_t)kMaxWorkers ? sft : -1;
    return -1;
}

bool server_tma_applies(uint64_t n, uint64_t bucket, int W) { return server_tma_nbt_shift(n, bucket, W) >= 0; }

// mode 1: dst = params (update with lr); mode 0: dst = acc (overwrite); mode 2: dst = acc (add into)
template <bool RANGE>
static cudaError_t launch_server_tma_codec(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                                           float* params, float lr, int mode, cudaStream_t stream)
{
    ServerTmaArgs a;
    a.ptrs = ptrs;
    a.params = params;
    a.n = n;
    a.ncode_words = (n * (uint64_t)bits + 31) / 32;
    a.nrows = (uint32_t)((n + 31) / 32);
    a.nrows_full = (uint32_t)(n / 32);
    a.ntiles = (a.nrows_full + kSrvTileRows - 1) / kSrvTileRows;
    a.nbuckets = (uint32_t)((n + bucket - 1) / bucket);
    const uint64_t rpb = bucket >= n ? a.nrows : bucket / 32;
    a.rows_per_bucket = (uint32_t)(rpb > 0xFFFFFFFFull ? 0xFFFFFFFFull : rpb);
    a.rpb_shift = -1;
    for (int sft = 0; sft < 32; ++sft)
        if (((uint64_t)1 << sft) == rpb) a.rpb_shift = sft;
    a.nbt_shift = server_tma_nbt_shift(n, bucket, W);
    if (a.nbt_shift < 0) return cudaErrorInvalidValue;
    a.W = W;
    a.neg_lr = -lr;
    a.bias_bits = 0x4B000000u;
    const WaitPolicy policy = wait_policy();
    a.poll_limit = policy.poll_limit;
    a.arm_only = policy.arm_only;
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    switch (bits) {
        case 1: return launch_server_tma_bits<1, RANGE>(params, a, mode, timeouts, stream);
        case 2: return launch_server_tma_bits<2, RANGE>(params, a, mode, timeouts, stream);
        case 3: return launch_server_tma_bits<3, RANGE>(params, a, mode, timeouts, stream);
        case 4: return launch_server_tma_bits<4, RANGE>(params, a, mode, timeouts, stream);
        case 5: return launch_server_tma_bits<5, RANGE>(params, a, mode, timeouts, stream);
        case 6: return launch_server_tma_bits<6, RANGE>(params, a, mode, timeouts, stream);
        case 7: return launch_server_tma_bits<7, RANGE>(params, a, mode, timeouts, stream);
        case 8: return launch_server_tma_bits<8, RANGE>(params, a, mode, timeouts, stream);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_server_tma(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                              float* params, float lr, int mode, cudaStream_t stream)
{
    return launch_server_tma_codec<false>(ptrs, W, bits, n, bucket, params, lr, mode, stream);
}

cudaError_t launch_server_range_tma(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                                    float* params, float lr, int mode, cudaStream_t stream)
{
    return launch_server_tma_codec<true>(ptrs, W, bits, n, bucket, params, lr, mode, stream);
}

// ---- downlink: de-quantize, sum, scale to the mean and quantize again -------------------------------
// (ReceiveQGThenSendQG of Algorithm 1, lines 1-5; steps 6-8 of Fig. 3.)  The decode half is the server
// kernel's: every warp stages the code words of its 32-row tiles by asynchronous copies, two stages
// ahead, and sums the W workers in registers.  The encode half is the quantize kernels' row code.  In
// between stands the bucket maximum: a CTA of WARPS warps takes 32 WARPS consecutive rows at a time, whole buckets, one
// 32-row tile per warp.  A bucket of 2^k rows is reduced by lane shuffles (at most 32 rows) or by the two, four or eight
// warps that hold it, through shared memory and a named barrier of just those warps; buckets of 24, 48 or 96 rows (three
// warps) by an atomic per row and the CTA's barrier.
// Persistent CTAs, no global load through registers.
struct RequantWarpArgs {
    ServerTmaArgs s;             // decode side: ptrs, nrows_full (= all rows), buckets, W, bias
    uint32_t* codes_out;
    float* scales_out;
    float mean_scale;
    uint32_t complete_rows;      // floor(n / 32)
    uint32_t nct;                // CTA tiles of 32 WARPS rows
    uint32_t warps_per_bucket;   // 1 (buckets of at most 32 rows), 2, 4 or 8
    RoundKeys rk;                // Philox round keys of the re-quantization's draws
    PhiloxHead head;             // and the launch-wide part of its blocks
};

template <int BITS, int WARPS>
struct RequantSmem {
    alignas(16) uint32_t code[WARPS][kCodeDepth][ServerGroup<BITS>::value][kSrvTileRows * BITS];
    float4 table[WARPS][2 * kMaxWorkers];
    uint32_t bmax[2][WARPS];                      // tile maxima, double-buffered by the parity of the turn
    uint32_t slot[3][4];                          // three warps: bucket maxima, rotating so that no reset races a use
};

template <int BITS, int WARPS, bool kUnit>
__global__ void __launch_bounds__(32 * WARPS, WARPS == 8 ? 2 : WARPS == 4 ? 4 : 5)
requantize_warp_kernel(const __grid_constant__ RequantWarpArgs ra)
{
    extern __shared__ uint8_t smem_raw[];
    RequantSmem<BITS, WARPS>& sm = *reinterpret_cast<RequantSmem<BITS, WARPS>*>(
        smem_raw + ((16u - (smem_u32(smem_raw) & 15u)) & 15u));
    const ServerTmaArgs& a = ra.s;
    constexpr int kGroup = ServerGroup<BITS>::value;
    constexpr uint32_t kWorkerWords = kSrvTileRows * BITS;
    constexpr uint32_t kCodeStageBytes = kGroup * kWorkerWords * 4;
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t wid = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);
    float4* table = sm.table[wid];
    const uint32_t code_base = smem_u32(&sm.code[wid][0][0][0]);
    if constexpr (WARPS == 3) {
        if (threadIdx.x < 12) (&sm.slot[0][0])[threadIdx.x] = 0u;
        __syncthreads();
    }
    grid_dependency_wait();            // nothing above touches global memory

    // this CTA's tiles of 32 WARPS rows: blockIdx.x, blockIdx.x + gridDim.x, ... (the grid works on one window of
    // consecutive tiles at a time, as in the server kernel); warp w takes rows 32 w .. 32 w + 31 of each
    const uint32_t base = ra.nct / gridDim.x, extra = ra.nct % gridDim.x;
    const uint32_t nct = base + (blockIdx.x < extra ? 1u : 0u);
    const uint32_t groups = ((uint32_t)a.W + kGroup - 1) / kGroup;      // code stages per tile
    const uint32_t nunits = nct * groups;
    const bool wide = ((uint32_t)a.W << a.nbt_shift) > 32u;
    const uint32_t lane_off = lane * 16u;
    const uint32_t last_row = a.nrows_full - 1;
    const uint32_t G = ra.warps_per_bucket;
    auto tile_loc = [&](uint32_t kk) {
        TileLoc t;
        t.map = nullptr;
        t.row0 = ((blockIdx.x + kk * gridDim.x) * WARPS + wid) * kSrvTileRows;
        t.nrows_full = ra.complete_rows;
        t.scale_idx = t.shift = 0;
        t.code_word0 = t.words_end = 0;
        return t;
    };
    auto fill = [&](uint32_t stage, uint32_t kk, int g0) {           // a tile beyond the last row has no codes
        const TileLoc t = tile_loc(kk);
        if (t.row0 < a.nrows_full) fill_code_stage<BITS, true>(a, stage, t, g0, lane_off);
    };

    const UnitBits<BITS, false> unit_bits(a.one);
    bool unit = false;                             // as in the server kernel
    uint32_t u = 0, rot = 0;
    if (nct > 0) {
        float2 s0[2];
        load_tile_scales<false, false>(a, tile_loc(0), lane, wide, s0);
#pragma unroll
        for (uint32_t u2 = 0; u2 < (uint32_t)kCodeDepth; ++u2) {
            if (u2 < nunits) fill(code_base + u2 * kCodeStageBytes, u2 / groups, (int)(u2 % groups) * kGroup);
            cp_async_commit();
        }
        unit = store_tile_scales<BITS, false, kUnit>(a, table, lane, wide, s0);
        __syncwarp();
    }
    uint32_t fill_tile = kCodeDepth / groups, fill_group = kCodeDepth % groups;

#pragma unroll 1
    for (uint32_t k = 0; k < nct; ++k, rot = rot == 2 ? 0 : rot + 1) {
        const TileLoc loc = tile_loc(k);
        const uint32_t row0 = loc.row0;
        const bool have_next = k + 1 < nct;
        float2 s_next[2];
        if (have_next) load_tile_scales<false, false>(a, tile_loc(k + 1), lane, wide, s_next);
        const uint32_t row_c = min(row0 + lane, last_row);
        const uint32_t bucket = bucket_of_row(a, row_c);
        const float4* my_table = table + (bucket - bucket_of_row(a, min(row0, last_row)));
        float2 v2[16];
#pragma unroll
        for (int p = 0; p < 16; ++p) v2[p] = make_float2(0.0f, 0.0f);

#pragma unroll 1
        for (uint32_t g = 0; g < groups; ++g, ++u) {
            const uint32_t cs = u % kCodeDepth;
            const uint32_t* cstage = &sm.code[wid][cs][0][0] + lane * BITS;
            cp_async_wait_group<kCodeDepth - 1>();
            __syncwarp();
            const int g0 = (int)g * kGroup;
            auto decode_worker = [&](int i, auto in_units) {
                uint32_t w[BITS];
                read_stage_words<BITS>(cstage + i * kWorkerWords, w);
                const float4 e = my_table[(uint32_t)(g0 + i) << a.nbt_shift];
                if constexpr (decltype(in_units)::value) {
                    add_decoded_row_unit<BITS, false>(w, e, unit_bits, v2);
                } else {
                    DecodeScale2 d;
                    d.two_h = make_float2(e.x, e.y); d.minus_h = make_float2(e.z, e.w);
                    add_decoded_row<BITS, false>(w, d, v2, a.bias_bits);
                }
            };
            const std::integral_constant<bool, kUnit> units;
            const bool in_units = !kUnit || __builtin_expect(unit, 1);
            if (in_units && g0 + kGroup <= a.W) {
#pragma unroll
                for (int i = 0; i < kGroup; ++i) decode_worker(i, units);
            } else if (in_units) {
#pragma unroll 1
                for (int i = 0; g0 + i < a.W; ++i) decode_worker(i, units);
            } else {
#pragma unroll 1
                for (int i = 0; i < kGroup && g0 + i < a.W; ++i) decode_worker(i, std::false_type());
            }
            __syncwarp();                          // every lane has read the stage: refill it
            if (u + kCodeDepth < nunits) fill(code_base + cs * kCodeStageBytes, fill_tile, (int)fill_group * kGroup);
            cp_async_commit();
            if (++fill_group == groups) { fill_group = 0; ++fill_tile; }
        }

        // the mean, and the bucket maximum of its magnitudes
        const uint32_t row = row0 + lane;
        const bool active = row < a.nrows_full;
        const int left = !active ? 0 : row < ra.complete_rows ? 32 : (int)(a.n - (uint64_t)row * 32);   // elements of the row
        float x[32];
        {
            const float factor = kUnit && unit ? a.unit_factor : ra.mean_scale;
            const float2 ms = make_float2(factor, factor);
#pragma unroll
            for (int p = 0; p < 16; ++p) {
                const float2 y = __fmul2_rn(v2[p], ms);
                x[2 * p] = y.x;
                x[2 * p + 1] = y.y;
            }
            if (row0 + kSrvTileRows > ra.complete_rows) {            // only in the gradient's last tiles:
#pragma unroll
                for (int j = 0; j < 32; ++j) x[j] = j < left ? x[j] : 0.0f;   // what is past the end is what its slot holds
            }
        }
        uint32_t m = __float_as_uint(row_abs_max(x));
        bool writer;
        if constexpr (WARPS == 3) {
            const uint32_t lb = bucket - ((blockIdx.x + k * gridDim.x) * (32u * WARPS)) / a.rows_per_bucket;
            uint32_t* slot = sm.slot[rot];
            if (a.rows_per_bucket == 32u * WARPS) {
                m = __reduce_max_sync(0xFFFFFFFFu, m);
                if (lane == 0) atomicMax(&slot[0], m);
            } else if (active) {
                atomicMax(&slot[lb], m);
            }
            named_barrier<1>(32 * WARPS);
            m = active ? slot[lb] : 0u;
            if (threadIdx.x < 4) sm.slot[rot == 0 ? 2 : rot - 1][threadIdx.x] = 0u;      // next used in two turns
            writer = row % a.rows_per_bucket == 0;
        } else if (G == 1) {
            const uint32_t rpb = min(a.rows_per_bucket, (uint32_t)kSrvTileRows);
            for (uint32_t d = rpb >> 1; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
            writer = (row & (a.rows_per_bucket - 1)) == 0;
        } else {
            m = __reduce_max_sync(0xFFFFFFFFu, m);
            uint32_t* slot = sm.bmax[k & 1];
            if (lane == 0) slot[wid] = m;
            const uint32_t first = wid & ~(G - 1);
            if (WARPS == 8 || G == 4 || first == 0) named_barrier<1>(32 * G);   // the warps that hold this bucket
            else named_barrier<2>(32 * G);
            m = max(slot[first], slot[first + 1]);
            if (WARPS == 8 || G == 4) m = max(m, max(slot[first + 2], slot[first + 3]));
            if constexpr (WARPS == 8) m = max(m, max(max(slot[4], slot[5]), max(slot[6], slot[7])));
            writer = (wid & (G - 1)) == 0 && lane == 0;
        }
        float sc = __uint_as_float(m);
        if (sc < flush_limit()) sc = 0.0f;
        if (active) {
            if (writer) ra.scales_out[bucket] = sc;
            const EncodeScale es = encode_scale<BITS>(sc);
            // (spreading the four Philox blocks over the decode of the workers, to fill its gaps, measured
            // 3 to 5 us slower per launch: the kernel then needs all 128 registers)
            uint32_t h[16];
            draw_row_blocks_head(4u * row, ra.head, ra.rk, h);     // the downlink draws from position 0
            uint32_t w[BITS];
            // (the encode's arithmetic in packed fp32x2 instructions: 0.5 to 1 us per launch at every width;
            // a fifth resident CTA, which 95 registers would allow, changes nothing: the kernel waits on
            // its arithmetic pipes, not on latency)
            encode_pack_row_best<BITS>(x, es, h, w);
            const uint64_t word0 = (uint64_t)row * BITS;
            if (left == 32) {
                store_row_words<BITS>(ra.codes_out, word0, w);
            } else {
                mask_row_words<BITS>(w, left * BITS);
#pragma unroll
                for (int j = 0; j < BITS; ++j)
                    if (word0 + j < a.ncode_words) ra.codes_out[word0 + j] = w[j];
            }
        }
        if (have_next) unit = store_tile_scales<BITS, false, kUnit>(a, table, lane, wide, s_next);
        __syncwarp();
    }
    cp_async_wait_group<0>();                                  // no code copy outlives the warp
}

template <int BITS, int WARPS, bool UNIT>
static cudaError_t launch_requantize_warp_inst(RequantWarpArgs& ra, cudaStream_t stream)
{
    auto kernel = requantize_warp_kernel<BITS, WARPS, UNIT>;
    constexpr size_t kSmemBytes = sizeof(RequantSmem<BITS, WARPS>) + 16;
    static std::atomic<int> grid_cap[64];                 // per device; 0 = not yet set up (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 32 * WARPS, kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    ra.nct = (ra.s.nrows_full + 32 * WARPS - 1) / (32 * WARPS);
    unsigned grid = (unsigned)cap;
    if (grid > ra.nct) grid = ra.nct;
    return launch_pdl_smem(kernel, grid, 32 * WARPS, kSmemBytes, stream, ra);
}

template <int BITS>
static cudaError_t launch_requantize_warp_bits(RequantWarpArgs& ra, int warps, cudaStream_t stream)
{
    if constexpr (UnitDecode<BITS, false>::kExists) {
        if (sum_in_units<BITS>(ra.s, ra.mean_scale))
            return warps == 3 ? launch_requantize_warp_inst<BITS, 3, true>(ra, stream)
                 : warps == 8 ? launch_requantize_warp_inst<BITS, 8, true>(ra, stream)
                              : launch_requantize_warp_inst<BITS, 4, true>(ra, stream);
    }
    return warps == 3 ? launch_requantize_warp_inst<BITS, 3, false>(ra, stream)
         : warps == 8 ? launch_requantize_warp_inst<BITS, 8, false>(ra, stream)
                      : launch_requantize_warp_inst<BITS, 4, false>(ra, stream);
}

// Warps of a CTA for buckets of `rpb` rows, 0 where the kernel does not take them: whole buckets fill the CTA's rows, and a
// warp's 32 rows touch at most two buckets (or a power of two of them).
static int requantize_warps(uint64_t rpb)
{
    if (rpb == 24 || rpb == 48 || rpb == 96) return 3;
    if ((rpb & (rpb - 1)) != 0 || rpb > 256) return 0;
    return rpb == 256 ? 8 : 4;
}

// At least 512 complete rows, fewer than 2^30 (so the draws' block numbers have no high half), buckets as above, those
// below 32 rows few enough per tile for the warp's table; and where it is the faster one.  Against a CTA per tile
// (mqg_requantize.cu) a warp's copies and constants are ahead of their use, which short launches gain from - bucket 1024, two
// bits, 1 / 8 / 16 workers 0.88 / 0.83 / 0.77 of the other's time at 1.5 M elements - and long ones when there is much to sum:
// 25 M elements, bucket 2048, four bits, 8 / 16 workers 44 / 68 against 52 / 86 us, eight bits, 4 workers 35 against 39 us.
// Otherwise the other's smaller CTAs with fewer registers win: 25 M elements, one bit, 4 / 16 workers 28 / 54 against 32 / 62 us,
// two bits, 4 workers 32 against 35 us; 1 M elements, six bits, one worker 0.93.  Three warps, whose CTAs are smaller still: 24 and 48
// rows, 0.7 M elements, four bits, 1 / 8 / 16 workers 1.02 / 0.88 / 0.84, 4 M 1.06 / 0.90 / 0.86; 96 rows 0.94 to 0.64 at 1 M.  Eight
// warps: a bucket to a CTA, two CTAs to an SM, so that a launch of 2.2 to 2.8 rounds of 296 waits for its third: 6 M elements,
// four bits, 4 / 8 workers 1.19 / 1.06, at 4 and 7 M and 8 workers 0.89 and 0.93.
bool requantize_warp_applies(uint64_t n, uint64_t bucket, int W, int bits)
{
    if (n / 32 < 512 || n / 32 >= (1ull << 30) - 1 || bucket >= n || bucket % 32 != 0) return false;
    const uint64_t rpb = bucket / 32;
    const int warps = requantize_warps(rpb);
    if (warps == 0 || (rpb < 24 && (uint64_t)W * (32 / rpb) > 2 * (uint64_t)kMaxWorkers)) return false;
    const bool several = W >= 8 && bits >= 2, six = bits == 6 && W <= 2;
    const bool much = several && W * bits >= 32 && (bits != 6 || W >= 16) && (bits >= 3 || n < 5ull << 19);
    if (rpb == 24 || rpb == 48) return n < 1ull << 20 ? several : much;
    if (n < 1ull << 20) return warps != 8 || !six;
    if (n < 3ull << 19) return !six;
    if (warps == 3) return much;
    if (warps == 8) return several && W * bits >= 24 && (n < 660 * 8192 || n >= 840 * 8192);
    return bits == 4 || (bits >= 2 && W * bits >= 24) || (several && n < 16ull << 20);
}

cudaError_t launch_requantize_warp(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                                   float mean_scale, uint64_t seed, uint32_t* codes_out, float* scales_out,
                                   uint32_t worker, uint32_t step, cudaStream_t stream)
{
    RequantWarpArgs ra;
    memset(&ra, 0, sizeof(ra));
    ServerTmaArgs& a = ra.s;
    a.ptrs = ptrs;
    a.n = n;
    a.ncode_words = (n * (uint64_t)bits + 31) / 32;
    a.nrows = a.nrows_full = (uint32_t)((n + 31) / 32);
    ra.complete_rows = (uint32_t)(n / 32);
    a.nbuckets = (uint32_t)((n + bucket - 1) / bucket);
    const uint64_t rpb = bucket / 32;
    const int warps = requantize_warps(rpb);
    a.rows_per_bucket = (uint32_t)rpb;
    a.rpb_shift = -1;
    for (int sft = 0; sft < 32; ++sft)
        if (((uint64_t)1 << sft) == rpb) a.rpb_shift = sft;
    // log2 of the buckets a tile of 32 rows touches
    a.nbt_shift = rpb == 24 || rpb == 48 ? 1 : 0;
    while (rpb < 24 && (rpb << a.nbt_shift) < 32) ++a.nbt_shift;
    a.W = W;
    a.bias_bits = 0x4B000000u;
    ra.codes_out = codes_out; ra.scales_out = scales_out;
    ra.mean_scale = mean_scale;
    ra.warps_per_bucket = rpb <= 32 ? 1u : (uint32_t)(rpb / 32);
    uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
    for (int r = 0; r < 10; ++r) {
        ra.rk.k0[r] = k0; ra.rk.k1[r] = k1;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    ra.rk.worker = worker; ra.rk.step = step;
    ra.head = philox_head(0u, worker, ra.rk.k0[0]);
    switch (bits) {
#define MQG_REQUANT_CASE(B) \
        case B: return launch_requantize_warp_bits<B>(ra, warps, stream)
        MQG_REQUANT_CASE(1); MQG_REQUANT_CASE(2); MQG_REQUANT_CASE(3); MQG_REQUANT_CASE(4);
        MQG_REQUANT_CASE(5); MQG_REQUANT_CASE(6); MQG_REQUANT_CASE(7); MQG_REQUANT_CASE(8);
#undef MQG_REQUANT_CASE
    }
    return cudaErrorInvalidValue;
}

// ---- several long segments of a per-layer step in one launch --------------------------------------
template <int BITS, bool UNIT, bool FLAT>
static cudaError_t launch_server_segs_inst(const ServerSegTable& tab, const ServerShortSegs& ss, const ServerTmaArgs& a,
                                           unsigned int* timeouts, cudaStream_t stream)
{
    auto kernel = server_tma_segments_kernel<BITS, UNIT, FLAT>;
    constexpr size_t kSmemBytes = sizeof(ServerSmem<BITS, FLAT>) + 1024;   // + slack to round the base up
    static std::atomic<int> grid_cap[64];                 // per device; 0 = not yet set up (zero-initialised)
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    int cap = grid_cap[dev].load(std::memory_order_relaxed);
    if (cap == 0) {
        int occ = 0, sms = 0;
        err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, kSrvThreads, kSmemBytes);
        if (err != cudaSuccess) return err;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        cap = sms * (occ > 0 ? occ : 1);
        grid_cap[dev].store(cap, std::memory_order_relaxed);   // every thread computes the same value
    }
    uint64_t grid = (uint64_t)cap;
    const uint64_t warps = (uint64_t)a.ntiles + (uint64_t)tab.nseg * (FLAT ? 2 : 1) + ss.pieces;   // at least one tile, last row or short piece per warp
    if (grid * kSrvWarps > warps) grid = (warps + kSrvWarps - 1) / kSrvWarps;
    return launch_pdl_smem(kernel, (unsigned)grid, kSrvThreads, kSmemBytes, stream, tab, ss, a, timeouts);
}

int flat_server_form(uint64_t on, uint64_t off, int W, int bits)
{
    // The table-driven launch is for short calls: one tensor, that launch / this form, one worker 3.4 / 3.9, 4.7 / 4.0, 9.9 / 4.9
    // us for 0.2, 0.4 and 1.6 M elements, eight 3.8 / 5.2, 6.4 / 6.6, 10.5 / 7.6 us for 0.2, 0.8 and 1.6 M, sixteen 8.2 / 9.6,
    // 12.9 / 11.2 us for 0.8 and 1.6 M; 50 M elements and eight workers 631 / 110 us.  (A table of a few long tensors that rides
    // along with the launch of the others is a tail of 6 us: 16 M elements, 40,000 of them off the boundaries, one worker 24.4
    // against 18.5 us.)
    if (off == 0 || on + off < (W <= 4 ? 1ull << 19 : 1ull << 20)) return 0;
    // Those on the boundaries go along, which saves 2 to 4 us for a second launch, unless their codes are many: the flat form
    // copies them four bytes at a time.  Apart / together, 1.5 M elements off the boundaries: eight workers, four bits, 1, 8
    // and 16 M on them 11.0 / 9.3, 21.5 / 21.1, 40.3 / 42.8 us, eight bits and 8 M 29.9 / 31.6, sixteen workers, four bits, 16 M
    // 58.3 / 67.3 us.  Up to four workers the parameters are most of the bytes: four bits, four workers, 40 M 70.8 / 69.9 us.
    return W >= 8 && on * (uint64_t)(W * bits) >= 512ull << 20 ? 1 : 2;
}

cudaError_t launch_server_tma_segments(const WorkerPtrs& ptrs, int W, int bits, const ServerSegHost* segs, int nseg,
                                       const SegmentTable* short_tab, int short_first, float* params, float lr,
                                       bool flat, cudaStream_t stream)
{
    if (nseg < 1 || nseg > kMaxSrvSegs) return cudaErrorInvalidValue;
    ServerShortSegs ss;
    memset(&ss, 0, sizeof(ss));
    if (short_tab != nullptr) {
        const uint64_t pieces = 8ull * short_tab->tile_start[short_tab->nseg];
        if (pieces > 0x7FFFFFFFull) return cudaErrorInvalidValue;
        ss.tab = *short_tab;
        ss.scale_first = short_first;
        ss.pieces = (uint32_t)pieces;
    }
    ServerSegTable tab;
    memset(&tab, 0, sizeof(tab));
    tab.nseg = nseg;
    uint64_t tiles = 0;
    for (int j = 0; j < nseg; ++j) {
        const ServerSegHost& h = segs[j];
        ServerSegEntry& e = tab.e[j];
        const uint64_t head = flat ? (0 - h.elem0) % 32 : 0;          // elements up to the next row of `params`
        if (h.n < head + 32) return cudaErrorInvalidValue;
        const uint64_t nrows_full = (h.n - head) / 32;
        if (nrows_full > 0x7FFFFFFFull) return cudaErrorInvalidValue;
        const char* why = nullptr;
        if (!encode_rows_map(&tab.map[j], params + h.elem0 + head, nrows_full, 4, 32, kSrvTileRows, &why))
            return cudaErrorNotSupported;
        e.tile_start = (uint32_t)tiles;
        e.nrows_full = (uint32_t)nrows_full;
        e.scale_idx = h.scale_idx;
        e.ragged = (uint32_t)((h.n - head) % 32);
        e.head = (uint32_t)head;
        e.shift = (uint32_t)(head * bits) & 31u;
        e.code_word0 = h.code_word0 + (head * bits >> 5);
        e.words0 = h.code_word0;
        e.words_end = h.code_word0 + (h.n * (uint64_t)bits + 31) / 32;
        e.elem0 = h.elem0;
        tiles += (nrows_full + kSrvTileRows - 1) / kSrvTileRows;
        if (tiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    }
    tab.e[nseg].tile_start = (uint32_t)tiles;
    ServerTmaArgs a;
    memset(&a, 0, sizeof(a));
    a.ptrs = ptrs;
    a.params = params;
    a.nrows = a.nrows_full = 1;          // not used by a launch over segments
    a.ntiles = (uint32_t)tiles;
    a.nbuckets = 1;
    a.rows_per_bucket = 1; a.rpb_shift = 0;
    a.nbt_shift = 0;                     // a tile lies in one bucket: table entry = worker
    a.W = W;
    a.neg_lr = -lr;
    a.bias_bits = 0x4B000000u;
    const WaitPolicy policy = wait_policy();
    a.poll_limit = policy.poll_limit;
    a.arm_only = policy.arm_only;
    unsigned int* timeouts = wait_timeout_counter();
    if (timeouts == nullptr) return cudaErrorNotSupported;
    switch (bits) {
#define MQG_SEGS_CASE(B) \
        case B: \
            if constexpr (UnitDecode<B, false>::kExists) \
                if (sum_in_units<B>(a, -lr)) \
                    return flat ? launch_server_segs_inst<B, true, true>(tab, ss, a, timeouts, stream) \
                                : launch_server_segs_inst<B, true, false>(tab, ss, a, timeouts, stream); \
            return flat ? launch_server_segs_inst<B, false, true>(tab, ss, a, timeouts, stream) \
                        : launch_server_segs_inst<B, false, false>(tab, ss, a, timeouts, stream)
        MQG_SEGS_CASE(1); MQG_SEGS_CASE(2); MQG_SEGS_CASE(3); MQG_SEGS_CASE(4);
        MQG_SEGS_CASE(5); MQG_SEGS_CASE(6); MQG_SEGS_CASE(7); MQG_SEGS_CASE(8);
#undef MQG_SEGS_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace mqg
