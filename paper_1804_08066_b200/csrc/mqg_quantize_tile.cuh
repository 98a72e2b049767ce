// The tile code of the TMA-fed quantize kernels (one tile of whole buckets per CTA turn: scale,
// draws, encode, pack), shared by the kernels of mqg_quantize.cu, mqg_quantize_workers.cu and mqg_segments_workers.cu.
#pragma once

#include <type_traits>

#include "mqg_common.cuh"
#include "mqg_internal.h"
#include "mqg_tma.cuh"

namespace mqg {

struct QuantizeArgs {
    const void* grad;
    uint32_t* codes;
    float* scales;
    uint64_t n;             // elements
    uint64_t nrows;         // ceil(n / 32)
    uint64_t nbuckets;      // ceil(n / bucket)
    uint64_t ncode_words;   // ceil(n * bits / 32)
    uint64_t elem_offset;
    uint32_t rows_per_bucket;   // bucket / 32 (a single ragged bucket counts as "all rows")
    uint32_t tile_rows;         // rows per tile: a multiple of rows_per_bucket, <= 512
    uint32_t buckets_per_tile;
    uint64_t nrows_full;    // floor(n / 32): rows the tensor map covers
    uint32_t ntiles;
    DrawKey key;
    uint32_t poll_limit;        // polls of one barrier wait before the CTA gives up (TMA kernels)
    uint32_t arm_only;          // test hook: 1 = arm the barriers but issue no copy
    uint32_t row_elems;         // 32, or 64 (kBf16Wide): what a "row" of the counts above holds
};


// ---------------------------------------------------------------------------------------
// The same computation fed by TMA: a persistent CTA walks tiles blockIdx.x, +gridDim.x, ...;
// one elected thread keeps STAGES tiled bulk copies (cp.async.bulk.tensor, 128- or 64-byte
// swizzle) in flight into a shared-memory ring, each completing on its own mbarrier, so the
// compute warps never issue a global load and never wait for DRAM latency in steady state.
// One __syncthreads per tile publishes the bucket maxima and releases the stage for refill.
// ---------------------------------------------------------------------------------------
template <int DTYPE>
__device__ __forceinline__ void read_row_swizzled(const uint8_t* stage, int row, float (&x)[32])
{
    if constexpr (DTYPE == 0) {
        read_row(reinterpret_cast<const float4*>(stage), row, x);
    } else {
        const uint4* t = reinterpret_cast<const uint4*>(stage);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const uint4 v = t[row * 4 + (c ^ ((row >> 1) & 3))];
            const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                x[8 * c + 2 * k] = bf16_lo(u[k]);
                x[8 * c + 2 * k + 1] = bf16_hi(u[k]);
            }
        }
    }
}

// A bf16 row as it lies in the stage: element pairs, two to a word.
__device__ __forceinline__ void read_row_words(const uint8_t* stage, int row, uint32_t (&u)[16])
{
    const uint4* t = reinterpret_cast<const uint4*>(stage);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        const uint4 v = t[row * 4 + (c ^ ((row >> 1) & 3))];
        u[4 * c] = v.x; u[4 * c + 1] = v.y; u[4 * c + 2] = v.z; u[4 * c + 3] = v.w;
    }
}

__device__ __forceinline__ void widen_row(const uint32_t (&u)[16], float (&x)[32])
{
#pragma unroll
    for (int k = 0; k < 16; ++k) { x[2 * k] = bf16_lo(u[k]); x[2 * k + 1] = bf16_hi(u[k]); }
}

// Largest magnitude of a bf16 row: two elements per instruction (the sign of the running maximum is an exclusive or
// and means nothing; the magnitude is the maximum).
__device__ __forceinline__ float row_abs_max_bf16(const uint32_t (&u)[16])
{
    auto max2 = [](uint32_t a, uint32_t b) {
        uint32_t r;
        asm("max.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
        return r;
    };
    uint32_t m[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) m[k] = max2(u[2 * k], u[2 * k + 1]);
#pragma unroll
    for (int d = 4; d > 0; d >>= 1)
#pragma unroll
        for (int k = 0; k < d; ++k) m[k] = max2(m[k], m[k + d]);
    return max3_abs(0.0f, bf16_lo(m[0]), bf16_hi(m[0]));      // from 0: a row that is NaN throughout does not count
}

constexpr int kBf16Wide = 2;                 // as DTYPE of the tile, the shared memory and the kernels: rows of 64 elements

// The one row of a gradient that is shorter than the others is not covered by the tensor map.  Before the tile's copy is
// waited for, the warp that holds it requests it, zeros behind its end, by asynchronous copies of four bytes a lane into a
// row of the warp's beside the stages.  (Into the stage by its owner after the wait is one round trip more: with the row
// then read where it is, 131,073 elements took 2.09 against 2.28 us, eight workers 2.86 against 3.15, the range 1.95 against 2.14;
// moved into the stage, as it is now, 2.2 for one worker.)  `row` is the gradient's, of row_bytes
// bytes.
static __device__ __noinline__ void fetch_ragged_row(uint32_t to, const uint8_t* grad, uint64_t row, uint64_t total_bytes,
                                                 uint32_t row_bytes)
{
    const uint32_t b = 4u * (threadIdx.x & 31u);
    if (b >= row_bytes) return;
    const uint64_t at = row * row_bytes + b;
    const uint32_t left = at < total_bytes ? (uint32_t)min(total_bytes - at, (uint64_t)4) : 0u;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 ::"r"(to + b), "l"(grad + (left != 0 ? at : 0)), "r"(left) : "memory");
}

// The warp moves that row into row `row` of the tile's stage, once the tile's copy, which fills it with zeros, has landed; its
// owner reads it like any other.  (Read from where it is, after or instead of the stage's, the choice between the two cost
// every row of the tiles that may have one 10 to 26 instructions.)
static __device__ __noinline__ void put_ragged_row(uint8_t* stage, uint32_t row, const uint8_t* from, uint32_t row_bytes)
{
    cp_async_wait_all();
    __syncwarp();
    const uint32_t lane = threadIdx.x & 31u, chunk = lane >> 2;
    const uint32_t at = row_bytes == 128 ? row * 8 + (chunk ^ (row & 7u)) : row * 4 + (chunk ^ ((row >> 1) & 3u));
    if (4 * lane < row_bytes)
        reinterpret_cast<uint32_t*>(stage)[at * 4 + (lane & 3u)] = reinterpret_cast<const uint32_t*>(from)[lane];
    fence_proxy_async();             // orders these stores before the bulk copy that refills the stage
    __syncwarp();
}

// The same in one step, by its owner, for 128-byte rows whose launches are long (rows of 64, and mqg_segments_workers.cu):
// there the other tiles' code decides, which the forms above lengthened (50 M bf16 elements 28.7 against 28.0 us).
static __device__ __noinline__ void stage_ragged_row(uint8_t* stage, uint32_t row, const uint8_t* grad, uint64_t from,
                                                     uint64_t total_bytes)
{
    const uint32_t* src = reinterpret_cast<const uint32_t*>(grad + from * 128);
    const uint32_t left = (uint32_t)(total_bytes - from * 128);              // fewer than 128
    uint32_t v[32];                  // all in flight at once
#pragma unroll
    for (uint32_t w = 0; w < 32; ++w) v[w] = 4 * w + 4 <= left ? __ldcg(src + w) : 0u;
    const uint32_t half = left % 4 >= 2 ? *reinterpret_cast<const uint16_t*>(src + left / 4) : 0u;
#pragma unroll
    for (uint32_t w = 0; w < 32; ++w)
        reinterpret_cast<uint32_t*>(stage)[(row * 8 + ((w >> 2) ^ (row & 7u))) * 4 + (w & 3u)] = w == left / 4 ? half : v[w];
    fence_proxy_async();             // orders these stores before the bulk copy that refills the stage
}

// Whether this thread's warp holds that row, in the tile that does; `first` is the row of the warp's lane 0.
__device__ __forceinline__ bool warp_has_row(uint64_t row, uint32_t first) { return (uint32_t)row - first < 32u; }

// How the rows of a bucket are reduced: a bucket is an aligned power-of-two group of at most 32 rows (lane
// shuffles), a whole number of warps (one shared-memory atomic per warp), or any other number of rows (one
// shared-memory atomic per row; at least three rows, so at most 42 buckets per tile of 128).
enum : int { kByShuffle = 0, kByWarps = 1, kByRows = 2 };
enum : int { kMaxAbs = 0, kRange = 1, kNorm = 2 };
constexpr int kSlots = 44;

// STAGES: depth of the shared-memory ring, two but for short launches of 256 fp32 rows to a tile (one_stage).
template <int DTYPE, int THREADS, int STAGES = 2>
struct TmaQuantizeShared {
    static constexpr int kRowBytes = DTYPE == 1 ? 64 : 128;
    static constexpr int kStages = STAGES;
    alignas(1024) uint8_t stage[kStages][THREADS * kRowBytes];
    uint32_t slots[3][kSlots];             // bucket maxima, rotating so no reset races a use
    uint32_t slots_lo[3][kSlots];          // bucket minima of the (min, max) variant, as ordered bits
    float row_sums[THREADS];               // L2 norm, reduction by rows
    alignas(16) uint8_t ragged[THREADS / 32][128];      // fetch_ragged_row
    alignas(8) uint64_t bar[kStages];
};

// Above 48 KB the shared memory is dynamic (with slack to round the base up).
template <typename Shared>
__host__ __device__ constexpr size_t dynamic_bytes() { return sizeof(Shared) > 48 * 1024 ? sizeof(Shared) + 1024 : 0; }
template <typename Shared>
__device__ __forceinline__ Shared& tile_shared()
{
    if constexpr (dynamic_bytes<Shared>() == 0) {
        __shared__ Shared sh;
        return sh;
    } else {
        extern __shared__ uint8_t tile_smem[];
        return *reinterpret_cast<Shared*>(tile_smem + ((1024u - (smem_u32(tile_smem) & 1023u)) & 1023u));
    }
}
// Gradients of whole rows run kernels without the code for a last row that is shorter (it costs 1 to 6 % of a launch, 0.1 us of
// a short one) - but for the range of fp32 rows by shuffles or warps, which the compiler makes 3 to 16 % slower without it.
template <int DTYPE, int THREADS, int RED, int MODE>
constexpr bool keeps_ragged_code() { return MODE == kRange && DTYPE == 0 && THREADS == 128 && RED != kByRows; }
template <int N>
using Int = std::integral_constant<int, N>;

// Whether tiles of up to 256 fp32 rows keep to one stage, refilled behind the tile's arithmetic, instead of two.  Two pay when the
// gradients come from DRAM and cost when they are in L2, i.e. from 18 M elements on; bucket 8192, four bits, one / two stages
// against the one stage of before: 4, 12 and 33 M elements 0.99 / 1.07, 0.99 / 1.05 and 1.00 / 0.87 of the time, the range 0.98 / 1.02,
// 1.00 / 1.02 and 1.00 / 0.93, the norm 1.00 / 0.99, 0.98 / 0.98 and 0.98 / 0.88.
inline bool one_stage(uint64_t rows) { return rows < (18u << 20) / 32; }

template <int DTYPE, int THREADS>
constexpr int quantize_min_ctas() { return DTYPE == kBf16Wide ? (THREADS == 128 ? 5 : 2) : THREADS == 512 ? 1 : 512 / THREADS; }

// The tile's rows from row `row0` on into a stage: a bulk copy, or two where the tile has more than the 256 rows that the
// box of a copy may have.
__device__ __forceinline__ void load_tile_rows(uint32_t stage, const CUtensorMap* map, uint32_t row0, uint32_t tile_rows,
                                               uint32_t row_bytes, bool halves, uint32_t bar)
{
    tma_load_2d(stage, map, 0, (int)row0, bar);
    if (halves) tma_load_2d(stage + (tile_rows >> 1) * row_bytes, map, 0, (int)(row0 + (tile_rows >> 1)), bar);
}

// Kernel-constant inputs of the TMA kernel beyond QuantizeArgs: the ten Philox round keys are
// computed on the host so the kernel reads them as constant operands.
struct TmaQuantizeConsts {
    RoundKeys rk;
    uint32_t full_tiles;         // leading tiles in which every thread has a complete row
    uint32_t ragged_tile;        // the tile whose last row is shorter than the others; 2^32 - 1 if there is none
    uint32_t blk0_lo, blk0_hi;   // Philox block index of element 0: elem_offset / 8; the launch's blocks
                                 // all have the high half blk0_hi (tma_path_applies)
    PhiloxHead head;             // launch-wide part of the blocks of worker rk.worker
};

// What a tile needs to know about the worker it belongs to.  The one-worker kernel builds it
// from its kernel parameters (so every member stays a constant operand), the batched kernel from
// its table.
struct WorkerView {
    const CUtensorMap* map;
    const void* grad;
    uint32_t* codes;
    float* scales;
    PhiloxHead head;             // launch-wide part of this worker's Philox blocks
    uint32_t blk0_lo;            // low half of the Philox block index of the gradient's element 0
};

// One tile, the k-th of this CTA, tile `tile` of worker `wv`.  FULL: every thread owns a complete
// row (no bounds checks).  RED: how a bucket's rows are reduced.  After the tile's rows are in registers thread 0 calls
// `refill(stage, bar)` to start the copy that uses the stage next.  Returns false if the tile's copy never landed.
template <int BITS, int DTYPE, int THREADS, bool FULL, int RED, bool RAGGED, bool NORM = false,
          typename Shared, typename Refill>
__device__ __forceinline__ bool quantize_tile(Shared& sh, const WorkerView wv,
                                              const QuantizeArgs& a, const TmaQuantizeConsts& c,
                                              uint32_t k, uint32_t rot, uint32_t tile, Refill&& refill,
                                              uint32_t local_bucket, bool scale_writer)
{
    constexpr int kQuantStages = Shared::kStages;
    constexpr bool SHUFFLE = RED == kByShuffle;
    const uint32_t t = threadIdx.x;
    const uint32_t row = tile * a.tile_rows + t;
    const bool active = FULL || (t < a.tile_rows && row < (uint32_t)a.nrows);
    const bool tail = RAGGED && !FULL && tile == c.ragged_tile;  // a tile with a row that the copy does not cover
    const uint32_t stg = k % kQuantStages, parity = (k / kQuantStages) & 1;
    const uint32_t bar = smem_u32(&sh.bar[stg]);
    uint8_t* stage = sh.stage[stg];

    // The row's draws depend on nothing but its number.  From three bits on they are computed before the
    // tile's data is waited for: 16 more live registers (four CTAs per SM instead of five) against the
    // overlap of the Philox rounds with the wait.  Measured per 100 MB gradient in the batched launch with the
    // SM clock at its maximum: 17.0 against 18.0 us at K = 4, 18.3 against 18.6 us at K = 6, 19.7 against
    // 20.0 us at K = 8; no difference at one and two bits, which keep the fifth CTA.  (In a long run the power
    // limit sets the clock and both forms take the same time: the instruction count decides there.)
    // bf16 input (half the bytes per tile, no wait to cover) keeps the draws after the wait at every width:
    // 32.3 / 32.1 / 32.7 / 32.4 us per 50 M elements at K = 3 / 4 / 6 / 8 against 33.2 / 32.8 / 33.6 / 32.8 us.
    constexpr bool kEarlyDraw = !NORM && DTYPE == 0 && BITS >= 3;
    uint32_t h[16];
    if (kEarlyDraw && active) draw_row_blocks_head(wv.blk0_lo + 4u * row, wv.head, c.rk, h);
    if (tail && warp_has_row(a.nrows_full, row - (t & 31u)))
        fetch_ragged_row(smem_u32(sh.ragged[t >> 5]), static_cast<const uint8_t*>(wv.grad), a.nrows_full,
                         a.n * (DTYPE == 0 ? 4 : 2), DTYPE == 0 ? 128 : 64);
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) ok = mbar_wait(bar, parity, a.poll_limit);
    if (tail && warp_has_row(a.nrows_full, row - (t & 31u)))
        put_ragged_row(stage, (uint32_t)a.nrows_full - tile * a.tile_rows, sh.ragged[t >> 5], DTYPE == 0 ? 128 : 64);

    // bf16 rows whose maximum is wanted stay packed until the encode: half the registers across the barrier, and the
    // maximum takes two elements per instruction (30.0 against 30.5 us per 50 M elements at K = 4)
    constexpr bool kPackedRow = DTYPE == 1 && !NORM;
    float x[32];
    uint32_t raw[16];
    if (active) {
        if (kPackedRow) read_row_words(stage, (int)t, raw);
        else read_row_swizzled<DTYPE>(stage, (int)t, x);
    } else {
#pragma unroll
        for (int j = 0; j < 32; ++j) x[j] = 0.0f;
#pragma unroll
        for (int j = 0; j < 16; ++j) raw[j] = 0u;
    }
    uint32_t m;
    uint32_t* slot = sh.slots[rot];          // rot = k % 3
    if constexpr (NORM) {
        // L2-norm scale: the fixed tree over the rows' sums of squares - partner distance 1, 2, 4, ...
        // inside the warp, then (buckets of whole warps) the warp sums, one slot per warp.
        // The row's draws depend on nothing but its number: they are computed here, before the chain of
        // 32 dependent fused multiply-adds, so that the Philox rounds fill the chain's latency gaps.
        // (one launch per worker at n = 25 M: 22.3 / 22.5 / 23.0 us at K = 1 / 4 / 8 against 22.6 / 22.6 / 24.9 us)
        if (active) draw_row_blocks_head(wv.blk0_lo + 4u * row, wv.head, c.rk, h);
        float ss = row_sum_squares(x);
        if constexpr (RED == kByRows) {
            sh.row_sums[t] = ss;
        } else {
            const uint32_t lanes = SHUFFLE ? a.rows_per_bucket : 32u;
            for (uint32_t d = 1; d < lanes; d <<= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xFFFFFFFFu, ss, d));
            if (!SHUFFLE && (t & 31) == 0) slot[t >> 5] = __float_as_uint(ss);
        }
        m = __float_as_uint(ss);
    } else {
        m = __float_as_uint(kPackedRow ? row_abs_max_bf16(raw) : row_abs_max(x));
        if (SHUFFLE) {
            for (uint32_t d = a.rows_per_bucket >> 1; d > 0; d >>= 1)
                m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
        } else if (RED == kByRows) {
            if (active) atomicMax(&slot[local_bucket], m);
        } else {
            m = __reduce_max_sync(0xFFFFFFFFu, m);
            if ((t & 31) == 0) atomicMax(&slot[local_bucket], m);
        }
    }
    if (__syncthreads_or(!ok)) return false;
    if (t == 0) refill(smem_u32(stage), bar);                    // every thread has read the stage
    if (!SHUFFLE) {
        if constexpr (NORM && RED == kByRows) {
            // a bucket's tree is a warp's work: lane l on rows 4l .. 4l + 3 of it (at most 128), zeros beyond
            const uint32_t lane = t & 31u, rpb = a.rows_per_bucket;
            for (uint32_t b = t >> 5; b < a.buckets_per_tile; b += THREADS / 32) {
                float v[4];
#pragma unroll
                for (uint32_t i = 0; i < 4; ++i) v[i] = 4 * lane + i < rpb ? sh.row_sums[b * rpb + 4 * lane + i] : 0.0f;
                float s = __fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3]));
#pragma unroll
                for (uint32_t d = 1; d < 32; d <<= 1) s = __fadd_rn(s, __shfl_xor_sync(0xFFFFFFFFu, s, d));
                if (lane == 0) slot[b] = __float_as_uint(s);
            }
            __syncthreads();
            m = slot[local_bucket];
        } else if constexpr (NORM) {
            // tree over the bucket's warp sums, zero leaves up to four or eight (plain stores: nothing to reset;
            // the slot array is written again two barriers from here)
            constexpr uint32_t kWarps = THREADS / 32;
            static_assert(kWarps == 4 || kWarps == 8, "the tree is written for four or eight warps");     // (no norm of longer buckets)
            const uint32_t wpb = a.rows_per_bucket >> 5, first = local_bucket * wpb;
            float v[kWarps];
#pragma unroll
            for (uint32_t i = 0; i < kWarps; ++i)
                v[i] = (i < wpb && first + i < kWarps) ? __uint_as_float(slot[first + i]) : 0.0f;
            float root = __fadd_rn(__fadd_rn(v[0], v[1]), __fadd_rn(v[2], v[3]));
            if constexpr (kWarps == 8)
                root = __fadd_rn(root, __fadd_rn(__fadd_rn(v[4], v[5]), __fadd_rn(v[6], v[7])));
            m = __float_as_uint(root);
        } else {
            m = slot[local_bucket];
            constexpr uint32_t kUsed = RED == kByRows ? kSlots : THREADS / 32;
            if (t < kUsed) sh.slots[rot == 0 ? 2 : rot - 1][t] = 0u;        // next used by this CTA's tile k + 2
        }
    }
    if (!active) return true;

    float sc = __uint_as_float(m);
    if constexpr (NORM) sc = sc < flush_limit() ? 0.0f : __fsqrt_rn(sc);         // flush decided on the sum
    else if (sc < flush_limit()) sc = 0.0f;
    const uint32_t bucket = tile * a.buckets_per_tile + local_bucket;
    if (scale_writer && (FULL || bucket < a.nbuckets)) wv.scales[bucket] = sc;

    const EncodeScale es = encode_scale<BITS>(sc);
    // Philox blocks of the row: elem_offset / 8 + 4 * row + 0 .. 3, all in the launch's high half
    if constexpr (!NORM && !kEarlyDraw)
        draw_row_blocks_head(wv.blk0_lo + 4u * row, wv.head, c.rk, h);
    if (kPackedRow) widen_row(raw, x);
    uint32_t w[BITS];
    // The encode's arithmetic runs in packed fp32x2 instructions at every width: 14.3 instead of 17.0 - 17.6
    // executed instructions per element (13.6 with the integer form up to seven bits).  With the SM clock at its maximum this gains only at one and two bits
    // (16.6 against 17.2 us per 100 MB gradient at K = 1; from K = 4 on the constant pairs compete with the
    // early draws for registers), but a launch that runs for more than a few tens of milliseconds is held at
    // the board's power limit, where the clock falls until the power fits and fewer instructions per element
    // mean less time: 19.6 against 20.5 us at K = 3, 19.4 against 20.4 us at K = 4, 20.5 against 21.2 us at
    // K = 5, 20.6 against 21.6 us at K = 8 (batched launch, 0.3 s of launches back to back, 1650 - 1720 MHz).
    encode_pack_row_best<BITS>(x, es, h, w);
    const uint64_t word0 = (uint64_t)row * BITS;
    if (FULL || (uint64_t)row * 32 + 32 <= a.n) {
        store_row_words<BITS>(wv.codes, word0, w);
    } else {
        mask_row_words<BITS>(w, (int)(a.n - (uint64_t)row * 32) * BITS);
#pragma unroll
        for (int j = 0; j < BITS; ++j)
            if (word0 + j < a.ncode_words) wv.codes[word0 + j] = w[j];
    }
    return true;
}

// The same tile for the (min, max) nearest-rounding variant: two reductions instead of one, two
// floats per bucket (ranges[2b] = lo, ranges[2b + 1] = hi), no random draws.  Padding must not
// take part in the range: the elements a ragged row lacks repeat its first element, and threads
// without a row contribute the identities.  sh.slots holds maxima, sh.slots_lo minima, both as
// ordered bits; the kernel initialises them to the identities.
template <int BITS, int DTYPE, int THREADS, bool FULL, int RED, bool RAGGED, typename Shared, typename Refill>
__device__ __forceinline__ bool range_quantize_tile(Shared& sh, const WorkerView wv,
                                                    const QuantizeArgs& a, const TmaQuantizeConsts& c, uint32_t k,
                                                    uint32_t rot, uint32_t tile, Refill&& refill, uint32_t local_bucket,
                                                    bool scale_writer)
{
    constexpr int kQuantStages = Shared::kStages;
    constexpr bool SHUFFLE = RED == kByShuffle;
    const uint32_t t = threadIdx.x;
    const uint32_t row = tile * a.tile_rows + t;
    const bool active = FULL || (t < a.tile_rows && row < (uint32_t)a.nrows);
    const bool tail = RAGGED && !FULL && tile == c.ragged_tile;  // a tile with a row that the copy does not cover
    const uint32_t stg = k % kQuantStages, parity = (k / kQuantStages) & 1;
    const uint32_t bar = smem_u32(&sh.bar[stg]);
    uint8_t* stage = sh.stage[stg];

    if (tail && warp_has_row(a.nrows_full, row - (t & 31u)))
        fetch_ragged_row(smem_u32(sh.ragged[t >> 5]), static_cast<const uint8_t*>(wv.grad), a.nrows_full,
                         a.n * (DTYPE == 0 ? 4 : 2), DTYPE == 0 ? 128 : 64);
    bool ok = mbar_try_wait(bar, parity);
    if (!ok) ok = mbar_wait(bar, parity, a.poll_limit);
    if (tail && warp_has_row(a.nrows_full, row - (t & 31u)))
        put_ragged_row(stage, (uint32_t)a.nrows_full - tile * a.tile_rows, sh.ragged[t >> 5], DTYPE == 0 ? 128 : 64);

    float x[32];
    uint32_t mlo = kOrderedMinIdentity, mhi = kOrderedMaxIdentity;
    if (active) {
        read_row_swizzled<DTYPE>(stage, (int)t, x);
        if (!FULL) {
            const uint64_t left = a.n - (uint64_t)row * 32;      // >= 1
#pragma unroll
            for (int j = 1; j < 32; ++j) x[j] = ((uint64_t)j < left) ? x[j] : x[0];
        }
        float lo, hi;
        row_min_max(x, lo, hi);
        mlo = ordered_bits(lo); mhi = ordered_bits(hi);
    }
    uint32_t* slot_hi = sh.slots[rot];       // rot = k % 3
    uint32_t* slot_lo = sh.slots_lo[rot];
    if (SHUFFLE) {
        for (uint32_t d = a.rows_per_bucket >> 1; d > 0; d >>= 1) {
            mlo = min(mlo, __shfl_xor_sync(0xFFFFFFFFu, mlo, d));
            mhi = max(mhi, __shfl_xor_sync(0xFFFFFFFFu, mhi, d));
        }
    } else if (RED == kByRows) {
        if (active) { atomicMin(&slot_lo[local_bucket], mlo); atomicMax(&slot_hi[local_bucket], mhi); }
    } else {
        mlo = __reduce_min_sync(0xFFFFFFFFu, mlo);
        mhi = __reduce_max_sync(0xFFFFFFFFu, mhi);
        if ((t & 31) == 0) { atomicMin(&slot_lo[local_bucket], mlo); atomicMax(&slot_hi[local_bucket], mhi); }
    }
    if (__syncthreads_or(!ok)) return false;
    if (t == 0) refill(smem_u32(stage), bar);                    // every thread has read the stage
    if (!SHUFFLE) {
        mlo = slot_lo[local_bucket]; mhi = slot_hi[local_bucket];
        if (t < (RED == kByRows ? kSlots : THREADS / 32)) {      // next used by this CTA's tile k + 2
            sh.slots[rot == 0 ? 2 : rot - 1][t] = kOrderedMaxIdentity;
            sh.slots_lo[rot == 0 ? 2 : rot - 1][t] = kOrderedMinIdentity;
        }
    }
    if (!active) return true;

    // a zero of either sign is stored as +0
    const float lo = __fadd_rn(from_ordered_bits(mlo), 0.0f), hi = __fadd_rn(from_ordered_bits(mhi), 0.0f);
    const uint32_t bucket = tile * a.buckets_per_tile + local_bucket;
    if (scale_writer && (FULL || bucket < a.nbuckets))
        reinterpret_cast<float2*>(wv.scales)[bucket] = make_float2(lo, hi);

    const RangeEncodeScale es = range_encode_scale<BITS>(lo, hi);
    uint32_t w[BITS];
    range_encode_pack_row<BITS>(x, es, w);
    const uint64_t word0 = (uint64_t)row * BITS;
    if (FULL || (uint64_t)row * 32 + 32 <= a.n) {
        store_row_words<BITS>(wv.codes, word0, w);
    } else {
        mask_row_words<BITS>(w, (int)(a.n - (uint64_t)row * 32) * BITS);
#pragma unroll
        for (int j = 0; j < BITS; ++j)
            if (word0 + j < a.ncode_words) wv.codes[word0 + j] = w[j];
    }
    return true;
}

// MODE: kMaxAbs = the main codec, kRange = the (min, max) variant, kNorm = the L2-norm scale variant.  (Rows of 64 bf16
// elements below exist for the main codec only: the variants' long bf16 launches were not tried with them.)

// ---------------------------------------------------------------------------------------
// bf16 gradients long enough to fill the device: a thread owns 64 consecutive elements, 128 bytes of the stage as in
// fp32, and keeps them packed until their half is encoded.  About a third of the executed instructions of a row are
// the tile's bookkeeping (waits, barrier, reduction, division, addresses), and they are paid once per 64 elements
// here instead of once per 32.  (122 to 128 registers left to itself: four CTAs per SM, 28.3 us per 50 M elements at
// K = 4; held to 102, five CTAs, 27.8 us; to 85, six CTAs, 29.5 us; rows of 32 29.8 us.)
// ---------------------------------------------------------------------------------------
template <int BITS, int THREADS, bool FULL, int RED, bool RAGGED, typename Shared, typename Refill>
__device__ __forceinline__ bool quantize_wide_tile(Shared& sh, const WorkerView wv,
                                                   const QuantizeArgs& a, const TmaQuantizeConsts& c, uint32_t k,
                                                   uint32_t rot, uint32_t tile, Refill&& refill, uint32_t local_bucket,
                                                   bool scale_writer)
{
    constexpr int kQuantStages = Shared::kStages;
    const uint32_t t = threadIdx.x;
    const uint32_t row = tile * a.tile_rows + t;
    const bool active = FULL || (t < a.tile_rows && row < (uint32_t)a.nrows);
    const uint32_t stg = k % kQuantStages, parity = (k / kQuantStages) & 1;
    const uint32_t bar = smem_u32(&sh.bar[stg]);
    uint8_t* stage = sh.stage[stg];

    bool ok = mbar_try_wait(bar, parity);
    if (!ok) ok = mbar_wait(bar, parity, a.poll_limit);

    uint32_t raw[2][16];
    if (active) {
        if (RAGGED && !FULL && row >= (uint32_t)a.nrows_full)      // a row that the copy does not cover
            stage_ragged_row(stage, t, static_cast<const uint8_t*>(wv.grad), row, a.n * 2);
        const uint4* s = reinterpret_cast<const uint4*>(stage);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint4 v = s[swz((int)t, i)];
            uint32_t* to = &raw[i >> 2][(i & 3) * 4];
            to[0] = v.x; to[1] = v.y; to[2] = v.z; to[3] = v.w;
        }
    } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) raw[0][j] = raw[1][j] = 0u;
    }
    uint32_t m = __float_as_uint(fmaxf(row_abs_max_bf16(raw[0]), row_abs_max_bf16(raw[1])));
    uint32_t* slot = sh.slots[rot];          // rot = k % 3
    if (RED == kByShuffle) {
        for (uint32_t d = a.rows_per_bucket >> 1; d > 0; d >>= 1) m = max(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
    } else if (RED == kByRows) {
        if (active) atomicMax(&slot[local_bucket], m);
    } else {
        m = __reduce_max_sync(0xFFFFFFFFu, m);
        if ((t & 31) == 0) atomicMax(&slot[local_bucket], m);
    }
    if (__syncthreads_or(!ok)) return false;
    if (t == 0) refill(smem_u32(stage), bar);                    // every thread has read the stage
    if (RED != kByShuffle) {
        m = slot[local_bucket];
        constexpr uint32_t kUsed = RED == kByRows ? kSlots : THREADS / 32;
        if (t < kUsed) sh.slots[rot == 0 ? 2 : rot - 1][t] = 0u;        // next used by this CTA's tile k + 2
    }
    if (!active) return true;

    float sc = __uint_as_float(m);
    if (sc < flush_limit()) sc = 0.0f;
    const uint32_t bucket = tile * a.buckets_per_tile + local_bucket;
    if (scale_writer && (FULL || bucket < a.nbuckets)) wv.scales[bucket] = sc;
    const EncodeScale es = encode_scale<BITS>(sc);
    uint32_t w[2 * BITS];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
        float x[32];
        uint32_t h[16], wh[BITS];
        draw_row_blocks_head(wv.blk0_lo + 8u * row + 4u * half, wv.head, c.rk, h);
        widen_row(raw[half], x);
        encode_pack_row_best<BITS>(x, es, h, wh);
#pragma unroll
        for (int j = 0; j < BITS; ++j) w[half * BITS + j] = wh[j];
    }
    const uint64_t word0 = (uint64_t)row * (2 * BITS);
    if (FULL || (uint64_t)row * 64 + 64 <= a.n) {
        store_row_words<2 * BITS>(wv.codes, word0, w);
    } else {
        mask_row_words<2 * BITS>(w, (int)(a.n - (uint64_t)row * 64) * BITS);
#pragma unroll
        for (int j = 0; j < 2 * BITS; ++j)
            if (word0 + j < a.ncode_words) wv.codes[word0 + j] = w[j];
    }
    return true;
}

// One tile in the given mode.
template <int BITS, int DTYPE, int THREADS, bool FULL, int RED, int MODE, bool RAGGED, typename Shared, typename Refill>
__device__ __forceinline__ bool mode_tile(Shared& sh, const WorkerView& wv, const QuantizeArgs& a,
                                          const TmaQuantizeConsts& c, uint32_t k, uint32_t rot, uint32_t tile,
                                          Refill&& refill, uint32_t local_bucket, bool scale_writer)
{
    if constexpr (DTYPE == kBf16Wide)
        return quantize_wide_tile<BITS, THREADS, FULL, RED, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket, scale_writer);
    else if constexpr (MODE == kRange)
        return range_quantize_tile<BITS, DTYPE, THREADS, FULL, RED, RAGGED>(sh, wv, a, c, k, rot, tile, refill, local_bucket,
                                                                    scale_writer);
    else
        return quantize_tile<BITS, DTYPE, THREADS, FULL, RED, RAGGED, MODE == kNorm>(sh, wv, a, c, k, rot, tile, refill,
                                                                             local_bucket, scale_writer);
}

// First contents of a CTA's slots: the identities of the reductions.
template <int DTYPE, int THREADS, typename Shared>
__device__ __forceinline__ void init_slots(Shared& sh)
{
    for (uint32_t i = threadIdx.x; i < 3u * kSlots; i += THREADS) {
        (&sh.slots[0][0])[i] = 0u;         // = kOrderedMaxIdentity
        (&sh.slots_lo[0][0])[i] = kOrderedMinIdentity;
    }
}

// Host side, shared by the launchers of mqg_quantize.cu and mqg_quantize_workers.cu.
bool tma_path_applies(uint64_t n, uint64_t rpb, uint64_t elem_offset);
uint64_t fill_args(QuantizeArgs& a, const void* grad, uint64_t n, int bits, uint64_t bucket, uint64_t seed,
                   uint32_t* codes, float* scales, uint32_t worker, uint32_t step, uint64_t elem_offset,
                   uint32_t row_elems = 32);
// Whether the launch (all workers' n together: total) takes rows of 64 bf16 elements.
bool bf16_wide_applies(uint64_t n, uint64_t total, uint64_t bucket, int dtype);
int fill_tma_args(QuantizeArgs& a, TmaQuantizeConsts& c, uint64_t rpb);
inline uint32_t box_rows(const QuantizeArgs& a) { return a.tile_rows <= 256 ? a.tile_rows : a.tile_rows / 2; }
inline int reduction_of(uint64_t rpb)
{
    return (rpb & (rpb - 1)) == 0 && rpb <= 32 ? kByShuffle : rpb % 32 == 0 ? kByWarps : kByRows;
}

}  // namespace mqg
