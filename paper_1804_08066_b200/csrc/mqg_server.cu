// Server side: unpack + de-quantize the W workers' buffers, sum them in worker order and apply
// the SGD update, in one pass (De-quantize, sum and update of Algorithm 1,
// ReceiveQGThenSendQG / steps 6-7 of Fig. 3).
//
// The bulk-copy kernel of mqg_server_tma.cu takes the shapes it can; the direct kernel here takes the others
// (long ones the row kernel): any bucket, any number of workers, gradients of less than four tiles, segments that start anywhere, the
// sum as an extra output.  A thread owns 8 consecutive elements, so that its codes are K whole bytes of every
// worker's stream, and requests everything it needs - parameters, code words of eight workers at a time -
// before it uses any of it: a launch on a short gradient is one round trip to memory and a short chain of
// arithmetic.
#include "mqg_segments.cuh"
#include "mqg_tma.cuh"

namespace mqg {

constexpr int kDirectThreads = 256;
constexpr int kDirectElems = 8;                                   // per thread
constexpr int kDirectBlocksPerTile = kMaxTileRows * 32 / (kDirectThreads * kDirectElems);   // per segment tile

struct DirectArgs {
    WorkerPtrs ptrs;         // RANGE: scales[w] = worker w's (lo, hi) pairs
    float* params;           // may be null (accumulate only)
    float* acc;              // may be null when params is given
    uint64_t n, ncode_words;
    uint32_t rows_per_bucket;
    int rpb_shift;           // log2(rows_per_bucket) if a power of two, else -1
    int scale_base;          // segments: index of the table's first segment in scales[]
    int W;
    int add_into;            // the sum continues from acc
    int warp_in_bucket;      // every warp's elements lie in one bucket
    float neg_lr;
};

// Eight floats at p, of which `left` (>= 1) exist.
__device__ __forceinline__ void load8(const float* p, uint64_t left, float2 (&v)[4])
{
    if (left >= 8 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
        const float4 lo = __ldcg(reinterpret_cast<const float4*>(p)), hi = __ldcg(reinterpret_cast<const float4*>(p) + 1);
        v[0] = make_float2(lo.x, lo.y); v[1] = make_float2(lo.z, lo.w);
        v[2] = make_float2(hi.x, hi.y); v[3] = make_float2(hi.z, hi.w);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            v[j].x = 2 * j < left ? __ldcg(p + 2 * j) : 0.0f;
            v[j].y = 2 * j + 1 < left ? __ldcg(p + 2 * j + 1) : 0.0f;
        }
    }
}

__device__ __forceinline__ void store8(float* p, uint64_t left, const float2 (&v)[4])
{
    if (left >= 8 && (reinterpret_cast<uintptr_t>(p) & 15u) == 0) {
        reinterpret_cast<float4*>(p)[0] = make_float4(v[0].x, v[0].y, v[1].x, v[1].y);
        reinterpret_cast<float4*>(p)[1] = make_float4(v[2].x, v[2].y, v[3].x, v[3].y);
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (2 * j < left) p[2 * j] = v[j].x;
            if (2 * j + 1 < left) p[2 * j + 1] = v[j].y;
        }
    }
}

// v <- v + the eight de-quantized codes that start `shift` bits into words[].
template <int BITS, bool RANGE, int WORDS>
__device__ __forceinline__ void add_decoded8(const uint32_t (&words)[WORDS], uint32_t shift, const DecodeScale& d,
                                             float2 (&v)[4])
{
    constexpr uint32_t kMask = (1u << BITS) - 1u, kTwo23 = 0x4B000000u;
    uint32_t win[2];                                              // the 8 K bits from bit 0 on
    win[0] = WORDS > 1 ? __funnelshift_r(words[0], words[WORDS > 1 ? 1 : 0], shift) : words[0] >> shift;
    win[1] = WORDS > 2 ? __funnelshift_r(words[1], words[WORDS > 2 ? 2 : 0], shift)
                       : WORDS > 1 ? words[WORDS > 1 ? 1 : 0] >> shift : 0u;
    if constexpr (BITS == 1 && !RANGE) {
#pragma unroll
        for (int p = 0; p < 4; ++p)
            v[p] = __fadd2_rn(v[p], make_float2(one_bit_value(d.minus_h, win[0] << (31 - 2 * p)),
                                                one_bit_value(d.minus_h, win[0] << (30 - 2 * p))));
    } else {
        const float2 th = make_float2(d.two_h, d.two_h), mh = make_float2(d.minus_h, d.minus_h);
        auto code = [&](int j) -> float {                             // the float 2^23 + q of code j
            const int o = j * BITS;
            const uint32_t q = o + BITS <= 32 ? win[0] >> o : o >= 32 ? win[1] >> (o - 32)
                                                                      : __funnelshift_r(win[0], win[1], o);
            return __uint_as_float((q & kMask) | kTwo23);
        };
#pragma unroll
        for (int p = 0; p < 4; ++p)
            v[p] = accumulate2<BITS, RANGE>(v[p], make_float2(code(2 * p), code(2 * p + 1)), th, mh);
    }
}

// SEG: tiles come from a segment table (one scale per segment) instead of uniform buckets.
// A launch is bound by its latency: at n = 2^20 and four workers it moves 10 MB in one wave of
// resident threads.
template <int BITS, bool RANGE, bool SEG>
__global__ void __launch_bounds__(kDirectThreads)
server_direct_kernel(const __grid_constant__ DirectArgs a, const __grid_constant__ SegmentTable tab)
{
    // words that hold K bytes which start at any byte of the first one (K = 1, 2, 4, 8: inside one / two words)
    constexpr int kWords = BITS == 1 || BITS == 2 || BITS == 4 ? 1 : BITS == 7 ? 3 : 2;
    constexpr int kBatch = 8;
    grid_dependency_wait();

    // threads beyond the end keep going with clamped addresses: the warp's shuffles need them
    uint64_t elem0, left, byte0, words_end, scale_idx;
    bool active;
    if constexpr (SEG) {
        const TileGeom g = locate_tile<BITS>(tab, blockIdx.x / kDirectBlocksPerTile);
        const uint32_t local = (blockIdx.x % kDirectBlocksPerTile) * kDirectThreads + threadIdx.x;
        active = (uint64_t)local * kDirectElems < g.valid;
        elem0 = g.elem0 + (uint64_t)local * kDirectElems;
        left = active ? g.valid - (uint64_t)local * kDirectElems : 0;
        byte0 = g.word0 * 4 + (uint64_t)local * BITS;
        words_end = g.words_end;
        scale_idx = (uint64_t)a.scale_base + g.seg;
    } else {
        const uint64_t unit = (uint64_t)blockIdx.x * kDirectThreads + threadIdx.x;
        elem0 = unit * kDirectElems;
        active = elem0 < a.n;
        left = active ? a.n - elem0 : 0;
        byte0 = unit * BITS;
        words_end = a.ncode_words;
        const uint64_t row = (active ? unit : (a.n - 1) / kDirectElems) >> 2;
        scale_idx = a.rpb_shift >= 0 ? row >> a.rpb_shift : row / a.rows_per_bucket;
    }
    const uint64_t word0 = byte0 >> 2;
    const uint32_t shift = ((uint32_t)byte0 & 3u) * 8u, lane = threadIdx.x & 31u;

    float2 p[4], v[4];
    if (a.params != nullptr) load8(a.params + elem0, left, p);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = make_float2(0.0f, 0.0f);
    if (a.add_into) {
        load8(a.acc + elem0, left, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = make_float2(sum_start<BITS, RANGE>(v[j].x), sum_start<BITS, RANGE>(v[j].y));
    }

    auto load_scale = [&](int w) -> float2 {
        if (RANGE) return __ldcg(reinterpret_cast<const float2*>(a.ptrs.scales[w]) + scale_idx);
        return make_float2(__ldcg(a.ptrs.scales[w] + scale_idx), 0.0f);
    };
    auto constants = [](float2 s) { return RANGE ? range_decode_scale<BITS>(s.x, s.y) : decode_scale<BITS>(s.x); };
    // A warp's 256 elements that lie in one bucket share the bucket's constants: lane w divides for worker w.
    DecodeScale mine = {0.0f, 0.0f};
    if (SEG || a.warp_in_bucket) {
        const float2 s = load_scale((int)lane < a.W ? (int)lane : a.W - 1);
        mine = constants(s);
    }

#pragma unroll 1
    for (int w0 = 0; w0 < a.W; w0 += kBatch) {
        uint32_t cw[kBatch][kWords];
        const int many = min(kBatch, a.W - w0);
#pragma unroll
        for (int i = 0; i < kBatch; ++i)
#pragma unroll
            for (int k = 0; k < kWords; ++k)
                cw[i][k] = i < many && word0 + k < words_end ? __ldcg(a.ptrs.codes[w0 + i] + word0 + k) : 0u;
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (i < many) {
                DecodeScale d;
                if (SEG || a.warp_in_bucket) {
                    d.two_h = __shfl_sync(0xFFFFFFFFu, mine.two_h, w0 + i);
                    d.minus_h = __shfl_sync(0xFFFFFFFFu, mine.minus_h, w0 + i);
                } else {
                    d = constants(load_scale(w0 + i));
                }
                add_decoded8<BITS, RANGE>(cw[i], shift, d, v);
            }
        }
    }
    if (!active) return;
    if (a.acc != nullptr) store8(a.acc + elem0, left, v);
    if (a.params != nullptr) {
        const float2 nlr = make_float2(a.neg_lr, a.neg_lr);
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = __ffma2_rn(nlr, v[j], p[j]);
        store8(a.params + elem0, left, p);
    }
}

struct ServerArgs {
    WorkerPtrs ptrs;
    float* params;           // may be null (accumulate only)
    float* acc;              // may be null when params != null
    uint64_t n, nrows, ncode_words;
    uint32_t rows_per_bucket;
    int W;
    int add_into;
    float neg_lr;
};

// Sum of the W de-quantized rows in worker order, continuing from v[] when have_init.
template <int BITS, bool RANGE>
__device__ __forceinline__ void accumulate_row(const ServerArgs& a, uint64_t scale_idx,
                                               uint64_t word0, uint64_t words_end, bool full_row,
                                               float (&v)[32], bool have_init)
{
    float2 v2[16];
    if (have_init) pairs_from_floats(v, v2);
    else {
#pragma unroll
        for (int p = 0; p < 16; ++p) v2[p] = make_float2(0.0f, 0.0f);
    }
    // four workers at a time: their code words and scales are all requested before the first one is
    // decoded, so that a row waits for global memory once per four workers, not once per worker
    constexpr int kBatch = 4;
    for (int w0 = 0; w0 < a.W; w0 += kBatch) {
        uint32_t w[kBatch][BITS];
        float2 sc[kBatch];
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            const int wk = min(w0 + i, a.W - 1);            // a worker past the last one repeats it (not summed)
            if (full_row) load_row_words<BITS>(a.ptrs.codes[wk], word0, w[i]);
            else {
#pragma unroll
                for (int k = 0; k < BITS; ++k)
                    w[i][k] = (word0 + k < words_end) ? __ldg(a.ptrs.codes[wk] + word0 + k) : 0u;
            }
            if (RANGE) sc[i] = __ldg(reinterpret_cast<const float2*>(a.ptrs.scales[wk]) + scale_idx);
            else sc[i] = make_float2(__ldg(a.ptrs.scales[wk] + scale_idx), 0.0f);
        }
#pragma unroll
        for (int i = 0; i < kBatch; ++i) {
            if (w0 + i < a.W) {
                const DecodeScale d = RANGE ? range_decode_scale<BITS>(sc[i].x, sc[i].y) : decode_scale<BITS>(sc[i].x);
                add_decoded_row<BITS, RANGE>(w[i], widen(d), v2);
            }
        }
    }
    floats_from_pairs(v2, v);
}

// The row kernel, for long gradients in shapes the bulk-copy kernel does not take: a thread owns a row of 32
// elements, whose parameters move through a swizzled shared-memory tile.  Fewer instructions per element than
// the direct kernel, a longer chain per thread.
// MODE 0: acc = sum (optionally continuing from acc).  MODE 1: params update, acc optional.
template <int BITS, int MODE, bool RANGE>
__global__ void __launch_bounds__(kMaxTileRows)
server_row_kernel(const __grid_constant__ ServerArgs a)
{
    __shared__ __align__(1024) float4 tile[kMaxTileRows * 8];

    const uint32_t t = threadIdx.x;
    grid_dependency_wait();
    const uint64_t row0 = (uint64_t)blockIdx.x * kMaxTileRows;
    const uint64_t rows_left = a.nrows - row0;
    const int rows = (int)(rows_left < (uint64_t)kMaxTileRows ? rows_left : (uint64_t)kMaxTileRows);
    const uint64_t elem0 = row0 * 32, valid = a.n - elem0;
    const uint64_t word0 = (row0 + t) * BITS, words_end = a.ncode_words;
    const uint64_t scale_idx = (row0 + t) / a.rows_per_bucket;
    const bool active = t < (uint32_t)rows;
    const bool full_row = 32ull * t + 32 <= valid;

    float v[32];
    if constexpr (MODE == 0) {
        float* acc = a.acc + elem0;
        if (a.add_into) {
            load_tile_f32<kMaxTileRows>(tile, acc, valid, rows);
            __syncthreads();
            if (active) read_row(tile, (int)t, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = sum_start<BITS, RANGE>(v[j]);
        }
        if (active) {
            accumulate_row<BITS, RANGE>(a, scale_idx, word0, words_end, full_row, v, a.add_into != 0);
            write_row(tile, (int)t, v);
        }
        __syncthreads();
        store_tile_f32<kMaxTileRows>(tile, acc, valid, rows);
    } else {
        float* params = a.params + elem0;
        load_tile_f32<kMaxTileRows, false>(tile, params, valid, rows);    // in flight during the decode
        if (active) accumulate_row<BITS, RANGE>(a, scale_idx, word0, words_end, full_row, v, false);
        cp_async_wait_all();
        __syncthreads();
        if (active) {
            float p[32];
            read_row(tile, (int)t, p);
            const float nlr = a.neg_lr;
#pragma unroll
            for (int j = 0; j < 32; ++j) p[j] = __fmaf_rn(nlr, v[j], p[j]);
            write_row(tile, (int)t, p);
        }
        __syncthreads();
        store_tile_f32<kMaxTileRows>(tile, params, valid, rows);
        if (a.acc != nullptr) {
            __syncthreads();
            if (active) write_row(tile, (int)t, v);
            __syncthreads();
            store_tile_f32<kMaxTileRows>(tile, a.acc + elem0, valid, rows);
        }
    }
}

__global__ void __launch_bounds__(256)
apply_kernel(float* __restrict__ params, const float* __restrict__ acc, float lr, uint64_t n)
{
    const float nlr = -lr;
    const uint64_t n4 = n / 4;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    grid_dependency_wait();
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += stride) {
        float4 p = __ldcg(reinterpret_cast<const float4*>(params) + i);
        const float4 g = __ldcs(reinterpret_cast<const float4*>(acc) + i);
        p.x = __fmaf_rn(nlr, g.x, p.x);
        p.y = __fmaf_rn(nlr, g.y, p.y);
        p.z = __fmaf_rn(nlr, g.z, p.z);
        p.w = __fmaf_rn(nlr, g.w, p.w);
        reinterpret_cast<float4*>(params)[i] = p;
    }
    if (blockIdx.x == 0 && threadIdx.x < (n & 3)) {
        const uint64_t i = n4 * 4 + threadIdx.x;
        params[i] = __fmaf_rn(nlr, __ldcg(acc + i), __ldcg(params + i));
    }
}

template <bool RANGE, bool SEG>
static cudaError_t launch_direct(int bits, const DirectArgs& a, const SegmentTable& tab, uint64_t blocks,
                                 cudaStream_t stream)
{
    if (blocks == 0) return cudaSuccess;
    if (blocks > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)blocks;
    switch (bits) {
#define MQG_DIRECT_CASE(B) \
        case B: return launch_pdl(server_direct_kernel<B, RANGE, SEG>, grid, kDirectThreads, stream, a, tab)
        MQG_DIRECT_CASE(1); MQG_DIRECT_CASE(2); MQG_DIRECT_CASE(3); MQG_DIRECT_CASE(4);
        MQG_DIRECT_CASE(5); MQG_DIRECT_CASE(6); MQG_DIRECT_CASE(7); MQG_DIRECT_CASE(8);
#undef MQG_DIRECT_CASE
    }
    return cudaErrorInvalidValue;
}

// Whether every warp of the direct kernel works inside one bucket.
static bool warp_in_one_bucket(uint64_t n, uint64_t bucket) { return bucket >= n || bucket % (32 * kDirectElems) == 0; }

template <bool RANGE>
static cudaError_t server_direct(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket, float* params,
                                 float lr, float* acc, int add_into, cudaStream_t stream)
{
    DirectArgs a;
    a.ptrs = ptrs;
    a.params = params; a.acc = acc;
    a.n = n;
    a.ncode_words = (n * (uint64_t)bits + 31) / 32;
    // bucket % 32 == 0, or a single bucket (bucket >= n): every row lies in one bucket
    const uint64_t nrows = (n + 31) / 32, rpb = bucket >= n ? nrows : bucket / 32;
    a.rows_per_bucket = (uint32_t)(rpb > 0xFFFFFFFFull ? 0xFFFFFFFFull : rpb);
    a.rpb_shift = -1;
    for (int s = 0; s < 32; ++s)
        if ((1ull << s) == rpb) a.rpb_shift = s;
    a.scale_base = 0;
    a.W = W; a.add_into = add_into; a.neg_lr = -lr;
    a.warp_in_bucket = warp_in_one_bucket(n, bucket);
    SegmentTable tab;
    tab.nseg = 0; tab.uniform_bucket = 0; tab.n_total = n; tab.tiles_per_bucket = 0;
    const uint64_t per_block = (uint64_t)kDirectThreads * kDirectElems;
    return launch_direct<RANGE, false>(bits, a, tab, (n + per_block - 1) / per_block, stream);
}

// Where the row kernel takes over from the direct one.  Direct / row in us, four bits.  Several buckets among a warp's 256
// elements (bucket 96; direct divides for every worker and thread): W = 1 4.5 / 4.7, 5.0 / 4.8 for n = 1.5 and 2 * 2^20,
// W = 8 5.8 / 6.1, 8.6 / 7.9 for n = 1 and 1.5 * 2^20, W = 32 12.7 / 14.4, 14.4 / 14.5 for n = 0.5 and 0.75 * 2^20; the
// (min, max) variant within 4 % of that, and at n = 25 M 53 / 41 us with W = 1, 134 / 69 us with W = 8.  One bucket to a
// warp, the sum as an extra output (bucket 2048): W = 1 4.8 / 4.8, 7.2 / 6.2, 12.1 / 10.6 for n = 1, 2 and 4 * 2^20,
// W = 4 11.5 / 12.8 for n = 4 * 2^20, W = 8 4.9 / 7.0, 7.9 / 9.2 for n = 1 and 2 * 2^20.
static bool row_kernel_preferred(uint64_t n, int W, bool warp_in_bucket, bool sum_out)
{
    if (!warp_in_bucket) return n * (uint64_t)(W + 16) >= (27ull << 20);
    return W <= 2 ? n >= (1ull << 21) : !sum_out && n * (uint64_t)(W + 4) >= (1ull << 25);
}

template <bool RANGE>
static cudaError_t server_rows(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket, float* params,
                               float lr, float* acc, int add_into, cudaStream_t stream)
{
    ServerArgs a;
    a.ptrs = ptrs;
    a.params = params; a.acc = acc;
    a.n = n;
    a.nrows = (n + 31) / 32;
    a.ncode_words = (n * (uint64_t)bits + 31) / 32;
    const uint64_t rpb = (bucket >= n) ? a.nrows : bucket / 32;
    a.rows_per_bucket = (uint32_t)(rpb > 0xFFFFFFFFull ? 0xFFFFFFFFull : rpb);
    a.W = W; a.add_into = add_into; a.neg_lr = -lr;
    const uint64_t tiles = (a.nrows + kMaxTileRows - 1) / kMaxTileRows;
    if (tiles > 0x7FFFFFFFull) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)tiles;
    switch (bits) {
#define MQG_ROW_CASE(B) \
        case B: return params == nullptr ? launch_pdl(server_row_kernel<B, 0, RANGE>, grid, kMaxTileRows, stream, a) \
                                         : launch_pdl(server_row_kernel<B, 1, RANGE>, grid, kMaxTileRows, stream, a)
        MQG_ROW_CASE(1); MQG_ROW_CASE(2); MQG_ROW_CASE(3); MQG_ROW_CASE(4);
        MQG_ROW_CASE(5); MQG_ROW_CASE(6); MQG_ROW_CASE(7); MQG_ROW_CASE(8);
#undef MQG_ROW_CASE
    }
    return cudaErrorInvalidValue;
}

// The sum as an extra output of the update: from 2^25 codes on, the bulk-copy kernel for the sum and a pass of
// its own for the update (the same roundings) are faster than the direct kernel although they read the sum
// again: 18 against 20 us at n = 2^22, W = 8, seven bits; 28 against 29 us at n = 2^23, W = 4; no difference at W = 1.
static bool sum_then_apply(uint64_t n, int W, const float* params, const float* acc)
{
    return params != nullptr && acc != nullptr && n * (uint64_t)W >= (1ull << 25);
}

template <bool RANGE>
static cudaError_t server_any(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket, float* params,
                              float lr, float* acc, int add_into, cudaStream_t stream)
{
    const bool split = sum_then_apply(n, W, params, acc);
    if (server_tma_applies(n, bucket, W) && (params == nullptr || acc == nullptr || split)) {
        float* dst = acc != nullptr ? acc : params;
        const int mode = acc == nullptr ? 1 : add_into ? 2 : 0;
        const cudaError_t err = RANGE ? launch_server_range_tma(ptrs, W, bits, n, bucket, dst, lr, mode, stream)
                                      : launch_server_tma(ptrs, W, bits, n, bucket, dst, lr, mode, stream);
        return err == cudaSuccess && split ? launch_apply(params, acc, lr, n, stream) : err;
    }
    if (row_kernel_preferred(n, W, warp_in_one_bucket(n, bucket), params != nullptr && acc != nullptr))
        return server_rows<RANGE>(ptrs, W, bits, n, bucket, params, lr, acc, add_into, stream);
    return server_direct<RANGE>(ptrs, W, bits, n, bucket, params, lr, acc, add_into, stream);
}

cudaError_t launch_server(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                          float* params, float lr, float* acc, int add_into, cudaStream_t stream)
{
    return server_any<false>(ptrs, W, bits, n, bucket, params, lr, acc, add_into, stream);
}

cudaError_t launch_server_range(const WorkerPtrs& ptrs, int W, int bits, uint64_t n, uint64_t bucket,
                                float* params, float lr, float* acc, int add_into, cudaStream_t stream)
{
    return server_any<true>(ptrs, W, bits, n, bucket, params, lr, acc, add_into, stream);
}

cudaError_t launch_server_segments(const WorkerPtrs& ptrs, int W, int bits, const SegmentTable& tab,
                                   int scale_base, float* params, float lr, float* acc,
                                   cudaStream_t stream)
{
    DirectArgs a;
    a.ptrs = ptrs;
    a.params = params; a.acc = acc;
    a.n = 0; a.ncode_words = 0; a.rows_per_bucket = 1; a.rpb_shift = 0;
    a.scale_base = scale_base;
    a.W = W; a.add_into = 0; a.neg_lr = -lr;
    a.warp_in_bucket = 1;
    return launch_direct<false, true>(bits, a, tab, (uint64_t)tab.tile_start[tab.nseg] * kDirectBlocksPerTile, stream);
}

cudaError_t launch_apply(float* params, const float* acc, float lr, uint64_t n, cudaStream_t stream)
{
    const uint64_t n4 = n / 4;
    uint64_t blocks = (n4 + 255) / 256;
    if (blocks < 1) blocks = 1;
    int dev = 0, sms = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err == cudaSuccess) err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    if (blocks > (uint64_t)sms * 16) blocks = (uint64_t)sms * 16;
    return launch_pdl(apply_kernel, (unsigned)blocks, 256, stream, params, acc, lr, n);
}

}  // namespace mqg
