// C ABI of libmqgrad: argument checks, dispatch to the kernel launchers, error reporting.
#include <cstdarg>
#include <cstdio>
#include <cstring>

#include "../../include/mqgrad.h"
#include "mqg_common.cuh"
#include "mqg_internal.h"
#include "mqg_tma.cuh"

namespace {

thread_local char g_err[256] = "";

mqg_status fail(mqg_status code, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

mqg_status cuda_fail(const char* what, cudaError_t err)
{
    return fail(MQG_ERR_CUDA, "%s: %s", what, cudaGetErrorString(err));
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
bool aligned4(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 3u) == 0; }
bool aligned8(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 7u) == 0; }

mqg_status check_bits(int bits)
{
    if (bits < 1 || bits > 8) return fail(MQG_ERR_BITS, "bits = %d is outside 1..8", bits);
    return MQG_OK;
}

mqg_status check_bucket(uint64_t n, uint64_t bucket)
{
    if (bucket == 0) return fail(MQG_ERR_INVALID, "bucket must be >= 1");
    if (bucket < n && bucket % 32 != 0)
        return fail(MQG_ERR_INVALID, "bucket = %llu must be a multiple of 32 (or >= n)",
                    (unsigned long long)bucket);
    return MQG_OK;
}

// With `empty` (nothing to process) only W is checked: the buffers may be null.
mqg_status check_workers(const uint32_t* const* codes, const float* const* scales, int W,
                         bool empty, mqg::WorkerPtrs* out)
{
    if (W < 1 || W > MQG_MAX_WORKERS)
        return fail(MQG_ERR_TOO_MANY_WORKERS, "W = %d is outside 1..%d", W, MQG_MAX_WORKERS);
    if (empty) return MQG_OK;
    if (!codes || !scales) return fail(MQG_ERR_INVALID, "codes / scales pointer table is null");
    for (int w = 0; w < W; ++w) {
        if (!codes[w] || !scales[w])
            return fail(MQG_ERR_INVALID, "worker %d: codes or scales buffer is null", w);
        if (!aligned16(codes[w])) return fail(MQG_ERR_ALIGN, "worker %d: codes not 16-byte aligned", w);
        if (!aligned4(scales[w])) return fail(MQG_ERR_ALIGN, "worker %d: scales not 4-byte aligned", w);
        out->codes[w] = codes[w];
        out->scales[w] = scales[w];
    }
    for (int w = W; w < mqg::kMaxWorkers; ++w) { out->codes[w] = nullptr; out->scales[w] = nullptr; }
    return MQG_OK;
}

uint64_t eff_bucket(uint64_t n, uint64_t bucket) { return bucket < n ? bucket : n; }

// Shapes outside the one-pass kernel, for several workers (few elements, a bucket of an odd number of rows above 128, draws
// off a block boundary): a bucket per CTA, all workers in one launch, where a bucket fills the CTA's warps or there are
// so few of them that one launch instead of W decides.  A launch takes about 3.3 us, a CTA per bucket 5 ns, whatever it
// holds: spans / launches 4.2 / 8.8 us for one bucket of 6581 elements, 7.6 / 8.4 us for 508 buckets of 128, 8.5 / 6.8 us
// for 625 and 22 / 6.8 us for 2032 of 32, all at W = 2; the same ratios at W = 8 and 32.  The (min, max) variant also for
// one worker, which takes four launches otherwise.
bool worker_spans_preferred(uint64_t n, uint64_t bucket)
{
    const uint64_t b = eff_bucket(n, bucket);
    return mqg::bucket_spans_apply(n, bucket) && (b > 4096 || (n < 65536 && n <= 512 * b));
}


mqg_status check_segments(int nseg, const uint64_t* seg_off, const uint64_t* code_off, int bits)
{
    if (nseg < 0) return fail(MQG_ERR_INVALID, "nseg = %d is negative", nseg);
    if (nseg == 0) return MQG_OK;
    if (!seg_off || !code_off) return fail(MQG_ERR_INVALID, "segment table is null");
    for (int j = 0; j < nseg; ++j) {
        if (seg_off[j + 1] < seg_off[j]) return fail(MQG_ERR_INVALID, "seg_off decreases at %d", j);
        const uint64_t len = seg_off[j + 1] - seg_off[j];
        const uint64_t need = (len * (uint64_t)bits + 31) / 32;
        if (code_off[j + 1] < code_off[j] || code_off[j + 1] - code_off[j] < need)
            return fail(MQG_ERR_INVALID, "code_off leaves segment %d fewer than %llu words", j,
                        (unsigned long long)need);
    }
    return MQG_OK;
}

// The per-layer quantizers: max-abs scales (workspace == nullptr), or L2-norm scales of one worker.
mqg_status quantize_segments(const void* const* grads, int W, int nseg, const uint64_t* seg_off, const uint64_t* code_off,
                             int bits, uint64_t seed, uint32_t* const* codes, float* const* scales, mqg_dtype dtype,
                             uint32_t first_worker, uint32_t step, uint64_t elem_offset, float* workspace,
                             cudaStream_t stream, const char* what)
{
    if (mqg_status st = check_segments(nseg, seg_off, code_off, bits)) return st;
    if (nseg == 0) return MQG_OK;
    const cudaError_t err = mqg::launch_quantize_segments(grads, W, nseg, seg_off, code_off, bits, seed, codes, scales,
                                                          (int)dtype, first_worker, step, elem_offset, workspace, stream);
    return err == cudaSuccess ? MQG_OK : cuda_fail(what, err);
}

// Validates a segment table and cuts it into chunks of at most kMaxSegmentsPerLaunch segments;
// calls fn(table, first_segment_index) for each chunk.  Segments for which skip(j) holds get no
// tiles in the tables, exactly like empty segments: another launch takes care of them.  skip is
// only called once the table has been checked.
template <typename Fn, typename Skip>
mqg_status for_each_chunk(int nseg, const uint64_t* seg_off, const uint64_t* code_off, int bits,
                          Fn&& fn, Skip&& skip)
{
    if (mqg_status st = check_segments(nseg, seg_off, code_off, bits)) return st;
    const uint64_t tile_elems = (uint64_t)mqg::kMaxTileRows * 32;
    int j = 0;
    while (j < nseg) {
        mqg::SegmentTable tab;
        std::memset(&tab, 0, sizeof(tab));
        int k = 0;
        uint64_t tiles = 0;
        while (j + k < nseg && k < mqg::kMaxSegmentsPerLaunch) {
            const uint64_t len = seg_off[j + k + 1] - seg_off[j + k];
            const uint64_t t = skip(j + k) ? 0 : (len + tile_elems - 1) / tile_elems;
            if (tiles + t > 0x7FFFFFFFull) break;
            tab.tile_start[k] = (uint32_t)tiles;
            tab.seg_off[k] = seg_off[j + k];
            tab.code_off[k] = code_off[j + k];
            tiles += t;
            ++k;
        }
        if (k == 0) return fail(MQG_ERR_INVALID, "segment %d is too large for one launch", j);
        tab.tile_start[k] = (uint32_t)tiles;
        tab.seg_off[k] = seg_off[j + k];
        tab.nseg = k;
        const mqg_status st = fn(tab, j);
        if (st != MQG_OK) return st;
        j += k;
    }
    return MQG_OK;
}

}  // namespace

int mqg::report_error(int code, const char* fmt, ...)
{
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_err, sizeof(g_err), fmt, ap);
    va_end(ap);
    return code;
}

extern "C" {

size_t mqg_code_words(uint64_t n, int bits) { return (size_t)((n * (uint64_t)bits + 31) / 32); }

size_t mqg_num_buckets(uint64_t n, uint64_t bucket)
{
    return bucket ? (size_t)((n + bucket - 1) / bucket) : 0;
}

size_t mqg_wire_bytes(uint64_t n, int bits, uint64_t bucket)
{
    return 4 * mqg_code_words(n, bits) + 4 * mqg_num_buckets(n, bucket);
}

const char* mqg_last_error(void) { return g_err; }

int mqg_version(void) { return 100; }

mqg_status mqg_device_timeouts(unsigned int* count)
{
    if (!count) return fail(MQG_ERR_INVALID, "count is null");
    const cudaError_t err = mqg::read_wait_timeouts(count);
    if (err != cudaSuccess) return cuda_fail("mqg_device_timeouts", err);
    return MQG_OK;
}

mqg_status mqg_check_timeouts(unsigned int* count, int reset)
{
    unsigned int c = 0;
    const cudaError_t err = mqg::read_wait_timeouts(&c, reset != 0);
    if (err != cudaSuccess) return cuda_fail("mqg_check_timeouts", err);
    if (count) *count = c;
    if (c != 0) return fail(MQG_ERR_TIMEOUT, "%u bounded wait(s) of a kernel ran out on this device", c);
    return MQG_OK;
}

mqg_status mqg_test_wait_override(uint32_t poll_limit, int arm_only)
{
    mqg::set_wait_policy(poll_limit, arm_only != 0 ? 1u : 0u);
    return MQG_OK;
}

mqg_status mqg_quantize(const void* grad, uint64_t n, int bits, uint64_t bucket, uint64_t seed,
                        uint32_t* codes, float* scales, mqg_dtype dtype, uint32_t worker,
                        uint32_t step, uint64_t elem_offset, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (n == 0) return MQG_OK;
    if (!grad || !codes || !scales) return fail(MQG_ERR_INVALID, "grad, codes or scales is null");
    if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
    if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
    if (!aligned4(scales)) return fail(MQG_ERR_ALIGN, "scales not 4-byte aligned");
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const uint64_t eff = bucket < n ? bucket : n;
    cudaError_t err;
    if (eff <= (uint64_t)mqg::kMaxFusedBucket || mqg::quantize_long_fused_applies(n, bucket, elem_offset))
        err = mqg::launch_quantize_fused(grad, n, bits, bucket, seed, codes, scales, (int)dtype,
                                         worker, step, elem_offset, stream);
    else if (mqg::bucket_spans_apply(n, bucket))
        err = mqg::launch_bucket_spans(&grad, 1, n, bits, bucket, seed, &codes, &scales, 0, (int)dtype, worker, step,
                                       elem_offset, stream);
    else
        err = mqg::launch_quantize_big_buckets(grad, n, bits, bucket, seed, codes, scales, (int)dtype,
                                               worker, step, elem_offset, stream);
    if (err != cudaSuccess) return cuda_fail("mqg_quantize", err);
    return MQG_OK;
}

mqg_status mqg_quantize_workers(const void* const* grads, int W, uint64_t n, int bits, uint64_t bucket,
                                uint64_t seed, uint32_t* const* codes, float* const* scales,
                                mqg_dtype dtype, uint32_t first_worker, uint32_t step,
                                uint64_t elem_offset, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (W < 1 || W > MQG_MAX_WORKERS)
        return fail(MQG_ERR_TOO_MANY_WORKERS, "W = %d outside 1..%d", W, MQG_MAX_WORKERS);
    if (n == 0) return MQG_OK;
    if (!grads || !codes || !scales) return fail(MQG_ERR_INVALID, "grads, codes or scales is null");
    for (int w = 0; w < W; ++w) {
        if (!grads[w] || !codes[w] || !scales[w])
            return fail(MQG_ERR_INVALID, "worker %d: grad, codes or scales is null", w);
        if (!aligned16(grads[w])) return fail(MQG_ERR_ALIGN, "worker %d: grad not 16-byte aligned", w);
        if (!aligned16(codes[w])) return fail(MQG_ERR_ALIGN, "worker %d: codes not 16-byte aligned", w);
        if (!aligned4(scales[w])) return fail(MQG_ERR_ALIGN, "worker %d: scales not 4-byte aligned", w);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (mqg::quantize_workers_applies(W, n, bucket, elem_offset, 0)) {
        const cudaError_t err = mqg::launch_quantize_workers(grads, W, n, bits, bucket, seed, codes, scales,
                                                             (int)dtype, first_worker, step, elem_offset,
                                                             0, stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers", err);
        return MQG_OK;
    }
    if (W > 1 && worker_spans_preferred(n, bucket)) {
        const cudaError_t err = mqg::launch_bucket_spans(grads, W, n, bits, bucket, seed, codes, scales, 0, (int)dtype,
                                                         first_worker, step, elem_offset, stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers", err);
        return MQG_OK;
    }
    // shapes the batched kernels do not take: one launch per worker, same results
    for (int w = 0; w < W; ++w) {
        const mqg_status st = mqg_quantize(grads[w], n, bits, bucket, seed, codes[w], scales[w], dtype,
                                           first_worker + (uint32_t)w, step, elem_offset, cuda_stream);
        if (st != MQG_OK) return st;
    }
    return MQG_OK;
}

mqg_status mqg_quantize_minmax(const void* grad, uint64_t n, int bits, uint64_t bucket, uint32_t* codes,
                               float* ranges, mqg_dtype dtype, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (n == 0) return MQG_OK;
    if (!grad || !codes || !ranges) return fail(MQG_ERR_INVALID, "grad, codes or ranges is null");
    if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
    if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
    if (!aligned8(ranges)) return fail(MQG_ERR_ALIGN, "ranges not 8-byte aligned");
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    const cudaError_t err = mqg::quantize_range_fused_applies(n, bucket)
        ? mqg::launch_quantize_range_fused(grad, n, bits, bucket, codes, ranges, (int)dtype, stream)
        : worker_spans_preferred(n, bucket)
        ? mqg::launch_bucket_spans(&grad, 1, n, bits, bucket, 0, &codes, &ranges, 1, (int)dtype, 0, 0, 0, stream)
        : mqg::launch_quantize_range_general(grad, n, bits, bucket, codes, ranges, (int)dtype, stream);
    if (err != cudaSuccess) return cuda_fail("mqg_quantize_minmax", err);
    return MQG_OK;
}

mqg_status mqg_quantize_workers_minmax(const void* const* grads, int W, uint64_t n, int bits, uint64_t bucket,
                                       uint32_t* const* codes, float* const* ranges, mqg_dtype dtype,
                                       void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (W < 1 || W > MQG_MAX_WORKERS)
        return fail(MQG_ERR_TOO_MANY_WORKERS, "W = %d outside 1..%d", W, MQG_MAX_WORKERS);
    if (n == 0) return MQG_OK;
    if (!grads || !codes || !ranges) return fail(MQG_ERR_INVALID, "grads, codes or ranges is null");
    for (int w = 0; w < W; ++w) {
        if (!grads[w] || !codes[w] || !ranges[w])
            return fail(MQG_ERR_INVALID, "worker %d: grad, codes or ranges is null", w);
        if (!aligned16(grads[w])) return fail(MQG_ERR_ALIGN, "worker %d: grad not 16-byte aligned", w);
        if (!aligned16(codes[w])) return fail(MQG_ERR_ALIGN, "worker %d: codes not 16-byte aligned", w);
        if (!aligned8(ranges[w])) return fail(MQG_ERR_ALIGN, "worker %d: ranges not 8-byte aligned", w);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (mqg::quantize_workers_applies(W, n, bucket, 0, 1)) {
        const cudaError_t err = mqg::launch_quantize_workers(grads, W, n, bits, bucket, 0, codes, ranges,
                                                             (int)dtype, 0, 0, 0, 1, stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers_minmax", err);
        return MQG_OK;
    }
    if (worker_spans_preferred(n, bucket)) {
        const cudaError_t err = mqg::launch_bucket_spans(grads, W, n, bits, bucket, 0, codes, ranges, 1, (int)dtype, 0, 0, 0,
                                                         stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers_minmax", err);
        return MQG_OK;
    }
    // shapes the batched kernels do not take: one call per worker, same results
    for (int w = 0; w < W; ++w) {
        const mqg_status st = mqg_quantize_minmax(grads[w], n, bits, bucket, codes[w], ranges[w], dtype, cuda_stream);
        if (st != MQG_OK) return st;
    }
    return MQG_OK;
}

// The variant's worker tables: as check_workers, with the stricter alignment of the range pairs.
static mqg_status check_range_workers(const uint32_t* const* codes, const float* const* ranges, int W,
                                      bool empty, mqg::WorkerPtrs* out)
{
    if (mqg_status st = check_workers(codes, ranges, W, empty, out)) return st;
    if (empty) return MQG_OK;
    for (int w = 0; w < W; ++w)
        if (!aligned8(ranges[w])) return fail(MQG_ERR_ALIGN, "worker %d: ranges not 8-byte aligned", w);
    return MQG_OK;
}

mqg_status mqg_dequant_accumulate_minmax(const uint32_t* const* codes, const float* const* ranges, int W,
                                         int bits, uint64_t n, float* acc, uint64_t bucket,
                                         int add_into_acc, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_range_workers(codes, ranges, W, n == 0, &ptrs)) return st;
    if (n == 0) return MQG_OK;
    if (!acc) return fail(MQG_ERR_INVALID, "acc is null");
    if (!aligned16(acc)) return fail(MQG_ERR_ALIGN, "acc not 16-byte aligned");
    const cudaError_t err = mqg::launch_server_range(ptrs, W, bits, n, bucket, nullptr, 0.0f, acc,
                                                     add_into_acc ? 1 : 0,
                                                     static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_dequant_accumulate_minmax", err);
    return MQG_OK;
}

mqg_status mqg_server_step_minmax(const uint32_t* const* codes, const float* const* ranges, int W, int bits,
                                  uint64_t n, uint64_t bucket, float* params, float lr, float* acc_out,
                                  void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_range_workers(codes, ranges, W, n == 0, &ptrs)) return st;
    if (n == 0) return MQG_OK;
    if (!params) return fail(MQG_ERR_INVALID, "params is null");
    if (!aligned16(params)) return fail(MQG_ERR_ALIGN, "params not 16-byte aligned");
    if (acc_out && !aligned16(acc_out)) return fail(MQG_ERR_ALIGN, "acc_out not 16-byte aligned");
    const cudaError_t err = mqg::launch_server_range(ptrs, W, bits, n, bucket, params, lr, acc_out, 0,
                                                     static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_server_step_minmax", err);
    return MQG_OK;
}

mqg_status mqg_dequant_accumulate(const uint32_t* const* codes, const float* const* scales, int W,
                                  int bits, uint64_t n, float* acc, uint64_t bucket,
                                  int add_into_acc, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_workers(codes, scales, W, n == 0, &ptrs)) return st;
    if (n == 0) return MQG_OK;
    if (!acc) return fail(MQG_ERR_INVALID, "acc is null");
    if (!aligned16(acc)) return fail(MQG_ERR_ALIGN, "acc not 16-byte aligned");
    const cudaError_t err = mqg::launch_server(ptrs, W, bits, n, bucket, nullptr, 0.0f, acc,
                                               add_into_acc ? 1 : 0,
                                               static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_dequant_accumulate", err);
    return MQG_OK;
}

mqg_status mqg_apply(float* params, const float* acc, float lr, uint64_t n, void* cuda_stream)
{
    if (n == 0) return MQG_OK;
    if (!params || !acc) return fail(MQG_ERR_INVALID, "params or acc is null");
    if (!aligned16(params) || !aligned16(acc)) return fail(MQG_ERR_ALIGN, "params / acc not 16-byte aligned");
    const cudaError_t err = mqg::launch_apply(params, acc, lr, n, static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_apply", err);
    return MQG_OK;
}

mqg_status mqg_server_step(const uint32_t* const* codes, const float* const* scales, int W, int bits,
                           uint64_t n, uint64_t bucket, float* params, float lr, float* acc_out,
                           void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_workers(codes, scales, W, n == 0, &ptrs)) return st;
    if (n == 0) return MQG_OK;
    if (!params) return fail(MQG_ERR_INVALID, "params is null");
    if (!aligned16(params)) return fail(MQG_ERR_ALIGN, "params not 16-byte aligned");
    if (acc_out && !aligned16(acc_out)) return fail(MQG_ERR_ALIGN, "acc_out not 16-byte aligned");
    const cudaError_t err = mqg::launch_server(ptrs, W, bits, n, bucket, params, lr, acc_out, 0,
                                               static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_server_step", err);
    return MQG_OK;
}

mqg_status mqg_server_requantize(const uint32_t* const* codes, const float* const* scales, int W,
                                 int bits, uint64_t n, uint64_t bucket, float mean_scale,
                                 uint64_t seed, uint32_t* codes_out, float* scales_out,
                                 uint32_t worker, uint32_t step, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_workers(codes, scales, W, n == 0, &ptrs)) return st;
    if (n == 0) return MQG_OK;
    const uint64_t eff = bucket < n ? bucket : n;
    if (eff > (uint64_t)mqg::kMaxFusedBucket)
        return fail(MQG_ERR_INVALID, "mqg_server_requantize supports buckets of at most %d elements",
                    mqg::kMaxFusedBucket);
    if (!codes_out || !scales_out) return fail(MQG_ERR_INVALID, "codes_out or scales_out is null");
    if (!aligned16(codes_out)) return fail(MQG_ERR_ALIGN, "codes_out not 16-byte aligned");
    if (!aligned4(scales_out)) return fail(MQG_ERR_ALIGN, "scales_out not 4-byte aligned");
    const cudaError_t err = mqg::launch_requantize(ptrs, W, bits, n, bucket, mean_scale, seed, codes_out,
                                                   scales_out, worker, step,
                                                   static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_server_requantize", err);
    return MQG_OK;
}

mqg_status mqg_quantize_segments(const void* grad, int nseg, const uint64_t* seg_off,
                                 const uint64_t* code_off, int bits, uint64_t seed,
                                 uint32_t* codes, float* scales, mqg_dtype dtype, uint32_t worker,
                                 uint32_t step, uint64_t elem_offset, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (nseg > 0) {
        if (!grad || !codes || !scales) return fail(MQG_ERR_INVALID, "grad, codes or scales is null");
        if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
        if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
        if (!aligned4(scales)) return fail(MQG_ERR_ALIGN, "scales not 4-byte aligned");
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    return quantize_segments(&grad, 1, nseg, seg_off, code_off, bits, seed, &codes, &scales, dtype, worker, step,
                             elem_offset, nullptr, stream, "mqg_quantize_segments");
}

mqg_status mqg_quantize_segments_workers(const void* const* grads, int W, int nseg, const uint64_t* seg_off,
                                         const uint64_t* code_off, int bits, uint64_t seed,
                                         uint32_t* const* codes, float* const* scales, mqg_dtype dtype,
                                         uint32_t first_worker, uint32_t step, uint64_t elem_offset,
                                         void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (W < 1 || W > MQG_MAX_WORKERS)
        return fail(MQG_ERR_TOO_MANY_WORKERS, "W = %d is outside 1..%d", W, MQG_MAX_WORKERS);
    if (nseg < 0) return fail(MQG_ERR_INVALID, "nseg = %d is negative", nseg);
    if (nseg == 0) return MQG_OK;
    if (!grads || !codes || !scales) return fail(MQG_ERR_INVALID, "grads, codes or scales pointer table is null");
    for (int w = 0; w < W; ++w) {
        if (!grads[w] || !codes[w] || !scales[w])
            return fail(MQG_ERR_INVALID, "worker %d: grad, codes or scales is null", w);
        if (!aligned16(grads[w])) return fail(MQG_ERR_ALIGN, "worker %d: grad not 16-byte aligned", w);
        if (!aligned16(codes[w])) return fail(MQG_ERR_ALIGN, "worker %d: codes not 16-byte aligned", w);
        if (!aligned4(scales[w])) return fail(MQG_ERR_ALIGN, "worker %d: scales not 4-byte aligned", w);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    return quantize_segments(grads, W, nseg, seg_off, code_off, bits, seed, codes, scales, dtype, first_worker, step,
                             elem_offset, nullptr, stream, "mqg_quantize_segments_workers");
}

mqg_status mqg_quantize_l2(const void* grad, uint64_t n, int bits, uint64_t bucket, uint64_t seed,
                           uint32_t* codes, float* scales, mqg_dtype dtype, uint32_t worker,
                           uint32_t step, uint64_t elem_offset, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (n == 0) return MQG_OK;
    if ((bucket < n ? bucket : n) > (uint64_t)mqg::kMaxFusedBucket)
        return fail(MQG_ERR_INVALID, "mqg_quantize_l2 supports buckets of at most %d elements; use "
                    "mqg_quantize_segments_l2 for longer ones", mqg::kMaxFusedBucket);
    if (!grad || !codes || !scales) return fail(MQG_ERR_INVALID, "grad, codes or scales is null");
    if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
    if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
    if (!aligned4(scales)) return fail(MQG_ERR_ALIGN, "scales not 4-byte aligned");
    const cudaError_t err = mqg::launch_quantize_l2(grad, n, bits, bucket, seed, codes, scales, (int)dtype,
                                                    worker, step, elem_offset,
                                                    static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_quantize_l2", err);
    return MQG_OK;
}

mqg_status mqg_quantize_workers_l2(const void* const* grads, int W, uint64_t n, int bits, uint64_t bucket,
                                   uint64_t seed, uint32_t* const* codes, float* const* scales,
                                   mqg_dtype dtype, uint32_t first_worker, uint32_t step,
                                   uint64_t elem_offset, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (W < 1 || W > MQG_MAX_WORKERS)
        return fail(MQG_ERR_TOO_MANY_WORKERS, "W = %d outside 1..%d", W, MQG_MAX_WORKERS);
    if (n == 0) return MQG_OK;
    if ((bucket < n ? bucket : n) > (uint64_t)mqg::kMaxFusedBucket)
        return fail(MQG_ERR_INVALID, "mqg_quantize_workers_l2 supports buckets of at most %d elements; use "
                    "mqg_quantize_segments_l2 for longer ones", mqg::kMaxFusedBucket);
    if (!grads || !codes || !scales) return fail(MQG_ERR_INVALID, "grads, codes or scales is null");
    for (int w = 0; w < W; ++w) {
        if (!grads[w] || !codes[w] || !scales[w])
            return fail(MQG_ERR_INVALID, "worker %d: grad, codes or scales is null", w);
        if (!aligned16(grads[w])) return fail(MQG_ERR_ALIGN, "worker %d: grad not 16-byte aligned", w);
        if (!aligned16(codes[w])) return fail(MQG_ERR_ALIGN, "worker %d: codes not 16-byte aligned", w);
        if (!aligned4(scales[w])) return fail(MQG_ERR_ALIGN, "worker %d: scales not 4-byte aligned", w);
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    if (mqg::quantize_workers_applies(W, n, bucket, elem_offset, 2)) {
        const cudaError_t err = mqg::launch_quantize_workers(grads, W, n, bits, bucket, seed, codes, scales,
                                                             (int)dtype, first_worker, step, elem_offset,
                                                             2, stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers_l2", err);
        return MQG_OK;
    }
    if (W > 1 && worker_spans_preferred(n, bucket)) {
        const cudaError_t err = mqg::launch_bucket_spans(grads, W, n, bits, bucket, seed, codes, scales, 2, (int)dtype,
                                                         first_worker, step, elem_offset, stream);
        if (err != cudaSuccess) return cuda_fail("mqg_quantize_workers_l2", err);
        return MQG_OK;
    }
    // shapes the batched kernels do not take: one launch per worker, same results
    for (int w = 0; w < W; ++w) {
        const mqg_status st = mqg_quantize_l2(grads[w], n, bits, bucket, seed, codes[w], scales[w], dtype,
                                              first_worker + (uint32_t)w, step, elem_offset, cuda_stream);
        if (st != MQG_OK) return st;
    }
    return MQG_OK;
}

mqg_status mqg_quantize_1bit_ef(const void* grad, float* residual, uint64_t n, uint64_t bucket,
                                uint32_t* codes, float* ranges, mqg_dtype dtype, void* cuda_stream)
{
    if (mqg_status st = check_bucket(n, bucket)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (n == 0) return MQG_OK;
    if ((bucket < n ? bucket : n) > (uint64_t)mqg::kMaxFusedBucket)
        return fail(MQG_ERR_INVALID, "mqg_quantize_1bit_ef supports buckets of at most %d elements",
                    mqg::kMaxFusedBucket);
    if (!grad || !residual || !codes || !ranges)
        return fail(MQG_ERR_INVALID, "grad, residual, codes or ranges is null");
    if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
    if (!aligned16(residual)) return fail(MQG_ERR_ALIGN, "residual not 16-byte aligned");
    if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
    if (!aligned8(ranges)) return fail(MQG_ERR_ALIGN, "ranges not 8-byte aligned");
    const cudaError_t err = mqg::launch_quantize_onebit_ef(grad, residual, n, bucket, codes, ranges, (int)dtype,
                                                           static_cast<cudaStream_t>(cuda_stream));
    if (err != cudaSuccess) return cuda_fail("mqg_quantize_1bit_ef", err);
    return MQG_OK;
}

size_t mqg_l2_workspace_floats(int nseg, const uint64_t* seg_off)
{
    if (nseg <= 0 || !seg_off) return 0;
    const uint64_t tile_elems = (uint64_t)mqg::kMaxTileRows * 32;
    uint64_t tiles = 0;
    for (int j = 0; j < nseg; ++j)
        if (seg_off[j + 1] > seg_off[j]) tiles += (seg_off[j + 1] - seg_off[j] + tile_elems - 1) / tile_elems;
    return (size_t)tiles;
}

mqg_status mqg_quantize_segments_l2(const void* grad, int nseg, const uint64_t* seg_off,
                                    const uint64_t* code_off, int bits, uint64_t seed,
                                    uint32_t* codes, float* scales, mqg_dtype dtype, uint32_t worker,
                                    uint32_t step, uint64_t elem_offset, float* workspace,
                                    size_t workspace_floats, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    if (dtype != MQG_F32 && dtype != MQG_BF16) return fail(MQG_ERR_INVALID, "unknown dtype %d", (int)dtype);
    if (nseg > 0) {
        if (!grad || !codes || !scales) return fail(MQG_ERR_INVALID, "grad, codes or scales is null");
        if (!aligned16(grad)) return fail(MQG_ERR_ALIGN, "grad not 16-byte aligned");
        if (!aligned16(codes)) return fail(MQG_ERR_ALIGN, "codes not 16-byte aligned");
        if (!aligned4(scales)) return fail(MQG_ERR_ALIGN, "scales not 4-byte aligned");
        if (!seg_off || !code_off) return fail(MQG_ERR_INVALID, "segment table is null");
        const size_t need = mqg_l2_workspace_floats(nseg, seg_off);
        if (need > workspace_floats)
            return fail(MQG_ERR_INVALID, "workspace holds %llu floats, %llu needed (mqg_l2_workspace_floats)",
                        (unsigned long long)workspace_floats, (unsigned long long)need);
        if (need != 0 && !workspace) return fail(MQG_ERR_INVALID, "workspace is null");
        if (!aligned4(workspace)) return fail(MQG_ERR_ALIGN, "workspace not 4-byte aligned");
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    float none = 0.0f;                    // a table of empty segments needs no workspace, but a pointer that says which codec
    return quantize_segments(&grad, 1, nseg, seg_off, code_off, bits, seed, &codes, &scales, dtype, worker, step,
                             elem_offset, workspace ? workspace : &none, stream, "mqg_quantize_segments_l2");
}

mqg_status mqg_server_step_segments(const uint32_t* const* codes, const float* const* scales, int W,
                                    int bits, int nseg, const uint64_t* seg_off,
                                    const uint64_t* code_off, float* params, float lr,
                                    float* acc_out, void* cuda_stream)
{
    if (mqg_status st = check_bits(bits)) return st;
    mqg::WorkerPtrs ptrs;
    if (mqg_status st = check_workers(codes, scales, W, nseg <= 0, &ptrs)) return st;
    if (nseg > 0) {
        if (!params) return fail(MQG_ERR_INVALID, "params is null");
        if (!aligned16(params)) return fail(MQG_ERR_ALIGN, "params not 16-byte aligned");
        if (acc_out && !aligned16(acc_out)) return fail(MQG_ERR_ALIGN, "acc_out not 16-byte aligned");
    }
    cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
    // A long segment is a gradient with a single bucket: the long segments go to the TMA-fed server kernel together, in one
    // launch, those off a 16-byte boundary in another of its form for segments that start anywhere (flat_server_form); all other
    // segments share the table-driven launch.  The results are the same bit for bit either way.
    constexpr uint64_t kOwnLaunchElems = mqg::kEntrySegmentElems;
    auto is_long = [&](int j) {
        const uint64_t len = seg_off[j + 1] - seg_off[j];
        return !acc_out && len >= kOwnLaunchElems && mqg::server_tma_applies(len, len);
    };
    bool alike = true;                   // the workers' buffers start at the same place between two 16-byte boundaries
    for (int w = 1; w < W; ++w) alike = alike && ((reinterpret_cast<uintptr_t>(codes[w]) ^ reinterpret_cast<uintptr_t>(codes[0])) & 15u) == 0;
    auto aligned = [&](int j) { return alike && aligned16(params + seg_off[j]) && aligned16(codes[0] + code_off[j]); };
    if (mqg_status st = check_segments(nseg, seg_off, code_off, bits)) return st;
    uint64_t on = 0, off = 0;            // elements of the long segments on and off the boundaries
    for (int j = 0; j < nseg; ++j)
        if (is_long(j)) (aligned(j) ? on : off) += seg_off[j + 1] - seg_off[j];
    const int flat = mqg::flat_server_form(on, off, W, bits);
    const bool any_long = on != 0 || flat != 0;
    enum { kTable, kBulk, kFlat };
    auto form = [&](int j) { return !is_long(j) ? kTable : aligned(j) ? (flat == 2 ? kFlat : kBulk) : flat != 0 ? kFlat : kTable; };
    // The other segments: table-driven launches - except that ONE table of short segments rides along
    // with the (first) launch of the long ones, so that a typical layered step is a single launch.
    mqg::SegmentTable folded;
    int folded_first = -1;
    const mqg_status st = for_each_chunk(nseg, seg_off, code_off, bits,
        [&](const mqg::SegmentTable& tab, int first) -> mqg_status {
            if (tab.tile_start[tab.nseg] == 0) return MQG_OK;
            if (any_long && folded_first < 0) {
                folded = tab;
                folded_first = first;
                return MQG_OK;
            }
            const cudaError_t err = mqg::launch_server_segments(ptrs, W, bits, tab, first, params, lr, acc_out, stream);
            return err == cudaSuccess ? MQG_OK : cuda_fail("mqg_server_step_segments", err);
        }, [&](int j) { return form(j) != kTable; });
    if (st != MQG_OK) return st;
    // The long ones, a launch for every kMaxServerSegsPerLaunch of them.  No heap here: the C ABI throws nothing.
    mqg::ServerSegHost longs[mqg::kMaxServerSegsPerLaunch];
    for (const auto which : {kBulk, kFlat}) {
        if (which == kBulk ? on == 0 || flat == 2 : flat == 0) continue;
        int count = 0;
        for (int j = 0; j <= nseg; ++j) {
            if (j < nseg && form(j) == which)
                longs[count++] = {seg_off[j + 1] - seg_off[j], seg_off[j], code_off[j], (uint32_t)j};
            if (count == 0 || (count < mqg::kMaxServerSegsPerLaunch && j < nseg)) continue;
            const cudaError_t err = mqg::launch_server_tma_segments(ptrs, W, bits, longs, count,
                                                                    folded_first >= 0 ? &folded : nullptr, folded_first, params,
                                                                    lr, which == kFlat, stream);
            if (err != cudaSuccess) return cuda_fail("mqg_server_step_segments", err);
            folded_first = -1;
            count = 0;
        }
    }
    return MQG_OK;
}

}  // extern "C"
