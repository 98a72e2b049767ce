// TMA (cp.async.bulk) and mbarrier wrappers for sm_100a, plus the host-side tensor-map
// encoder.  Loads are plain per-CTA copies (no cluster multicast anywhere).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace mqg {

// Upper bound on polls of one mbarrier wait.  Each try_wait already blocks for a
// hardware-defined interval, so this is seconds of wall time; a copy that has not landed
// by then never will.
constexpr uint32_t kMaxWaitPolls = 1u << 22;

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Orders this thread's earlier generic-proxy accesses to shared memory before later
// async-proxy (TMA) accesses.
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}

// Bounded wait: false if the phase did not complete within `limit` polls.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t limit = kMaxWaitPolls)
{
    for (uint32_t i = 0; i < limit; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// 2-D tiled load global -> shared, completion counted in bytes on `bar`.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar) : "memory");
}

// 2-D tiled store shared -> global (bulk async-group completion).
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, int x, int y, uint32_t src)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];"
                 ::"l"(map), "r"(x), "r"(y), "r"(src) : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

// Wait until at most N of this thread's bulk groups still READ their shared-memory source.
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }

template <int N>
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void prefetch_tensormap(const CUtensorMap* map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}

// Programmatic dependent launch.  A kernel launched with launch_pdl() is set up while the previous kernel of
// the stream is still running, starts the moment that kernel's last CTA has gone, and blocks in
// grid_dependency_wait() until its writes are visible.  Every access to global memory must come after
// that wait.  No kernel releases its dependents early (griddepcontrol.launch_dependents): the next launch's
// CTAs then take the SMs in the order in which this launch's CTAs retire and crowd on those that come free
// first.  Without it a step on 300,000 elements, W = 8, takes 6.9 against 9.1 us (batched quantize, server), on
// 2^20, W = 4, 8.3 against 9.2 us, the per-layer quantizer of 11 M elements, W = 2, 74 against 79 us; long
// launches are the same.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- host side ------------------------------------------------------------------------
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_grid(void (*kernel)(KArgs...), dim3 grid, unsigned block, size_t dynamic_smem,
                            cudaStream_t stream, Args&&... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = dynamic_smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

// The same on a grid of one dimension, without and with dynamic shared memory.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, cudaStream_t stream, Args&&... args)
{
    return launch_pdl_grid(kernel, dim3(grid), block, 0, stream, args...);
}
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_smem(void (*kernel)(KArgs...), unsigned grid, unsigned block, size_t dynamic_smem,
                            cudaStream_t stream, Args&&... args)
{
    return launch_pdl_grid(kernel, dim3(grid), block, dynamic_smem, stream, args...);
}

// Encodes a 2-D row-major tensor map: `rows` rows of `row_elems` elements (row_bytes =
// 64 or 128 selects the matching swizzle), box = box_rows x row_elems.  Returns false with a
// message if the driver entry point is missing or the encode fails.
bool encode_rows_map(CUtensorMap* map, const void* base, uint64_t rows, int elem_bytes,
                     uint32_t row_elems, uint32_t box_rows, const char** why);

// Device address of the current device's counter of kernel waits that gave up (a word in the
// library's own device image; kernels receive the pointer as an argument).  nullptr on error.
unsigned int* wait_timeout_counter();

// Reads that counter (synchronises with the device) and, with `reset`, clears it.
cudaError_t read_wait_timeouts(unsigned int* count, bool reset = false);

// What the launchers put into their kernels' arguments: the poll limit of a barrier wait, and
// whether the staging copies are issued at all.  The defaults are kMaxWaitPolls and true; the
// test hook mqg_test_wait_override() changes them for the whole process, so that a test can make
// a wait run out with nothing in flight.
struct WaitPolicy {
    uint32_t poll_limit;
    uint32_t arm_only;       // 1: barriers are armed for their bytes but no copy is issued
};
WaitPolicy wait_policy();
void set_wait_policy(uint32_t poll_limit, uint32_t arm_only);

}  // namespace mqg
