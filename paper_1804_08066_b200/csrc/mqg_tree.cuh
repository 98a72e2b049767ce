// Fixed-order float sums over the rows of a bucket, shared by the codec variants whose scale or
// reconstruction values are sums (L2 norm, class means): the per-row values are the leaves of a
// balanced binary tree of adjacent pairs, the leaf count padded with zeros to a power of two.
// Adding +0 is exact, so evaluating more (all-zero) leaves or levels than the padded tree has
// does not change the result.
#pragma once

#include "mqg_common.cuh"

namespace mqg {

// Five tree levels inside a warp: lane l holds the sum of rows (l & ~(2d - 1)) .. + 2d - 1 after
// the step with distance d.  Both partners compute the same sum (addition commutes bit for bit).
__device__ __forceinline__ float warp_tree(float a, uint32_t levels_end)
{
    for (uint32_t d = 1; d < levels_end; d <<= 1)
        a = __fadd_rn(a, __shfl_xor_sync(0xFFFFFFFFu, a, d));
    return a;
}

// Tree over `count` <= 8 values v[first .. first + count) padded with zeros to eight leaves.
__device__ __forceinline__ float tree8(const float* v, uint32_t first, uint32_t count)
{
    float x[8];
#pragma unroll
    for (uint32_t i = 0; i < 8; ++i) x[i] = i < count ? v[first + i] : 0.0f;
    return __fadd_rn(__fadd_rn(__fadd_rn(x[0], x[1]), __fadd_rn(x[2], x[3])),
                     __fadd_rn(__fadd_rn(x[4], x[5]), __fadd_rn(x[6], x[7])));
}

// The buckets' sums of N values per row, from the per-row values of a tile of THREADS (at most 256) rows that
// holds whole buckets of `rpb` rows (thread t owns row t of the tile; threads without a row pass 0).  Every
// thread of the CTA must call it.  s_part: N * THREADS floats of shared memory, free for reuse after the next
// barrier only.
template <int THREADS, int N>
__device__ __forceinline__ void bucket_tree_sums(float (&a)[N], uint32_t rpb, float* s_part)
{
    const uint32_t t = threadIdx.x;
    if ((rpb & (rpb - 1)) == 0 && rpb <= 32) {
#pragma unroll
        for (int i = 0; i < N; ++i) a[i] = warp_tree(a[i], rpb);
        return;
    }
    if (rpb % 32 == 0) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
            a[i] = warp_tree(a[i], 32);
            if ((t & 31) == 0) s_part[i * THREADS + (t >> 5)] = a[i];
        }
        __syncthreads();
        const uint32_t wpb = rpb / 32;
        const uint32_t first = (t / rpb) * wpb;
#pragma unroll
        for (int i = 0; i < N; ++i)
            a[i] = first + wpb <= THREADS / 32 ? tree8(s_part + i * THREADS, first, wpb) : 0.0f;
        return;
    }
    // any other shape: a bucket's tree is the work of an aligned group of 2^k lanes, 8 rows of it per lane, zeros
    // beyond; there are more groups than buckets
#pragma unroll
    for (int i = 0; i < N; ++i) s_part[i * THREADS + t] = a[i];
    __syncthreads();
    const uint32_t buckets = THREADS / rpb;
    uint32_t lanes = 1;
    while (8 * lanes < rpb) lanes <<= 1;
    const uint32_t b = t / lanes, row = 8 * (t & (lanes - 1));
    const uint32_t left = b < buckets && row < rpb ? min(8u, rpb - row) : 0u;
    float* p = s_part + (left != 0 ? b * rpb : 0u);
#pragma unroll
    for (int i = 0; i < N; ++i, p += THREADS) {
        const float s = warp_tree(tree8(p, row, left), lanes);
        __syncwarp();                              // every lane has read the bucket's values
        if (row == 0 && left != 0) p[0] = s;
    }
    __syncthreads();
    const uint32_t mine = t / rpb;
#pragma unroll
    for (int i = 0; i < N; ++i) a[i] = mine < buckets ? s_part[i * THREADS + mine * rpb] : 0.0f;
}

__device__ __forceinline__ float bucket_tree_sum(float a, uint32_t rpb, float* s_part)
{
    float v[1] = {a};
    bucket_tree_sums<kMaxTileRows, 1>(v, rpb, s_part);
    return v[0];
}

}  // namespace mqg
