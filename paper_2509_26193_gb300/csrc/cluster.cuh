// Whole passes over a small network in one launch: a cluster of kBlocks blocks whose
// hardware barrier separates the steps that a larger network runs as kernels of their own.
//
// A small update with delivery and deletion is a chain of about 40 kernels and memsets of
// 2 to 8 us each (launch, one wave of work, drain), whatever the network's size, and the
// host cannot launch them faster than it takes the GPU to run them. A cluster barrier
// costs well under a microsecond, so the same steps cost little but their work.
//
// Measured (two updates with delivery, a partial and a full deletion, clustered network,
// theta 0.5; us, general kernels -> cluster kernels of 8 x 1024, 16 x 1024 and 16 x 512
// threads): 1,000 neurons 402 -> 238 / 253 / 217, 8,000 533 -> 358 / 344 / 328, 16,000
// 634 -> 516 / 479 / 476, 32,000 853 -> 883 / 759 / 797, 50,000 1156 -> 1366 / 1162 / 1218:
// hence 16 x 512, up to kSmallN = 40,960 neurons (internal.h). Replayed from a graph,
// without launch gaps (an update and a full deletion): 131 -> 87, 146 -> 109 (4,000), 178 ->
// 149, 252 -> 232, 399 -> 387, 437 -> 496 (40,000); deliveries then choose for themselves
// (deliver_small in synapses.cu).
#pragma once

#include <cooperative_groups.h>

#include "internal.h"

namespace rl {

namespace cluster_form {

constexpr int kBlocks = 16; // more than the portable 8: placeable
constexpr int kThreads = 512;

// Allows kernel k its cluster size and tells whether the current context can hold one such
// cluster: not every part of a GPU can (an SM limit, a partition). False leaves no error
// pending. 0.4 us on the host.
template <class Kernel>
inline bool placeable(Kernel *k)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kBlocks);
    cfg.blockDim = dim3(kThreads);
    cudaLaunchAttribute size = {};
    size.id = cudaLaunchAttributeClusterDimension;
    size.val.clusterDim.x = kBlocks;
    size.val.clusterDim.y = size.val.clusterDim.z = 1;
    cfg.attrs = &size;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return clusters > 0;
}

// Orders the cluster's global and shared memory accesses across all of its threads.
__device__ __forceinline__ void sync() { cooperative_groups::this_cluster().sync(); }

__device__ __forceinline__ int64_t first() // this thread's first element
{
    return (int64_t)cooperative_groups::this_cluster().block_rank() * kThreads + threadIdx.x;
}
constexpr int64_t kStride = (int64_t)kBlocks * kThreads;

struct I32 {
    int32_t v;
};
struct I64x2 {
    long long a, b;
};
__device__ __forceinline__ I32 add(I32 x, I32 y) { return I32{x.v + y.v}; }
__device__ __forceinline__ I32 up(I32 x, int o) { return I32{__shfl_up_sync(0xffffffffu, x.v, o)}; }
__device__ __forceinline__ I64x2 add(I64x2 x, I64x2 y) { return I64x2{x.a + y.a, x.b + y.b}; }
__device__ __forceinline__ I64x2 up(I64x2 x, int o)
{
    return I64x2{__shfl_up_sync(0xffffffffu, x.a, o), __shfl_up_sync(0xffffffffu, x.b, o)};
}

// Exclusive scan over the elements 0 .. n - 1 by the whole cluster: load(i) is called once
// per element, then again(i) (the same value) and emit(i, prefix, value, total), by the
// same thread. Returns the total. One cluster barrier, between the load and the emit
// calls: whatever load wrote, every emit may read. A barrier (sync) has to follow before
// the next scan and before the kernel ends. T: zero when value-initialised, add and up.
template <class T, class Load, class Again, class Emit>
__device__ __forceinline__ T scan(int64_t n, Load load, Again again, Emit emit)
{
    namespace cg = cooperative_groups;
    __shared__ T s_warp[kThreads / 32];
    __shared__ T s_total; // read by every block of the cluster
    cg::cluster_group cl = cg::this_cluster();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t per_block = (n + kBlocks - 1) / kBlocks;
    const int64_t per = (per_block + kThreads - 1) / kThreads;
    const int64_t lo = min(n, (int64_t)cl.block_rank() * per_block);
    const int64_t hi = min(n, lo + per_block);
    const int64_t i0 = min(hi, lo + (int64_t)threadIdx.x * per), i1 = min(hi, i0 + per);
    T sum{};
    for (int64_t i = i0; i < i1; ++i) sum = add(sum, load(i));
    T inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T t = up(inc, o);
        if (lane >= o) inc = add(inc, t);
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    T run{};
    for (int w = 0; w < warp; ++w) run = add(run, s_warp[w]);
    if (threadIdx.x == kThreads - 1) s_total = add(run, inc);
    cl.sync();
    T before{}, total{};
    for (int b = 0; b < kBlocks; ++b) {
        const T t = *cl.map_shared_rank(&s_total, b);
        if (b < (int)cl.block_rank()) before = add(before, t);
        total = add(total, t);
    }
    run = add(before, run);
    // exclusive within the warp: the inclusive prefix of the lane below
    T low = up(inc, 1);
    if (lane > 0) run = add(run, low);
    for (int64_t i = i0; i < i1; ++i) {
        const T v = again(i);
        emit(i, run, v, total);
        run = add(run, v);
    }
    return total;
}

} // namespace cluster_form

} // namespace rl
