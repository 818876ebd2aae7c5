// What the sweeps over the master weights share: sums in a fixed order within a block, within a cluster of at most eight
// blocks (distributed shared memory) and over a grid, and their launches.
#pragma once

#include <cooperative_groups.h>

#include "common.cuh"

namespace {

constexpr int kSweepWarps = 16;
constexpr int kSweepThreads = 32 * kSweepWarps;
constexpr int kSweepBlocksPerSm = 2;                        // 64 registers; three blocks spill: 1e8 weights 131 -> 164 us
constexpr unsigned int kMaxParts = kSweepBlocksPerSm * 148;  // one part per block of a full grid
constexpr int kSmallParts = 8;                               // blocks of the cluster that sweeps a small tensor

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// Block-wide sums with a fixed order: a shuffle tree per warp, then every thread adds the sixteen warps' sums in
// the same tree, so that one barrier does and nobody waits for a broadcast.  The buffers alternate from call to
// call (`turn`): a buffer is written again two barriers later, when all have read it.
struct Reduce {
    double sum[2][kSweepWarps];
    uint2 cnt[2][kSweepWarps];
};
__device__ __forceinline__ double tree16(const double *v)
{
    double t[kSweepWarps / 2];
#pragma unroll
    for (int i = 0; i < kSweepWarps / 2; ++i) t[i] = v[i] + v[i + kSweepWarps / 2];
#pragma unroll
    for (int o = kSweepWarps / 4; o > 0; o >>= 1)
#pragma unroll
        for (int i = 0; i < o; ++i) t[i] += t[i + o];
    return t[0];
}
__device__ __forceinline__ double sweep_sum(double v, Reduce &red, unsigned int &turn)
{
    double *buf = red.sum[turn & 1];
    ++turn;
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = v;
    __syncthreads();
    return tree16(buf);
}
// The same for a sum and two counts of the block (below 2^32).
__device__ __forceinline__ double sweep_sum(double v, unsigned int &pos, unsigned int &neg, Reduce &red, unsigned int &turn)
{
    double *buf = red.sum[turn & 1];
    uint2 *cnt = red.cnt[turn & 1];
    ++turn;
    v = warp_sum(v);
    const unsigned int p = __reduce_add_sync(0xffffffffu, pos), q = __reduce_add_sync(0xffffffffu, neg);
    if ((threadIdx.x & 31) == 0) { buf[threadIdx.x >> 5] = v; cnt[threadIdx.x >> 5] = make_uint2(p, q); }
    __syncthreads();
    pos = neg = 0;
#pragma unroll
    for (int i = 0; i < kSweepWarps; ++i) { pos += cnt[i].x; neg += cnt[i].y; }
    return tree16(buf);
}

__device__ __forceinline__ uint32_t peer_smem(const void *p, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void st_peer(uint32_t addr, unsigned long long v)
{
    asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

// Eight values in the order of the shuffle tree that folds the parts of a larger tensor.
__device__ __forceinline__ double tree8(const double *p)
{
    return ((p[0] + p[4]) + (p[2] + p[6])) + ((p[1] + p[5]) + (p[3] + p[7]));
}

// cudaLaunchKernelEx with one attribute.
template <typename K, typename... A>
int launch_with(K kernel, unsigned int grid, cudaLaunchAttributeID id, cudaLaunchAttributeValue val, cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = id;
    attr[0].val = val;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSweepThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    TWN_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, args...));
    return TWN_OK;
}

}  // namespace
