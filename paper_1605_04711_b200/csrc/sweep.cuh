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

// A cluster of `grid` blocks.  It may start while the kernel before it drains (its blocks wait in pdl_begin), as the
// small kernels around it do: 6.2 -> 4.6 us per call for a stream of small ternarizations.
template <typename K, typename... A>
int launch_cluster(K kernel, unsigned int grid, cudaStream_t s, const A &...args)
{
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSweepThreads);
    cfg.stream = s;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    TWN_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, args...));
    return TWN_OK;
}
// A kernel of a chain of launches: launched programmatically, it is there when the one before it ends, and from here on what that
// wrote is visible.  It lets its own successor start by ending, not earlier: with a trigger at the start of every kernel the
// successors' blocks were resident and waiting three launches ahead, and a training layer of one 83x83x224 image (96 channels)
// took 59.6 us instead of 52.4, the 21 tensors of ResNet-18 35.6 instead of 31.1.
#ifdef __CUDACC__
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif
// A grid whose blocks all run at once and may wait for one another.
template <typename K, typename... A>
int launch_cooperative(K kernel, unsigned int grid, cudaStream_t s, size_t smem, const A &...args)
{
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSweepThreads);
    cfg.stream = s;
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    TWN_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, args...));
    return TWN_OK;
}

// ---- the codes --------------------------------------------------------------
// Bit position of element e (0..15) inside its word: even elements fill the low
// half-word, odd elements the high half-word, each from the top down, so that a left
// shift by 2*(e/2) brings the element's field to the top two bits of its half-word.
__host__ __device__ __forceinline__ int field_pos(int e) { return 14 - 2 * (e >> 1) + 16 * (e & 1); }

// A "quarter byte" holds the 2-bit fields (bit 0 = kept, bit 1 = negative: 00 / 01 / 11) of four consecutive
// weights: low nibble = elements 0 (upper) and 2, high nibble = elements 1 (upper) and 3.
//
// Bits 0..15 of x -> the even bits of the result.
__device__ __forceinline__ uint32_t spread16(uint32_t x)
{
    x = (x | (x << 8)) & 0x00FF00FFu;
    x = (x | (x << 4)) & 0x0F0F0F0Fu;
    x = (x | (x << 2)) & 0x33333333u;
    return (x | (x << 1)) & 0x55555555u;
}

// Quarter bytes B0..B3 of sixteen consecutive weights -> the word of
// those 16 elements: low half = low nibbles, high half = high nibbles, B0's on top.
__device__ __forceinline__ uint32_t bytes_to_word(uint32_t r)
{
    r = __byte_perm(r, 0u, 0x0123);
    uint32_t lo = r & 0x0F0F0F0Fu, hi = (r >> 4) & 0x0F0F0F0Fu;
    lo = (lo | (lo >> 4)) & 0x00FF00FFu;
    lo = (lo | (lo >> 8)) & 0x0000FFFFu;
    hi = (hi | (hi >> 4)) & 0x00FF00FFu;
    hi = (hi | (hi >> 8)) & 0x0000FFFFu;
    return lo | (hi << 16);
}

// int8 image of the four fields of a quarter byte, in element order:
// 00 -> 0x00, 01 -> 0x01, 11 -> 0xFF
__device__ __forceinline__ uint32_t fields_to_i8x4(uint32_t c8)
{
    uint32_t r = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const uint32_t f = (c8 >> (2 - 2 * (e >> 1) + 4 * (e & 1))) & 3u;
        const uint32_t b = (f & 1u) ? ((f & 2u) ? 0xFFu : 0x01u) : 0u;
        r |= b << (8 * e);
    }
    return r;
}

// The codes of four quarters (sixteen weights) of a thread against a threshold: a byte per quarter; adds the kept
// magnitudes to k and counts.  Bound by instruction issue, above all by the half-rate integer pipe: a comparison, a
// select, three shifts and two merges per weight took 29 us for 20 million weights that are in L2.  Here a weight costs
// that pipe two instructions, the comparison (as 1.0 or 0.0) and a funnel shift that collects the signs; the masking and
// the collection of the kept bits are multiplications.
__device__ __forceinline__ uint32_t code_quarters(const float4 (&v)[4], float thr, double (&k)[4], unsigned int &pos, unsigned int &neg)
{
    float kept_bits = 0.0f;          // below 2^16, exact
    uint32_t sign_bits = 0;
#pragma unroll
    for (int i = 3; i >= 0; --i) {
        const float w4[4] = {v[i].y, v[i].w, v[i].x, v[i].z};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            float keep;
            asm("set.gt.f32.f32 %0, %1, %2;" : "=f"(keep) : "f"(fabsf(w4[x])), "f"(thr));
            k[x] += (double)(fabsf(w4[x]) * keep);
            kept_bits = fmaf(kept_bits, 2.0f, keep);
            sign_bits = __funnelshift_l(__float_as_uint(w4[x]), sign_bits, 1);
        }
    }
    const uint32_t kb = (uint32_t)kept_bits, nb = sign_bits & kb;
    const unsigned int n_neg = __popc(nb);
    neg += n_neg;
    pos += __popc(kb) - n_neg;
    return spread16(kb) | (spread16(nb) << 1);
}

// A word's four quarters sit in the bytes of four neighbouring lanes: a 4x4 byte transpose (lanes l^2, then l^1) leaves
// lane l with word l/4 of its warp's share of quarter-row l%4.
__device__ __forceinline__ uint32_t exchange_quarters(uint32_t bytes)
{
    const int lane = threadIdx.x;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, bytes, 2);
    bytes = __byte_perm(bytes, y, (lane & 2) ? 0x3276 : 0x5410);
    const uint32_t z = __shfl_xor_sync(0xffffffffu, bytes, 1);
    bytes = __byte_perm(bytes, z, (lane & 1) ? 0x3715 : 0x6240);
    return bytes_to_word(bytes);
}

}  // namespace
