// Ternary-weight contraction for problems that do not fill the GPU (Eq. 2; Algorithm 1 TernaryForward /
// TernaryBackward): one tile per block, the reduction split over the blocks of a cluster.
//
// What bounds such a problem is latency, not a pipe: in tconv_kernel a block walks the whole reduction of its tile
// alone (255-280 cycles per 64-element k-block of 128 pixels), and the first tile of its long straight-line epilogue
// costs 4400 cycles of cold instruction fetch.  1x1024x512 took 10.9 us there on 4 blocks, 14x14x256 at batch 8 14.2 us
// on 26 (both with k-blocks of 430-540 cycles; the second 10.9 now).  Here
//   - a tile is 128 output channels x PIX pixels with PIX = 32 ... 256, so that small problems still make blocks;
//   - a cluster of S = 1 ... 8 blocks shares a tile, every block reduces a contiguous share of the k-blocks;
//   - every block leaves its fp32 accumulator in shared memory as [pixel][channel] and finishes PIX / S of the pixels:
//     the other blocks push their partial sums of those into its memory, one bulk copy each, announced at an mbarrier
//     (reading them from the peers cost 2-3 us of latency, pushing them by plain stores more than that); it adds
//     the S partial sums in rank order (deterministic), applies alpha, the affine, the residual and the ReLU and stores
//     four channels per thread.  The stores are coalesced as they are, so there is no store map and any pitch, dtype
//     and embedding goes this way.
// The roles of the main loop are those of tconv_kernel: the decoded weights are the A operand in tensor memory, the
// activations the B operand in shared memory (TMA, 128-byte swizzle).
//
//   warp 0       TMA producer
//   warp 1       allocates tensor memory, issues tcgen05.mma
//   warps 2-9    decode, two groups on alternate k-blocks; afterwards they drain the accumulator
//   all warps    the final sums and the epilogue
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstddef>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "tconv_host.cuh"

using namespace twn_detail;

namespace {

constexpr int kChan = 128;
constexpr int kBlockK = 64;
constexpr int kSets = 2;                 // decode groups, on k-blocks in turn (three or four: no gain, 1 us more set-up)
constexpr int kThreads = 32 * (2 + 4 * kSets);
constexpr int kAColsPerBlock = kBlockK / 2;
constexpr int kMaxBlocks = 512;          // k-blocks of a block whose code offsets are tabulated
constexpr int kPitch = 132;              // floats per pixel of the staged accumulator: 16-byte rows, no bank conflicts

template <int PIX> struct Cfg;           // stages of one k-block; two blocks share an SM's tensor memory up to 128 pixels
template <> struct Cfg<32> { static constexpr int kStages = 6, kTmem = 256; };
template <> struct Cfg<64> { static constexpr int kStages = 6, kTmem = 256; };
template <> struct Cfg<128> { static constexpr int kStages = 4, kTmem = 256; };
template <> struct Cfg<256> { static constexpr int kStages = 4, kTmem = 512; };

struct SplitParams {
    int n_tiles;                      // channel tiles
    int lgBW, lgBH;                   // pixel tile = BW x BH x BB, product PIX
    int n_cblk;                       // k-blocks per tap
    const uint32_t *T;
    long long wpr;
    int sw, sh;
    int Bv, OH, OW, osh, osw;         // images; embedding of the virtual output grid in the output tensor
    // The classes of the output grid, one for all but strided backward passes.  Their tiles follow one another, and
    // each has its own run of taps, so their reductions differ in length.
    int n_classes;
    struct { int tile0, tw, th, Hv, Wv, ooh, oow, tap0, kb, kb_per_block; } cls[kMaxClasses];
    long long ldy;
    int Cout;
    const double *alpha;
    const float *scale, *shift;
    const void *residual;
    int res_dtype, res_gate, relu, out_dtype;
    int vec;                          // four channels at a time are aligned in Y and the residual
    void *Y;
    __nv_bfloat16 *pool;              // 2x2 max pooling of the output [Bv, PH, PW, Cout]: whole windows in every block's share
    int PH, PW;
    int32_t *status;
    Tap taps[kMaxTaps];
};

template <int PIX>
struct __align__(1024) SplitSmem {
    static constexpr int kXBytes = PIX * kBlockK * 2;
    union {
        uint8_t x[Cfg<PIX>::kStages][kXBytes];
        float acc[PIX * kPitch];      // after the last MMA has read the operands
    };
    unsigned long long full[Cfg<PIX>::kStages], empty[Cfg<PIX>::kStages], acc_full, recv_full;
    uint32_t kword[kMaxBlocks];
    uint32_t off[PIX];                // element offset of every pixel of the tile in the output, ~0 outside it
    uint32_t tmem_base;
    volatile int abort_flag;
    alignas(128) float recv[1];       // the other blocks' partial sums of this block's pixels: (S - 1) x (PIX / S) rows
};
template <int PIX> constexpr int smem_bytes(int splits)
{
    return (int)offsetof(SplitSmem<PIX>, recv) + PIX / splits * (splits - 1) * kPitch * 4 + 1024;
}

__device__ __forceinline__ uint32_t peer(uint32_t addr, int rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }

// Four channels of a pixel: affine, residual, ReLU, store.  Returns them as stored where that is bf16, four at a time.
__device__ __forceinline__ uint2 finish(const SplitParams &P, size_t off, int left, const float4 a, const float (&sc)[4], const float (&sf)[4])
{
    float y[4] = {fmaf(a.x, sc[0], sf[0]), fmaf(a.y, sc[1], sf[1]), fmaf(a.z, sc[2], sf[2]), fmaf(a.w, sc[3], sf[3])};
    if (P.residual) {
        float r[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (P.res_dtype == TWN_BF16) {
            const __nv_bfloat16 *rp = reinterpret_cast<const __nv_bfloat16 *>(P.residual) + off;
            if (P.vec) {
                const uint2 u = *reinterpret_cast<const uint2 *>(rp);
                r[0] = __uint_as_float(u.x << 16); r[1] = __uint_as_float(u.x & 0xFFFF0000u);
                r[2] = __uint_as_float(u.y << 16); r[3] = __uint_as_float(u.y & 0xFFFF0000u);
            } else {
#pragma unroll
                for (int x = 0; x < 4; ++x) if (x < left) r[x] = __bfloat162float(rp[x]);
            }
        } else {
            const float *rp = reinterpret_cast<const float *>(P.residual) + off;
#pragma unroll
            for (int x = 0; x < 4; ++x) if (x < left) r[x] = rp[x];
        }
#pragma unroll
        for (int x = 0; x < 4; ++x) y[x] = P.res_gate ? (r[x] > 0.0f ? y[x] : 0.0f) : y[x] + r[x];
    }
    if (P.relu) {
#pragma unroll
        for (int x = 0; x < 4; ++x) y[x] = relu_f32(y[x]);
    }
    if (P.out_dtype == TWN_BF16) {
        __nv_bfloat16 *yp = reinterpret_cast<__nv_bfloat16 *>(P.Y) + off;
        if (P.vec) {
            const uint2 packed = make_uint2(pack_bf16x2(y[0], y[1]), pack_bf16x2(y[2], y[3]));
            *reinterpret_cast<uint2 *>(yp) = packed;
            return packed;
        } else {
#pragma unroll
            for (int x = 0; x < 4; ++x) if (x < left) yp[x] = __float2bfloat16_rn(y[x]);
        }
    } else {
        float *yp = reinterpret_cast<float *>(P.Y) + off;
        if (P.vec) {
            *reinterpret_cast<float4 *>(yp) = make_float4(y[0], y[1], y[2], y[3]);
        } else {
#pragma unroll
            for (int x = 0; x < 4; ++x) if (x < left) yp[x] = y[x];
        }
    }
    return make_uint2(0u, 0u);
}

// Adds the S partial sums of a block's pixels, in rank order, and finishes them.  A warp takes every tenth pixel, 32
// lanes x 4 channels; four 16-byte loads are in flight per thread.
struct Sums {
    const float *own, *recv;          // this lane's channels of the first pixel: this block's sums, the first peer's
    const uint32_t *off;
    int per, rank, n0, left;
};
template <int S>
__device__ __forceinline__ void final_sums(const SplitParams &P, const Sums &m, const float (&sc)[4], const float (&sf)[4])
{
    constexpr int kPix = S == 1 ? 4 : S == 2 ? 2 : 1, kStep = kThreads / 32;
#pragma unroll 1
    for (int base = threadIdx.x >> 5; base < m.per; base += kPix * kStep) {
        float4 v[kPix][S];
#pragma unroll
        for (int u = 0; u < kPix; ++u)
#pragma unroll
            for (int r = 0; r < S; ++r) {
                const int i = base + u * kStep < m.per ? base + u * kStep : base;
                const float *src = r == m.rank ? m.own : m.recv + (r < m.rank ? r : r - 1) * m.per * kPitch;
                v[u][r] = *reinterpret_cast<const float4 *>(src + i * kPitch);
            }
#pragma unroll
        for (int u = 0; u < kPix; ++u) {
            if (base + u * kStep >= m.per) break;
            const uint32_t off = m.off[base + u * kStep];
            float4 a = v[u][0];
#pragma unroll
            for (int r = 1; r < S; ++r) { a.x += v[u][r].x; a.y += v[u][r].y; a.z += v[u][r].z; a.w += v[u][r].w; }
            if (off != 0xFFFFFFFFu) finish(P, (size_t)off + m.n0, m.left, a, sc, sf);
        }
    }
}

// The same for a pooled output: a warp takes every tenth window of the block's pixels, its four pixels one after the other.
// `p0` is the block's first pixel, which starts a row pair of the tile.
template <int S>
__device__ __forceinline__ void final_sums_pool(const SplitParams &P, const Sums &m, const float (&sc)[4], const float (&sf)[4], int p0, int h0, int w0, int b0)
{
#pragma unroll 1
    for (int win = threadIdx.x >> 5; win < m.per / 4; win += kThreads / 32) {
        const int x = win & ((1 << (P.lgBW - 1)) - 1), y = win >> (P.lgBW - 1);
        const int first = (y << (P.lgBW + 1)) + 2 * x;              // in the block's share
        uint2 best = make_uint2(0xFF80FF80u, 0xFF80FF80u);
        bool whole = false;
        constexpr int kPix = S <= 4 ? 4 : 1;                         // pixels whose partial sums are in registers at once
#pragma unroll 1
        for (int q0 = 0; q0 < 4; q0 += kPix) {
            float4 v[kPix][S];
#pragma unroll
            for (int u = 0; u < kPix; ++u)
#pragma unroll
                for (int r = 0; r < S; ++r) {
                    const int q = q0 + u;
                    const float *src = r == m.rank ? m.own : m.recv + (r < m.rank ? r : r - 1) * m.per * kPitch;
                    v[u][r] = *reinterpret_cast<const float4 *>(src + (first + (q & 1) + ((q >> 1) << P.lgBW)) * kPitch);
                }
#pragma unroll
            for (int u = 0; u < kPix; ++u) {
                const int q = q0 + u;
                float4 a = v[u][0];
#pragma unroll
                for (int r = 1; r < S; ++r) { a.x += v[u][r].x; a.y += v[u][r].y; a.z += v[u][r].z; a.w += v[u][r].w; }
                const uint32_t off = m.off[first + (q & 1) + ((q >> 1) << P.lgBW)];
                whole = off != 0xFFFFFFFFu;                              // of the last pixel: the tile starts on a window
                if (!whole) continue;
                const uint2 z = finish(P, (size_t)off + m.n0, m.left, a, sc, sf);
                best.x = max_first_bf16x2(best.x, z.x);
                best.y = max_first_bf16x2(best.y, z.y);
            }
        }
        if (whole) {
            const int p = p0 + first, lgHW = P.lgBW + P.lgBH;
            const int gw = (w0 + (p & ((1 << P.lgBW) - 1))) >> 1, gh = (h0 + ((p >> P.lgBW) & ((1 << P.lgBH) - 1))) >> 1, gb = b0 + (p >> lgHW);
            *reinterpret_cast<uint2 *>(P.pool + (((size_t)gb * P.PH + gh) * P.PW + gw) * P.Cout + m.n0) =
                make_uint2(no_max_to_zero(best.x), no_max_to_zero(best.y));
        }
    }
}

// RUN: code words on whose boundaries every k-block starts.  A kernel for each: the fetch stands six times in the decode loop, and
// with the loads of other boundaries in it layers that never take them lost 1.5 % (3552x1174x72 8.18 -> 8.33 us).
template <int PIX, int BITS, bool POOL, int RUN>
__global__ void __launch_bounds__(kThreads, PIX <= 128 ? 2 : 1)
tconv_split_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ SplitParams P, int splits)
{
    using L = SplitSmem<PIX>;
    constexpr int kStages = Cfg<PIX>::kStages;
    constexpr int kCodesPerWord = 32 / BITS, kWordsPerBlock = kBlockK / kCodesPerWord;
    static_assert(PIX + kStages * kAColsPerBlock <= Cfg<PIX>::kTmem, "tensor memory budget");
    pdl_launch_dependents();
    extern __shared__ uint8_t smem_raw[];
    L *sm = reinterpret_cast<L *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    volatile int *abort_flag = &sm->abort_flag;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // a cluster's blocks are consecutive: rank = block mod splits
    const int tile = (int)blockIdx.x / splits, rank = (int)blockIdx.x - tile * splits;
    int ci = 0;
    while (ci + 1 < P.n_classes && tile >= P.cls[ci + 1].tile0) ++ci;
    const auto &C = P.cls[ci];
    const int nt = (tile - C.tile0) % P.n_tiles;
    int pt = (tile - C.tile0) / P.n_tiles;
    const int twi = pt % C.tw; pt /= C.tw;
    const int thi = pt % C.th, tbi = pt / C.th;
    const int w0 = twi << P.lgBW, h0 = thi << P.lgBH, b0 = tbi * (PIX >> (P.lgBW + P.lgBH));
    const int k0 = rank * C.kb_per_block;
    const int k1 = k0 + C.kb_per_block < C.kb ? k0 + C.kb_per_block : C.kb;
    const int n_kb = k1 > k0 ? k1 - k0 : 0;
    const int per = PIX / splits;                    // pixels that this block finishes
    const uint32_t share_bytes = (uint32_t)(per * kPitch * 4);

    if (tid == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&map_x)) : "memory");
        for (int s = 0; s < kStages; ++s) { mbar_init(&sm->full[s], 1 + 4); mbar_init(&sm->empty[s], 1); }
        mbar_init(&sm->acc_full, 1);
        mbar_init(&sm->recv_full, 1);
        sm->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (splits > 1) mbar_expect_tx(&sm->recv_full, (uint32_t)(splits - 1) * share_bytes);
    }
    for (int i = tid; i < n_kb; i += kThreads) {
        const int t = (k0 + i) / P.n_cblk, cb = k0 + i - t * P.n_cblk;
        sm->kword[i] = (uint32_t)(P.taps[C.tap0 + t].koff / kCodesPerWord) + cb * kWordsPerBlock;
    }
    for (int p = tid; p < PIX; p += kThreads) {
        const int wv = w0 + (p & ((1 << P.lgBW) - 1)), hv = h0 + ((p >> P.lgBW) & ((1 << P.lgBH) - 1)), bv = b0 + (p >> (P.lgBW + P.lgBH));
        sm->off[p] = wv < C.Wv && hv < C.Hv && bv < P.Bv
                         ? (uint32_t)((((long long)bv * P.OH + (hv * P.osh + C.ooh)) * P.OW + (wv * P.osw + C.oow)) * P.ldy)
                         : 0xFFFFFFFFu;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm->tmem_base)), "r"((uint32_t)Cfg<PIX>::kTmem) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (splits > 1) cluster_arrive();                // recv_full may be signalled: waited for before the sums are pushed
    pdl_wait();
    const uint32_t tmem = sm->tmem_base, tmem_a = tmem + PIX;

    if (warp == 0) {
        if (elect_one()) {
            int t = k0 / P.n_cblk, cb = k0 - t * P.n_cblk;
            for (int i = 0; i < n_kb; ++i) {
                const int s = i % kStages;
                if (i >= kStages && !mbar_wait(&sm->empty[s], ((i / kStages) & 1) ^ 1, abort_flag, P.status)) break;
                mbar_expect_tx(&sm->full[s], L::kXBytes);
                const Tap tap = P.taps[C.tap0 + t];
                tma_load_4d(sm->x[s], &map_x, &sm->full[s], cb * kBlockK, w0 * P.sw + tap.dw, h0 * P.sh + tap.dh, b0);
                if (++cb == P.n_cblk) { cb = 0; ++t; }
            }
        }
        __syncwarp();
    } else if (warp == 1) {
        if (elect_one()) {                               // see tc_mma_ts
            constexpr uint32_t idesc = make_idesc(kChan, PIX);
            const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sm->x[0]));
            const uint32_t b_lo0 = (uint32_t)bdesc0, b_hi = (uint32_t)(bdesc0 >> 32);
            bool ok = true;
            for (int i = 0; i < n_kb; ++i) {
                const int s = i % kStages;
                if (!mbar_wait(&sm->full[s], (i / kStages) & 1, abort_flag, P.status, 0)) { ok = false; break; }
                tc_fence_after();
                const uint32_t b_lo = b_lo0 + (uint32_t)(s * (L::kXBytes >> 4));
                if (i == 0) tc_mma_block<true>(tmem, tmem_a + s * kAColsPerBlock, b_lo, b_hi, idesc);
                else tc_mma_block<false>(tmem, tmem_a + s * kAColsPerBlock, b_lo, b_hi, idesc);
                tc_commit(&sm->empty[s]);
            }
            if (ok && n_kb > 0) tc_commit(&sm->acc_full);
        }
        __syncwarp();
    } else {
        const int q = warp & 3, set = (warp - 2) >> 2;
        const uint32_t lane_base = ((uint32_t)(q * 32) << 16);
        {
            // decode: as in tconv_kernel, the code words of this group's next k-blocks are fetched ahead
            const long long n = (long long)nt * kChan + q * 32 + lane;
            const uint32_t *rowp = P.T + (n < P.Cout ? n : P.Cout - 1) * P.wpr;
            auto fetch = [&](uint4 &c, int i) {
                const long long word = sm->kword[i < n_kb ? i : n_kb - 1], last = P.wpr - 1;
                if (BITS == 2) {
                    if (RUN == 4) {
                        ld_nc_v4(c, rowp + word);
                    } else if (RUN == 2) {
                        ld_nc_v2(c.x, c.y, rowp + word);
                        ld_nc_v2(c.z, c.w, rowp + (word + 2 < P.wpr ? word + 2 : word));
                    } else {
                        ld_nc_u32(c.x, rowp + (word + 0 < last ? word + 0 : last));
                        ld_nc_u32(c.y, rowp + (word + 1 < last ? word + 1 : last));
                        ld_nc_u32(c.z, rowp + (word + 2 < last ? word + 2 : last));
                        ld_nc_u32(c.w, rowp + (word + 3 < last ? word + 3 : last));
                    }
                } else if (RUN == 2) {
                    ld_nc_v2(c.x, c.y, rowp + word);
                } else {
                    ld_nc_u32(c.x, rowp + (word + 0 < last ? word + 0 : last));
                    ld_nc_u32(c.y, rowp + (word + 1 < last ? word + 1 : last));
                }
            };
            uint4 c0, c1, c2;
            if (n_kb > 0) { fetch(c0, set); fetch(c1, set + kSets); fetch(c2, set + 2 * kSets); }
            auto decode = [&](const uint4 &c, int i) -> bool {
                const int s = i % kStages;
                if (i >= kStages && !mbar_wait_warp(&sm->empty[s], ((i / kStages) & 1) ^ 1, abort_flag, P.status, 32)) return false;
                tc_fence_after();
                const uint32_t wv[4] = {c.x, c.y, c.z, c.w};
                uint32_t out[32];
                decode_kblock<BITS>(wv, out);
                tmem_st32(tmem_a + lane_base + s * kAColsPerBlock, out);
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->full[s]);
                return true;
            };
            // three buffers in turn, each refilled where it was used: no register is copied while its load is in flight
#pragma unroll 1
            for (int i = set; i < n_kb; i += 3 * kSets) {
                if (!decode(c0, i)) break;
                fetch(c0, i + 3 * kSets);
                if (i + kSets >= n_kb || !decode(c1, i + kSets)) break;
                fetch(c1, i + 4 * kSets);
                if (i + 2 * kSets >= n_kb || !decode(c2, i + 2 * kSets)) break;
                fetch(c2, i + 5 * kSets);
            }
        }
        // the accumulator -> shared memory, [pixel][channel]; the two warps of a lane quadrant take alternate chunks.
        // acc_full also says that the operands under `acc` have been read.
        const bool have = n_kb > 0 && mbar_wait_warp(&sm->acc_full, 0, abort_flag, P.status, 32);
        tc_fence_after();
        if (nt * kChan + q * 32 < P.Cout) {
#pragma unroll 1
            for (int c = set; c < PIX / 32; c += kSets) {
                uint32_t v[32];
                if (have) {
                    tmem_ld32(tmem + lane_base + c * 32, v);
                    tmem_wait_ld(v);
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0u;
                }
                float *dst = sm->acc + (c * 32) * kPitch + q * 32 + lane;
#pragma unroll
                for (int j = 0; j < 32; ++j) dst[j * kPitch] = __uint_as_float(v[j]);
            }
        }
        tc_fence_before();
        if (splits > 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();
    if (splits > 1) {
        cluster_wait();
        if (tid < splits && tid != rank) {
            // this block's partial sums of the pixels of block `tid`
            const uint32_t slot = (uint32_t)(rank < tid ? rank : rank - 1);
            asm volatile(
                "cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                ::"r"(peer(smem_u32(sm->recv) + slot * share_bytes, tid)), "r"(smem_u32(sm->acc) + (uint32_t)tid * share_bytes),
                  "r"(share_bytes), "r"(peer(smem_u32(&sm->recv_full), tid)) : "memory");
        }
        __syncwarp();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)Cfg<PIX>::kTmem) : "memory");
    }

    // ---- final sums and epilogue: four channels of a pixel per thread and round
    const float alpha = (P.alpha ? (float)__ldg(P.alpha) : 1.0f) * (1.0f / decoded_unit<BITS>());
    const int n0 = nt * kChan + lane * 4;
    float sc[4], sf[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
        const bool in = n0 + x < P.Cout;
        sc[x] = alpha * (P.scale && in ? __ldg(P.scale + n0 + x) : 1.0f);
        sf[x] = P.shift && in ? __ldg(P.shift + n0 + x) : 0.0f;
    }
    if (splits > 1) {
        mbar_wait_warp(&sm->recv_full, 0, abort_flag, P.status, 32);
        cluster_arrive();                            // this block has received: see the wait below
    }
    if (n0 < P.Cout) {
        const Sums sums = {sm->acc + (rank * per) * kPitch + lane * 4, sm->recv + lane * 4, sm->off + rank * per, per, rank, n0, P.Cout - n0};
        if (POOL) {
            if (splits == 1) final_sums_pool<1>(P, sums, sc, sf, rank * per, h0, w0, b0);
            else if (splits == 2) final_sums_pool<2>(P, sums, sc, sf, rank * per, h0, w0, b0);
            else if (splits == 4) final_sums_pool<4>(P, sums, sc, sf, rank * per, h0, w0, b0);
            else final_sums_pool<8>(P, sums, sc, sf, rank * per, h0, w0, b0);
        } else if (splits == 1) final_sums<1>(P, sums, sc, sf);
        else if (splits == 2) final_sums<2>(P, sums, sc, sf);
        else if (splits == 4) final_sums<4>(P, sums, sc, sf);
        else final_sums<8>(P, sums, sc, sf);
    }
    __syncwarp();
    if (splits > 1) cluster_wait();                  // all have received, so nothing reads this block's memory any more
    if (sm->abort_flag)
        for (int i = 0; i < 64; ++i) __nanosleep(1000);      // copies still in flight land before the memory is released
}

template <int PIX, int BITS, bool POOL, int RUN>
int launch_t(const Geometry &g, SplitParams &P, const void *X, int splits, const twn_device_info &dev, cudaStream_t s)
{
    static bool attr_set[64] = {false};
    auto kernel = tconv_split_kernel<PIX, BITS, POOL, RUN>;
    // At most two blocks on an SM, as many as its tensor memory holds: a block that waits for tensor memory in one
    // cluster while its peers wait for it must never be possible.
    constexpr int kFloor = 78 * 1024, kMost = std::max(kFloor, PIX == 256 ? smem_bytes<PIX>(2) : smem_bytes<PIX>(8));
    static_assert(kMost <= 232448 && 3 * (kFloor + 1024) > 233472, "shared memory");
    if (!attr_set[dev.ordinal]) {
        TWN_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost));
        attr_set[dev.ordinal] = true;
    }
    pick_tile(g, PIX, &P.lgBW, &P.lgBH);
    const int BW = 1 << P.lgBW, BH = 1 << P.lgBH, BB = PIX >> (P.lgBW + P.lgBH);
    long long tiles = 0;
    for (int c = 0; c < P.n_classes; ++c) {
        auto &C = P.cls[c];
        C.tile0 = (int)tiles;
        C.tw = (C.Wv + BW - 1) / BW;
        C.th = (C.Hv + BH - 1) / BH;
        C.kb_per_block = (C.kb + splits - 1) / splits;
        tiles += (long long)P.n_tiles * C.tw * C.th * ((g.Bv + BB - 1) / BB);
        if (tiles > 0x7fffffffLL) return TWN_ERR_INVALID_ARG;
    }
    if (tiles <= 0 || tiles * splits > 0x7fffffffLL) return TWN_ERR_INVALID_ARG;
    CUtensorMap map_x;
    cuuint64_t dims[4] = {(cuuint64_t)g.XC, (cuuint64_t)g.XW, (cuuint64_t)g.XH, (cuuint64_t)g.XB};
    const long long rowp = g.x_row_pitch ? g.x_row_pitch : g.XW * g.ldx;
    const long long imgp = g.x_img_pitch ? g.x_img_pitch : g.XH * rowp;
    cuuint64_t strides[3] = {(cuuint64_t)g.ldx * 2, (cuuint64_t)rowp * 2, (cuuint64_t)imgp * 2};
    cuuint32_t box[4] = {(cuuint32_t)kBlockK, (cuuint32_t)(BW * g.sw), (cuuint32_t)(BH * g.sh), (cuuint32_t)BB};
    cuuint32_t estr[4] = {1, (cuuint32_t)g.sw, (cuuint32_t)g.sh, 1};
    if (encode_fn()(&map_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(X), dims, strides, box, estr,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return TWN_ERR_INVALID_ARG;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * splits));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = (size_t)std::max(kFloor, smem_bytes<PIX>(splits));
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)splits;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    TWN_CUDA_OK(cudaLaunchKernelEx(&cfg, kernel, map_x, P, splits));
    return TWN_OK;
}

template <int BITS, bool POOL, int RUN>
int launch_pix(const Geometry &g, SplitParams &P, const void *X, const SplitPlan &plan, const twn_device_info &dev, cudaStream_t s)
{
    switch (plan.pix) {
        case 32: return launch_t<32, BITS, POOL, RUN>(g, P, X, plan.splits, dev, s);
        case 64: return launch_t<64, BITS, POOL, RUN>(g, P, X, plan.splits, dev, s);
        case 128: return launch_t<128, BITS, POOL, RUN>(g, P, X, plan.splits, dev, s);
        default: return launch_t<256, BITS, POOL, RUN>(g, P, X, plan.splits, dev, s);
    }
}

}  // namespace

namespace twn_detail {

// The tile and the split by a model of the launch's time, fitted to 791 launches of 82 shapes (1 to 16384 rows or 1 to
// 128 images, reductions of 64 to 19200; half of its errors are under 7 %):
//   us = -1.0 + g * (E + n R (1 + 0.25 min(1, L))) + X
// with n k-blocks per block; L blocks per SM and g = max(1, 0.61 L + 0.43), because two blocks on an SM overlap, or
// for blocks that have an SM to themselves the number of rounds, where clusters do not fill every SM; E and R what a
// block and a k-block take (few pixels make a k-block hardly cheaper: its decoding and its issue stay); X the exchange.
// What it picks takes 3 % longer on average than the best of what was measured, and a third less than without this kernel.
// The constants are those of the kernel before one elected thread issued and its code buffers rotated (0.5 us of a call of 36
// k-blocks); on 140 calls of all sizes forced into the kernel as it is, the model is 0.2 % high on average, half of its errors
// are under 7 % and a tenth over 18 % (calls of 10 to 20 us 5 % low), and what the three kernels' models pick together is 1.1 %
// behind the best of the four on average (26 % at worst: 80x19x19x96 -> 48, 3x3 stride 2, 10.0 us split, 7.9 in the general kernel).
SplitPlan plan_conv_split(const Geometry &g, int sm_count, bool in_order)
{
    static const int pixels[4] = {32, 64, 128, 256};
    static const double E[4] = {3.89, 4.47, 5.51, 7.73}, R[4] = {0.241, 0.249, 0.255, 0.275};
    SplitPlan best = {0, 0, 1e30};
    // A pooled output: up to 64 channels, where half of a tile of the general kernel is idle (14x14x64, 3x3 on 64: 16 images 7.2 us, 5.3 here, 64 images 7.8 and
    // 6.6; 12x12x64, 5x5 on 32: 32 images 8.7 and 7.4, 100 images 10.7 and 10.5, in LeNet-5 behind its first layer 2.2 us less).
    // Wider pooled layers were not timed here and stay in the general kernel, which does not split their sums: a test compares a
    // VGG-7's at 24 images bit by bit with sums in order.  Callers who ask for that order get it there as well.
    if (g.bn_partial || (g.pool && (in_order || g.code_bits != 2 || g.Cout > 64))) return best;
    // with classes: as many tiles as the largest has each (it comes first), the longest reduction and the mean one
    const int classes = g.n_classes > 0 ? g.n_classes : 1;
    const long long cblk = (g.Cin + kBlockK - 1) / kBlockK;
    long long kb = g.n_classes > 0 ? 0 : g.n_taps * cblk;
    for (int c = 0; c < g.n_classes; ++c) kb = std::max(kb, g.cls[c].n_taps * cblk);
    const double mean = g.n_classes > 0 && kb > 0 ? (double)g.n_taps * cblk / classes / kb : 1.0;
    const int n_tiles = (g.Cout + kChan - 1) / kChan;
    for (int i = 0; i < 4; ++i) {
        int a, b;
        const int pix = pixels[i];
        const long long tiles = pick_tile(g, pix, &a, &b) * n_tiles;
        for (int splits = 1; splits <= (in_order ? 1 : pix == 256 ? 2 : 8); splits *= 2) {
            const long long n = (kb + splits - 1) / splits;
            if ((splits > 1 && splits > kb) || n > kMaxBlocks) continue;
            if (g.pool && pix / splits < 2 << a) continue;
            const double ctas = (double)tiles * classes * splits, L = ctas / sm_count;
            const bool alone = pix == 256 || (pix == 128 && splits >= 4);
            // clusters of 4 and 8 fill 128 and 112 of 148 SMs
            const double slots = sm_count * (splits == 8 ? 112.0 / 148 : splits == 4 ? 128.0 / 148 : splits == 2 ? 144.0 / 148 : 1.0);
            const double rounds = alone ? std::ceil(ctas / slots) : std::max(1.0, 0.607 * L + 0.428);
            const double x = splits > 1 ? 0.58 + pix * (0.0004 + 0.0008 * splits) : 0.0;
            const double r = n * R[i] * (1.0 + 0.25 * std::min(1.0, L));
            const double us = -1.0 + std::max(E[i] + r, rounds * (E[i] + mean * r)) + x * (alone ? rounds : 1.0);
            if (us < best.us) best = SplitPlan{pix, splits, us};
        }
    }
    return best;
}

int launch_conv_split(const Geometry &g, const void *X, const uint32_t *T, const EpilogueArgs &epi, void *Y,
                      int32_t *dev_status, const twn_device_info &dev, cudaStream_t s, const SplitPlan &plan)
{
    SplitParams P;
    P.n_tiles = (g.Cout + kChan - 1) / kChan;
    P.n_cblk = (int)((g.Cin + kBlockK - 1) / kBlockK);
    P.n_classes = g.n_classes > 0 ? g.n_classes : 1;
    for (int c = 0; c < P.n_classes; ++c) {
        const TapClass k = g.n_classes > 0 ? g.cls[c] : TapClass{g.Hv, g.Wv, g.ooh, g.oow, 0, g.n_taps};
        P.cls[c].Hv = k.Hv; P.cls[c].Wv = k.Wv; P.cls[c].ooh = k.ooh; P.cls[c].oow = k.oow;
        P.cls[c].tap0 = k.tap0;
        P.cls[c].kb = k.n_taps * P.n_cblk;
    }
    const int run = code_run(g);
    for (int t = 0; t < g.n_taps; ++t) P.taps[t] = g.taps[t];
    P.T = T;
    P.wpr = g.ld_codes / (g.code_bits == 1 ? 32 : 16);
    P.sw = g.sw; P.sh = g.sh;
    P.Bv = g.Bv;
    P.OH = g.OH; P.OW = g.OW; P.osh = g.osh; P.osw = g.osw;
    P.ldy = g.ldy;
    P.Cout = g.Cout;
    P.alpha = epi.alpha; P.scale = epi.scale; P.shift = epi.shift;
    P.residual = epi.residual; P.res_dtype = epi.res_dtype; P.res_gate = epi.res_gate;
    P.relu = epi.relu; P.out_dtype = epi.out_dtype;
    const int es = epi.out_dtype == TWN_BF16 ? 2 : 4;
    P.vec = g.Cout % 4 == 0 && g.ldy % 4 == 0 && reinterpret_cast<uintptr_t>(Y) % (4 * es) == 0 &&
            (!epi.residual || reinterpret_cast<uintptr_t>(epi.residual) % 8 == 0);
    P.Y = Y;
    P.pool = static_cast<__nv_bfloat16 *>(g.pool);
    P.PH = g.Hv / 2; P.PW = g.Wv / 2;
    if (g.pool && !P.vec) return TWN_ERR_CUDA;       // the caller has looked at the alignment
    P.status = dev_status;
    const bool b1 = g.code_bits == 1;
    if (g.pool)
        return run == 4 ? launch_pix<2, true, 4>(g, P, X, plan, dev, s) : run == 2 ? launch_pix<2, true, 2>(g, P, X, plan, dev, s)
                                                                      : launch_pix<2, true, 1>(g, P, X, plan, dev, s);
    if (b1) return run == 2 ? launch_pix<1, false, 2>(g, P, X, plan, dev, s) : launch_pix<1, false, 1>(g, P, X, plan, dev, s);
    return run == 4 ? launch_pix<2, false, 4>(g, P, X, plan, dev, s) : run == 2 ? launch_pix<2, false, 2>(g, P, X, plan, dev, s)
                                                                   : launch_pix<2, false, 1>(g, P, X, plan, dev, s);
}

}  // namespace twn_detail
