// Binary precision weights (Sec. 3: the BPWN baseline binarizes the weights with the sign function;
// like the ternary weights they carry one scale per layer) fused with 1-bit packing, and the helpers
// for the 1-bit format (unpack, re-layout for the backward-for-data pass).
//
//   B_i = +1 if W_i >= 0, -1 if W_i < 0;      alpha = (1/n) sum |W_i|
//
// Neither needs a threshold, so one sweep over the fp32 master weights does both: 4 bytes read and
// 1/32 byte written per weight, bound by HBM bandwidth.  A thread holds eight quarters of four weights; their 32 signs
// are collected by funnel shifts, and an 8x8 transpose of 4-bit groups among eight lanes leaves every lane with one
// whole word.  (A warp vote per word of 32 costs a 4-byte load, a vote and a select per weight of a lane, and rows that
// are no whole words were voted one word at a time.)
// sum |W| has a fixed order: per-thread fp64 sums, the trees of sweep.cuh, one part per block.  The blocks meet through
// the workspace and a launch that folds them, those of a small tensor as one cluster through distributed shared memory.
#include <algorithm>

#include "sweep.cuh"

namespace {

constexpr int kThreads = 256;            // the helpers below
constexpr int kGroupWords = 512;         // words of a group: eight quarter-words per thread
// workspace: kMaxParts fp64 sums, then kMaxParts negative counts (the size is that of an earlier layout)
constexpr size_t kBinWorkspaceBytes = 256 + 2 * size_t(2048) * 8;

__host__ __device__ inline int bit_of_element(int e) { return 15 - (e >> 1) + 16 * (e & 1); }

struct BinParams {
    const float *W;
    uint32_t *packed;
    twn_stats_t *stats;
    double *part_sum;
    unsigned long long *part_neg;
    unsigned long long n, words;         // weights; words that hold codes
    long long rows, cols, wpr;
    unsigned int wpr_used, parts, part_words;
    bool vec4, dense;                    // quarters start on 16-byte boundaries; word w holds weights 32 w ..
};

// Word w: its index in the packed matrix, its first weight and how many weights it holds.
struct BinPlace {
    unsigned long long out, f;
    unsigned int valid;
};
__device__ __forceinline__ BinPlace bin_place(const BinParams &P, unsigned long long w)
{
    BinPlace p;
    if (P.dense) {
        p.out = w;
        p.f = 32ull * w;
        p.valid = (unsigned int)min(32ull, P.n - p.f);
    } else {
        const unsigned long long row = w >> 32 ? w / P.wpr_used : (unsigned int)w / P.wpr_used;
        const unsigned long long j = w - row * P.wpr_used;
        p.out = row * P.wpr + j;
        p.f = row * P.cols + 32 * j;
        p.valid = (unsigned int)min(32ull, (unsigned long long)P.cols - 32 * j);
    }
    return p;
}

// Eight nibbles of x, exchanged among the lanes of an aligned group of eight: lane l gets nibble l of every lane.
__device__ __forceinline__ uint32_t exchange_nibbles(uint32_t x)
{
    const int lane = threadIdx.x;
    uint32_t y = __shfl_xor_sync(0xffffffffu, x, 4);
    x = __byte_perm(x, y, (lane & 4) ? 0x3276 : 0x5410);
    y = __shfl_xor_sync(0xffffffffu, x, 2);
    x = __byte_perm(x, y, (lane & 2) ? 0x3715 : 0x6240);
    y = __shfl_xor_sync(0xffffffffu, x, 1);
    return (lane & 1) ? ((x & 0xF0F0F0F0u) | ((y >> 4) & 0x0F0F0F0Fu)) : ((x & 0x0F0F0F0Fu) | ((y << 4) & 0xF0F0F0F0u));
}

__device__ __forceinline__ void write_binary(const BinParams &P, double s, unsigned long long n_neg)
{
    P.stats->delta = 0.0;
    P.stats->alpha = P.n > 0 ? s / (double)P.n : 0.0;
    P.stats->sum_abs = s;
    P.stats->sum_abs_kept = s;
    P.stats->n_neg = n_neg;
    P.stats->n_zero = 0;
    P.stats->n_pos = P.n - n_neg;
    P.stats->status = isfinite(s) ? TWN_OK : TWN_ERR_NONFINITE;
    P.stats->reserved = 0;
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kSweepThreads, kSweepBlocksPerSm)
binarize_kernel(const __grid_constant__ BinParams P)
{
    __shared__ Reduce red;
    __shared__ double sum_s[kSmallParts];
    __shared__ unsigned long long neg_s[kSmallParts];
    const unsigned int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x, G = gridDim.x;
    unsigned int turn = 0;
    if (CLUSTER) {
        if (tid < kSmallParts) { sum_s[tid] = 0.0; neg_s[tid] = 0ull; }
        pdl_begin();
        cluster_arrive();
    } else {
        chain_wait();
    }
    // padding words of the rows
    const unsigned int pad = (unsigned int)(P.wpr - P.wpr_used);
    if (pad && P.packed)
        for (unsigned long long i = (unsigned long long)b * kSweepThreads + tid; i < (unsigned long long)P.rows * pad; i += (unsigned long long)G * kSweepThreads) {
            const unsigned long long r = i >> 32 ? i / pad : (unsigned int)i / pad;
            P.packed[r * P.wpr + P.wpr_used + (i - r * pad)] = 0u;
        }
    double own = 0.0;
    unsigned long long own_neg = 0;
    for (unsigned int part = b; part < P.parts; part += G) {
        const unsigned long long w0 = (unsigned long long)part * P.part_words;
        const unsigned long long w1 = min(w0 + P.part_words, P.words);
        double a[4] = {0.0, 0.0, 0.0, 0.0};
        unsigned int neg = 0, none = 0;
        for (unsigned long long wg = w0; wg < w1; wg += kGroupWords) {
            float4 v[8];
            if (P.dense && P.vec4 && wg + kGroupWords <= w1 && (wg + kGroupWords) * 32 <= P.n) {
                const float4 *v4 = reinterpret_cast<const float4 *>(P.W) + wg * 8 + tid;
#pragma unroll
                for (int k = 0; k < 8; ++k) v[k] = __ldg(v4 + k * kSweepThreads);
            } else {
                // quarter-words that are not whole are masked; addresses stay inside the part
                unsigned long long f[8];
                unsigned int left[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const unsigned long long w = wg + (k * kSweepThreads + tid) / 8;
                    const unsigned int e = 4 * (tid & 7);
                    const BinPlace p = bin_place(P, min(w, w1 - 1));
                    left[k] = w < w1 && p.valid > e ? p.valid - e : 0;
                    f[k] = left[k] ? p.f + e : p.f;
                }
                if (P.vec4 && !P.dense) {
#pragma unroll
                    for (int k = 0; k < 8; ++k) v[k] = __ldg(reinterpret_cast<const float4 *>(P.W + f[k]));
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k) {
                        v[k].x = left[k] > 0 ? __ldg(P.W + f[k]) : 0.0f;
                        v[k].y = left[k] > 1 ? __ldg(P.W + f[k] + 1) : 0.0f;
                        v[k].z = left[k] > 2 ? __ldg(P.W + f[k] + 2) : 0.0f;
                        v[k].w = left[k] > 3 ? __ldg(P.W + f[k] + 3) : 0.0f;
                    }
                }
#pragma unroll
                for (int k = 0; k < 8; ++k)
                    if (left[k] < 4) {
                        if (left[k] < 1) v[k].x = 0.0f;
                        if (left[k] < 2) v[k].y = 0.0f;
                        if (left[k] < 3) v[k].z = 0.0f;
                        v[k].w = 0.0f;
                    }
            }
            // nibble k of `signs`: elements 0, 2, 1, 3 of quarter k, the first on the left
            uint32_t signs = 0;
#pragma unroll
            for (int k = 7; k >= 0; --k) {
                const float x4[4] = {v[k].x, v[k].z, v[k].y, v[k].w};
#pragma unroll
                for (int x = 0; x < 4; ++x) {
                    a[x] += (double)fabsf(x4[x]);
                    // "negative" is w < 0, which -0.0 is not: adding zero makes it +0.0
                    signs = __funnelshift_l(__float_as_uint(__fadd_rn(x4[x], 0.0f)), signs, 1);
                }
            }
            neg += __popc(signs);
            // Lane l now has word l % 8 of the eight that its group shares, a quarter per nibble, the first on the right:
            // reverse the nibbles, then even elements to the low half and odd ones to the high half.
            uint32_t x = __byte_perm(exchange_nibbles(signs), 0u, 0x0123);
            x = ((x >> 4) & 0x0F0F0F0Fu) | ((x << 4) & 0xF0F0F0F0u);
            uint32_t even = (x >> 2) & 0x33333333u, odd = x & 0x33333333u;
            even = (even | (even >> 2)) & 0x0F0F0F0Fu; odd = (odd | (odd >> 2)) & 0x0F0F0F0Fu;
            even = (even | (even >> 4)) & 0x00FF00FFu; odd = (odd | (odd >> 4)) & 0x00FF00FFu;
            even = (even | (even >> 8)) & 0x0000FFFFu; odd = (odd | (odd >> 8)) & 0x0000FFFFu;
            const unsigned long long w = wg + (lane & 7) * (kSweepThreads / 8) + warp * 4 + (lane >> 3);
            if (w < w1) P.packed[P.dense ? w : bin_place(P, w).out] = even | (odd << 16);
        }
        const double s = sweep_sum((a[0] + a[1]) + (a[2] + a[3]), neg, none, red, turn);
        if (CLUSTER) {
            own = s;                     // a block of the cluster has at most one part
            own_neg = neg;
        } else if (tid == 0) {
            P.part_sum[part] = s;
            P.part_neg[part] = neg;
        }
    }
    if (CLUSTER) {
        cluster_wait();
        if (tid == 0) {
            st_peer(peer_smem(&sum_s[b], 0), __double_as_longlong(own));
            st_peer(peer_smem(&neg_s[b], 0), own_neg);
        }
        cluster_arrive();
        cluster_wait();
        if (b != 0 || tid != 0) return;
        unsigned long long c = 0;
        for (int i = 0; i < kSmallParts; ++i) c += neg_s[i];
        write_binary(P, tree8(sum_s), c);
    }
}
// The parts' sums of a larger tensor: a launch of its own that is there when the sweep ends (in one cooperative launch with a
// grid-wide barrier 663 thousand weights took 8.3 us, 6.4 now).
__global__ void __launch_bounds__(kSweepThreads)
binarize_fold_kernel(const BinParams P)
{
    __shared__ Reduce red;
    unsigned int turn = 0;
    chain_wait();
    double s = 0.0;
    unsigned int lo = 0, hi = 0;         // of at most kMaxParts counts below 2^32: no carry gets lost
    for (unsigned int i = threadIdx.x; i < P.parts; i += kSweepThreads) {
        s += __ldcg(P.part_sum + i);
        const unsigned long long k = __ldcg(P.part_neg + i);
        lo += (unsigned int)(k & 0xFFFFFull);
        hi += (unsigned int)(k >> 20);
    }
    s = sweep_sum(s, lo, hi, red, turn);
    if (threadIdx.x == 0) write_binary(P, s, lo + ((unsigned long long)hi << 20));
}

__global__ void __launch_bounds__(kThreads)
unpack_b1_kernel(const uint32_t *__restrict__ packed, long long rows, long long cols, long long ld_codes,
                 int8_t *__restrict__ codes)
{
    const long long wpr = ld_codes >> 5, total = rows * cols;
    for (long long i = (long long)blockIdx.x * kThreads + threadIdx.x; i < total; i += (long long)gridDim.x * kThreads) {
        const long long r = i / cols, c = i - r * cols;
        const uint32_t w = __ldg(packed + r * wpr + (c >> 5));
        codes[i] = ((w >> bit_of_element((int)(c & 31))) & 1u) ? -1 : 1;
    }
}

// [Cout][taps][Cin] -> [Cin][taps][Cout]: a thread builds one word of the output
__global__ void __launch_bounds__(kThreads)
transpose_b1_kernel(const uint32_t *__restrict__ in, long long ld_in, int Cout, int Cin, int taps,
                    uint32_t *__restrict__ out, long long ld_out)
{
    const long long wpr_in = ld_in >> 5, wpr_out = ld_out >> 5, total = (long long)Cin * wpr_out;
    for (long long w = (long long)blockIdx.x * kThreads + threadIdx.x; w < total; w += (long long)gridDim.x * kThreads) {
        const long long c = w / wpr_out, j0 = (w - c * wpr_out) << 5;
        uint32_t word = 0u;
        for (int e = 0; e < 32; ++e) {
            const long long j = j0 + e;                       // column of the output row: tap * Cout + o
            if (j >= (long long)taps * Cout) break;
            const long long t = j / Cout, o = j - t * Cout;
            const long long src = t * Cin + c;                // column of input row o
            const uint32_t bit = (__ldg(in + o * wpr_in + (src >> 5)) >> bit_of_element((int)(src & 31))) & 1u;
            word |= bit << bit_of_element(e);
        }
        out[w] = word;
    }
}

int grid_for_words(long long work, int sms)
{
    long long g = (work + kThreads - 1) / kThreads;
    const long long cap = (long long)sms * 8;
    if (g > cap) g = cap;
    if (g < 1) g = 1;
    return (int)g;
}

}  // namespace

extern "C" size_t twn_binarize_workspace_bytes(void) { return kBinWorkspaceBytes; }

extern "C" int twn_binarize(const float *W, int64_t rows, int64_t cols, twn_stats_t *stats, uint32_t *packed,
                            int64_t ld_codes, void *workspace, size_t workspace_bytes, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0 && stats != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ld_codes >= cols && ld_codes % 128 == 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(cols == 0 || rows <= (int64_t)0x3fffffffffffLL / (cols > ld_codes ? cols : ld_codes), TWN_ERR_INVALID_ARG);
    const long long n = (long long)rows * cols;
    TWN_REQUIRE(n == 0 || (W != nullptr && packed != nullptr), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace != nullptr && workspace_bytes >= kBinWorkspaceBytes, TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(W, 4) && twn_aligned(packed, 16) && twn_aligned(stats, 8) && twn_aligned(workspace, 256),
                TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    BinParams P;
    P.W = W; P.packed = packed; P.stats = stats;
    P.part_sum = static_cast<double *>(workspace);
    P.part_neg = reinterpret_cast<unsigned long long *>(P.part_sum + kMaxParts);
    P.n = (unsigned long long)n;
    P.rows = rows; P.cols = cols; P.wpr = ld_codes / 32;
    const unsigned long long used = (unsigned long long)(cols + 31) / 32;
    P.words = (unsigned long long)rows * used;
    // whole groups per part, at most one part per block of a full grid
    const unsigned long long part = std::max(1ull, ((P.words + kMaxParts - 1) / kMaxParts + kGroupWords - 1) / kGroupWords) * kGroupWords;
    TWN_REQUIRE(used <= 0xFFFFFFFFull && part <= 0x04000000ull, TWN_ERR_TOO_LARGE);
    P.wpr_used = (unsigned int)used;
    P.part_words = (unsigned int)part;
    P.parts = (unsigned int)std::max(1ull, (P.words + part - 1) / part);
    P.vec4 = twn_aligned(W, 16) && (rows == 1 || cols % 4 == 0);
    P.dense = rows == 1 || ld_codes == cols;
    if (P.parts <= (unsigned int)kSmallParts) {
        unsigned int grid = 1;
        while (grid < P.parts) grid *= 2;
        return launch_cluster(binarize_kernel<true>, grid, twn_cu(stream), P);
    }
    TWN_CUDA_OK(twn_launch_pdl(true, binarize_kernel<false>, (int)std::min(P.parts, (unsigned int)(dev.sm_count * kSweepBlocksPerSm)),
                               kSweepThreads, 0, twn_cu(stream), P));
    TWN_CUDA_OK(twn_launch_pdl(true, binarize_fold_kernel, 1, kSweepThreads, 0, twn_cu(stream), P));
    return TWN_OK;
}

extern "C" int twn_unpack_b1(const uint32_t *packed, int64_t rows, int64_t cols, int64_t ld_codes, int8_t *codes,
                             twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0 && ld_codes >= cols && ld_codes % 128 == 0, TWN_ERR_INVALID_ARG);
    if (rows == 0 || cols == 0) return TWN_OK;
    TWN_REQUIRE(packed && codes, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed, 16), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    unpack_b1_kernel<<<grid_for_words((long long)rows * cols, dev.sm_count), kThreads, 0, twn_cu(stream)>>>(
        packed, rows, cols, ld_codes, codes);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

extern "C" int twn_transpose_codes_b1(const uint32_t *packed_fwd, int64_t ld_fwd, const twn_conv_desc_t *d,
                                      uint32_t *packed_bwd, int64_t ld_bwd, twn_stream_t stream)
{
    TWN_REQUIRE(d != nullptr && packed_fwd && packed_bwd, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->Cin > 0 && d->Cout > 0 && d->kh > 0 && d->kw > 0, TWN_ERR_INVALID_ARG);
    const long long taps = (long long)d->kh * d->kw;
    TWN_REQUIRE(ld_fwd % 128 == 0 && ld_bwd % 128 == 0 && ld_fwd >= taps * d->Cin && ld_bwd >= taps * d->Cout,
                TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->Cin <= 0x7fffffffLL && d->Cout <= 0x7fffffffLL && taps <= 4096, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed_fwd, 16) && twn_aligned(packed_bwd, 16), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    const long long words = d->Cin * (ld_bwd / 32);
    transpose_b1_kernel<<<grid_for_words(words, dev.sm_count), kThreads, 0, twn_cu(stream)>>>(
        packed_fwd, ld_fwd, (int)d->Cout, (int)d->Cin, (int)taps, packed_bwd, ld_bwd);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}
