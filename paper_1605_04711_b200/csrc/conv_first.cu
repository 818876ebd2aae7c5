// Forward pass of a layer on few input channels, straight from the image (the first layers of LeNet-5 and VGG-7), with the
// 2x2 pooling of its output beside it where that is asked for.
//
// What bounds such a layer is its output: a reduction of 25 or 27 elements is a few microseconds of any matrix pipe, and the
// patch matrix that twn_gemm needs is written, read and launched for it.  128x32x32x3 -> 128, 3x3: 18.6 us that way, 10.9 here (5.2
// for its 34 MB at the copy rate; two rounds of units, the second 73 % full, at half an instruction a cycle and scheduler);
// 100x28x28x1 -> 32, 5x5, with its pooling 12.1 us in three launches, 3.8 here.  So the patches are gathered from a piece of the image
// in shared memory into the registers of warp-wide MMAs (m16n8k16: 16 pixels, eight channels; the operands of tcgen05 would have
// to be written to shared memory once more first), and everything after that stays in the thread that holds the sum:
//   - a warp's unit is eight 2x2 windows of output pixels: rows g and g + 8 of its two pixel tiles are the four pixels of
//     window g, so their maximum is taken in registers;
//   - channels are dealt to the columns so that a thread holds eight neighbouring ones: 16-byte stores, 64 bytes a pixel and
//     instruction;
//   - the decoded weights of up to 128 channels lie in shared memory as the threads' operands; a warp walks units, each with its
//     own piece of the image, the next one's on its way meanwhile: no barrier (a piece for a block, loaded between two of them, and
//     the weights in registers: 128x32x32x3 -> 128 15.6 us).
#include <cuda_bf16.h>
#include <string.h>

#include <algorithm>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "tconv_host.cuh"

namespace {

constexpr int kT = 256, kWarps = kT / 32;
constexpr int kMostK = 64, kMostCin = 8;     // elements of a filter, channels: a unit's piece of the image is 5 KB at most
constexpr int kMostPiece = 2560;             // elements of it (8 x 1 filters on 8 channels, stride 2: 2480)
constexpr int kAhead = 8;                    // elements of the next piece that a lane holds; more are loaded when they are needed

struct FirstParams {
    const __nv_bfloat16 *X;
    const uint32_t *T;
    const double *alpha;
    const float *scale, *shift;
    __nv_bfloat16 *Y, *Yp;
    int B, H, W, Cin, Ho, Wo, PH, PW, Cout, kw, K, sh, sw, ph, pw;
    int wpr;                                 // code words of a filter's row
    int lgUx, nx, ny, units;                 // a unit: 2^lgUx windows by the rest of eight; units of an image, units
    int rows, pitch;                         // its piece of the image: rows, elements of a row
    int splits, groups;                      // blocks that share units, each its own channels: so many groups of 32
};

__device__ __forceinline__ uint32_t ld_shared_u16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}
template <bool ACC>
__device__ __forceinline__ void mma_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    if (!ACC)
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%10, %10, %10, %10};"
                     : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
                     : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.0f));
    else
        asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// KS steps of 16 reduction elements
template <int KS, bool RELU, bool POOL>
__global__ void __launch_bounds__(kT, 2)
conv_first_kernel(const FirstParams P)
{
    extern __shared__ __align__(16) unsigned char first_smem[];
    uint2 *const wt = reinterpret_cast<uint2 *>(first_smem);                // decoded weights: [group][step][channel tile][lane]
    float *const affine = reinterpret_cast<float *>(wt + P.groups * KS * 4 * 32);  // scale and shift of the block's channels
    int *const koff = reinterpret_cast<int *>(affine + 2 * 32 * P.groups);  // byte offset of a filter element in a piece
    const int size = P.rows * P.pitch;
    uint32_t *const place = reinterpret_cast<uint32_t *>(koff + kMostK);    // row and element of the row of a piece's elements
    uint16_t *const pieces = reinterpret_cast<uint16_t *>(place + (size + 31) / 32 * 32);
    pdl_launch_dependents();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const int ch0 = (int)(blockIdx.x % P.splits) * (32 * P.groups);
    uint16_t *const mine = pieces + warp * ((size + 7) / 8 * 8);
    if (threadIdx.x < kMostK) {
        const int k = (int)threadIdx.x, c = k % P.Cin, tap = k / P.Cin, r = tap / P.kw, s = tap - r * P.kw;
        koff[k] = k < P.K ? 2 * (r * P.pitch + s * P.Cin + c) : 0;
    }
    for (int i = threadIdx.x; i < size; i += kT) {
        const int r = i / P.pitch;
        place[i] = (uint32_t)r << 16 | (uint32_t)(i - r * P.pitch);
    }
    pdl_wait();
    if (threadIdx.x < 32 * P.groups) {
        const int n = ch0 + (int)threadIdx.x;
        const float alpha = (P.alpha ? (float)__ldg(P.alpha) : 1.0f) * (1.0f / kDecodedUnit);
        affine[threadIdx.x] = (P.scale && n < P.Cout ? __ldg(P.scale + n) : 1.0f) * alpha;
        affine[32 * P.groups + threadIdx.x] = P.shift && n < P.Cout ? __ldg(P.shift + n) : 0.0f;
    }
    // column n of channel tile j is channel 8 (n / 2) + 2 j + n % 2 of its group
    for (int i = warp; i < P.groups * KS * 4; i += kWarps) {
        const int j = i & 3, ks = (i >> 2) % KS, cg = (i >> 2) / KS;
        const int n = ch0 + cg * 32 + (g >> 1) * 8 + j * 2 + (g & 1);
        const uint32_t w = __ldg(P.T + (size_t)(n < P.Cout ? n : P.Cout - 1) * P.wpr + ks);
        wt[i * 32 + lane] = make_uint2(pair_to_bf16x2(w, t), pair_to_bf16x2(w, t + 4));
    }
    __syncthreads();
    // where this thread's elements of a patch lie, from the patch's first; past the filter's end they count as zero
    int off[KS][4];
    uint32_t keep[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int k = ks * 16 + 2 * t + (e & 1) + (e >> 1) * 8;
            off[ks][e] = koff[k];
            if (ks == KS - 1 && k >= P.K) keep[e >> 1] &= e & 1 ? 0x0000FFFFu : 0xFFFF0000u;
        }

    const int dx = 2 * P.sw * P.Cin, dy = 2 * P.sh * P.pitch;      // bytes to the pixel on the right and below
    const int line = P.W * P.Cin, Uy = 8 >> P.lgUx;
    const int lx = g & ((1 << P.lgUx) - 1), ly = g >> P.lgUx;
    const uint32_t base = smem_u32(mine) + 2 * ly * dy + 2 * lx * dx;
    const uint32_t right = (uint32_t)P.Cout, below = (uint32_t)P.Wo * P.Cout;
    // element i of the piece of a unit; x0 and y0 place the piece in image b, whose first row is `src`
    struct Where { int b, xi, yi; };
    auto where = [&](int unit) -> Where {
        const int q = unit / P.nx, b = q / P.ny;
        return {b, unit - q * P.nx, q - b * P.ny};
    };
    auto element = [&](const Where &w, int i) -> uint16_t {
        const uint32_t at = place[i];
        const int y = 2 * (w.yi * Uy) * P.sh - P.ph + (int)(at >> 16), x = (2 * (w.xi << P.lgUx) * P.sw - P.pw) * P.Cin + (int)(at & 0xFFFF);
        const uint16_t *src = reinterpret_cast<const uint16_t *>(P.X) + ((size_t)w.b * P.H + y) * line + x;
        return y >= 0 && y < P.H && x >= 0 && x < line ? __ldg(src) : (uint16_t)0;
    };
    const int stride = (int)(gridDim.x / P.splits) * kWarps;
    int unit = (int)(blockIdx.x / P.splits) * kWarps + warp;
    uint16_t ahead[kAhead];
    Where at = where(unit);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) ahead[i] = unit < P.units && lane + 32 * i < size ? element(at, lane + 32 * i) : (uint16_t)0;
#pragma unroll 1
    for (; unit < P.units; unit += stride) {
        const int wy = at.yi * Uy + ly, wx = (at.xi << P.lgUx) + lx, b = at.b;
        __syncwarp();                                            // the piece before has been read
#pragma unroll
        for (int i = 0; i < kAhead; ++i)
            if (lane + 32 * i < size) mine[lane + 32 * i] = ahead[i];
        for (int i = lane + 32 * kAhead; i < size; i += 32) mine[i] = element(at, i);
        __syncwarp();
        if (unit + stride < P.units) {
            at = where(unit + stride);
#pragma unroll
            for (int i = 0; i < kAhead; ++i)
                if (lane + 32 * i < size) ahead[i] = element(at, lane + 32 * i);
        }
        uint32_t first = base;
        if (KS > 2) asm volatile("" : "+r"(first));              // 32 addresses are kept in registers, 48 or 64 would be spilled
        uint32_t a[2][KS][4];
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                for (int q = 0; q < 4; ++q) {                    // q: column half * 2 + pixel of the row
                    const uint32_t p = first + m * dy + (q & 1) * dx;
                    a[m][ks][q] = __byte_perm(ld_shared_u16(p + off[ks][(q >> 1) * 2]), ld_shared_u16(p + off[ks][(q >> 1) * 2 + 1]), 0x5410);
                    if (ks == KS - 1) a[m][ks][q] &= keep[q >> 1];
                }
        const int oy = 2 * wy, ox = 2 * wx;
        const uint32_t y_at = (((uint32_t)b * P.Ho + oy) * P.Wo + ox) * P.Cout + ch0 + t * 8;
        const uint32_t p_at = (((uint32_t)b * P.PH + wy) * P.PW + wx) * P.Cout + ch0 + t * 8;
        const bool row0 = oy < P.Ho, row1 = oy + 1 < P.Ho, col0 = ox < P.Wo, col1 = ox + 1 < P.Wo;
#pragma unroll 1
        for (int cg = 0; cg < P.groups; ++cg) {
            float d[2][4][4];
#pragma unroll
            for (int ks = 0; ks < KS; ++ks)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const uint2 w = wt[((cg * KS + ks) * 4 + j) * 32 + lane];
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        if (ks == 0) mma_16816<false>(d[m][j], a[m][ks], w.x, w.y);
                        else mma_16816<true>(d[m][j], a[m][ks], w.x, w.y);
                    }
                }
            const bool on = ch0 + cg * 32 + t * 8 < P.Cout;
            const float4 *const sc = reinterpret_cast<const float4 *>(affine + cg * 32 + t * 8);
            const float4 sc0 = sc[0], sc1 = sc[1], sf0 = sc[8 * P.groups], sf1 = sc[8 * P.groups + 1];
            const float s[8] = {sc0.x, sc0.y, sc0.z, sc0.w, sc1.x, sc1.y, sc1.z, sc1.w};
            const float f[8] = {sf0.x, sf0.y, sf0.z, sf0.w, sf1.x, sf1.y, sf1.z, sf1.w};
            uint32_t best[4] = {0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u};
#pragma unroll
            for (int q = 0; q < 4; ++q) {                        // the window's pixels in scan order
                uint32_t v[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t y0 = __float_as_uint(d[q >> 1][j][(q & 1) * 2]), y1 = __float_as_uint(d[q >> 1][j][(q & 1) * 2 + 1]);
                    fma_f32x2(y0, y1, s[2 * j], s[2 * j + 1], f[2 * j], f[2 * j + 1]);
                    v[j] = RELU ? pack_bf16x2_relu(__uint_as_float(y0), __uint_as_float(y1)) : pack_bf16x2(__uint_as_float(y0), __uint_as_float(y1));
                    if (POOL) best[j] = max_first_bf16x2(best[j], v[j]);
                }
                if (on && (q >> 1 ? row1 : row0) && (q & 1 ? col1 : col0))
                    *reinterpret_cast<uint4 *>(P.Y + (y_at + (q >> 1 ? below : 0u) + (q & 1 ? right : 0u) + cg * 32)) = make_uint4(v[0], v[1], v[2], v[3]);
            }
            if (POOL && on && row1 && col1)
                *reinterpret_cast<uint4 *>(P.Yp + (p_at + cg * 32)) =
                    make_uint4(no_max_to_zero(best[0]), no_max_to_zero(best[1]), no_max_to_zero(best[2]), no_max_to_zero(best[3]));
        }
    }
}

template <int KS>
int launch_first(FirstParams &P, int relu, const twn_device_info &dev, cudaStream_t s)
{
    const int all = (P.Cout + 31) / 32;
    P.splits = (all + 3) / 4;
    P.groups = (all + P.splits - 1) / P.splits;
    const int size = P.rows * P.pitch;
    const size_t smem = (size_t)(P.groups * (KS * 4 * 32 * 8 + 2 * 32 * 4) + kMostK * 4 + (size + 31) / 32 * 128 + kWarps * ((size + 7) / 8 * 16));
    const long long blocks = std::min(((long long)P.units + kWarps - 1) / kWarps, std::max(1LL, 2LL * dev.sm_count / P.splits)) * P.splits;
    if (blocks > 0x7fffffffLL) return TWN_ERR_TOO_LARGE;
    constexpr size_t kMostSmem = 4 * (KS * 4 * 32 * 8 + 2 * 32 * 4) + kMostK * 4 + kMostPiece * 4 + kWarps * kMostPiece * 2;
    static_assert(2 * (kMostSmem + 1024) <= 233472, "two blocks on an SM");
    static bool attr_set[64] = {false};
    constexpr decltype(&conv_first_kernel<KS, false, false>) kernels[2][2] = {
        {conv_first_kernel<KS, false, false>, conv_first_kernel<KS, false, true>},
        {conv_first_kernel<KS, true, false>, conv_first_kernel<KS, true, true>}};
    if (!attr_set[dev.ordinal]) {
        for (int i = 0; i < 4; ++i)
            TWN_CUDA_OK(cudaFuncSetAttribute(kernels[i / 2][i % 2], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMostSmem));
        attr_set[dev.ordinal] = true;
    }
    TWN_CUDA_OK(twn_launch_pdl(true, kernels[relu][P.Yp != nullptr], (int)blocks, kT, smem, s, P));
    return TWN_OK;
}

}  // namespace

extern "C" int twn_conv2d_fwd_image(const twn_conv_desc_t *d, const void *X, const uint32_t *T_fwd, int64_t ld_codes,
                                    const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y, void *Yp, twn_stream_t stream)
{
    TWN_REQUIRE(d && X && T_fwd && epi && Y, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->B > 0 && d->H > 0 && d->W > 0 && d->Cin > 0 && d->Cout > 0 && d->kh > 0 && d->kw > 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->B <= 0x7fffffffLL && d->H <= 0xffffff && d->W <= 0xffffff && d->Cin <= kMostCin && d->Cout <= 0xffffff, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->stride_h >= 1 && d->stride_w >= 1 && d->stride_h <= 2 && d->stride_w <= 2 && d->pad_h >= 0 && d->pad_w >= 0 &&
                    d->kh <= kMostK && d->kw <= kMostK && d->kh * d->kw * d->Cin <= kMostK && d->pad_h < d->kh && d->pad_w < d->kw,
                TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->H + 2 * d->pad_h >= d->kh && d->W + 2 * d->pad_w >= d->kw, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->Cout % 8 == 0 && ld_codes % 64 == 0 && ld_codes >= d->kh * d->kw * d->Cin, TWN_ERR_INVALID_ARG);
    int rc = twn_detail::check_epilogue(epi);
    if (rc != TWN_OK) return rc;
    TWN_REQUIRE(epi->out_dtype == TWN_BF16 && !epi->residual, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(X, 2) && twn_aligned(T_fwd, 16) && twn_aligned(Y, 16) && twn_aligned(Yp, 16) && twn_aligned(stats, 8),
                TWN_ERR_MISALIGNED);
    FirstParams P;
    memset(&P, 0, sizeof P);
    P.Ho = (int)((d->H + 2 * d->pad_h - d->kh) / d->stride_h + 1);
    P.Wo = (int)((d->W + 2 * d->pad_w - d->kw) / d->stride_w + 1);
    P.PH = P.Ho / 2; P.PW = P.Wo / 2;
    TWN_REQUIRE(!Yp || (P.PH > 0 && P.PW > 0), TWN_ERR_INVALID_ARG);
    twn_device_info dev;
    rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    P.X = static_cast<const __nv_bfloat16 *>(X);
    P.T = T_fwd;
    P.alpha = stats ? &stats->alpha : nullptr;
    P.scale = epi->scale; P.shift = epi->shift;
    P.Y = static_cast<__nv_bfloat16 *>(Y); P.Yp = static_cast<__nv_bfloat16 *>(Yp);
    P.B = (int)d->B; P.H = (int)d->H; P.W = (int)d->W; P.Cin = (int)d->Cin; P.Cout = (int)d->Cout;
    P.kw = (int)d->kw; P.K = (int)(d->kh * d->kw * d->Cin);
    P.sh = (int)d->stride_h; P.sw = (int)d->stride_w; P.ph = (int)d->pad_h; P.pw = (int)d->pad_w;
    P.wpr = (int)(ld_codes / 16);
    // Offsets of outputs in 32 bits, the general kernel's limit.  (Those past an output's edge may wrap: they are not stored to.)
    // It leaves less than 2^29 units, each of at least one pixel of at least eight channels.
    TWN_REQUIRE((double)d->B * P.Ho * P.Wo * d->Cout < 4294967295.0, TWN_ERR_TOO_LARGE);
    // A unit: eight windows in the shape that covers the output with the fewest (12 by 12 windows: 18 units of 4 x 2, 24 of 8 x 1),
    // the wider of equals.
    const int wins_x = (P.Wo + 1) / 2, wins_y = (P.Ho + 1) / 2;
    long long best = -1;
    for (int lg = 3; lg >= 0; --lg) {
        const long long nx = (wins_x + (1 << lg) - 1) >> lg, ny = (wins_y + (8 >> lg) - 1) / (8 >> lg);
        const int rows = (2 * (8 >> lg) - 1) * P.sh + (int)d->kh, pitch = ((2 << lg) - 1) * P.sw * P.Cin + P.kw * P.Cin;
        if (best >= 0 && (nx * ny >= best || rows * pitch > kMostPiece)) continue;
        best = nx * ny;
        P.lgUx = lg; P.nx = (int)nx; P.ny = (int)ny; P.rows = rows; P.pitch = pitch;
    }
    if (P.rows * P.pitch > kMostPiece) return TWN_ERR_TOO_LARGE;
    P.units = (int)(best * d->B);
    const cudaStream_t s = twn_cu(stream);
    switch ((P.K + 15) / 16) {
        case 1: return launch_first<1>(P, epi->relu, dev, s);
        case 2: return launch_first<2>(P, epi->relu, dev, s);
        case 3: return launch_first<3>(P, epi->relu, dev, s);
        default: return launch_first<4>(P, epi->relu, dev, s);
    }
}
