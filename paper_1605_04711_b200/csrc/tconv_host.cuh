// Host-side description of one contraction launch, shared by the tensor-core kernels of the
// ternary-weight contraction: the sum over taps, the virtual output grid and its embedding in
// the output tensor, and the tensor-map encoder of the driver.
#pragma once

#include <cuda.h>
#include <stdint.h>
#include <string.h>

#include "common.cuh"

namespace twn_detail {

constexpr int kMaxTaps = 64;

struct Tap {
    int16_t dh, dw;   // input pixel offset of this tap
    int32_t koff;     // first code column of this tap in a packed row
};

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

inline EncodeTiledFn encode_fn()
{
    static EncodeTiledFn fn = nullptr;
    static bool tried = false;
    if (!tried) {
        tried = true;
        void *p = nullptr;
        cudaDriverEntryPointQueryResult qr;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &qr) == cudaSuccess &&
            qr == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}

// Part of a virtual output grid that is contracted with its own taps: a residue class of a strided
// backward-for-data pass.
constexpr int kMaxClasses = 4;
struct TapClass {
    int Hv, Wv, ooh, oow, tap0, n_taps;
};

struct Geometry {
    // input tensor X: NHWC [XB, XH, XW, XC] with pixel pitch ldx (elements)
    long long XB, XH, XW, XC, ldx;
    long long x_row_pitch, x_img_pitch;   // elements between rows / images; 0 = dense (XW*ldx, XH*XW*ldx)
    // virtual output grid and embedding
    int Bv, Hv, Wv, OH, OW, osh, osw, ooh, oow;
    long long ldy;
    int sh, sw;      // input step per virtual output pixel
    int Cout;
    long long ld_codes, code_cols;  // packed row pitch and used columns
    int code_bits;   // 2: ternary codes, 16 per word; 1: binary codes, 32 per word
    // 2x2 max pooling of the output, written beside it (optional): bf16 [Bv, Hv / 2, Wv / 2, Cout]
    void *pool;
    // batch statistics of the pre-activation output (optional): per-tile partial sums, then the totals
    float *bn_partial;
    size_t bn_partial_bytes;
    double *bn_sum, *bn_sumsq;
    int n_taps;
    Tap taps[kMaxTaps];
    long long Cin;   // channels per tap
    int beside;      // launches that run at the same time as this one (0 or 1: none)
    // 0: one class, described by the fields above; else all of them in one launch (split kernel, general kernel of 128 pixels)
    int n_classes;
    TapClass cls[kMaxClasses];
};

// Words of a packed row on whose boundaries every k-block of 64 codes starts: 4, 2 or 1 (binary codes: 2 or 1).  A k-block's
// codes come with as many loads, and a warp's load costs the 32 rows that it touches, not their bytes.  Layers of 32 (mod 64)
// channels, two loads instead of four: 16x14x14x224 -> 256, 3x3, 20.9 -> 14.4 us (split kernel), 64x14x14x608 -> 512 63.9 -> 61.1,
// 100x14x14x288 -> 688, 5x5, 179.8 -> 173.1 (general kernel), 4x14x14x96 -> 96 5.7 -> 5.2.
inline int code_run(const Geometry &g)
{
    const int word = g.code_bits == 1 ? 32 : 16;
    int run = 64 / word;
    for (int t = 0; t < g.n_taps; ++t)
        while (g.taps[t].koff % (run * word) != 0) run /= 2;
    return run;
}

// Picks the pixel-tile shape BW x BH x BB (BW and BH powers of two, product `pix`) that needs the
// fewest tiles.
inline long long pick_tile(const Geometry &g, int pix, int *lgBW, int *lgBH)
{
    // A call plans with half a dozen of these, and a small call takes the GPU no longer than planning took the host when every
    // candidate cost three 64-bit divisions (1.1 us of 5.0): shifts, and one division by three where the tile is 3 * 2^k images.
    int lg = 0;
    while (((pix >> lg) & 1) == 0) ++lg;      // BW * BH divides the power-of-two part of `pix`
    const int odd = pix >> lg;                // 1 or 3
    const auto up = [](int n, int sh) { return (long long)(((unsigned)n + ((1u << sh) - 1)) >> sh); };
    long long rows[9], images[9];
    for (int i = 0; i <= lg; ++i) {
        rows[i] = up(g.Hv, i);
        images[i] = up(g.Bv, i);
        if (odd == 3) images[i] = (images[i] + 2) / 3;
    }
    long long best = -1;
    int bw = 0, bh = 0;
    for (int a = 0; a <= lg && g.sw << a <= 256; ++a) {
        // pooled from chunks of 32 pixels of a tile: those have to hold whole windows
        if (g.pool && (a < 1 || a > 4)) continue;
        const long long cols = up(g.Wv, a);
        for (int b = g.pool ? 1 : 0; a + b <= lg && g.sh << b <= 256; ++b) {
            if (odd << (lg - a - b) > 256) continue;
            const long long tiles = cols * rows[b] * images[lg - a - b];
            // prefer fewer tiles, then wider rows
            if (best < 0 || tiles < best || (tiles == best && a > bw)) { best = tiles; bw = a; bh = b; }
        }
    }
    *lgBW = bw; *lgBH = bh;
    return best;
}

// What every contraction asks of an epilogue; NULL stands for the default one.
inline int check_epilogue(const twn_epilogue_t *e)
{
    if (!e) return TWN_OK;
    TWN_REQUIRE(e->out_dtype == TWN_F32 || e->out_dtype == TWN_BF16, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(e->residual_dtype == TWN_F32 || e->residual_dtype == TWN_BF16, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(e->relu == 0 || e->relu == 1, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(e->residual_op >= 0 && e->residual_op <= (TWN_RESIDUAL_GATE | TWN_SUM_IN_ORDER), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(e->scale, 4) && twn_aligned(e->shift, 4) && twn_aligned(e->residual, 4), TWN_ERR_MISALIGNED);
    return TWN_OK;
}

// What follows the contraction (twn_epilogue_t with the device scalar alpha resolved).
struct EpilogueArgs {
    const double *alpha;          // device scalar (twn_stats_t::alpha) or nullptr for 1
    const float *scale, *shift;
    const void *residual;
    int res_dtype, res_gate, relu, out_dtype;
    bool in_order;                // every sum runs over the taps, then the channels (TWN_SUM_IN_ORDER): no split
};

// Contraction with the layer's decoded weights resident in shared memory (tconv_res.cu).  Launches
// and returns TWN_OK with *handled = true when the launch fits that kernel (unit input stride, decoded
// weights of 64 output channels that fit in shared memory, outputs that TMA can store; not several taps
// of several channel blocks whose sums must stay in order) and should not take longer than `rival_us`;
// otherwise *handled = false and nothing has been launched.  With `us_only` nothing is launched in either
// case: *handled says whether it would be, *us_only then what it should take.
int launch_conv_resident(const Geometry &g, const void *X, const uint32_t *T, const EpilogueArgs &epi, void *Y,
                         int32_t *dev_status, const twn_device_info &dev, cudaStream_t s, double rival_us, bool *handled,
                         double *us_only);

// Contraction for problems that do not fill the GPU (tconv_split.cu): tiles of 128 channels x `pix` pixels (32, 64, 128
// or 256), the reduction of each split over a cluster of `splits` blocks (1, 2, 4 or 8; 256 pixels: 1 or 2).  Takes every
// geometry but batch statistics, reductions of more than 512 k-blocks per block, and pooled outputs of more than 64 channels, of
// binary codes or with their sums in order.
struct SplitPlan {
    int pix, splits;
    double us;        // what the launch should take
};
SplitPlan plan_conv_split(const Geometry &g, int sm_count, bool in_order);
int launch_conv_split(const Geometry &g, const void *X, const uint32_t *T, const EpilogueArgs &epi, void *Y,
                      int32_t *dev_status, const twn_device_info &dev, cudaStream_t s, const SplitPlan &plan);

}  // namespace twn_detail
