// Ternary-weight contraction on the 5th-generation tensor cores (Eq. 2 forward block;
// Algorithm 1 TernaryForward / TernaryBackward):  Y = epilogue(alpha * X (*) T).
//
// One persistent, warp-specialised kernel serves the inner product, the convolution
// forward pass and the backward-for-data pass.  All three are written as a sum over
// "taps": for output pixel p and output channel n
//     acc[n, p] = sum_t sum_c  T[n, koff_t + c] * X[pixel(p) * stride + (dh_t, dw_t), c]
// with X an NHWC bf16 tensor addressed through a 4-D TMA tensor map (out-of-range
// pixels and channels read as zero) and T the packed 2-bit codes, one row per n.
//
// The weights are the A operand of tcgen05.mma and live in tensor memory: decode
// warps turn the packed codes into exact bf16 {-1, 0, +1} in registers and write them
// with tcgen05.st.  The activations are the B operand, staged by TMA into 128-byte
// swizzled shared memory.  The accumulator (fp32, tensor memory) therefore holds
// D[n, p]: a lane is an output channel, a column a pixel.  In the epilogue each thread
// owns one channel, so alpha, the per-channel affine and ReLU cost one register each,
// and a warp's store of one pixel covers 32 consecutive channels (128 contiguous bytes).
//
//   warp 0            TMA producer: one activation tile per k-block
//   warp 1            allocates tensor memory, issues tcgen05.mma, commits to mbarriers
//   warps 2-5 (2-9)   decode: packed codes (global, L2) -> bf16 pairs -> tensor memory; one group
//                     of four warps (one per lane quadrant), or two groups that take the stages
//                     in turn
//   last eight warps  epilogue, two per lane quadrant: tensor memory -> registers -> per-warp
//                     staging buffer -> TMA store
//
// Three tile shapes (template parameter PIX = pixels per tile; the channel tile is always 128).
// A k-block takes 256 pixels 517 cycles of 512 of MMA, 192 pixels 444 of 384 (the activation feed: 24 KB from L2), 128 pixels
// 255 to 280 of 256.
//   PIX = 256: one accumulator (256 of the 512 tensor-memory columns, the rest holds decoded
//              weights), five stages; the epilogue of a tile is not overlapped with the next
//              tile's MMAs.  Long reductions with many tiles.
//   PIX = 192: two accumulators and four stages fill the tensor memory exactly; the epilogue
//              overlaps the next tile.
//   PIX = 128: two accumulators, four stages of two k-blocks each.
// The host picks the shape per launch with a model of its time.
//
// Every wait on an mbarrier is bounded (about a second); on expiry the kernel records
// TWN_ERR_TIMEOUT, all roles leave their loops, tensor memory is freed and the grid exits.
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstddef>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "tc_ptx.cuh"
#include "tconv_host.cuh"

using namespace twn_detail;


namespace {

constexpr int kChan = 128;          // output channels per tile (UMMA M)
constexpr int kBlockK = 64;         // reduction elements per k-block (128 bytes of bf16)
// Groups of 4 decode warps in a block: one, or two that take the stages in turn.  Two where the epilogue overlaps the next
// tile's reduction (128 pixels: 0 to 28 % faster on 40 shapes, 16384x576x1000 30.7 -> 22.0 us, 3x3 64x7x7x512 17.8 -> 16.1; 192
// pixels: 24 % slower without on the latter, 3 % faster on 1x1 64x28x28x512); 256 pixels are bound by their MMAs with one.
__host__ __device__ constexpr int first_epi_warp(int ds) { return 2 + 4 * ds; }
constexpr int kEpiSets = 2;         // epilogue warps per lane quadrant; each drains every other 32-pixel chunk
__host__ __device__ constexpr int threads_conv(int ds) { return 32 * (first_epi_warp(ds) + 4 * kEpiSets); }
constexpr int kEpiWarps = 4 * kEpiSets;
constexpr int kStageBytes = 2048;   // one output staging buffer of a warp: 32 channels x 32 pixels of bf16 or 16 pixels of fp32
constexpr int kWordTab = 128;       // k-blocks per tile whose code offsets are tabulated in shared memory
constexpr int kAColsPerBlock = kBlockK / 2;    // 32 columns of bf16 pairs per k-block
constexpr uint32_t kTmemCols = 512;

template <int PIX> struct Cfg;
template <> struct Cfg<128> {
    static constexpr int kStages = 4;   // operand ring depth (shared and tensor memory)
    static constexpr int kSub = 2;      // k-blocks per stage: one wait and one commit per 8 MMAs
    static constexpr int kAccBufs = 2;  // the epilogue of a tile overlaps the MMAs of the next
    static constexpr int kOutBufs = 4;  // output staging buffers per epilogue warp
    static constexpr int kDecodeGroups = 2;
};
template <> struct Cfg<256> {
    static constexpr int kStages = 5;
    static constexpr int kSub = 1;
    static constexpr int kAccBufs = 1;
    static constexpr int kOutBufs = 2;
    static constexpr int kDecodeGroups = 1;
};
// 192 pixels: the largest tile that leaves room for two accumulators beside four stages of
// decoded weights (2 x 192 + 4 x 32 = 512 columns); the pixel tile is 3 * 2^k images deep.
template <> struct Cfg<192> {
    static constexpr int kStages = 4;
    static constexpr int kSub = 1;
    static constexpr int kAccBufs = 2;
    static constexpr int kOutBufs = 4;
    static constexpr int kDecodeGroups = 2;
};

struct ConvParams {
    // tiles
    int n_tiles, tw, th, tb, total_tiles;
    int lgBW, lgBH;               // pixel tile = BB x BH x BW, powers of two, product PIX
    // reduction
    int n_taps, n_cblk;           // k-blocks per tile = n_taps * n_cblk
    int code_run;                 // words of the packed row on whose boundaries every k-block starts: 1, 2, 4; 8: k-block u follows
                                  // k-block u - 1, and every other one starts on such a boundary
    const uint32_t *T;            // packed codes, one row of `wpr` words per output channel
    long long wpr;
    int sw, sh;                   // input pixel = output pixel * (sh, sw) + (dh, dw)
    // virtual output grid and its embedding in the output tensor
    int Bv, Hv, Wv;
    int OH, OW, osh, osw, ooh, oow;
    long long ldy;                // output pixel pitch in elements
    int Cout;
    // epilogue
    const double *alpha;          // device scalar (twn_stats_t::alpha) or nullptr for 1
    const float *scale, *shift;
    const void *residual;
    int res_dtype, relu, out_dtype;
    int res_gate;                 // 0: the residual is added; 1: it gates the result (kept where residual > 0)
    void *Y;
    int32_t *status;
    // optional batch statistics: [tile][epilogue warp of the quadrant][128 channels][sum, sum of squares]
    float *bn_partial;
    // output path: 1 = each epilogue warp stages its 32 channels x 32 pixels in shared memory and
    // writes them with a TMA store (box = 32 channels x sbw x sbh x sbb pixels); 0 = per-thread stores
    int tma_store;
    // optional 2x2 max pooling of the output (with `fragments`): a chunk of 32 pixels is 2^lg_sbw x 2^lg_sbh x the rest images
    __nv_bfloat16 *pool;
    int PH, PW, lg_sbw, lg_sbh;
    int res_tma;                  // 1: the residual (bf16) is staged by per-warp TMA loads, two chunks deep
    int fragments;                // 1: bf16 in and out by TMA, no batch statistics: chunks are drained as matrix fragments
    Tap taps[kMaxTaps];
};

// The classes of a strided backward pass: their tiles follow one another, those without taps last; each class has its own run of
// taps and place in the output.  (An argument of its own: launches without classes do without it.)
struct ClassTable {
    int n, live_tiles;            // classes; tiles of those with taps
    struct { int tile0, tw, th, Hv, Wv, ooh, oow, tap0, kb0, kb, stages; } cls[kMaxClasses];
};
struct NoClasses {};

template <int PIX>
struct __align__(1024) SmemLayout {
    static constexpr int kStages = Cfg<PIX>::kStages, kSub = Cfg<PIX>::kSub;
    static constexpr int kXBytes = PIX * kBlockK * 2;
    uint8_t x[kStages][kSub][kXBytes];           // swizzled activation tiles
    // TMA and decode -> MMA: the activation tile has landed (one arrival with its byte count) and the
    // four decode warps have put the stage's weights into tensor memory (one arrival each).  One
    // barrier for both: every wait of the issuing warp is latency that the tensor core may sit out.
    unsigned long long full[kStages];
    unsigned long long empty[kStages];     // MMA commit -> TMA and decode: both operand slots are free
    unsigned long long acc_full[2];        // MMA commit -> epilogue
    unsigned long long acc_empty[2];       // epilogue -> MMA
    // per-warp output staging for TMA stores: [pixels][32 channels].  The stores of the epilogue
    // queue behind the producer's tile loads in the copy engine, so while the main loop of the next
    // tile runs a store takes long to release its buffer: the overlapped tile shapes keep four.
    // The fragment path swizzles them (64 bytes), hence the alignment.
    alignas(1024) uint8_t stage_out[kEpiWarps][Cfg<PIX>::kOutBufs][kStageBytes];
    alignas(1024) __nv_bfloat16 stage_res[kEpiWarps][2][32 * 32];  // per-warp residual staging: [32 pixels][32 channels]
    unsigned long long res_full[kEpiWarps][2];
    uint32_t kword[kWordTab];              // first code word of k-block u in a packed row, u < kWordTab
    uint32_t tmem_base;
    volatile int abort_flag;
};

static_assert(offsetof(SmemLayout<128>, stage_res) % 128 == 0 && offsetof(SmemLayout<256>, stage_res) % 128 == 0 &&
                  offsetof(SmemLayout<192>, stage_res) % 128 == 0 && offsetof(SmemLayout<192>, stage_out) % 128 == 0 &&
                  sizeof(SmemLayout<256>) + 1024 <= 232448 && sizeof(SmemLayout<128>) + 1024 <= 232448 &&
                  sizeof(SmemLayout<192>) + 1024 <= 232448 &&
                  offsetof(SmemLayout<128>, stage_out) % 128 == 0 && offsetof(SmemLayout<256>, stage_out) % 128 == 0,
              "TMA and vector accesses need aligned shared-memory regions");

// CLASSES: the residue classes of a strided backward pass in one launch, the longest reductions first; fragments alone.
// WORDS: the ternary codes come word by word (in a kernel of its own where they do: with the wider loads beside them those layers
// lost 2 %, 64x28x28x192 <- 272, 3x3, 52.7 -> 54.2 us).
template <int PIX, int BITS, bool CLASSES, bool WORDS>
__global__ void __launch_bounds__(threads_conv(Cfg<PIX>::kDecodeGroups), 1)
tconv_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_y,
             const __grid_constant__ CUtensorMap map_r, const __grid_constant__ ConvParams P,
             const __grid_constant__ std::conditional_t<CLASSES, ClassTable, NoClasses> K)
{
    using L = SmemLayout<PIX>;
    constexpr int kStages = Cfg<PIX>::kStages, kSub = Cfg<PIX>::kSub, kAccBufs = Cfg<PIX>::kAccBufs, DS = Cfg<PIX>::kDecodeGroups;
    constexpr int kOutBufs = Cfg<PIX>::kOutBufs;
    constexpr int kXBytes = L::kXBytes;
    constexpr int kAColsPerStage = kSub * kAColsPerBlock;
    constexpr int kCodesPerWord = 32 / BITS, kWordsPerBlock = kBlockK / kCodesPerWord;   // 16 and 4, or 32 and 2
    static_assert(kAccBufs * PIX + kStages * kAColsPerStage <= (int)kTmemCols, "tensor memory budget");
    

    pdl_launch_dependents();
    extern __shared__ uint8_t smem_raw[];
    L *sm = reinterpret_cast<L *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    volatile int *abort_flag = &sm->abort_flag;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int kb_all = P.n_taps * P.n_cblk;             // k-blocks per tile (of all classes)
    // the class of a tile, from that of an earlier one
    auto seek = [&](int &c, int tile) {
        if constexpr (CLASSES)
            while (c + 1 < K.n && tile >= K.cls[c + 1].tile0) ++c;
    };
    int live_tiles = P.total_tiles;
    if constexpr (CLASSES) live_tiles = K.live_tiles;

    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            mbar_init(&sm->full[s], 1 + 4);
            mbar_init(&sm->empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&sm->acc_full[b], 1);
            mbar_init(&sm->acc_empty[b], kEpiWarps);
        }
        for (int b = 0; b < 2 * kEpiWarps; ++b) mbar_init(&sm->res_full[0][0] + b, 1);
        sm->abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // code-word offset of every k-block, in the order the k-blocks are consumed: taps outer,
    // channel blocks inner
    constexpr int kFirstEpiWarp = first_epi_warp(DS), kThreadsConv = threads_conv(DS);
    for (int u = threadIdx.x; u < kb_all && u < kWordTab; u += kThreadsConv) {
        const int t = u / P.n_cblk, cb = u - t * P.n_cblk;
        sm->kword[u] = (uint32_t)(P.taps[t].koff / kCodesPerWord) + cb * kWordsPerBlock;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&sm->tmem_base)), "r"(kTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    // the set-up above touched no global memory; everything below may read what the previous kernel wrote
    pdl_wait();
    const uint32_t tmem = sm->tmem_base;
    const uint32_t tmem_acc = tmem;                       // kAccBufs x PIX columns
    const uint32_t tmem_a = tmem + kAccBufs * PIX;        // kStages x kAColsPerStage columns

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (elect_one()) {
            uint32_t it = 0;
            bool ok = true;
            const uint32_t block_bytes = kXBytes;
            int ci = 0;
            for (int tile = blockIdx.x; tile < live_tiles && ok; tile += gridDim.x) {
                int tw = P.tw, th = P.th, tap0 = 0, kbpt = kb_all, spt = (kb_all + kSub - 1) / kSub, pt = tile;
                if constexpr (CLASSES) {
                    seek(ci, tile);
                    const auto &C = K.cls[ci];
                    tw = C.tw; th = C.th; tap0 = C.tap0; kbpt = C.kb; spt = C.stages; pt -= C.tile0;
                }
                pt /= P.n_tiles;
                const int twi = pt % tw; pt /= tw;
                const int thi = pt % th;
                const int tbi = pt / th;
                const int w0 = (twi << P.lgBW) * P.sw;
                const int h0 = (thi << P.lgBH) * P.sh;
                const int b0 = tbi * (PIX >> (P.lgBW + P.lgBH));
                int t = 0, cb = 0;
                for (int st = 0; st < spt; ++st, ++it) {
                    const int s = it % kStages;
                    const uint32_t ph = (it / kStages) & 1u;
                    const int nsb = (kbpt - st * kSub) < kSub ? (kbpt - st * kSub) : kSub;
                    if (!mbar_wait(&sm->empty[s], ph ^ 1u, abort_flag, P.status)) { ok = false; break; }
                    mbar_expect_tx(&sm->full[s], nsb * block_bytes);
                    for (int sb = 0; sb < nsb; ++sb) {
                        const Tap tap = P.taps[tap0 + t];
                        tma_load_4d(sm->x[s][sb], &map_x, &sm->full[s], cb * kBlockK, w0 + tap.dw, h0 + tap.dh, b0);
                        if (++cb == P.n_cblk) { cb = 0; ++t; }
                    }
                }
            }
        }
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer: one thread (see tc_mma_ts)
        // One wait and one commit per stage, constant accumulate flags.  With no taps at all
        // (no k-blocks) nothing is accumulated and the epilogue does not wait.
        if (kb_all > 0 && elect_one()) {
            constexpr uint32_t idesc = make_idesc(kChan, PIX);
            const uint64_t bdesc0 = smem_desc_sw128(smem_u32(sm->x[0][0]));
            const uint32_t b_lo0 = (uint32_t)bdesc0, b_hi = (uint32_t)(bdesc0 >> 32);
            uint32_t it = 0, lt = 0;
            bool ok = true;
            // in registers: what this thread waits for between two tiles, the tensor core waits for
            int first[kMaxClasses], kbs[kMaxClasses];
            kbs[0] = kb_all;
            if constexpr (CLASSES)
                for (int c = 0; c < kMaxClasses; ++c) {
                    first[c] = c < K.n ? K.cls[c].tile0 : 0x7fffffff;
                    kbs[c] = K.cls[c].kb;
                }
            for (int tile = blockIdx.x; tile < live_tiles && ok; tile += gridDim.x, ++lt) {
                int kbpt = kbs[0];
                if (CLASSES) {
#pragma unroll
                    for (int c = 1; c < kMaxClasses; ++c) kbpt = tile >= first[c] ? kbs[c] : kbpt;
                }
                const int spt = (kbpt + kSub - 1) / kSub;
                const int buf = lt % kAccBufs;
                const uint32_t aph = (lt / kAccBufs) & 1u;
                if (!mbar_wait(&sm->acc_empty[buf], aph ^ 1u, abort_flag, P.status, 0)) break;
                tc_fence_after();
                const uint32_t d_tmem = tmem_acc + buf * PIX;
                for (int st = 0; st < spt; ++st, ++it) {
                    const int s = it % kStages;
                    const uint32_t ph = (it / kStages) & 1u;
                    if (!mbar_wait(&sm->full[s], ph, abort_flag, P.status, 0)) { ok = false; break; }
                    tc_fence_after();
                    const uint32_t b_lo = b_lo0 + (uint32_t)(s * ((kSub * kXBytes) >> 4));
                    const uint32_t a_tmem = tmem_a + s * kAColsPerStage;
                    if (st == 0) tc_mma_block<true>(d_tmem, a_tmem, b_lo, b_hi, idesc);
                    else tc_mma_block<false>(d_tmem, a_tmem, b_lo, b_hi, idesc);
                    if (kSub > 1 && kbpt - st * kSub > 1)
                        tc_mma_block<false>(d_tmem, a_tmem + kAColsPerBlock, b_lo + (kXBytes >> 4), b_hi, idesc);
                    tc_commit(&sm->empty[s]);
                }
                if (ok) tc_commit(&sm->acc_full[buf]);
            }
        }
        __syncwarp();
    } else if (warp < kFirstEpiWarp) {
        // ------------------------------------------------ decode: codes -> bf16 -> tensor memory
        // One group of four warps, or two on alternate stages.  Each thread owns one channel row: it
        // reads the row's codes of a stage (16 bytes per k-block of ternary codes, a stage's two
        // k-blocks at once where they lie so) straight from global memory (L2-resident, fetched two
        // or three of its stages ahead), so decoding depends only on a free tensor-memory slot, not
        // on the activation pipeline.
        const int q = warp & 3;                 // tensor-memory lane quadrant of this warp
        const int set = (warp - 2) >> 2;
        constexpr int dsets = DS;               // groups of this kernel; the loops below are stepped by it
        const int row = q * 32 + lane;          // channel row inside the tile
        const uint32_t lane_base = tmem_a + ((uint32_t)(q * 32) << 16);

        // Code words are fetched with explicit non-coherent loads straight into the registers that
        // hold them until they are decoded, from addresses clamped into the packed matrix: no
        // branch and no register copy stands between a load and its use, so its latency stays
        // hidden.  What a clamped fetch returns is either never decoded (no such stage) or feeds
        // channels that are never stored, or multiplies activations that the TMA zero-fills.
        struct Codes { uint4 v[kSub]; };
        int kbpt = kb_all, spt = (kb_all + kSub - 1) / kSub;        // of the tile being decoded
        int kbpt_f = kbpt, spt_f = spt, kb0_f = 0, tap0_f = 0;      // of the tile being fetched
        auto fetch = [&](Codes &c, const uint32_t *rowp, int st) {
            // A warp's load touches 32 rows, and that is what it costs: both k-blocks of a stage come with one 32-byte load
            // where the codes lie so.  With two of 16 bytes a k-block of 128 pixels took 320 cycles, 255 with one
            // (4001x4608x512 20.1 -> 17.7 us, 3x3 64x7x7x512 18.9 -> 16.0).
            if (kSub == 2 && !WORDS && P.code_run == 8) {
                if (BITS == 2) {
                    ld_nc_v8(c.v[0], c.v[kSub - 1], rowp + (CLASSES ? sm->kword[kb0_f + 2 * st] : 8 * st));
                } else {
                    uint4 both;
                    ld_nc_v4(both, rowp + (CLASSES ? sm->kword[kb0_f + 2 * st] : 4 * st));
                    c.v[0].x = both.x; c.v[0].y = both.y; c.v[kSub - 1].x = both.z; c.v[kSub - 1].y = both.w;
                }
                return;
            }
#pragma unroll
            for (int sb = 0; sb < kSub; ++sb) {
                int u = st * kSub + sb;
                u = u < kbpt_f ? u : kbpt_f - 1;
                long long word;
                if (kb_all <= kWordTab) {
                    word = sm->kword[kb0_f + u];
                } else {
                    const int t = u / P.n_cblk, cb = u - t * P.n_cblk;
                    word = (P.taps[tap0_f + t].koff / kCodesPerWord) + cb * kWordsPerBlock;
                }
                if (BITS == 2) {
                    if (!WORDS && P.code_run >= 4) {
                        ld_nc_v4(c.v[sb], rowp + word);
                    } else if (!WORDS && (PIX == 128 || P.code_run == 2)) {
                        ld_nc_v2(c.v[sb].x, c.v[sb].y, rowp + word);
                        ld_nc_v2(c.v[sb].z, c.v[sb].w, rowp + (word + 2 < P.wpr ? word + 2 : word));
                    } else {
                        const long long last = P.wpr - 1;
                        ld_nc_u32(c.v[sb].x, rowp + (word + 0 < last ? word + 0 : last));
                        ld_nc_u32(c.v[sb].y, rowp + (word + 1 < last ? word + 1 : last));
                        ld_nc_u32(c.v[sb].z, rowp + (word + 2 < last ? word + 2 : last));
                        ld_nc_u32(c.v[sb].w, rowp + (word + 3 < last ? word + 3 : last));
                    }
                } else {
                    if (P.code_run >= 2) {
                        ld_nc_v2(c.v[sb].x, c.v[sb].y, rowp + word);
                    } else {
                        const long long last = P.wpr - 1;
                        ld_nc_u32(c.v[sb].x, rowp + (word + 0 < last ? word + 0 : last));
                        ld_nc_u32(c.v[sb].y, rowp + (word + 1 < last ? word + 1 : last));
                    }
                }
            }
        };
        // position of this group's next stages: (tile, st), advanced dsets stages at a time
        int ci_c = 0, ci_f = 0;
        auto advance = [&](int &tile, int &st, int steps) {
            for (int i = 0; i < steps; ++i)
                if (++st >= spt) {
                    st = 0; tile += gridDim.x;
                    if constexpr (CLASSES)
                        if (tile < live_tiles) { seek(ci_c, tile); kbpt = K.cls[ci_c].kb; spt = K.cls[ci_c].stages; }
                }
        };
        // the fetch position also carries its row of the packed matrix: the channel tile of
        // `tile` is tile mod n_tiles, stepped without a division (one sits in the way of every
        // stage otherwise); rows past Cout read the last row and are never stored
        const int nt_step = (int)(gridDim.x % (unsigned)P.n_tiles);
        auto row_ptr = [&](int nt) -> const uint32_t * {
            long long n = (long long)nt * kChan + row;
            n = n < P.Cout ? n : P.Cout - 1;
            return P.T + n * P.wpr;
        };
        auto advance_f = [&](int &tile, int &st, int &nt, const uint32_t *&rowp, int steps) {
            for (int i = 0; i < steps; ++i)
                if (++st >= spt_f) {
                    st = 0; tile += gridDim.x;
                    nt += nt_step; if (nt >= P.n_tiles) nt -= P.n_tiles;     // (a class has whole sets of channel tiles)
                    rowp = row_ptr(nt);
                    if constexpr (CLASSES)
                        if (tile < live_tiles) {
                            seek(ci_f, tile);
                            kbpt_f = K.cls[ci_f].kb; spt_f = K.cls[ci_f].stages; kb0_f = K.cls[ci_f].kb0; tap0_f = K.cls[ci_f].tap0;
                        }
                }
        };
        int tile_c = blockIdx.x, st_c = 0;                   // the stage being decoded
        if constexpr (CLASSES)
            if (tile_c < live_tiles) {
                seek(ci_c, tile_c);
                kbpt = K.cls[ci_c].kb; spt = K.cls[ci_c].stages;
            }
        if (CLASSES ? tile_c < live_tiles : spt > 0) {
            // 256-pixel tiles: three code buffers in rotation, each refilled right after use for the
            // stage three of this group's stages ahead: no register is copied while its load is still
            // in flight.  The other shapes: two buffers, see below.
            advance(tile_c, st_c, set);
            int tile_f = tile_c, st_f = st_c;                // the stage being fetched
            if constexpr (CLASSES) {
                ci_f = ci_c;
                kbpt_f = kbpt; spt_f = spt; kb0_f = K.cls[ci_c].kb0; tap0_f = K.cls[ci_c].tap0;
            }
            int nt_f = tile_f % P.n_tiles;
            const uint32_t *rowp_f = row_ptr(nt_f);
            Codes c0, c1, c2;
            fetch(c0, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets);
            fetch(c1, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets);
            if (PIX == 256) { fetch(c2, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets); }
            uint32_t it = set;
            auto decode_stage = [&](const Codes &cur) -> bool {
                const int s = it % kStages;
                const uint32_t ph = (it / kStages) & 1u;
                const int nsb = (kbpt - st_c * kSub) < kSub ? (kbpt - st_c * kSub) : kSub;
                // the MMAs that read this slot's previous contents have completed
                if (!mbar_wait_warp(&sm->empty[s], ph ^ 1u, abort_flag, P.status, 32)) return false;
                tc_fence_after();
#pragma unroll
                for (int sb = 0; sb < kSub; ++sb) {
                    if (sb < nsb) {
                        const uint32_t wv[4] = {cur.v[sb].x, cur.v[sb].y, cur.v[sb].z, cur.v[sb].w};
                        uint32_t out[32];
                        decode_kblock<BITS>(wv, out);
                        tmem_st32(lane_base + s * kAColsPerStage + sb * kAColsPerBlock, out);
                    }
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->full[s]);
                advance(tile_c, st_c, dsets);
                it += dsets;
                return true;
            };
            if (PIX == 256) {
                // long reductions, no slack for a late code word: three buffers in rotation
                while (true) {
                    if (tile_c >= live_tiles || !decode_stage(c0)) break;
                    { fetch(c0, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets); }
                    if (tile_c >= live_tiles || !decode_stage(c1)) break;
                    { fetch(c1, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets); }
                    if (tile_c >= live_tiles || !decode_stage(c2)) break;
                    { fetch(c2, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets); }
                }
            } else {
                // The overlapped tile shapes are paced by this loop, and a loop that is a third as long
                // gains more than it loses by fetching only two stages ahead and moving the code words
                // one buffer down per stage (measured: 128-pixel tiles 6-20 % faster, 192-pixel tiles
                // unchanged).
#pragma unroll 1
                while (true) {
                    if (tile_c >= live_tiles || !decode_stage(c0)) break;
                    c0 = c1;
                    { fetch(c1, rowp_f, st_f); advance_f(tile_f, st_f, nt_f, rowp_f, dsets); }
                }
            }
        }
    } else {
        // ------------------------------------------------ epilogue
        // Eight warps, two per tensor-memory lane quadrant; the two warps of a quadrant take
        // alternate 32-pixel chunks of the accumulator.  Every warp works on its own: it drains
        // its 32 channels x 32 pixels with tcgen05.ld (the load of its next chunk is in flight
        // while the current one is processed), applies scale / shift / residual / ReLU, stages
        // the chunk in its own shared-memory buffer and writes it with its own TMA store
        // (box = 32 channels x 32 pixels).  No barrier joins the epilogue warps, so a warp never
        // waits for a slower one, and the accumulator goes back to the MMA warp as soon as the
        // last tensor-memory load of every warp has completed.
        const int q = warp & 3;
        const int es = (warp - kFirstEpiWarp) >> 2;          // which of the two warps of the quadrant
        const int ewi = warp - kFirstEpiWarp;                // buffer set of this warp
        // decoded ternary weights are +-2, so half of alpha scales the accumulators
        const float alpha = (P.alpha ? (float)(*P.alpha) : 1.0f) * (1.0f / decoded_unit<BITS>());
        const int BWm = (1 << P.lgBW) - 1, BHm = (1 << P.lgBH) - 1;
        const bool out_bf16 = P.out_dtype == TWN_BF16, res_bf16 = P.res_dtype == TWN_BF16;
        const bool need_off = !P.tma_store || (P.residual && !P.res_tma);
        // the ReLU of a bf16 output rides on the conversion; every other path clamps explicitly (a NaN stays a NaN in both)
        const bool relu_in_cvt = P.relu && out_bf16 && P.tma_store;
        const bool relu_here = P.relu && !relu_in_cvt;
        constexpr int kChunks = PIX / 32;
        constexpr int kMine = kChunks / kEpiSets;            // chunks of a tile this warp drains
        static_assert(kChunks % kEpiSets == 0, "the chunks of a tile are split evenly over the warps of a quadrant");
        uint8_t *const my_out = sm->stage_out[ewi][0];
        __nv_bfloat16 *const my_res = sm->stage_res[ewi][0];
        unsigned long long *const my_res_full = sm->res_full[ewi];
        uint32_t lt = 0;
        uint32_t nst = 0;      // staging buffers this warp has filled so far (selects the buffer)
        uint32_t nres = 0;     // residual chunks this warp has consumed so far (buffer and phase)
        bool alive = true;
        int ci = 0;
        for (int tile = blockIdx.x; tile < P.total_tiles && alive; tile += gridDim.x, ++lt) {
            const int nt = tile % P.n_tiles;
            int pt = tile, kbpt = kb_all, tw = P.tw, th = P.th;
            int sto_w = 0, sto_h = 0;                            // of a store's coordinates; without classes in the tensor map
            if constexpr (CLASSES) {
                seek(ci, tile);
                const auto &C = K.cls[ci];
                pt -= C.tile0; kbpt = C.kb; tw = C.tw; th = C.th; sto_w = C.oow; sto_h = C.ooh;
            }
            pt /= P.n_tiles;
            const int twi = pt % tw; pt /= tw;
            const int thi = pt % th;
            const int tbi = pt / th;
            const int n = nt * kChan + q * 32 + lane;
            const bool n_ok = n < P.Cout;
            // a warp whose 32 channels all lie past Cout hands the accumulator back but loads,
            // computes and stores nothing
            const bool warp_on = nt * kChan + q * 32 < P.Cout;
            const float sc = ((P.scale && n_ok) ? __ldg(P.scale + n) : 1.0f) * alpha;
            const float sf = (P.shift && n_ok) ? __ldg(P.shift + n) : 0.0f;
            const int p_w0 = twi << P.lgBW, p_h0 = thi << P.lgBH, p_b0 = tbi * (PIX >> (P.lgBW + P.lgBH));
            const int c_n0 = nt * kChan + q * 32;            // first channel of this warp
            // residual chunk `c` of this tile -> buffer `slot` of this warp (one lane)
            auto res_load = [&](int c, uint32_t slot) {
                const int p0 = c * 32;
                mbar_expect_tx(&my_res_full[slot], 32 * 32 * 2);
                tma_load_4d(my_res + slot * (32 * 32), &map_r, &my_res_full[slot], c_n0,
                            (p_w0 + (p0 & BWm)) * P.osw + sto_w, (p_h0 + ((p0 >> P.lgBW) & BHm)) * P.osh + sto_h,
                            p_b0 + (p0 >> (P.lgBW + P.lgBH)));
            };
            // both buffers are free here: the warp has read the last chunk of its previous tile
            const bool use_res_tma = P.res_tma && warp_on;
            if (use_res_tma && lane == 0) {
                res_load(es, nres & 1u);
                if (kMine > 1) res_load(es + kEpiSets, (nres + 1) & 1u);
            }
            const int buf = lt % kAccBufs;
            if (kbpt > 0 && !mbar_wait_warp(&sm->acc_full[buf], (lt / kAccBufs) & 1u, abort_flag, P.status, 32)) break;
            tc_fence_after();
            float *const y32 = reinterpret_cast<float *>(P.Y) + n;
            __nv_bfloat16 *const y16 = reinterpret_cast<__nv_bfloat16 *>(P.Y) + n;
            const uint32_t t_acc = tmem_acc + ((uint32_t)(q * 32) << 16) + buf * PIX;
            uint32_t v[32];
            float bn_s1 = 0.0f, bn_s2 = 0.0f;      // this thread's channel: sum and sum of squares over its pixels of the tile
            // the chunk loop stays rolled: the epilogue is straight-line code that every warp walks
            // once per chunk, so its size is instruction-fetch time
#pragma unroll 1
            for (int i = 0; i < kMine; ++i) {
                const int c = es + i * kEpiSets;
                if (kbpt > 0) {
                    if (warp_on) {
                        if (CLASSES || P.fragments) {
                            tmem_ld_16x256b_x4(t_acc + c * 32, v);
                            tmem_ld_16x256b_x4(t_acc + (16u << 16) + c * 32, v + 16);
                        } else {
                            tmem_ld32(t_acc + c * 32, v);
                        }
                        tmem_wait_ld(v);
                    }
                    if (i + 1 == kMine) {
                        // this warp's share of the accumulator is in registers: hand it back
                        tc_fence_before();
                        __syncwarp();
                        if (lane == 0) mbar_arrive(&sm->acc_empty[buf]);
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = 0u;
                }
                if (!warp_on) continue;
                if (CLASSES || P.fragments) {
                    // The accumulator's rows are channels, the output's rows pixels: the chunk has to be transposed.  The
                    // 16x256b load leaves a thread two neighbouring pixels of channels g, g + 8, g + 16, g + 24: packed,
                    // that is the operand of stmatrix.trans.  Four of those store the chunk, four ldmatrix.trans fetch
                    // its residual; with a channel per thread (below) each takes 32 two-byte accesses.  Layers gain 3-15 %
                    // (64x14x14x256 3x3 19.2 -> 17.8 us, 100000x640x256 50.8 -> 43.0); fp32 outputs would store as often
                    // and lose 3 %, and everything else is rare: they keep the path below, whose registers fit in the
                    // 96 that two decode groups leave (one loop for all cases spilled and lost 3-5 %).
                    // v[16 h + 4 k + 2 u + e]: channel g + 8 (2 h + u), pixel 8 k + 2 (ln % 4) + e
                    uint32_t ln;
                    asm volatile("mov.u32 %0, %%laneid;" : "=r"(ln));      // read here: nothing of it is kept in registers
                    // this lane's row of the 8x8 matrices: pixel ln % 8 of eight, channels 8 (ln / 8) ...
                    const uint32_t mat = (ln & 7) * 64 + (((ln >> 3) ^ ((ln >> 1) & 3)) << 4);
#pragma unroll
                    for (int m = 0; m < 4; ++m) {
                        const float scm = __shfl_sync(0xffffffffu, sc, (ln >> 2) + 8 * m);
                        const float sfm = __shfl_sync(0xffffffffu, sf, (ln >> 2) + 8 * m);
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            const int j = m / 2 * 16 + k * 4 + m % 2 * 2;
                            fma_f32x2(v[j], v[j + 1], scm, scm, sfm, sfm);
                        }
                    }
                    if (use_res_tma) {
                        if (!mbar_wait_warp(&my_res_full[nres & 1u], (nres >> 1) & 1u, abort_flag, P.status, 32)) { alive = false; break; }
                        const uint32_t rs = smem_u32(my_res) + (nres & 1u) * (32 * 32 * 2) + mat;
#pragma unroll
                        for (int k = 0; k < 4; ++k) {
                            uint32_t rr[4];
                            ldmatrix_x4_trans(rs + k * 512, rr);
#pragma unroll
                            for (int m = 0; m < 4; ++m) {
                                const int j = m / 2 * 16 + k * 4 + m % 2 * 2;
                                const float r0 = __uint_as_float(rr[m] << 16), r1 = __uint_as_float(rr[m] & 0xFFFF0000u);
                                const float y0 = __uint_as_float(v[j]), y1 = __uint_as_float(v[j + 1]);
                                v[j] = __float_as_uint(P.res_gate ? (r0 > 0.0f ? y0 : 0.0f) : y0 + r0);
                                v[j + 1] = __float_as_uint(P.res_gate ? (r1 > 0.0f ? y1 : 0.0f) : y1 + r1);
                            }
                        }
                        // the buffer is free again: fetch the residual of the chunk after the next
                        __syncwarp();
                        if (lane == 0 && i + 2 < kMine) res_load(c + 2 * kEpiSets, nres & 1u);
                        ++nres;
                    }
                    // the buffer was last read by the store this warp issued kOutBufs chunks ago
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kOutBufs - 1) : "memory");
                    __syncwarp();
                    uint8_t *const sbuf = my_out + (nst % kOutBufs) * kStageBytes;
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        uint32_t w[4];
#pragma unroll
                        for (int m = 0; m < 4; ++m) {
                            const int j = m / 2 * 16 + k * 4 + m % 2 * 2;
                            w[m] = relu_in_cvt ? pack_bf16x2_relu(__uint_as_float(v[j]), __uint_as_float(v[j + 1]))
                                               : pack_bf16x2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                        }
                        stmatrix_x4_trans(smem_u32(sbuf) + mat + k * 512, w);
                    }
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) {
                        const int p0 = c * 32;
                        tma_store_4d(&map_y, sbuf, c_n0, (p_w0 + (p0 & BWm)) * P.osw + sto_w, (p_h0 + ((p0 >> P.lgBW) & BHm)) * P.osh + sto_h,
                                     p_b0 + (p0 >> (P.lgBW + P.lgBH)));
                    }
                    if (PIX == 128 && !CLASSES && P.pool) {
                        // The chunk's eight windows from the staged output: a lane takes one, eight channels of it.  A sweep of
                        // its own reads the whole output again: 12.5 us for 128x32x32x128, 8.8 for 128x16x16x256, 5.7 for
                        // 128x8x8x512; here 1.7, 1.5 and 0.7.
                        const int o = (int)ln >> 2, cg = (int)ln & 3;
                        const int ox = o & ((1 << (P.lg_sbw - 1)) - 1), oy = (o >> (P.lg_sbw - 1)) & ((1 << (P.lg_sbh - 1)) - 1),
                                  ob = o >> (P.lg_sbw + P.lg_sbh - 2);
                        const int q0 = (((ob << P.lg_sbh) + 2 * oy) << P.lg_sbw) + 2 * ox, p0 = c * 32;
                        uint32_t best[4] = {0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u, 0xFF80FF80u};
#pragma unroll
                        for (int t = 0; t < 4; ++t) {
                            const int q = q0 + (t & 1) + ((t >> 1) << P.lg_sbw);
                            const uint4 x = ld_shared_v4(smem_u32(sbuf) + q * 64 + ((cg ^ ((q >> 1) & 3)) << 4));
                            best[0] = max_first_bf16x2(best[0], x.x); best[1] = max_first_bf16x2(best[1], x.y);
                            best[2] = max_first_bf16x2(best[2], x.z); best[3] = max_first_bf16x2(best[3], x.w);
                        }
                        const int gx = ((p_w0 + (p0 & BWm)) >> 1) + ox, gy = ((p_h0 + ((p0 >> P.lgBW) & BHm)) >> 1) + oy,
                                  gb = p_b0 + (p0 >> (P.lgBW + P.lgBH)) + ob, gc = c_n0 + 8 * cg;
                        if (gx < P.PW && gy < P.PH && gb < P.Bv && gc < P.Cout)
                            *reinterpret_cast<uint4 *>(P.pool + (((size_t)gb * P.PH + gy) * P.PW + gx) * P.Cout + gc) =
                                make_uint4(no_max_to_zero(best[0]), no_max_to_zero(best[1]), no_max_to_zero(best[2]), no_max_to_zero(best[3]));
                    }
                    ++nst;
                    continue;
                }
                // output offset of pixel `lane` of this chunk (per-thread stores and residual loads
                // exchange them by shuffle), ~0 = outside the output
                uint32_t my_off = 0xFFFFFFFFu;
                if (need_off) {
                    const int p = c * 32 + lane;
                    const int wv = p_w0 + (p & BWm);
                    const int hv = p_h0 + ((p >> P.lgBW) & BHm);
                    const int bv = p_b0 + (p >> (P.lgBW + P.lgBH));
                    if (wv < P.Wv && hv < P.Hv && bv < P.Bv)
                        my_off = (uint32_t)((((long long)bv * P.OH + (hv * P.osh + P.ooh)) * P.OW + (wv * P.osw + P.oow)) * P.ldy);
                }
                if (use_res_tma) {
                    if (!mbar_wait_warp(&my_res_full[nres & 1u], (nres >> 1) & 1u, abort_flag, P.status, 32)) { alive = false; break; }
                }
                if (P.bn_partial) {
                    // Batch statistics of z = acc * scale' + shift, the value before the residual and the ReLU,
                    // over the pixels that exist (a ragged tile computes on zero-filled pixels too).  Lane j
                    // decides for pixel j of the chunk, a vote makes the mask warp-wide.
                    const int p = c * 32 + lane;
                    const bool in_range = (p_w0 + (p & BWm)) < P.Wv && (p_h0 + ((p >> P.lgBW) & BHm)) < P.Hv &&
                                          (p_b0 + (p >> (P.lgBW + P.lgBH))) < P.Bv;
                    const uint32_t live = __ballot_sync(0xffffffffu, in_range);
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float z = fmaf(__uint_as_float(v[j]), sc, sf);
                        if ((live >> j) & 1u) { bn_s1 += z; bn_s2 = fmaf(z, z, bn_s2); }
                    }
                }
                // The inner loops are kept free of conditionals: every instruction issued here is
                // exposed latency of this warp's chunk.
                if (use_res_tma) {
                    const __nv_bfloat16 *rs = my_res + (nres & 1u) * (32 * 32) + lane;
                    if (P.res_gate) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const float y = fmaf(__uint_as_float(v[j]), sc, sf);
                            v[j] = __float_as_uint(__bfloat162float(rs[j * 32]) > 0.0f ? y : 0.0f);
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j)
                            v[j] = __float_as_uint(fmaf(__uint_as_float(v[j]), sc, sf) + __bfloat162float(rs[j * 32]));
                    }
                    // the buffer is free again: fetch the residual of the chunk after the next
                    __syncwarp();
                    if (lane == 0 && i + 2 < kMine) res_load(c + 2 * kEpiSets, nres & 1u);
                    ++nres;
                } else if (P.residual) {
                    // y = acc * scale' + shift + residual (residual fetched with the per-pixel offsets)
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const uint32_t o = __shfl_sync(0xffffffffu, my_off, j);
                        float r = 0.0f;
                        if (o != 0xFFFFFFFFu && n_ok)
                            r = res_bf16 ? __bfloat162float(reinterpret_cast<const __nv_bfloat16 *>(P.residual)[(size_t)o + n])
                                         : reinterpret_cast<const float *>(P.residual)[(size_t)o + n];
                        const float y = fmaf(__uint_as_float(v[j]), sc, sf);
                        v[j] = __float_as_uint(P.res_gate ? (r > 0.0f ? y : 0.0f) : y + r);
                    }
                } else {
                    // two pixels per instruction
#pragma unroll
                    for (int j = 0; j < 32; j += 2) fma_f32x2(v[j], v[j + 1], sc, sc, sf, sf);
                }
                if (relu_here) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(relu_f32(__uint_as_float(v[j])));
                }
                if (P.tma_store) {
                    // a staging buffer holds 32 pixels of bf16 or 16 of fp32: one or two rounds per chunk
                    const int rounds = out_bf16 ? 1 : 2;
                    for (int h = 0; h < rounds; ++h) {
                        // the buffer was last read by the store this warp issued kOutBufs rounds ago
                        if (lane == 0) asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(kOutBufs - 1) : "memory");
                        __syncwarp();
                        uint8_t *const sbuf = my_out + (nst % kOutBufs) * kStageBytes;
                        if (out_bf16) {
                            uint16_t *const st16 = reinterpret_cast<uint16_t *>(sbuf) + lane;
#pragma unroll
                            for (int j = 0; j < 32; j += 2) {
                                // one packed conversion per two pixels
                                const uint32_t pk = relu_in_cvt ? pack_bf16x2_relu(__uint_as_float(v[j]), __uint_as_float(v[j + 1]))
                                                                : pack_bf16x2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]));
                                st16[j * 32] = (uint16_t)pk;
                                st16[(j + 1) * 32] = (uint16_t)(pk >> 16);
                            }
                        } else {
                            uint32_t *const st32 = reinterpret_cast<uint32_t *>(sbuf) + lane;
                            if (h == 0) {
#pragma unroll
                                for (int j = 0; j < 16; ++j) st32[j * 32] = v[j];
                            } else {
#pragma unroll
                                for (int j = 0; j < 16; ++j) st32[j * 32] = v[16 + j];
                            }
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) {
                            const int p0 = c * 32 + h * 16;
                            tma_store_4d(&map_y, sbuf, c_n0, (p_w0 + (p0 & BWm)) * P.osw + sto_w,
                                         (p_h0 + ((p0 >> P.lgBW) & BHm)) * P.osh + sto_h, p_b0 + (p0 >> (P.lgBW + P.lgBH)));
                        }
                        ++nst;
                    }
                } else {
                    if (out_bf16) {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const uint32_t o = __shfl_sync(0xffffffffu, my_off, j);
                            if (o != 0xFFFFFFFFu && n_ok) y16[o] = __float2bfloat16_rn(__uint_as_float(v[j]));
                        }
                    } else {
#pragma unroll
                        for (int j = 0; j < 32; ++j) {
                            const uint32_t o = __shfl_sync(0xffffffffu, my_off, j);
                            if (o != 0xFFFFFFFFu && n_ok) y32[o] = __uint_as_float(v[j]);
                        }
                    }
                }
            }
            if (!CLASSES && P.bn_partial && warp_on)
                *reinterpret_cast<float2 *>(P.bn_partial + ((size_t)tile * kEpiSets + es) * (2 * kChan) + (q * 32 + lane) * 2) =
                    make_float2(bn_s1, bn_s2);
            __syncwarp();
        }
        // all bulk stores of this thread have been written before the block may exit
        if (P.tma_store && lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }

    // ---------------------------------------------------- teardown
    tc_fence_before();
    __syncthreads();
    if (sm->abort_flag) {
        // give copies and MMAs still in flight time to land before the memory is released
        for (int i = 0; i < 64; ++i) __nanosleep(1000);
        __syncthreads();
    }
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
    }
}

// Totals of the per-tile statistics: one warp per channel, the lanes take the tiles in turn and a shuffle tree
// adds the 32 partial totals: a fixed order, so the result is the same bits on every run.
__global__ void __launch_bounds__(256)
bn_reduce_kernel(const float *__restrict__ partial, int total_tiles, int n_tiles, int Cout,
                 double *__restrict__ sum, double *__restrict__ sumsq)
{
    const int lane = threadIdx.x & 31;
    const int c = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (c >= Cout) return;
    const int nt = c / kChan, within = c - nt * kChan;
    double s1 = 0.0, s2 = 0.0;
    for (int tile = nt + lane * n_tiles; tile < total_tiles; tile += 32 * n_tiles)
#pragma unroll
        for (int es = 0; es < kEpiSets; ++es) {
            const float2 v = __ldg(reinterpret_cast<const float2 *>(partial + ((size_t)tile * kEpiSets + es) * (2 * kChan) + within * 2));
            s1 += (double)v.x; s2 += (double)v.y;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_down_sync(0xffffffffu, s1, o);
        s2 += __shfl_down_sync(0xffffffffu, s2, o);
    }
    if (lane == 0) { sum[c] = s1; sumsq[c] = s2; }
}

// ---------------------------------------------------------------- host side
template <int PIX, int BITS, bool CLASSES = false, bool WORDS = false>
int launch_conv_t(const Geometry &g, ConvParams &P, const void *X, const twn_device_info &dev,
                  EncodeTiledFn enc, cudaStream_t s, ClassTable *table = nullptr)
{
    static bool attr_set[64] = {false};
    const int smem_bytes = (int)sizeof(SmemLayout<PIX>) + 1024;
    if (!attr_set[dev.ordinal]) {
        TWN_CUDA_OK(cudaFuncSetAttribute(tconv_kernel<PIX, BITS, CLASSES, WORDS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes));
        attr_set[dev.ordinal] = true;
    }
    pick_tile(g, PIX, &P.lgBW, &P.lgBH);
    const int BW = 1 << P.lgBW, BH = 1 << P.lgBH, BB = PIX >> (P.lgBW + P.lgBH);
    P.tw = (g.Wv + BW - 1) / BW;
    P.th = (g.Hv + BH - 1) / BH;
    P.tb = (g.Bv + BB - 1) / BB;
    long long total = (long long)P.n_tiles * P.tw * P.th * P.tb;
    if (CLASSES) {
        total = 0;
        for (int c = 0; c < table->n; ++c) {
            auto &C = table->cls[c];
            if (total > 0x7fffffffLL) return TWN_ERR_INVALID_ARG;
            C.tile0 = (int)total;
            C.tw = (C.Wv + BW - 1) / BW;
            C.th = (C.Hv + BH - 1) / BH;
            total += (long long)P.n_tiles * C.tw * C.th * P.tb;
            if (C.kb > 0) table->live_tiles = (int)std::min(total, 0x7fffffffLL);
        }
    }
    if (total <= 0 || total > 0x7fffffffLL) return TWN_ERR_INVALID_ARG;
    P.total_tiles = (int)total;

    // activations: (C, W, H, B), 64-channel boxes with 128-byte swizzle, zero fill outside
    CUtensorMap map_x;
    {
        cuuint64_t dims[4] = {(cuuint64_t)g.XC, (cuuint64_t)g.XW, (cuuint64_t)g.XH, (cuuint64_t)g.XB};
        const long long rowp = g.x_row_pitch ? g.x_row_pitch : g.XW * g.ldx;
        const long long imgp = g.x_img_pitch ? g.x_img_pitch : g.XH * rowp;
        cuuint64_t strides[3] = {(cuuint64_t)g.ldx * 2, (cuuint64_t)rowp * 2, (cuuint64_t)imgp * 2};
        // with a traversal stride the box counts traversed elements: N loaded elements need N * stride
        cuuint32_t box[4] = {(cuuint32_t)kBlockK, (cuuint32_t)(BW * g.sw), (cuuint32_t)(BH * g.sh), (cuuint32_t)BB};
        cuuint32_t estr[4] = {1, (cuuint32_t)g.sw, (cuuint32_t)g.sh, 1};
        if (enc(&map_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(X), dims, strides, box, estr,
                CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
            return TWN_ERR_INVALID_ARG;
    }
    // output: TMA stores when the pitch allows it.  The virtual output grid may be embedded in
    // the tensor with a stride and an offset (backward for data of a strided layer): the map
    // then starts at the offset pixel and traverses with that stride.
    // (the channel extent must be a whole number of 16-byte units: the store clips at that granularity)
    CUtensorMap map_y = map_x, map_r = map_x;
    const int es = P.out_dtype == TWN_BF16 ? 2 : 4;
    P.tma_store = 0;
    P.res_tma = 0;
    // a bf16 residual is as addressable as a bf16 output of the same pitch, but for its base
    P.fragments = es == 2 && !P.bn_partial &&
                  (!P.residual || (P.res_dtype == TWN_BF16 && reinterpret_cast<uintptr_t>(P.residual) % 16 == 0));
    const CUtensorMapSwizzle swz = P.fragments ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_NONE;
    const long long base_pix = (long long)g.ooh * g.OW + g.oow;
    if ((g.ldy * es) % 16 == 0 && ((long long)g.Cout * es) % 16 == 0 && (reinterpret_cast<uintptr_t>(P.Y) % 16) == 0 &&
        g.OW > g.oow && g.OH > g.ooh) {
        // 2^lg consecutive tile pixels are a sub-box sbw x sbh x sbb of the tile box, 32 channels wide
        // (one epilogue warp): a staging buffer holds 32 pixels of bf16 or 16 of fp32, a residual
        // buffer 32 pixels
        auto sub_box = [&](int lg, cuuint32_t *bx) {
            const int lg_sbw = P.lgBW < lg ? P.lgBW : lg;
            const int lg_sbh = P.lgBH < lg - lg_sbw ? P.lgBH : lg - lg_sbw;
            const int lg_sbb = lg - lg_sbw - lg_sbh;
            bx[0] = 32u; bx[1] = (cuuint32_t)((1 << lg_sbw) * g.osw);
            bx[2] = (cuuint32_t)((1 << lg_sbh) * g.osh); bx[3] = 1u << lg_sbb;
        };
        cuuint64_t dims[4] = {(cuuint64_t)g.Cout, (cuuint64_t)(g.OW - g.oow), (cuuint64_t)(g.OH - g.ooh), (cuuint64_t)g.Bv};
        cuuint32_t box[4], rbox[4];
        sub_box(es == 2 ? 5 : 4, box);
        sub_box(5, rbox);
        cuuint32_t estr[4] = {1, (cuuint32_t)g.osw, (cuuint32_t)g.osh, 1};
        if (box[1] <= 256 && box[2] <= 256 && rbox[1] <= 256 && rbox[2] <= 256) {
            cuuint64_t strides[3] = {(cuuint64_t)g.ldy * es, (cuuint64_t)g.OW * g.ldy * es, (cuuint64_t)g.OH * g.OW * g.ldy * es};
            void *ybase = static_cast<char *>(P.Y) + base_pix * g.ldy * es;
            if (enc(&map_y, es == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, ybase, dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
                    CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
                P.tma_store = 1;
            // a bf16 residual of the same geometry is staged the same way
            if (P.tma_store && P.residual && P.res_dtype == TWN_BF16 && (g.ldy * 2) % 16 == 0 &&
                ((long long)g.Cout * 2) % 16 == 0 && (reinterpret_cast<uintptr_t>(P.residual) % 16) == 0) {
                cuuint64_t rstrides[3] = {(cuuint64_t)g.ldy * 2, (cuuint64_t)g.OW * g.ldy * 2, (cuuint64_t)g.OH * g.OW * g.ldy * 2};
                void *rbase = const_cast<char *>(static_cast<const char *>(P.residual)) + base_pix * g.ldy * 2;
                if (enc(&map_r, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, rbase, dims, rstrides, rbox, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS)
                    P.res_tma = 1;
            }
        }
    }
    P.fragments = P.fragments && P.tma_store;
    if (g.pool) {
        if (!P.fragments) return TWN_ERR_CUDA;       // the caller has looked at everything that could be in the way
        P.pool = static_cast<__nv_bfloat16 *>(g.pool);
        P.PH = g.Hv / 2; P.PW = g.Wv / 2;
        P.lg_sbw = P.lgBW;
        P.lg_sbh = std::min(P.lgBH, 5 - P.lgBW);
    }
    if (CLASSES && !P.fragments) return TWN_ERR_CUDA;       // the caller has looked at what fragments need
    if (P.fragments && P.residual && !P.res_tma) return TWN_ERR_CUDA;      // the same geometry could be encoded for Y
    const int grid = dev.sm_count < P.total_tiles ? dev.sm_count : P.total_tiles;
    // Programmatic dependent launch pays when the blocks cover the GPU (set-up and launch latency hide behind the
    // previous kernel's last tiles); a launch of a few blocks measured slower with it (an inner product of 8 blocks
    // after a convolution: 21 us instead of 12), so those launch the plain way.
    const bool kPdlConv = grid * 2 >= dev.sm_count;
    if (P.bn_partial && (size_t)P.total_tiles * kEpiSets * 2 * kChan * sizeof(float) > g.bn_partial_bytes) return TWN_ERR_WORKSPACE;
    std::conditional_t<CLASSES, ClassTable, NoClasses> classes;
    if constexpr (CLASSES) classes = *table;
    TWN_CUDA_OK(twn_launch_pdl(kPdlConv, tconv_kernel<PIX, BITS, CLASSES, WORDS>, grid, threads_conv(Cfg<PIX>::kDecodeGroups), (size_t)smem_bytes, s,
                               map_x, map_y, map_r, P, classes));
    if (P.bn_partial)
        bn_reduce_kernel<<<(g.Cout + 7) / 8, 256, 0, s>>>(P.bn_partial, P.total_tiles, P.n_tiles, g.Cout, g.bn_sum, g.bn_sumsq);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

EpilogueArgs epilogue_args(const twn_stats_t *stats, const twn_epilogue_t *epi, int out_dtype_default)
{
    EpilogueArgs ea;
    ea.alpha = stats ? &stats->alpha : nullptr;
    ea.scale = epi ? epi->scale : nullptr;
    ea.shift = epi ? epi->shift : nullptr;
    ea.residual = epi ? epi->residual : nullptr;
    ea.res_dtype = epi ? epi->residual_dtype : TWN_F32;
    ea.res_gate = (epi && epi->residual) ? epi->residual_op & TWN_RESIDUAL_GATE : 0;
    ea.in_order = epi && (epi->residual_op & TWN_SUM_IN_ORDER);
    ea.relu = epi ? epi->relu : 0;
    ea.out_dtype = epi ? epi->out_dtype : out_dtype_default;
    return ea;
}

// With `us_only`, nothing is launched: it receives what the launch that the same call would make should take.
int launch_conv(const Geometry &g, const void *X, const uint32_t *T, const twn_stats_t *stats,
                const twn_epilogue_t *epi, void *Y, int out_dtype_default, int32_t *dev_status, cudaStream_t s,
                double *us_only = nullptr)
{
    twn_device_info dev;
    int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    EncodeTiledFn enc = encode_fn();
    if (!enc) return TWN_ERR_CUDA;

    // the epilogue keeps output offsets in 32 bits
    if ((long long)g.Bv * g.OH * g.OW * g.ldy >= 0xFFFFFFFFLL) return TWN_ERR_INVALID_ARG;
    const EpilogueArgs ea = epilogue_args(stats, epi, out_dtype_default);
    // problems that do not fill the GPU: small tiles, the reduction split over a cluster
    const bool classes = g.n_classes > 0;
    const SplitPlan split = classes ? SplitPlan{0, 0, 1e30} : plan_conv_split(g, dev.sm_count / (g.beside > 1 ? g.beside : 1), ea.in_order);
    ConvParams P;
    memset(&P, 0, sizeof P);
    P.n_tiles = (g.Cout + kChan - 1) / kChan;
    P.n_taps = g.n_taps;
    P.n_cblk = (int)((g.Cin + kBlockK - 1) / kBlockK);
    P.code_run = code_run(g);
    // (a pair of k-blocks: 8 words of ternary codes, 4 of binary ones)
    if (P.code_run * (g.code_bits == 1 ? 2 : 1) == 4 && g.ld_codes % 128 == 0 && reinterpret_cast<uintptr_t>(T) % 32 == 0) {
        bool follow = true;
        if (classes) {
            // taps in any order: a pair of k-blocks is one of a tap
            follow = P.n_cblk % 2 == 0 && g.n_taps * P.n_cblk <= kWordTab;
            for (int t = 0; t < g.n_taps; ++t) follow &= g.taps[t].koff % (2 * kBlockK) == 0;
        } else {
            for (int t = 0; t < g.n_taps; ++t) follow &= g.taps[t].koff == t * P.n_cblk * kBlockK;
        }
        if (follow) P.code_run = 8;
    }
    // Tile shape by a model of the launch's time: a fixed part and, per round of tiles, an epilogue and the k-blocks, or where
    // the epilogue of one tile overlaps the reduction of the next at least the epilogue.  Fitted to 40 launches (convolutions of
    // 16 to 128 images, inner products of 333 to 50176 rows) forced to each shape, three inputs in turn; what it picks takes 0.7 %
    // longer on average than the best of the three, 9 % at most (32x32x128, 128 images).
    int a, b;
    const long long kb = (long long)P.n_taps * P.n_cblk;
    const long long sms = dev.sm_count;
    const bool half = g.Cout <= kChan / 2;           // half of the epilogue warps idle
    const long long t128 = pick_tile(g, 128, &a, &b) * P.n_tiles, t256 = pick_tile(g, 256, &a, &b) * P.n_tiles;
    const long long t192 = pick_tile(g, 192, &a, &b) * P.n_tiles;
    auto time_us = [&](long long tiles, double fixed, double per_tile, double per_block, double least) {
        return fixed + (double)((tiles + sms - 1) / sms) * std::max(per_tile + per_block * (double)kb, least);
    };
    // (k-blocks off the 16-byte boundaries come with two or four loads, which the smaller shapes wait for: 7 further shapes, all of
    // them measured with four)
    const bool words = P.code_run * (g.code_bits == 1 ? 2 : 1) < 4;
    const double u128 = time_us(t128, 4.3, 1.4, words ? 0.225 : 0.155, 1.85),
                 u192 = time_us(t192, 5.1, 1.6, words ? 0.24 : 0.225, half ? 1.76 : 2.43),
                 u256 = time_us(t256, 5.4, half ? 2.4 : 2.8, 0.293, 3.0);
    // Another shape than 128 pixels has to gain more than a launch loses whose code is not that of the launches before it (1.5
    // us): VGG-7 at 128 images takes 189.7 us when its five layers run in the 128-pixel kernel, 200.3 with two of the others
    // between them, although alone each layer is within 10 % in its best shape.  What a call loses with it whose neighbours are
    // of its own kind: of 140 calls of all sizes, each alone in a graph of twelve, it decides ten, where the three models are
    // close, and those are 3 % faster with it on average (81x81x384, 5x5: 48.4 us, 64.7 without; 6 of the ten between -2 and
    // -6 %); at worst 6 % slower (16384x4608x512: 63.8 / 60.1).
    constexpr double kOther = 1.5;
    // The classes of a strided backward pass in one launch: their tiles go round the blocks, the longest first, and end with half a
    // tile's difference.  Fitted to 97 shapes (1 to 128 images of 7 to 110 pixels, 32 to 768 channels, 1x1 to 5x5) forced to it: 7 %
    // off on average, 22 % at most.
    double all_classes = 0.0;
    ClassTable table;
    if (classes) {
        table.n = g.n_classes;
        table.live_tiles = 0;
        double work = 0.0, longest = 0.0;
        for (int c = 0; c < g.n_classes; ++c) {
            const TapClass &k = g.cls[c];
            table.cls[c].Hv = k.Hv; table.cls[c].Wv = k.Wv; table.cls[c].ooh = k.ooh; table.cls[c].oow = k.oow;
            table.cls[c].tap0 = k.tap0; table.cls[c].kb0 = k.tap0 * P.n_cblk;
            table.cls[c].kb = k.n_taps * P.n_cblk; table.cls[c].stages = (table.cls[c].kb + Cfg<128>::kSub - 1) / Cfg<128>::kSub;
            const double us = 1.24 + (words ? (P.code_run == 1 ? 0.257 : 0.218) : P.code_run == 8 ? 0.149 : 0.219) * (double)(k.n_taps * P.n_cblk);
            work += us * (double)t128;
            longest = std::max(longest, us);
        }
        all_classes = 4.56 + std::max(longest, work / (double)sms + 0.58 * longest);
        if (us_only) {
            // bf16 in and out by TMA, else not at all
            const bool fits = ea.out_dtype == TWN_BF16 && g.Cout % 8 == 0 && g.ldy % 8 == 0 && twn_aligned(Y, 16) &&
                              (!ea.residual || (ea.res_dtype == TWN_BF16 && twn_aligned(ea.residual, 16)));
            *us_only = fits ? all_classes : 1e30;
            return TWN_OK;
        }
    }
    int choice = u256 + kOther < u128 ? 1 : 0;
    if (u192 + (choice ? 0.0 : kOther) < (choice ? u256 : u128)) choice = 2;
    // Of the three shapes pooling is in that kernel alone: the others, whose epilogue is longer with it, lost 0.6 % on
    // 16384x4096x4096 to code that they do not run.
    if (g.pool || classes) choice = 0;
    const double us = choice == 0 ? u128 : choice == 1 ? u256 : u192;
    // Narrow layers and short reductions: the kernel that decodes its channels' codes once per block.  Up to 64 channels
    // the general kernel's half-empty tiles lose wherever that kernel runs; above, its own time decides.
    bool handled = false;
    if (!g.pool && !classes) rc = launch_conv_resident(g, X, T, ea, Y, dev_status, dev, s, half || split.us < us ? split.us : us, &handled, us_only);
    if (rc != TWN_OK || handled) return rc;
    // The more SMs the general kernel fills by itself, the clearer the modelled gain has to be: near the line the split
    // kernel's model is the optimistic one where most SMs are filled (3x3 3x56x56x64 -> 256: 66 % filled, 9.5 us split, 7.7 here,
    // modelled 8.4 and 8.7), and not where few are (1392x624x720: 45 %, 7.1 split, 8.4 here, modelled 6.5 and 7.2).
    const long long tiles = choice == 0 ? t128 : choice == 1 ? t256 : t192;
    const double fill = tiles < sms ? (double)tiles / (double)sms : 1.0;
    const bool take_split = split.us < (1.0 - 0.25 * fill * fill) * us;
    if (us_only) {
        *us_only = take_split ? split.us : us;
        return TWN_OK;
    }
    if (take_split) return launch_conv_split(g, X, T, ea, Y, dev_status, dev, s, split);
    P.T = T;
    P.wpr = g.ld_codes / (g.code_bits == 1 ? 32 : 16);
    P.sw = g.sw; P.sh = g.sh;
    P.Bv = g.Bv; P.Hv = g.Hv; P.Wv = g.Wv;
    P.OH = g.OH; P.OW = g.OW; P.osh = g.osh; P.osw = g.osw; P.ooh = g.ooh; P.oow = g.oow;
    P.ldy = g.ldy;
    P.Cout = g.Cout;
    P.alpha = ea.alpha; P.scale = ea.scale; P.shift = ea.shift;
    P.residual = ea.residual; P.res_dtype = ea.res_dtype; P.res_gate = ea.res_gate;
    P.relu = ea.relu; P.out_dtype = ea.out_dtype;
    P.Y = Y;
    P.status = dev_status;
    P.bn_partial = g.bn_partial;
    for (int t = 0; t < g.n_taps; ++t) P.taps[t] = g.taps[t];
    const bool by_word = P.code_run == 1;
    if (g.code_bits == 1) {
        if (classes) return launch_conv_t<128, 1, true>(g, P, X, dev, enc, s, &table);
        return choice == 1 ? launch_conv_t<256, 1>(g, P, X, dev, enc, s) : choice == 2 ? launch_conv_t<192, 1>(g, P, X, dev, enc, s)
                                                                                    : launch_conv_t<128, 1>(g, P, X, dev, enc, s);
    }
    if (classes) return by_word ? launch_conv_t<128, 2, true, true>(g, P, X, dev, enc, s, &table) : launch_conv_t<128, 2, true>(g, P, X, dev, enc, s, &table);
    if (choice != 0) return choice == 1 ? launch_conv_t<256, 2>(g, P, X, dev, enc, s) : launch_conv_t<192, 2>(g, P, X, dev, enc, s);
    return by_word ? launch_conv_t<128, 2, false, true>(g, P, X, dev, enc, s) : launch_conv_t<128, 2>(g, P, X, dev, enc, s);
}

// Helper streams for launches that are independent of one another (the residue classes of a
// strided backward-for-data pass write disjoint pixels).  They fork from the caller's stream
// through an event and join it again the same way, so the caller sees one stream-ordered
// operation; under stream capture the fork and the join become graph edges.  Created once per
// device; a mutex keeps two host threads from interleaving their use of the shared events.
struct ForkPool {
    cudaStream_t side[3];
    cudaEvent_t fork, join[3];
    bool ready = false, failed = false;
};
std::mutex g_fork_mutex;

ForkPool *fork_pool(int ordinal)
{
    static ForkPool pools[64];
    ForkPool &p = pools[ordinal];
    if (p.failed) return nullptr;
    if (!p.ready) {
        bool ok = cudaEventCreateWithFlags(&p.fork, cudaEventDisableTiming) == cudaSuccess;
        for (int i = 0; i < 3 && ok; ++i)
            ok = cudaStreamCreateWithFlags(&p.side[i], cudaStreamNonBlocking) == cudaSuccess &&
                 cudaEventCreateWithFlags(&p.join[i], cudaEventDisableTiming) == cudaSuccess;
        if (!ok) { p.failed = true; return nullptr; }
        p.ready = true;
    }
    return &p;
}

// Shared by the ternary (bits = 2) and binary (bits = 1) entry points.
int gemm_impl(const void *X, int64_t ldx, const uint32_t *T_packed, int64_t ld_codes,
              const twn_stats_t *stats, int64_t M, int64_t N, int64_t K,
              const twn_epilogue_t *epi, void *Y, int64_t ldy, int32_t *dev_status,
              twn_stream_t stream, int bits)
{
    TWN_REQUIRE(M >= 0 && N >= 0 && K >= 0, TWN_ERR_INVALID_ARG);
    if (M == 0 || N == 0) return TWN_OK;
    TWN_REQUIRE(X && T_packed && Y && K > 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ldx >= K && ldy >= N && ld_codes >= K && ld_codes % (bits == 1 ? 128 : 64) == 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(M <= 0x7fffffffLL && N <= 0x7fffffffLL && K <= 0x7fffffffLL, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ldx % 8 == 0, TWN_ERR_MISALIGNED);
    TWN_REQUIRE(twn_aligned(X, 16) && twn_aligned(T_packed, 16) && twn_aligned(Y, 4) && twn_aligned(stats, 8) &&
                    twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    int rc = check_epilogue(epi);
    if (rc != TWN_OK) return rc;
    Geometry g;
    memset(&g, 0, sizeof g);
    g.XB = 1; g.XH = 1; g.XW = M; g.XC = K; g.ldx = ldx;
    g.Bv = 1; g.Hv = 1; g.Wv = (int)M; g.OH = 1; g.OW = (int)M;
    g.osh = g.osw = 1; g.ooh = g.oow = 0; g.ldy = ldy;
    g.sh = g.sw = 1;
    g.Cout = (int)N; g.ld_codes = ld_codes; g.code_cols = K;
    g.n_taps = 1; g.taps[0] = Tap{0, 0, 0};
    g.Cin = K;
    g.code_bits = bits;
    return launch_conv(g, X, T_packed, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream));
}

}  // namespace

extern "C" int twn_gemm(const void *X, int64_t ldx, const uint32_t *T_packed, int64_t ld_codes,
                        const twn_stats_t *stats, int64_t M, int64_t N, int64_t K,
                        const twn_epilogue_t *epi, void *Y, int64_t ldy, int32_t *dev_status,
                        twn_stream_t stream)
{
    return gemm_impl(X, ldx, T_packed, ld_codes, stats, M, N, K, epi, Y, ldy, dev_status, stream, 2);
}

extern "C" int twn_gemm_b1(const void *X, int64_t ldx, const uint32_t *B_packed, int64_t ld_codes,
                           const twn_stats_t *stats, int64_t M, int64_t N, int64_t K,
                           const twn_epilogue_t *epi, void *Y, int64_t ldy, int32_t *dev_status,
                           twn_stream_t stream)
{
    return gemm_impl(X, ldx, B_packed, ld_codes, stats, M, N, K, epi, Y, ldy, dev_status, stream, 1);
}

namespace {

int conv_common_checks(const twn_conv_desc_t *d)
{
    TWN_REQUIRE(d != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->B > 0 && d->H > 0 && d->W > 0 && d->Cin > 0 && d->Cout > 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->kh > 0 && d->kw > 0 && d->stride_h > 0 && d->stride_w > 0 && d->pad_h >= 0 && d->pad_w >= 0,
                TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->stride_h <= 8 && d->stride_w <= 8, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->kh * d->kw <= kMaxTaps, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->H + 2 * d->pad_h >= d->kh && d->W + 2 * d->pad_w >= d->kw, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->B <= 0x7fffffffLL && d->H <= 0x7fffffffLL && d->W <= 0x7fffffffLL && d->Cin <= 0x7fffffffLL &&
                    d->Cout <= 0x7fffffffLL, TWN_ERR_INVALID_ARG);
    return TWN_OK;
}

}  // namespace

namespace {

struct BnArgs { double *sum, *sumsq; void *ws; size_t ws_bytes; };
struct PoolArgs { void *Yp; bool *done; };

int conv_fwd_impl(const twn_conv_desc_t *d, const void *X, const uint32_t *T_fwd, int64_t ld_codes,
                  const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y,
                  int32_t *dev_status, twn_stream_t stream, int bits, const BnArgs *bn = nullptr, const PoolArgs *pool = nullptr)
{
    int rc = conv_common_checks(d);
    if (rc != TWN_OK) return rc;
    TWN_REQUIRE(X && T_fwd && Y, TWN_ERR_INVALID_ARG);
    const long long taps = (long long)d->kh * d->kw;
    TWN_REQUIRE(ld_codes % (bits == 1 ? 128 : 64) == 0 && ld_codes >= taps * d->Cin, TWN_ERR_INVALID_ARG);
    // channel runs must start on 16-byte boundaries for TMA, tap columns on word boundaries
    TWN_REQUIRE(d->Cin % 8 == 0 && (taps == 1 || d->Cin % (bits == 1 ? 32 : 16) == 0), TWN_ERR_MISALIGNED);
    TWN_REQUIRE(twn_aligned(X, 16) && twn_aligned(T_fwd, 16) && twn_aligned(Y, 4) && twn_aligned(stats, 8) &&
                    twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    rc = check_epilogue(epi);
    if (rc != TWN_OK) return rc;
    const long long Ho = (d->H + 2 * d->pad_h - d->kh) / d->stride_h + 1;
    const long long Wo = (d->W + 2 * d->pad_w - d->kw) / d->stride_w + 1;
    Geometry g;
    memset(&g, 0, sizeof g);
    g.XB = d->B; g.XH = d->H; g.XW = d->W; g.XC = d->Cin; g.ldx = d->Cin;
    g.Bv = (int)d->B; g.Hv = (int)Ho; g.Wv = (int)Wo; g.OH = (int)Ho; g.OW = (int)Wo;
    g.osh = g.osw = 1; g.ooh = g.oow = 0; g.ldy = d->Cout;
    g.sh = d->stride_h; g.sw = d->stride_w;
    g.Cout = (int)d->Cout; g.ld_codes = ld_codes; g.code_cols = taps * d->Cin;
    g.Cin = d->Cin;
    for (int r = 0; r < d->kh; ++r)
        for (int s = 0; s < d->kw; ++s) {
            Tap &t = g.taps[g.n_taps++];
            t.dh = (int16_t)(r - d->pad_h);
            t.dw = (int16_t)(s - d->pad_w);
            t.koff = (int32_t)((r * d->kw + s) * d->Cin);
        }
    g.code_bits = bits;
    if (bn) {
        g.bn_partial = static_cast<float *>(bn->ws);
        g.bn_partial_bytes = bn->ws_bytes;
        g.bn_sum = bn->sum; g.bn_sumsq = bn->sumsq;
    }
    // Without padding in w the taps of a filter row read one run of kw * Cin elements, in the order of its codes: a "pixel" of as
    // many channels, Cin elements from the next, and one tap per row.  Where that fills the k-blocks of 64 better and a kernel is
    // modelled faster with it (5x5 on 32 channels: 15 k-blocks for 25; 100x12x12x32 -> 64, pooled, 10.6 -> 9.4
    // us; 128x30x30x16 -> 128 31.9 -> 19.5).  The order of a sum is the same.
    const long long run = d->kw * d->Cin;
    double alone = -1.0;             // what the layer takes by itself, where that has been looked up
    if (d->pad_w == 0 && d->kw > 1 && (run + 63) / 64 < d->kw * ((d->Cin + 63) / 64)) {
        Geometry rows = g;
        rows.XW = d->W - d->kw + 1; rows.XC = rows.Cin = run;
        rows.x_row_pitch = d->W * d->Cin; rows.x_img_pitch = d->H * d->W * d->Cin;
        rows.n_taps = d->kh;
        for (int r = 0; r < d->kh; ++r) rows.taps[r] = g.taps[r * d->kw];
        double by_tap = 0.0, by_row = 0.0;
        rc = launch_conv(g, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream), &by_tap);
        if (rc != TWN_OK) return rc;
        rc = launch_conv(rows, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream), &by_row);
        if (rc != TWN_OK) return rc;
        if (by_row < by_tap) g = rows;
        alone = std::min(by_row, by_tap);
    }
    if (pool) {
        // Pooled in the epilogue of the general or the split kernel, if that and no sweep should take less time than the kernel that
        // the layer would get by itself and a sweep (modelled as 2 us and 4.2 TB/s; 2.1 us for 100x8x8x64).  What TMA cannot store or the
        // fragments do not hold stays with the sweep.
        *pool->done = false;
        const double bytes = 2.5 * (double)g.Bv * g.Hv * g.Wv * g.Cout;
        if (epi && epi->out_dtype == TWN_BF16 && g.Cout % 8 == 0 && twn_aligned(Y, 16) && twn_aligned(pool->Yp, 16) &&
            (!epi->residual || (epi->residual_dtype == TWN_BF16 && twn_aligned(epi->residual, 16)))) {
            double apart = alone, here = 0.0;
            if (apart < 0.0) rc = launch_conv(g, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream), &apart);
            if (rc != TWN_OK) return rc;
            Geometry p = g;
            p.pool = pool->Yp;
            rc = launch_conv(p, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream), &here);
            if (rc != TWN_OK) return rc;
            if (here < apart + 2.0 + bytes / 4.2e6) {
                *pool->done = true;
                return launch_conv(p, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream));
            }
        }
    }
    return launch_conv(g, X, T_fwd, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream));
}

}  // namespace

extern "C" size_t twn_conv2d_fwd_bn_workspace_bytes(const twn_conv_desc_t *d)
{
    if (conv_common_checks(d) != TWN_OK) return 0;
    // the smallest pixel tile gives the most tiles: 128 pixels, whatever shape the launch then picks
    Geometry g;
    memset(&g, 0, sizeof g);
    g.Bv = (int)d->B;
    g.Hv = (int)((d->H + 2 * d->pad_h - d->kh) / d->stride_h + 1);
    g.Wv = (int)((d->W + 2 * d->pad_w - d->kw) / d->stride_w + 1);
    g.sh = d->stride_h; g.sw = d->stride_w;
    int a, b;
    const long long tiles = pick_tile(g, 128, &a, &b) * ((d->Cout + kChan - 1) / kChan);
    return (size_t)tiles * kEpiSets * 2 * kChan * sizeof(float);
}

extern "C" int twn_conv2d_fwd_bn(const twn_conv_desc_t *d, const void *X, const uint32_t *T_fwd, int64_t ld_codes,
                                 const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y, double *bn_sum,
                                 double *bn_sumsq, void *workspace, size_t workspace_bytes, int32_t *dev_status,
                                 twn_stream_t stream)
{
    TWN_REQUIRE(bn_sum && bn_sumsq && workspace, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(bn_sum, 8) && twn_aligned(bn_sumsq, 8) && twn_aligned(workspace, 16), TWN_ERR_MISALIGNED);
    TWN_REQUIRE(workspace_bytes >= twn_conv2d_fwd_bn_workspace_bytes(d) && workspace_bytes > 0, TWN_ERR_WORKSPACE);
    const BnArgs bn = {bn_sum, bn_sumsq, workspace, workspace_bytes};
    return conv_fwd_impl(d, X, T_fwd, ld_codes, stats, epi, Y, dev_status, stream, 2, &bn);
}

extern "C" int twn_conv2d_fwd(const twn_conv_desc_t *d, const void *X, const uint32_t *T_fwd, int64_t ld_codes,
                              const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y,
                              int32_t *dev_status, twn_stream_t stream)
{
    return conv_fwd_impl(d, X, T_fwd, ld_codes, stats, epi, Y, dev_status, stream, 2);
}

extern "C" int twn_conv2d_fwd_maxpool(const twn_conv_desc_t *d, const void *X, const uint32_t *T_fwd, int64_t ld_codes,
                                      const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y, void *Yp,
                                      int32_t *dev_status, twn_stream_t stream)
{
    const int rc0 = conv_common_checks(d);
    if (rc0 != TWN_OK) return rc0;
    TWN_REQUIRE(Yp && epi && epi->out_dtype == TWN_BF16, TWN_ERR_INVALID_ARG);
    const int64_t Ho = (d->H + 2 * d->pad_h - d->kh) / d->stride_h + 1, Wo = (d->W + 2 * d->pad_w - d->kw) / d->stride_w + 1;
    TWN_REQUIRE(Ho >= 2 && Wo >= 2, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(Yp, 4), TWN_ERR_MISALIGNED);
    bool done = false;
    const PoolArgs pool = {Yp, &done};
    const int rc = conv_fwd_impl(d, X, T_fwd, ld_codes, stats, epi, Y, dev_status, stream, 2, nullptr, &pool);
    return rc != TWN_OK || done ? rc : twn_maxpool2d_fwd(Y, d->B, Ho, Wo, d->Cout, 2, 2, 0, Yp, nullptr, stream);
}

extern "C" int twn_conv2d_fwd_b1(const twn_conv_desc_t *d, const void *X, const uint32_t *B_fwd, int64_t ld_codes,
                                 const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y,
                                 int32_t *dev_status, twn_stream_t stream)
{
    return conv_fwd_impl(d, X, B_fwd, ld_codes, stats, epi, Y, dev_status, stream, 1);
}

extern "C" int twn_conv2d_fwd_folded(const twn_conv_desc_t *d, const void *Xf, const uint32_t *Tf, int64_t ld_folded,
                                     const twn_stats_t *stats, const twn_epilogue_t *epi, void *Y,
                                     int32_t *dev_status, twn_stream_t stream)
{
    int64_t Hf, Wf, ldf;
    int rc = twn_fold_dims(d, &Hf, &Wf, &ldf);
    if (rc != TWN_OK) return rc;
    TWN_REQUIRE(Xf && Tf && Y && ld_folded == ldf, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(Xf, 16) && twn_aligned(Tf, 16) && twn_aligned(Y, 4) && twn_aligned(stats, 8) &&
                    twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    rc = check_epilogue(epi);
    if (rc != TWN_OK) return rc;
    const long long Ho = (d->H + 2 * d->pad_h - d->kh) / 2 + 1, Wo = (d->W + 2 * d->pad_w - d->kw) / 2 + 1;
    // A 64-"channel" tensor whose pixels are 16 elements apart: window position w reads folded
    // pixels w..w+3.  One tap per folded filter row, stride 1, no padding.
    Geometry g;
    memset(&g, 0, sizeof g);
    g.XB = d->B; g.XH = Hf; g.XW = Wo; g.XC = 64; g.ldx = 16;
    g.x_row_pitch = Wf * 16; g.x_img_pitch = Hf * Wf * 16;
    g.Bv = (int)d->B; g.Hv = (int)Ho; g.Wv = (int)Wo; g.OH = (int)Ho; g.OW = (int)Wo;
    g.osh = g.osw = 1; g.ooh = g.oow = 0; g.ldy = d->Cout;
    g.sh = g.sw = 1;
    g.Cout = (int)d->Cout; g.ld_codes = ldf; g.code_cols = ldf;
    g.Cin = 64;
    for (int r = 0; r < (int)(ldf / 64); ++r) {
        Tap &t = g.taps[g.n_taps++];
        t.dh = (int16_t)r;
        t.dw = 0;
        t.koff = (int32_t)(r * 64);
    }
    g.code_bits = 2;
    return launch_conv(g, Xf, Tf, stats, epi, Y, TWN_F32, dev_status, twn_cu(stream));
}

namespace {

int conv_bwd_data_impl(const twn_conv_desc_t *d, const void *dZ, const uint32_t *T_bwd, int64_t ld_codes,
                       const twn_stats_t *stats, const twn_epilogue_t *epi, void *dX,
                       int32_t *dev_status, twn_stream_t stream, int bits)
{
    int rc = conv_common_checks(d);
    if (rc != TWN_OK) return rc;
    TWN_REQUIRE(dZ && T_bwd && dX, TWN_ERR_INVALID_ARG);
    const long long taps = (long long)d->kh * d->kw;
    TWN_REQUIRE(ld_codes % (bits == 1 ? 128 : 64) == 0 && ld_codes >= taps * d->Cout, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->Cout % 8 == 0 && (taps == 1 || d->Cout % (bits == 1 ? 32 : 16) == 0), TWN_ERR_MISALIGNED);
    TWN_REQUIRE(twn_aligned(dZ, 16) && twn_aligned(T_bwd, 16) && twn_aligned(dX, 4) && twn_aligned(stats, 8) &&
                    twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    rc = check_epilogue(epi);
    if (rc != TWN_OK) return rc;
    const long long Ho = (d->H + 2 * d->pad_h - d->kh) / d->stride_h + 1;
    const long long Wo = (d->W + 2 * d->pad_w - d->kw) / d->stride_w + 1;
    // One residue class (ph, pw) of the input pixel modulo the stride at a time: inside a
    // class the adjoint is a stride-1 sum over the taps r with (ph + pad - r) divisible by
    // the stride, reading dZ at ho = h' + (ph + pad - r)/stride.  The classes write disjoint pixels.
    Geometry all;
    memset(&all, 0, sizeof all);
    all.XB = d->B; all.XH = Ho; all.XW = Wo; all.XC = d->Cout; all.ldx = d->Cout;
    all.Bv = (int)d->B;
    all.OH = (int)d->H; all.OW = (int)d->W;
    all.osh = d->stride_h; all.osw = d->stride_w;
    all.ldy = d->Cin;
    all.sh = all.sw = 1;
    all.Cout = (int)d->Cin; all.ld_codes = ld_codes; all.code_cols = taps * d->Cout;
    all.Cin = d->Cout;
    all.code_bits = bits;
    TapClass cls[64];
    int n_cls = 0;
    // A residue class no tap reaches gets epilogue(0); when the epilogue only adds a second gradient
    // branch that already lives in dX (in place), that leaves the class as it is: nothing to launch.
    const bool skip_empty = epi && epi->residual == dX && !(epi->residual_op & TWN_RESIDUAL_GATE) && !epi->scale && !epi->shift &&
                            !epi->relu && epi->residual_dtype == epi->out_dtype;
    for (int ph = 0; ph < d->stride_h; ++ph)
        for (int pw = 0; pw < d->stride_w; ++pw) {
            if (ph >= d->H || pw >= d->W) continue;
            TapClass c;
            c.Hv = (int)((d->H - ph + d->stride_h - 1) / d->stride_h);
            c.Wv = (int)((d->W - pw + d->stride_w - 1) / d->stride_w);
            c.ooh = ph; c.oow = pw;
            c.tap0 = all.n_taps;
            for (int r = 0; r < d->kh; ++r) {
                const int xh = ph + d->pad_h - r;
                if (((xh % d->stride_h) + d->stride_h) % d->stride_h != 0) continue;
                for (int s = 0; s < d->kw; ++s) {
                    const int xw = pw + d->pad_w - s;
                    if (((xw % d->stride_w) + d->stride_w) % d->stride_w != 0) continue;
                    Tap &t = all.taps[all.n_taps++];
                    t.dh = (int16_t)(xh / d->stride_h);
                    t.dw = (int16_t)(xw / d->stride_w);
                    t.koff = (int32_t)((r * d->kw + s) * d->Cout);
                }
            }
            c.n_taps = all.n_taps - c.tap0;
            if (c.n_taps == 0 && skip_empty) continue;
            cls[n_cls++] = c;
        }
    auto one_class = [&](const TapClass &c, int beside) {
        Geometry g = all;
        g.Hv = c.Hv; g.Wv = c.Wv; g.ooh = c.ooh; g.oow = c.oow;
        g.n_taps = c.n_taps;
        for (int t = 0; t < c.n_taps; ++t) g.taps[t] = all.taps[c.tap0 + t];
        g.beside = beside;
        return g;
    };
    cudaStream_t user = twn_cu(stream);
    if (n_cls <= 1) return n_cls == 0 ? TWN_OK : launch_conv(one_class(cls[0], 1), dZ, T_bwd, stats, epi, dX, TWN_F32, dev_status, user);
    twn_device_info dev;
    rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    if (n_cls <= kMaxClasses && encode_fn()) {
        // all classes in one launch
        if ((long long)all.Bv * all.OH * all.OW * all.ldy >= 0xFFFFFFFFLL) return TWN_ERR_INVALID_ARG;
        Geometry g = all;
        g.Hv = cls[0].Hv; g.Wv = cls[0].Wv;
        g.n_classes = n_cls;
        for (int c = 0; c < n_cls; ++c) g.cls[c] = cls[c];
        // (the longest reductions first in the general kernel, whose blocks walk the tiles in turn; the split kernel, a block for
        // each, is 1 to 2 % slower so)
        Geometry by_length = g;
        std::stable_sort(by_length.cls, by_length.cls + n_cls, [](const TapClass &a, const TapClass &b) { return a.n_taps > b.n_taps; });
        // Apart, the launches follow one another as far as each fills the SMs, and overlap at their ends: the sum of what the
        // kernels that they would run should take, less 1.2 us for each after the first.  Measured both ways on 180 shapes (1 to
        // 256 images of 7 to 112 pixels, 32 to 768 channels, 1x1 to 5x5), half of them not used in the fit, the way it takes is
        // 1.4 % behind the better one on average; at most 23 %, where classes of a few blocks each run side by side after all.
        // 64 images of 56x56x64 <- 128 take 30 us apart and 44 in one launch, 20 images 24 and 21, 5 of 76x76x640 <- 32 30 and 42,
        // 8 of 31x31x512 <- 192 (5x5) 30 and 19.
        const EpilogueArgs ea = epilogue_args(stats, epi, TWN_F32);
        const SplitPlan plan = plan_conv_split(g, dev.sm_count, ea.in_order);
        constexpr double kLeast = 2.8;           // no model goes below: a sum that has passed a limit stays above it (saves 2 us of host time)
        // In the general kernel, whose blocks walk tiles of all classes: 50x28x28x192 <- 384 takes 22.1 us so, 28.0 split and 35 apart,
        // 20 images of 56x56x64 <- 128 12.7, 17.4 and 24, 15x41x41x448 <- 240 28.8, 34.3 and 37.2.  It has to be modelled 5 % below
        // the split kernel and 10 % below launches apart (35 % where a class has no taps: those take less than their models say).  Of
        // 97 shapes measured all three ways the choice was 2.4 % behind the best on average, 6.3 % without this way, with a sum that ended
        // at the split kernel's time and left 4 % of all layers, most of them 1x1, split against this rule: of 34 such shapes 32 are
        // as fast or faster here, two 1.1 and 1.6 % slower, 12 % faster on average (22x32x32x544 <- 544 15.3 us, 19.8 split, 20.9 apart;
        // 105x12x12x368 <- 112, 3x3, 13.2, 18.7 and 27.1).
        double together = 0.0;
        rc = launch_conv(by_length, dZ, T_bwd, stats, epi, dX, TWN_F32, dev_status, user, &together);
        if (rc != TWN_OK) return rc;
        const double less = by_length.cls[n_cls - 1].n_taps == 0 ? 0.65 : 0.9;
        // The sum ends where it answers the only question left: whether the general kernel is far enough below launches apart, where
        // it is below the split kernel, else whether the split kernel is below them.
        const bool below_split = together < 0.95 * plan.us;
        const double enough = below_split ? together / less : plan.us;
        double apart = kLeast * n_cls - 1.2 * (n_cls - 1);
        for (int c = 0; c < n_cls && apart <= enough; ++c) {
            double us = 0.0;
            rc = launch_conv(one_class(cls[c], n_cls), dZ, T_bwd, stats, epi, dX, TWN_F32, dev_status, user, &us);
            if (rc != TWN_OK) return rc;
            apart += us - kLeast;
        }
        if (below_split && apart > enough) return launch_conv(by_length, dZ, T_bwd, stats, epi, dX, TWN_F32, dev_status, user);
        if (plan.pix && plan.us < apart)
            return launch_conv_split(g, dZ, T_bwd, ea, dX, dev_status, dev, user, plan);
    }
    // A launch per class, side by side on helper streams.
    std::unique_lock<std::mutex> lock(g_fork_mutex);
    ForkPool *pool = fork_pool(dev.ordinal);
    if (pool) {
        TWN_CUDA_OK(cudaEventRecord(pool->fork, user));
        for (int i = 0; i < 3; ++i) TWN_CUDA_OK(cudaStreamWaitEvent(pool->side[i], pool->fork, 0));
    }
    int first_error = TWN_OK;
    for (int c = 0; c < n_cls; ++c) {
        cudaStream_t s = (pool && c % 4 != 0) ? pool->side[c % 4 - 1] : user;
        rc = launch_conv(one_class(cls[c], pool ? std::min(n_cls, 4) : 1), dZ, T_bwd, stats, epi, dX, TWN_F32, dev_status, s);
        if (rc != TWN_OK && first_error == TWN_OK) first_error = rc;
    }
    if (pool) {
        // always rejoin, also after a failed launch: the caller's stream must not be left forked
        for (int i = 0; i < 3; ++i) {
            TWN_CUDA_OK(cudaEventRecord(pool->join[i], pool->side[i]));
            TWN_CUDA_OK(cudaStreamWaitEvent(user, pool->join[i], 0));
        }
    }
    return first_error;
}

}  // namespace

extern "C" int twn_conv2d_bwd_data(const twn_conv_desc_t *d, const void *dZ, const uint32_t *T_bwd, int64_t ld_codes,
                                   const twn_stats_t *stats, const twn_epilogue_t *epi, void *dX,
                                   int32_t *dev_status, twn_stream_t stream)
{
    return conv_bwd_data_impl(d, dZ, T_bwd, ld_codes, stats, epi, dX, dev_status, stream, 2);
}

extern "C" int twn_conv2d_bwd_data_b1(const twn_conv_desc_t *d, const void *dZ, const uint32_t *B_bwd, int64_t ld_codes,
                                      const twn_stats_t *stats, const twn_epilogue_t *epi, void *dX,
                                      int32_t *dev_status, twn_stream_t stream)
{
    return conv_bwd_data_impl(d, dZ, B_bwd, ld_codes, stats, epi, dX, dev_status, stream, 1);
}

