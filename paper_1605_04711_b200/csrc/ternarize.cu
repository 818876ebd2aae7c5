// Threshold ternarization fused with 2-bit packing (Sec. 2.3: Eq. 3, Eq. 5 and the
// threshold rule; Algorithm 1, first loop), the parameter update, plus the standalone pack / unpack /
// re-layout kernels.
//
// Ternarization is two phases, bound by HBM bandwidth:
//   phase 1  S = sum |W_i| in fp64  ->  delta = factor * S / n
//   phase 2  codes by Eq. 3, packed 16 per word; sum and count of the kept set
//            ->  alpha (Eq. 5)
// one launch each and one for the last fold, or, for small tensors, one launch of a cluster with its barrier in between; for
// tensors much larger than L2 one phase against an estimate of the threshold, with corrections (ternarize_once_kernel).
// Phase 2 walks every block's share back to front, so that what phase 1 read last comes from L1 and L2.
//
// All sums have a fixed order that depends on the shape of the tensor alone: a tensor is cut into at most
// kMaxParts parts, every part is summed by one block in a fixed way (per-thread strided sums, shuffle tree per
// warp, warps in order) and the parts are folded in a fixed way.  Which block takes a part does not matter, so a
// tensor gets the same bits alone and in a batch.  The kept sum of a tensor that is read once has an order of its own, but no
// rounding in it (read_once), so alpha is the same bits whichever call wrote it.  No floating-point atomics.
#include <algorithm>

#include "sweep.cuh"

namespace {

constexpr int kThreads = 256;       // pack, unpack
constexpr int kWarps = kThreads / 32;
constexpr int kTrThreads = 128;     // re-layouts
// A tensor of up to 8192 words (131072 weights) is "small": at most eight parts of up to 8 x 128 words, so that
// one cluster of eight blocks holds it in registers, eight quarter-words per thread.
constexpr int kSmallQuarters = 8, kQuarterWords = kSweepThreads / 4;
constexpr unsigned long long kSmallWords = kSmallParts * kSmallQuarters * kQuarterWords;
// workspace: [0,256) counters, then arrays of 8-byte partials
constexpr size_t kWorkspaceBytes = 65792;
static_assert(256 + 3 * kMaxParts * 8 <= kWorkspaceBytes, "the partial sums fit in the workspace");
constexpr int kMaxBatch = 32;

struct Workspace {
    unsigned int *done;             // parts whose second sums are written
    double *part_sum;
    double *part_kept;
    unsigned long long *part_cnt;   // negatives in the high half, positives in the low half
};

__host__ __device__ inline Workspace carve(void *ws, int t)
{
    char *b = static_cast<char *>(ws) + (size_t)t * kWorkspaceBytes;
    Workspace w;
    w.done = reinterpret_cast<unsigned int *>(b);
    w.part_sum = reinterpret_cast<double *>(b + 256);
    w.part_kept = w.part_sum + kMaxParts;
    w.part_cnt = reinterpret_cast<unsigned long long *>(w.part_kept + kMaxParts);
    return w;
}

// ---- the codes --------------------------------------------------------------
// inverse: word -> bytes B0..B3
__device__ __forceinline__ uint32_t word_to_bytes(uint32_t w)
{
    uint32_t lo = w & 0xFFFFu, hi = w >> 16;
    lo = (lo | (lo << 8)) & 0x00FF00FFu;
    lo = (lo | (lo << 4)) & 0x0F0F0F0Fu;
    hi = (hi | (hi << 8)) & 0x00FF00FFu;
    hi = (hi | (hi << 4)) & 0x0F0F0F0Fu;
    return __byte_perm(lo | (hi << 4), 0u, 0x0123);
}

// ---- parts ------------------------------------------------------------------
// A part is a run of consecutive packed words that hold codes (the padding words of a row belong to none); the
// weights of consecutive words follow one another in memory, so a part is a contiguous range of weights as well,
// whatever the row length.
struct Item {
    const float *W;
    twn_stats_t *stats;
    uint32_t *packed;
    int8_t *codes_i8;
    unsigned long long n, words;     // weights; words that hold codes
    long long rows, cols, wpr;
    unsigned int wpr_used;           // words of a row that hold codes
    unsigned int wpr_magic;          // floor(2^32 / wpr_used) + 1, 0 for one word per row
    unsigned int last_valid;         // weights of a row's last word; every other word holds 16
    unsigned int parts, part_words;
    unsigned int first_part;         // of this tensor, among the parts of the launch
    unsigned int first_pass;         // weights of a part that phase 1 reads without keeping them in L2
    bool small;
    bool vec4;                       // every word starts on a 16-byte boundary
    bool dense;                      // word w of the packed matrix holds weights 16 w ..
    bool linear;                     // word w of those that hold codes does: no row ends inside a word
};

template <int N>
struct Launch {
    int count;
    unsigned int parts;              // of all tensors
    double factor;
    Item item[N];
};

struct PartRange {
    unsigned long long w0, f0;       // first word, first weight
    unsigned long long out0;         // packed word of the first word's row
    unsigned int j0, words, len;     // the first word's position in its row; words, weights
};

__device__ __forceinline__ void row_of(const Item &it, unsigned long long w, unsigned long long &row, unsigned int &j)
{
    if (w >> 32) { row = w / it.wpr_used; j = (unsigned int)(w - row * it.wpr_used); }
    else { row = (unsigned int)w / it.wpr_used; j = (unsigned int)w - (unsigned int)row * it.wpr_used; }
}

__device__ __forceinline__ PartRange part_range(const Item &it, unsigned int part)
{
    PartRange r;
    r.w0 = (unsigned long long)part * it.part_words;
    const unsigned long long left = it.words > r.w0 ? it.words - r.w0 : 0;
    r.words = left < it.part_words ? (unsigned int)left : it.part_words;
    r.out0 = 0; r.j0 = 0; r.f0 = 0; r.len = 0;
    if (r.words == 0) return r;
    if (it.dense) {
        r.f0 = 16 * r.w0;
        r.len = (unsigned int)min(16ull * r.words, it.n - r.f0);
        return r;
    }
    unsigned long long row, row1;
    unsigned int j1;
    row_of(it, r.w0, row, r.j0);
    row_of(it, r.w0 + r.words, row1, j1);
    r.out0 = row * (unsigned long long)it.wpr;
    r.f0 = row * (unsigned long long)it.cols + 16ull * r.j0;
    const unsigned long long f1 = row1 * (unsigned long long)it.cols + 16ull * j1;
    r.len = (unsigned int)((f1 < it.n ? f1 : it.n) - r.f0);
    return r;
}

// Word `wl` of a part: its index in the packed matrix, its first weight (counted from the part's) and how many
// weights it holds.
struct Place {
    unsigned long long out;
    unsigned int f, valid;
};
__device__ __forceinline__ Place place_word(const Item &it, const PartRange &r, unsigned int wl)
{
    Place p;
    if (it.dense) {
        p.out = r.w0 + wl;
        p.f = 16 * wl;
        p.valid = min(16u, r.len - p.f);
    } else {
        const unsigned int jj = r.j0 + wl;
        // jj / wpr_used: the multiplication is at most one too high
        unsigned int ro = it.wpr_magic ? __umulhi(jj, it.wpr_magic) : jj;
        if (ro * it.wpr_used > jj) --ro;
        const unsigned int j = jj - ro * it.wpr_used;
        p.out = r.out0 + (unsigned long long)ro * (unsigned long long)it.wpr + j;
        // the low halves do: the difference is inside the part, which holds fewer than 2^32 weights
        p.f = ro * (unsigned int)it.cols + 16 * j - 16 * r.j0;
        p.valid = j + 1 == it.wpr_used ? it.last_valid : 16u;
    }
    return p;
}

// Quarter `q` (four weights) of a part, zeros where there is no weight.
__device__ __forceinline__ float4 load_quarter(const Item &it, const PartRange &r, unsigned int q)
{
    float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const unsigned int wl = q >> 2, e = 4 * (q & 3);
    if (wl < r.words) {
        const Place p = place_word(it, r, wl);
        if (p.valid > e) {
            const unsigned int left = p.valid - e;
            const float *w = it.W + r.f0 + (p.f + e);
            if (it.vec4 && left >= 4) {
                v = __ldg(reinterpret_cast<const float4 *>(w));
            } else {
                v.x = __ldg(w);
                if (left > 1) v.y = __ldg(w + 1);
                if (left > 2) v.z = __ldg(w + 2);
                if (left > 3) v.w = __ldg(w + 3);
            }
        }
    }
    return v;
}

// A 16-byte load of weights that need not stay in L2.
__device__ __forceinline__ float4 ld_stream(const float4 *p, unsigned long long policy)
{
    float4 v;
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p), "l"(policy));
    return v;
}
__device__ __forceinline__ unsigned long long evict_first_policy()
{
    unsigned long long p;
    asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}

// The four quarters that a thread has in a group of 512 words.  All loads of a thread are issued before any is used
// and none sits behind a branch of its own (with load_quarter's branches 96 million weights in rows of 8001 took
// 208 us, half of it waiting for one load at a time).  Rows that start off the 16-byte boundaries are read by two
// aligned vectors and shifted.
__device__ __forceinline__ void load_group(const Item &it, const PartRange &r, unsigned int w_grp, float4 (&v)[4])
{
    const unsigned int tid = threadIdx.x;
    const float *W = it.W + r.f0;
    if (it.dense && w_grp + 512 <= r.words && (w_grp + 512ull) * 16 <= r.len) {
        const float4 *v4 = reinterpret_cast<const float4 *>(W) + (size_t)w_grp * 4 + tid;
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = it.first_pass ? ld_stream(v4 + k * kSweepThreads, evict_first_policy()) : __ldg(v4 + k * kSweepThreads);
        return;
    }
    // what the branch-free paths may read: up to the end of the group's last word, and seven weights more
    const Place last = place_word(it, r, min(w_grp + 511, r.words - 1));
    if (r.f0 + last.f + 24 > it.n || it.dense) {
#pragma unroll 1
        for (int k = 0; k < 4; ++k) {
            const float4 x = load_quarter(it, r, w_grp * 4 + k * kSweepThreads + tid);
            if (k == 0) v[0] = x; else if (k == 1) v[1] = x; else if (k == 2) v[2] = x; else v[3] = x;
        }
        return;
    }
    unsigned int f[4], left[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const unsigned int q = w_grp * 4 + k * kSweepThreads + tid, wl = q >> 2, e = 4 * (q & 3);
        const Place p = place_word(it, r, min(wl, r.words - 1));
        left[k] = wl < r.words && p.valid > e ? p.valid - e : 0;
        f[k] = left[k] ? p.f + e : p.f;
    }
    if (it.vec4) {
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = __ldg(reinterpret_cast<const float4 *>(W + f[k]));
    } else {
        float4 a[4], b[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 *w4 = reinterpret_cast<const float4 *>(W + f[k] - ((r.f0 + f[k]) & 3));
            a[k] = __ldg(w4);
            b[k] = __ldg(w4 + 1);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const unsigned int mis = (unsigned int)(r.f0 + f[k]);
            const bool one = mis & 1, two = mis & 2;
            const float s0 = one ? a[k].y : a[k].x, s1 = one ? a[k].z : a[k].y, s2 = one ? a[k].w : a[k].z,
                        s3 = one ? b[k].x : a[k].w, s4 = one ? b[k].y : b[k].x, s5 = one ? b[k].z : b[k].y;
            v[k] = make_float4(two ? s2 : s0, two ? s3 : s1, two ? s4 : s2, two ? s5 : s3);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (left[k] < 1) v[k].x = 0.0f;
        if (left[k] < 2) v[k].y = 0.0f;
        if (left[k] < 3) v[k].z = 0.0f;
        if (left[k] < 4) v[k].w = 0.0f;
    }
}

struct AbsSum {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    __device__ __forceinline__ void add(const float4 v)
    {
        a0 += (double)fabsf(v.x); a1 += (double)fabsf(v.y); a2 += (double)fabsf(v.z); a3 += (double)fabsf(v.w);
    }
    __device__ __forceinline__ double total() const { return (a0 + a1) + (a2 + a3); }
};

// The kept weights of a part: per-thread sums and counts, and the codes of one group of 512 words.  A thread codes
// quarter-word q = k * 512 + tid of the group for k = 0..3, so a warp covers 512 consecutive bytes of weights at a
// time; each byte of `bytes` is one quarter.
struct Coder {
    double k[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned int pos = 0, neg = 0;
    __device__ __forceinline__ double kept() const { return (k[0] + k[1]) + (k[2] + k[3]); }
    __device__ __forceinline__ void group(const Item &it, const PartRange &r, unsigned int w_grp, const float4 (&v)[4], float thr)
    {
        const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
        const uint32_t bytes = code_quarters(v, thr, k, pos, neg);
        if (it.codes_i8) {
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
                const unsigned int q = i * kSweepThreads + tid, wl = w_grp + (q >> 2), e = 4 * (q & 3);
                if (wl >= r.words) continue;
                const Place p = place_word(it, r, wl);
                const uint32_t c4 = fields_to_i8x4((bytes >> (8 * i)) & 0xFFu);
                for (unsigned int x = 0; x < 4 && e + x < p.valid; ++x) it.codes_i8[r.f0 + p.f + e + x] = (int8_t)(c4 >> (8 * x));
            }
        }
        const uint32_t word = exchange_quarters(bytes);
        const unsigned int wl = w_grp + (lane & 3) * kQuarterWords + warp * 8 + (lane >> 2);
        if (wl < r.words) it.packed[it.dense ? r.w0 + wl : place_word(it, r, wl).out] = word;
    }
};

__device__ __forceinline__ double threshold(const Item &it, double s, double factor)
{
    return it.n > 0 ? factor * (s / (double)it.n) : 0.0;
}
__device__ __forceinline__ void write_threshold(const Item &it, double s, double delta)
{
    it.stats->sum_abs = s;
    it.stats->delta = delta;
    it.stats->status = isfinite(s) ? TWN_OK : TWN_ERR_NONFINITE;
    it.stats->reserved = 0;
}
__device__ __forceinline__ void write_kept(const Item &it, double kept, unsigned long long pos, unsigned long long neg)
{
    const unsigned long long n_kept = pos + neg;
    it.stats->sum_abs_kept = kept;
    it.stats->alpha = n_kept > 0 ? kept / (double)n_kept : 0.0;
    it.stats->n_pos = pos;
    it.stats->n_neg = neg;
    it.stats->n_zero = it.n - n_kept;
}

// The codes of a part against a threshold, back to front: what was read last comes from L2.  (A thread per word, as in
// ternarize_once_kernel, needs no exchange among lanes but more registers than two blocks leave: 8.4 million weights 12.6 us
// instead of 12.1, 28.7 million 40.8 instead of 38.3.)
__device__ __forceinline__ Coder code_part(const Item &it, const PartRange &r, float thr)
{
    Coder c;
    for (unsigned int grp = (r.words + 511) >> 9; grp-- > 0;) {
        float4 v[4];
        load_group(it, r, grp << 9, v);
        c.group(it, r, grp << 9, v, thr);
    }
    return c;
}

// padding words of the rows
__device__ __forceinline__ void write_padding(const Item &it, unsigned int b, unsigned int G)
{
    const unsigned int pad = (unsigned int)(it.wpr - it.wpr_used);
    if (pad == 0 || !it.packed) return;
    const unsigned long long total = (unsigned long long)it.rows * pad;
    for (unsigned long long i = (unsigned long long)b * kSweepThreads + threadIdx.x; i < total; i += (unsigned long long)G * kSweepThreads) {
        const unsigned long long r = i >> 32 ? i / pad : (unsigned int)i / pad;
        it.packed[r * it.wpr + it.wpr_used + (i - r * pad)] = 0u;
    }
}

// ---- small tensors: one cluster -------------------------------------------------
// Latency is all there is (50 thousand weights: 14.3 us as two sweeps over memory with a cleared ticket, 12 of them
// waiting for memory and launches).  A block keeps its part in registers between the phases, the sums travel through
// distributed shared memory, and the cluster's barrier (0.2 us) stands where larger tensors need the grid's.
template <int Q, bool SUMS>      // quarter-words per thread; false: the coding sweep alone
__global__ void __launch_bounds__(kSweepThreads, 1)
ternarize_small_kernel(const __grid_constant__ Launch<1> P)
{
    __shared__ Reduce red;
    __shared__ double sum_s[kSmallParts], kept_s[kSmallParts];
    __shared__ unsigned long long cnt_s[kSmallParts];
    const Item &it = P.item[0];
    const unsigned int b = blockIdx.x, G = gridDim.x, tid = threadIdx.x;
    unsigned int turn = 0;
    if (tid < kSmallParts) { sum_s[tid] = 0.0; kept_s[tid] = 0.0; cnt_s[tid] = 0ull; }
    pdl_begin();
    cluster_arrive();                    // from here on other blocks may write this block's sums
    PartRange r = part_range(it, b);
    float4 v[Q < 4 ? 4 : Q];
#pragma unroll
    for (int k = 0; k < (Q < 4 ? 4 : Q); ++k)
        v[k] = k < Q ? load_quarter(it, r, k * kSweepThreads + tid) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    write_padding(it, b, G);
    double delta;
    if (SUMS) {
        AbsSum a;
#pragma unroll
        for (int k = 0; k < Q; ++k) a.add(v[k]);
        const double part = sweep_sum(a.total(), red, turn);
        cluster_wait();
        if (tid < G) st_peer(peer_smem(&sum_s[b], tid), __double_as_longlong(part));
        cluster_arrive();
        cluster_wait();
        const double s = tree8(sum_s);
        delta = threshold(it, s, P.factor);
        if (b == 0 && tid == 0) write_threshold(it, s, delta);
    } else {
        cluster_wait();
        delta = __ldcg(&it.stats->delta);
    }
    // delta rounded toward -inf: for any float w,  w > delta  <=>  w > thr
    const float thr = __double2float_rd(delta);
    Coder c;
#pragma unroll
    for (int g = (Q + 3) / 4; g-- > 0;) {
        const float4 four[4] = {v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]};
        c.group(it, r, g * 512, four, thr);
    }
    const double kept = sweep_sum(c.kept(), c.pos, c.neg, red, turn);
    if (tid == 0) {
        st_peer(peer_smem(&kept_s[b], 0), __double_as_longlong(kept));
        st_peer(peer_smem(&cnt_s[b], 0), ((unsigned long long)c.neg << 32) + c.pos);
    }
    cluster_arrive();
    cluster_wait();
    if (b == 0 && tid == 0) {
        unsigned long long pos = 0, neg = 0;
#pragma unroll
        for (int i = 0; i < kSmallParts; ++i) { pos += cnt_s[i] & 0xFFFFFFFFull; neg += cnt_s[i] >> 32; }
        write_kept(it, tree8(kept_s), pos, neg);
    }
}

// ---- any tensor: a launch per phase ---------------------------------------------
// The tensor of part g, from the one of an earlier part (up) or of a later part (down) on.
template <int N> __device__ __forceinline__ int item_up(const Launch<N> &P, unsigned int g, int t)
{
    if (N > 1)
        while (t + 1 < P.count && g >= P.item[t + 1].first_part) ++t;
    return t;
}
template <int N> __device__ __forceinline__ int item_down(const Launch<N> &P, unsigned int g, int t)
{
    if (N > 1)
        while (g < P.item[t].first_part) --t;
    return t;
}

// sum |W| over the weights of a part: whole 16-byte vectors from the boundary below its first weight on, and by
// plain loads the weights before the first and after the last whole vector (small tensors: by quarter-words, as the
// kernel above adds them).
__device__ __forceinline__ double part_abs_sum(const Item &it, const PartRange &r)
{
    AbsSum a;
    if (it.small) {
#pragma unroll 1
        for (unsigned int q = threadIdx.x; q < 4 * r.words; q += kSweepThreads) a.add(load_quarter(it, r, q));
        return a.total();
    }
    const unsigned int head = (unsigned int)(r.f0 & 3ull);
    const float4 *v4 = reinterpret_cast<const float4 *>(it.W + (r.f0 - head));
    const unsigned long long end = (unsigned long long)head + r.len;
    const unsigned long long first = head ? 1 : 0, last = end >> 2;     // vectors [first, last) lie inside the part
    unsigned long long i = first + threadIdx.x;
    // a tensor larger than L2: what phase 2 reads last is not kept, so that what it reads first still is
    const unsigned long long pol = evict_first_policy();
    for (const unsigned long long end1 = min((unsigned long long)(it.first_pass >> 2), last); i + 3 * kSweepThreads < end1; i += 4 * kSweepThreads) {
        const float4 v0 = ld_stream(v4 + i, pol), v1 = ld_stream(v4 + i + kSweepThreads, pol),
                     v2 = ld_stream(v4 + i + 2 * kSweepThreads, pol), v3 = ld_stream(v4 + i + 3 * kSweepThreads, pol);
        a.add(v0); a.add(v1); a.add(v2); a.add(v3);
    }
    for (; i + 3 * kSweepThreads < last; i += 4 * kSweepThreads) {
        const float4 v0 = __ldg(v4 + i), v1 = __ldg(v4 + i + kSweepThreads), v2 = __ldg(v4 + i + 2 * kSweepThreads),
                     v3 = __ldg(v4 + i + 3 * kSweepThreads);
        a.add(v0); a.add(v1); a.add(v2); a.add(v3);
    }
    for (; i < last; i += kSweepThreads) a.add(__ldg(v4 + i));
    if (threadIdx.x < 8) {
        const unsigned int x = threadIdx.x & 3;
        const unsigned long long e = threadIdx.x < 4 ? x : 4 * last + x;
        const bool inside = e < end && (threadIdx.x < 4 ? (first && x >= head) : last >= first);
        if (inside) a.a0 += (double)fabsf(__ldg(reinterpret_cast<const float *>(v4) + e));
    }
    return a.total();
}

// Folds `parts` partial sums in a fixed order; the result is valid in every thread.
__device__ __forceinline__ double fold_parts(const double *p, unsigned int parts, Reduce &red, unsigned int &turn)
{
    double s = 0.0;
    for (unsigned int i = threadIdx.x; i < parts; i += kSweepThreads) s += __ldcg(p + i);
    return sweep_sum(s, red, turn);
}

// The last block's part: the second sums of a tensor's parts, in a fixed order.
__device__ __forceinline__ void fold_kept(const Item &it, const Workspace &ws, Reduce &red, unsigned long long (&cnt)[2][kSweepWarps], unsigned int &turn)
{
    double s = 0.0;
    unsigned long long pos = 0, neg = 0;
    for (unsigned int i = threadIdx.x; i < it.parts; i += kSweepThreads) {
        s += __ldcg(ws.part_kept + i);
        const unsigned long long c = __ldcg(ws.part_cnt + i);
        pos += c & 0xFFFFFFFFull;
        neg += c >> 32;
    }
    const double kept = sweep_sum(s, red, turn);
    pos = warp_sum(pos);
    neg = warp_sum(neg);
    if ((threadIdx.x & 31) == 0) { cnt[0][threadIdx.x >> 5] = pos; cnt[1][threadIdx.x >> 5] = neg; }
    __syncthreads();
    if (threadIdx.x == 0) {
        pos = neg = 0;
        for (int w = 0; w < kSweepWarps; ++w) { pos += cnt[0][w]; neg += cnt[1][w]; }
        write_kept(it, kept, pos, neg);
    }
}

// The warps' sums of up to kRun parts of a block.  Nothing joins the warps between the parts, so a warp's loads of its
// next part are not held up by a slower warp's reduction: with a block-wide sum per part, 1400 parts of the 21 tensors of
// ResNet-18 took 50 us.
constexpr int kRun = 32;
struct PartRun {
    double sum[kRun][kSweepWarps];
    uint2 cnt[kRun][kSweepWarps];
};

// The codes of a block's parts b, b + G, ..., back to front, and their sums into the workspace.
template <int N>
__device__ __forceinline__ void code_parts(const Launch<N> &P, void *ws_raw, unsigned int mine, const float *thr_s, PartRun &run)
{
    const unsigned int b = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int ti = P.count - 1;
    for (unsigned int left = mine; left > 0;) {
        const unsigned int n = min(left, (unsigned int)kRun);
        for (unsigned int i = 0; i < n; ++i) {
            const unsigned int g = b + (left - 1 - i) * G;
            ti = item_down(P, g, ti);
            const Item &it = P.item[ti];
            const Coder c = code_part(it, part_range(it, g - it.first_part), thr_s[N == 1 ? 0 : ti]);
            const double kept = warp_sum(c.kept());
            const unsigned int p = __reduce_add_sync(0xffffffffu, c.pos), q = __reduce_add_sync(0xffffffffu, c.neg);
            if (lane == 0) { run.sum[i][warp] = kept; run.cnt[i][warp] = make_uint2(p, q); }
        }
        __syncthreads();
        if (tid < n) {
            const unsigned int g = b + (left - 1 - tid) * G;
            const int t = item_up(P, g, ti);
            const Item &it = P.item[t];
            const Workspace ws = carve(ws_raw, t);
            unsigned int p = 0, q = 0;
#pragma unroll
            for (int w = 0; w < kSweepWarps; ++w) { p += run.cnt[tid][w].x; q += run.cnt[tid][w].y; }
            ws.part_kept[g - it.first_part] = tree16(run.sum[tid]);
            ws.part_cnt[g - it.first_part] = ((unsigned long long)q << 32) + p;
        }
        __syncthreads();
        left -= n;
    }
}

// Sums, codes, and the folds of both are launches of their own, each there when the one before it ends (programmatic launches):
// no block waits for another.  In a cooperative launch with grid-wide barriers a stream of calls came in steps of 2 us: 147
// thousand to 590 thousand weights 10.3 us so, 7.9 to 8.6 in three launches; the coding sweep of 590 thousand 8.3 and 5.2; the 21
// tensors of ResNet-18 39.1 and 35.7, their coding sweeps 28.0 and 20.1.
// N: tensors of the launch (1, or up to kMaxBatch).
template <int N>
__global__ void __launch_bounds__(kSweepThreads, kSweepBlocksPerSm)
sums_kernel(const __grid_constant__ Launch<N> P, void *ws_raw)
{
    __shared__ PartRun run;
    const unsigned int b = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned int mine = b < P.parts ? (P.parts - 1 - b) / G + 1 : 0;     // this block's parts: b, b + G, ...
    chain_wait();
    int ti = 0;
    for (unsigned int i0 = 0; i0 < mine; i0 += kRun) {
        const unsigned int n = min(mine - i0, (unsigned int)kRun);
        for (unsigned int i = 0; i < n; ++i) {
            const unsigned int g = b + (i0 + i) * G;
            ti = item_up(P, g, ti);
            const Item &it = P.item[ti];
            const double v = warp_sum(part_abs_sum(it, part_range(it, g - it.first_part)));
            if (lane == 0) run.sum[i][warp] = v;
        }
        __syncthreads();
        if (tid < n) {
            const unsigned int g = b + (i0 + tid) * G;
            const int t = item_down(P, g, ti);
            carve(ws_raw, t).part_sum[g - P.item[t].first_part] = tree16(run.sum[tid]);
        }
        __syncthreads();
    }
}
// the thresholds of a batch, one block per tensor
template <int N>
__global__ void __launch_bounds__(kSweepThreads)
sums_fold_kernel(const __grid_constant__ Launch<N> P, void *ws_raw)
{
    __shared__ Reduce red;
    unsigned int turn = 0;
    chain_wait();
    const Item &it = P.item[blockIdx.x];
    const double s = fold_parts(carve(ws_raw, (int)blockIdx.x).part_sum, it.parts, red, turn);
    if (threadIdx.x == 0) write_threshold(it, s, threshold(it, s, P.factor));
}

// The coding sweep, against the threshold that is in the stats, or (FOLD, one tensor) that every block folds for itself.
template <int N, bool FOLD>
__global__ void __launch_bounds__(kSweepThreads, kSweepBlocksPerSm)
codes_kernel(const __grid_constant__ Launch<N> P, void *ws_raw)
{
    static_assert(!FOLD || N == 1, "the thresholds of a batch have a launch");
    __shared__ Reduce red;
    __shared__ PartRun run;
    __shared__ float thr_s[N];
    const unsigned int b = blockIdx.x, G = gridDim.x;
    unsigned int turn = 0;
    chain_wait();
    // delta rounded toward -inf: for any float w,  w > delta  <=>  w > thr
    if (FOLD) {
        const double s = fold_parts(carve(ws_raw, 0).part_sum, P.item[0].parts, red, turn);
        const double delta = threshold(P.item[0], s, P.factor);
        if (b == 0 && threadIdx.x == 0) write_threshold(P.item[0], s, delta);
        if (threadIdx.x == 0) thr_s[0] = __double2float_rd(delta);
    } else if (threadIdx.x < (unsigned)P.count) {
        thr_s[threadIdx.x] = __double2float_rd(__ldcg(&P.item[threadIdx.x].stats->delta));
    }
    __syncthreads();
    code_parts(P, ws_raw, b < P.parts ? (P.parts - 1 - b) / G + 1 : 0, thr_s, run);
#pragma unroll 1
    for (int t = 0; t < P.count; ++t) write_padding(P.item[t], b, G);
}
template <int N>
__global__ void __launch_bounds__(kSweepThreads)
codes_fold_kernel(const __grid_constant__ Launch<N> P, void *ws_raw)
{
    __shared__ Reduce red;
    __shared__ unsigned long long red_cnt64[2][kSweepWarps];
    unsigned int turn = 0;
    chain_wait();
    fold_kept(P.item[blockIdx.x], carve(ws_raw, (int)blockIdx.x), red, red_cnt64, turn);
}

// ---- large tensors: one read ------------------------------------------------------
// A tensor that does not stay in L2 would cross HBM twice, because the threshold needs every weight before the first code.
// Here it crosses once: a sample (16 runs of 512 weights from every part) gives an estimate `mid` of the threshold and how far
// off it may be, the one sweep adds up |W|, codes against `mid` and marks the half-words with a weight within `half` of it; when
// the threshold is known, the weights of marked half-words that lie between it and `mid` get their other code, and sums and
// counts are put right.  Of normal weights 1.4 % of the half-words are marked; most are kept in shared memory, the others read
// again.  A threshold further than `half` from the estimate (an order of weights that the sample does not see, a NaN) costs a
// second sweep.  Codes, counts and kept sum are the same bits in any case: the kernel is not taken where the kept sum could be
// rounded (read_once).
// The sweep costs nearly as many issue slots as memory time, so a thread takes whole words (no exchange among lanes), their
// kept bits are collected by the fp32 adders (as sums of powers of two) and their signs two at a time.
//   12288 x 8192 (three tensors in turn) 137.7 -> 88.3 us, 66 at the copy rate.
// Where one read pays: 9.2 million weights in rows of 2301, cold, 28.9 us so, 27.0 in two sweeps; 14.2 million 24.9 / 26.7; 18.9 million 28.9 / 33.0
// (27.3 / 26.9 where they are in L2 from the call before); 33.6 million 39.1 / 51.5; rows of 8001 weights 145 / 192.
// Where it loses: a threshold outside the window (sorted weights, large ones that no run of the sample sees) 151 to 154 us against
// 136 in two sweeps, 33.6 million weights 60 / 49; every weight at the threshold 156 / 136.  Normal, Laplace, uniform, sparse
// weights, rows of different scale, outliers 84 to 92, Cauchy 99.
constexpr unsigned long long kOnceWeights = 16ull << 20;
constexpr unsigned int kOnceGroups = 128;        // groups of 512 words in a part (310 million weights in all; see read_once, too)
constexpr unsigned int kOnceKept = 64;           // marked half-words that a warp keeps beside their marks
constexpr unsigned int kOnceDense = 20;          // of a warp's 64 half-words in a group, marked ones from which its part is swept again
constexpr int kSampleRun = 512;                  // weights of a warp's sample

// In shared memory: the weights of each warp's first marks; of warp w in group g, for each half of a thread's word, the lanes
// with a weight near `mid`; how many of the warp's marks come before those.
struct Once {
    float4 (*kept)[kOnceKept][2];
    uint2 *mark;
    unsigned int *before;
};
__host__ __device__ constexpr unsigned int once_smem(unsigned int groups)
{
    return kSweepWarps * (kOnceKept * 2 * (unsigned int)sizeof(float4) + groups * (unsigned int)(sizeof(uint2) + 4));
}

__device__ __forceinline__ void ld_eight(float (&v)[8], const float *p, bool wide, unsigned long long policy)
{
    if (wide) {
        asm("ld.global.nc.L2::cache_hint.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8], %9;"
            : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "l"(p), "l"(policy));
    } else {
        const float4 x = ld_stream(reinterpret_cast<const float4 *>(p), policy), y = ld_stream(reinterpret_cast<const float4 *>(p) + 1, policy);
        v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
        v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
    }
}
// Half `h` of word `wl` of a part, zeros where there is no weight: aligned vectors, shifted into place.
__device__ __forceinline__ void load_eight(const Item &it, const PartRange &r, unsigned int wl, int h, float (&v)[8])
{
#pragma unroll
    for (int x = 0; x < 8; ++x) v[x] = 0.0f;
    if (wl >= r.words) return;
    const Place p = place_word(it, r, wl);
    const unsigned int left = p.valid > 8u * h ? p.valid - 8u * h : 0;
    if (left == 0) return;
    const unsigned long long at = r.f0 + p.f + 8 * h;
    if (at + 12 > it.n) {
        for (int x = 0; x < 8; ++x)
            if ((unsigned)x < left) v[x] = __ldg(it.W + at + x);
        return;
    }
    const float4 *p4 = reinterpret_cast<const float4 *>(it.W + (at & ~3ull));
    const unsigned int mis = (unsigned int)at & 3;
    const float4 q0 = __ldg(p4), q1 = __ldg(p4 + 1), q2 = __ldg(p4 + 2);
    const float s[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
    const bool one = mis & 1, two = mis & 2;
    float t[10];
#pragma unroll
    for (int x = 0; x < 10; ++x) t[x] = one ? s[x + 1] : s[x];
#pragma unroll
    for (int x = 0; x < 8; ++x) v[x] = (unsigned)x < left ? (two ? t[x + 2] : t[x]) : 0.0f;
}

// The codes of a word: bit 0 of the kept weights' fields, and the signs in the place of bit 1.
struct Word {
    float even = 8388608.0f, odd = 8388608.0f;       // 2^23 plus a sum of distinct powers of two below 2^15: exact
    uint32_t signs = 0;
    __device__ __forceinline__ uint32_t kept() const { return __byte_perm(__float_as_uint(even), __float_as_uint(odd), 0x5410) & 0x7FFF7FFFu; }
};

// Half `h` of a word: the sums, the codes against `mid`; whether a weight lies within `half` of `mid`.
__device__ __forceinline__ bool sweep_eight(const float (&v)[8], int h, float mid, float half, double (&a)[2], double (&k)[2], Word &w)
{
    float near[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const float m = fabsf(v[x]);
        const double d = (double)m;
        a[x & 1] += d;
        if (m > mid) {
            k[x & 1] += d;
            (x & 1 ? w.odd : w.even) += (float)(1 << (14 - 8 * h - (x & ~1)));
        }
        near[x] = fabsf(__fsub_rn(m, mid));
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int down = 2 * (4 * h + j);
        w.signs |= (__byte_perm(__float_as_uint(v[2 * j]), __float_as_uint(v[2 * j + 1]), 0x7632) >> down) & (0x80008000u >> down);
    }
    auto min3 = [](float x, float y, float z) {
        float r;
        asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(x), "f"(y), "f"(z));
        return r;
    };
    return min3(min3(near[0], near[1], near[2]), min3(near[3], near[4], near[5]), fminf(near[6], near[7])) <= half;
}

// A word's codes to memory, and its counts.
__device__ __forceinline__ void finish_word(const Item &it, const PartRange &r, unsigned int wl, const Word &w, unsigned int &pos, unsigned int &neg)
{
    const uint32_t kept = w.kept(), minus = w.signs & (kept << 1);
    const unsigned int n_neg = __popc(minus);
    neg += n_neg;
    pos += __popc(kept) - n_neg;
    if (wl >= r.words) return;
    if (it.dense && !it.codes_i8) {
        it.packed[r.w0 + wl] = kept | minus;
        return;
    }
    const Place p = place_word(it, r, wl);
    it.packed[p.out] = kept | minus;
    if (it.codes_i8)
#pragma unroll 1
        for (unsigned int e = 0; e < p.valid; ++e) {
            const uint32_t f = ((kept | minus) >> field_pos((int)e)) & 3u;
            it.codes_i8[r.f0 + p.f + e] = (int8_t)(f == 0 ? 0 : f == 1 ? 1 : -1);
        }
}

// A marked half-word coded against `mid`, now that the threshold is known.
__device__ __forceinline__ void correct(const Item &it, const PartRange &r, unsigned int wl, int h, const float (&v)[8], float mid, float thr,
                                        double &kept, unsigned int &pos, unsigned int &neg)
{
    uint32_t flip = 0;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
        const float mag = fabsf(v[x]);
        const bool now = mag > thr, minus = v[x] < 0.0f;
        if (now == (mag > mid)) continue;
        kept += now ? (double)mag : -(double)mag;
        const unsigned int one = now ? 1u : 0xFFFFFFFFu;
        if (minus) neg += one; else pos += one;
        flip |= (minus ? 3u : 1u) << field_pos(x);
    }
    if (!flip) return;
    const Place p = place_word(it, r, wl);
    atomicXor(it.packed + p.out, flip >> (8 * h));   // field_pos(8 + x) = field_pos(x) - 8; nobody waits for the word
    if (it.codes_i8)
        for (int x = 0; x < 8; ++x)
            if ((flip >> field_pos(x)) & 1u) it.codes_i8[r.f0 + p.f + 8 * h + x] = fabsf(v[x]) > thr ? (v[x] < 0.0f ? -1 : 1) : 0;
}

// sum |W| over a warp's run of the sample, 0 where the part is too short for one
__device__ __forceinline__ float sample_run(const Item &it, const PartRange &r)
{
    const unsigned int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (r.len < 2 * kSampleRun) return 0.0f;
    // the run starts on a 16-byte boundary of the tensor
    const unsigned long long at = (r.f0 + (unsigned long long)(r.len - kSampleRun - 4) * (2 * warp + 1) / (2 * kSweepWarps) + 3) & ~3ull;
    const float4 *p = reinterpret_cast<const float4 *>(it.W + at) + lane;
    float4 v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __ldg(p + 32 * k);
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) s += (fabsf(v[k].x) + fabsf(v[k].y)) + (fabsf(v[k].z) + fabsf(v[k].w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__global__ void __launch_bounds__(kSweepThreads, kSweepBlocksPerSm)
ternarize_once_kernel(const __grid_constant__ Launch<1> P, void *ws_raw)
{
    __shared__ Reduce red;
    __shared__ unsigned long long red_cnt64[2][kSweepWarps];
    __shared__ float run_s[kSweepWarps];
    __shared__ unsigned int last_s;
    extern __shared__ float4 once_raw[];
    const Item &it = P.item[0];
    const Workspace ws = carve(ws_raw, 0);
    const unsigned int b = blockIdx.x, G = gridDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned int turn = 0;
    if (b == 0 && tid == 0) *ws.done = 0u;
    const PartRange r = part_range(it, b);          // a block has one part
    const unsigned int groups = (r.words + 511) >> 9, most = it.part_words >> 9;
    uint2 *const mark0 = reinterpret_cast<uint2 *>(once_raw + kSweepWarps * kOnceKept * 2);
    const Once marks = {reinterpret_cast<float4 (*)[kOnceKept][2]>(once_raw), mark0, reinterpret_cast<unsigned int *>(mark0 + kSweepWarps * most)};


    // ---- the sample: per part its sum and the squared deviations of its runs (in the arrays of the final sums).  Loads of the
    // sweep that are issued before its barrier hold the barrier up by more than they gain (88 -> 94 us, the first 128 KB of every
    // part fetched into L2 88 -> 97).
    {
        const float s = sample_run(it, r);
        if (lane == 0) run_s[warp] = s;
        __syncthreads();
        if (tid == 0) {
            double sum = 0.0, dev = 0.0;
            for (int w = 0; w < kSweepWarps; ++w) sum += (double)run_s[w];
            for (int w = 0; w < kSweepWarps; ++w) {
                const double d = (double)run_s[w] - sum / kSweepWarps;
                dev += d * d;
            }
            ws.part_kept[b] = sum;
            ws.part_cnt[b] = (unsigned long long)__double_as_longlong(dev);
        }
    }
    cooperative_groups::this_grid().sync();
    float mid, half;
    {
        double sum = 0.0, dev = 0.0;
        unsigned int n = 0, unused = 0;
        for (unsigned int i = tid; i < it.parts; i += kSweepThreads) {
            sum += __ldcg(ws.part_kept + i);
            dev += __longlong_as_double((long long)__ldcg(ws.part_cnt + i));
            n += part_range(it, i).len >= 2 * kSampleRun ? kSweepWarps : 0;
        }
        sum = sweep_sum(sum, n, unused, red, turn);
        dev = sweep_sum(dev, red, turn);
        // 4.5 standard errors of a mean of n runs drawn from strata, and what the rounding of the runs' sums may be
        const double mean = sum / ((double)n * kSampleRun), se = sqrt(dev * (kSweepWarps / (kSweepWarps - 1.0))) / ((double)n * kSampleRun);
        mid = (float)(P.factor * mean);
        half = fminf((float)(P.factor * (4.5 * se + 2e-5 * mean)), 3.0e38f);
    }

    // ---- the sweep.  The registers of half a word take the next group's as soon as they are coded: a thread's loads never pause.
    double a[2] = {0.0, 0.0}, k[2] = {0.0, 0.0};
    unsigned int pos = 0, neg = 0;
    float v[2][8];
    {
        const unsigned int whole = it.linear ? r.len >> 13 : 0;        // groups of 512 words of 16 weights, in memory order
        const unsigned long long pol = evict_first_policy();
        const bool wide = (reinterpret_cast<uintptr_t>(it.W) & 31) == 0;
        const float *p = it.W + r.f0 + 16 * tid;
        unsigned int n_marks = 0;                                      // of this warp
        if (whole > 0) {
            ld_eight(v[0], p, wide, pol);
            ld_eight(v[1], p + 8, wide, pol);
        }
#pragma unroll 1
        for (unsigned int g = 0; g < groups; ++g) {
            p += 16 * kSweepThreads;
            if (g >= whole) {
                load_eight(it, r, (g << 9) + tid, 0, v[0]);
                load_eight(it, r, (g << 9) + tid, 1, v[1]);
            }
            Word w;
            unsigned int near[2];
            if (lane == 0) marks.before[g * kSweepWarps + warp] = n_marks;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const bool mine = sweep_eight(v[h], h, mid, half, a, k, w);
                near[h] = __ballot_sync(0xffffffffu, mine);
                if (near[h]) {
                    const unsigned int slot = n_marks + __popc(near[h] & ((1u << lane) - 1));
                    if (mine && slot < kOnceKept) {
                        marks.kept[warp][slot][0] = make_float4(v[h][0], v[h][1], v[h][2], v[h][3]);
                        marks.kept[warp][slot][1] = make_float4(v[h][4], v[h][5], v[h][6], v[h][7]);
                    }
                    n_marks += __popc(near[h]);
                }
                if (g + 1 < whole) ld_eight(v[h], p + 8 * h, wide, pol);
            }
            if (lane == 0) marks.mark[g * kSweepWarps + warp] = make_uint2(near[0], near[1]);
            finish_word(it, r, (g << 9) + tid, w, pos, neg);
        }
    }
    write_padding(it, b, G);
    double kept = k[0] + k[1];
    {
        const double s = sweep_sum(a[0] + a[1], red, turn);
        if (tid == 0) ws.part_sum[b] = s;
    }
    cooperative_groups::this_grid().sync();
    const double s = fold_parts(ws.part_sum, it.parts, red, turn);
    const double delta = threshold(it, s, P.factor);
    if (b == 0 && tid == 0) write_threshold(it, s, delta);
    const float thr = __double2float_rd(delta);

    // This warp's marks, none if the estimate was the threshold; a block with a warp that has too many sweeps its part again.
    // (12288 x 8192 with half of the half-words marked: 181 us by the list of marks, 133 with such blocks swept again; all marked
    // 260 and 156; all weights zero, so marked but none to correct, 246 and 87.  From about 20 of 64 on the second sweep is shorter.)
    unsigned int total = 0;
    if (groups && thr != mid) {
        const unsigned int last = (groups - 1) * kSweepWarps + warp;
        total = marks.before[last] + __popc(marks.mark[last].x) + __popc(marks.mark[last].y);
    }
    const bool dense = __syncthreads_or(total > kOnceDense * groups);
    if (!dense && fabsf(__fsub_rn(thr, mid)) <= half && thr <= 2.0f * mid) {     // (the last: read_once)
        // ---- put right what lies between.  x -> |x - mid| as computed here and in the sweep is monotonic on either side of
        // mid, so a weight between mid and thr is no further from mid than thr is: its half-word is marked.  A warp takes its own
        // marks, a lane every 32nd.
#pragma unroll 1
        for (unsigned int m = lane; m < total; m += 32) {
            unsigned int g = 0;                                        // the last group with no more than m marks before it
            for (unsigned int hi = groups; hi - g > 1;) {
                const unsigned int c = (g + hi) >> 1;
                if (marks.before[c * kSweepWarps + warp] <= m) g = c; else hi = c;
            }
            const uint2 mk = marks.mark[g * kSweepWarps + warp];
            unsigned int skip = m - marks.before[g * kSweepWarps + warp], lanes = mk.x;
            const int h = skip >= __popc(mk.x);
            if (h) { skip -= __popc(mk.x); lanes = mk.y; }
            for (; skip > 0; --skip) lanes &= lanes - 1;
            const unsigned int wl = (g << 9) + warp * 32 + __ffs(lanes) - 1;
            float m8[8];
            if (m < kOnceKept) {
                const float4 x = marks.kept[warp][m][0], y = marks.kept[warp][m][1];
                m8[0] = x.x; m8[1] = x.y; m8[2] = x.z; m8[3] = x.w;
                m8[4] = y.x; m8[5] = y.y; m8[6] = y.z; m8[7] = y.w;
            } else {
                load_eight(it, r, wl, h, m8);
            }
            correct(it, r, wl, h, m8, mid, thr, kept, pos, neg);
        }
    } else {
        const Coder c = code_part(it, r, thr);
        kept = c.kept(); pos = c.pos; neg = c.neg;
    }
    // pos and neg of a thread may be below zero after corrections: their sums over the block are counts again
    kept = sweep_sum(kept, pos, neg, red, turn);
    if (tid == 0) {
        ws.part_kept[b] = kept;
        ws.part_cnt[b] = ((unsigned long long)neg << 32) + pos;
        unsigned int old;
        asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(ws.done) : "memory");
        last_s = old == it.parts - 1;
    }
    __syncthreads();
    if (last_s) fold_kept(it, ws, red, red_cnt64, turn);
}

// ---- parameter update fused with the sums of the next iteration ----------------
// Last step of Algorithm 1 (UpdateParameters: SGD with momentum and L2 weight decay on the fp32
// master weights, Sec. 3):
//     g = dW + wd * W;   V' = mu * V + g;   W' = W - lr * V'
// every operation a separately rounded fp32 operation in this order (no fused multiply-add), so
// the result is defined to the bit.  The next iteration starts by ternarizing W', whose
// threshold needs sum |W'|: it is accumulated here while W' is still in registers, which saves
// the first phase of that ternarization (one read of the weights).
struct SgdItem {
    float *W;
    const float *dW;
    float *V;
    long long n;
    twn_stats_t *stats;
    unsigned int first_block;        // blocks [first_block, first_block of the next item) work on this tensor
};
template <int N>
struct SgdLaunch {
    int count;
    unsigned int blocks;
    float lr, mu, wd;
    double factor;
    SgdItem item[N];
};

__device__ __forceinline__ float sgd_one(float w, float g, float &v, float lr, float mu, float wd)
{
    const float grad = __fadd_rn(g, __fmul_rn(wd, w));
    v = __fadd_rn(__fmul_rn(mu, v), grad);
    return __fsub_rn(w, __fmul_rn(lr, v));
}

__device__ __forceinline__ void sgd_four(float4 &w, const float4 g, float4 &v, float lr, float mu, float wd, double &a0, double &a1)
{
    w.x = sgd_one(w.x, g.x, v.x, lr, mu, wd);
    w.y = sgd_one(w.y, g.y, v.y, lr, mu, wd);
    w.z = sgd_one(w.z, g.z, v.z, lr, mu, wd);
    w.w = sgd_one(w.w, g.w, v.w, lr, mu, wd);
    a0 += (double)fabsf(w.x); a1 += (double)fabsf(w.y); a0 += (double)fabsf(w.z); a1 += (double)fabsf(w.w);
}

__device__ __forceinline__ void write_next(const SgdItem &it, double factor, double s)
{
    it.stats->sum_abs = s;
    it.stats->delta = it.n > 0 ? factor * (s / (double)it.n) : 0.0;
    it.stats->status = isfinite(s) ? TWN_OK : TWN_ERR_NONFINITE;
    it.stats->reserved = 0;
}

// The blocks' sums meet through distributed shared memory where one cluster of at most eight blocks does, else in the
// workspace, where a launch of their own folds them, one block per tensor, that is there when this one ends (in a cooperative
// launch with a barrier 590 thousand weights took 6.2 us, 4.4 now, 8.4 million 32.4 and 30.3).
template <int N, bool CLUSTER>
__global__ void __launch_bounds__(kSweepThreads, kSweepBlocksPerSm)
sgd_update_kernel(const __grid_constant__ SgdLaunch<N> P, void *ws_raw)
{
    static_assert(!CLUSTER || N == 1, "a batch meets grid-wide");
    __shared__ Reduce red;
    __shared__ double sum_s[kSmallParts];
    unsigned int turn = 0;
    double own = 0.0;
    if (CLUSTER) {
        if (threadIdx.x < kSmallParts) sum_s[threadIdx.x] = 0.0;
        pdl_begin();
        cluster_arrive();
    } else {
        chain_wait();
    }
    for (unsigned int g = blockIdx.x; g < P.blocks; g += gridDim.x) {
        int t = 0;
        if (N > 1)
            while (t + 1 < P.count && g >= P.item[t + 1].first_block) ++t;
        const SgdItem &it = P.item[t];
        const unsigned int vb = g - it.first_block;
        const unsigned int vg = (t + 1 < P.count ? P.item[t + 1 < N ? t + 1 : 0].first_block : P.blocks) - it.first_block;
        const long long n4 = it.n >> 2;
        float4 *W4 = reinterpret_cast<float4 *>(it.W);
        float4 *V4 = reinterpret_cast<float4 *>(it.V);
        const float4 *G4 = reinterpret_cast<const float4 *>(it.dW);
        const long long stride = (long long)vg * kSweepThreads;
        double a0 = 0.0, a1 = 0.0;
        long long i = (long long)vb * kSweepThreads + threadIdx.x;
        // two iterations in flight: six 16-byte loads per thread, 1024 threads per SM
        for (; i + stride < n4; i += 2 * stride) {
            float4 w = W4[i], v = V4[i], w2 = W4[i + stride], v2 = V4[i + stride];
            const float4 d = __ldg(G4 + i), d2 = __ldg(G4 + i + stride);
            sgd_four(w, d, v, P.lr, P.mu, P.wd, a0, a1);
            W4[i] = w;
            V4[i] = v;
            sgd_four(w2, d2, v2, P.lr, P.mu, P.wd, a0, a1);
            W4[i + stride] = w2;
            V4[i + stride] = v2;
        }
        if (i < n4) {
            float4 w = W4[i], v = V4[i];
            sgd_four(w, __ldg(G4 + i), v, P.lr, P.mu, P.wd, a0, a1);
            W4[i] = w;
            V4[i] = v;
        }
        if (vb == 0) {
            const long long e = (n4 << 2) + threadIdx.x;
            if (e < it.n) {
                float v = it.V[e];
                const float w = sgd_one(it.W[e], __ldg(it.dW + e), v, P.lr, P.mu, P.wd);
                it.W[e] = w;
                it.V[e] = v;
                a0 += (double)fabsf(w);
            }
        }
        const double s = sweep_sum(a0 + a1, red, turn);
        if (CLUSTER) own = s;
        else if (threadIdx.x == 0) carve(ws_raw, t).part_sum[vb] = s;
    }
    if (CLUSTER) {
        // a block has at most one share
        cluster_wait();
        if (threadIdx.x == 0) st_peer(peer_smem(&sum_s[blockIdx.x], 0), __double_as_longlong(own));
        cluster_arrive();
        cluster_wait();
        if (blockIdx.x == 0 && threadIdx.x == 0 && P.item[0].stats) write_next(P.item[0], P.factor, tree8(sum_s));
    }
}
template <int N>
__global__ void __launch_bounds__(kSweepThreads)
sgd_fold_kernel(const __grid_constant__ SgdLaunch<N> P, void *ws_raw)
{
    __shared__ Reduce red;
    unsigned int turn = 0;
    chain_wait();
    const int t = (int)blockIdx.x;
    const SgdItem &it = P.item[t];
    if (!it.stats) return;
    const unsigned int vg = (t + 1 < P.count ? P.item[t + 1 < N ? t + 1 : 0].first_block : P.blocks) - it.first_block;
    const double s = fold_parts(carve(ws_raw, t).part_sum, vg, red, turn);
    if (threadIdx.x == 0) write_next(it, P.factor, s);
}

// ---- standalone pack / unpack / re-layout ----------------------------------
// Block-wide sum with a fixed order; the result is valid in thread 0.
template <typename T>
__device__ __forceinline__ T block_sum(T v, T *smem /* kWarps entries */)
{
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) smem[warp] = v;
    __syncthreads();
    T r = T(0);
    if (warp == 0) r = warp_sum(lane < kWarps ? smem[lane] : T(0));
    return r;
}

__device__ __forceinline__ uint32_t i8x4_to_fields(uint32_t x, uint32_t &bad)
{
    // a byte is valid iff (byte + 1) mod 256 <= 2
    const uint32_t inval = __vcmpgtu4(__vadd4(x, 0x01010101u), 0x02020202u);
    bad |= inval;
    x &= ~inval;
    // low two bits of bytes 0..3 -> fields in code8 order (low nibble e0, e2; high nibble e1, e3)
    const uint32_t y = x & 0x03030303u;
    return ((y & 3u) << 2) | ((y >> 16) & 3u) | ((y >> 2) & 0xC0u) | ((y >> 20) & 0x30u);
}

__global__ void __launch_bounds__(kThreads)
pack_kernel(const int8_t *__restrict__ codes, long long rows, long long cols, long long ld_codes,
            int vec_ok, uint32_t *__restrict__ packed, twn_stats_t *__restrict__ counts)
{
    __shared__ unsigned long long redu[kWarps];
    const long long wpr = ld_codes >> 4;
    const long long total_words = rows * wpr;
    unsigned long long npos = 0, nneg = 0;
    uint32_t bad = 0;
    for (long long w = (long long)blockIdx.x * kThreads + threadIdx.x; w < total_words;
         w += (long long)gridDim.x * kThreads) {
        const long long r = w / wpr;
        const long long j0 = (w - r * wpr) << 4;
        uint32_t word = 0;
        if (vec_ok && j0 + 16 <= cols) {
            const uint4 v = __ldg(reinterpret_cast<const uint4 *>(codes + r * cols + j0));
            word = bytes_to_word(i8x4_to_fields(v.x, bad) | (i8x4_to_fields(v.y, bad) << 8) |
                                 (i8x4_to_fields(v.z, bad) << 16) | (i8x4_to_fields(v.w, bad) << 24));
        } else {
            for (int e = 0; e < 16; ++e) {
                const long long j = j0 + e;
                if (j < cols) {
                    const uint32_t b = (uint8_t)codes[r * cols + j];
                    word |= ((i8x4_to_fields(b, bad) >> 2) & 3u) << field_pos(e);   // byte 0 -> bits 3:2
                }
            }
        }
        const uint32_t neg = __popc((word >> 1) & 0x55555555u);
        nneg += neg;
        npos += __popc(word & 0x55555555u) - neg;
        packed[w] = word;
    }
    if (counts) {
        const unsigned long long bp = block_sum(npos, redu);
        const unsigned long long bn = block_sum(nneg, redu);
        const int any_bad = __syncthreads_or(bad != 0);
        if (threadIdx.x == 0) {
            // integer atomics: order-independent, hence still deterministic
            atomicAdd(reinterpret_cast<unsigned long long *>(&counts->n_pos), bp);
            atomicAdd(reinterpret_cast<unsigned long long *>(&counts->n_neg), bn);
            if (any_bad) atomicMin(&counts->status, (int)TWN_ERR_BAD_CODE);
        }
    }
}

__global__ void finish_counts_kernel(twn_stats_t *counts, unsigned long long n)
{
    counts->n_zero = n - counts->n_pos - counts->n_neg;
}

__global__ void __launch_bounds__(kThreads)
unpack_kernel(const uint32_t *__restrict__ packed, long long rows, long long cols, long long ld_codes,
              int vec_ok, int8_t *__restrict__ codes, int32_t *__restrict__ dev_status)
{
    const long long wpr = ld_codes >> 4;
    const long long wpr_used = (cols + 15) >> 4;
    const long long total = rows * wpr_used;
    bool bad = false;
    for (long long t = (long long)blockIdx.x * kThreads + threadIdx.x; t < total;
         t += (long long)gridDim.x * kThreads) {
        const long long r = t / wpr_used;
        const long long wi = t - r * wpr_used;
        const uint32_t word = __ldg(packed + r * wpr + wi);
        // field 10: bit 1 set while bit 0 is clear
        const uint32_t inval = (word >> 1) & ~word & 0x55555555u;
        const long long j0 = wi << 4;
        const long long valid = cols - j0 >= 16 ? 16 : cols - j0;
        // fields of elements < valid: the top ceil(valid/2) of the low half, the top floor(valid/2) of the high half
        const uint32_t vmask = valid >= 16 ? 0xFFFFFFFFu
                                           : (((0xFFFFu << (16 - 2 * ((valid + 1) >> 1))) & 0xFFFFu) |
                                              (((0xFFFFu << (16 - 2 * (valid >> 1))) & 0xFFFFu) << 16));
        if (inval & vmask) bad = true;
        const uint32_t clean = word & ~(inval << 1);
        if (vec_ok && valid == 16) {
            const uint32_t by = word_to_bytes(clean);
            uint4 o;
            o.x = fields_to_i8x4(by & 0xFFu);
            o.y = fields_to_i8x4((by >> 8) & 0xFFu);
            o.z = fields_to_i8x4((by >> 16) & 0xFFu);
            o.w = fields_to_i8x4(by >> 24);
            *reinterpret_cast<uint4 *>(codes + r * cols + j0) = o;
        } else {
            for (int e = 0; e < valid; ++e) {
                const uint32_t f = (clean >> field_pos(e)) & 3u;
                codes[r * cols + j0 + e] = (int8_t)((f & 1u) ? ((f & 2u) ? -1 : 1) : 0);
            }
        }
    }
    if (dev_status && __syncthreads_or(bad) && threadIdx.x == 0) atomicMin(dev_status, (int)TWN_ERR_BAD_CODE);
}

// out row c, column t*Cout + o  <-  in row o, column t*Cin + c   (t = tap index)
// (32-bit index arithmetic: a filter bank has far fewer than 2^31 codes)
// `vb` of `vg`: this block's index among the blocks that work on this filter bank.
__device__ __forceinline__ void transpose_codes_body(const uint32_t *__restrict__ in, int ld_in, int Cout, int Cin,
                                                     int taps, uint32_t *__restrict__ out, int ld_out,
                                                     unsigned int vb, unsigned int vg)
{
    const int wpr_out = ld_out >> 4, wpr_in = ld_in >> 4;
    const int total = Cin * wpr_out;
    const int cols_out = taps * Cout;
    for (int w = vb * kTrThreads + threadIdx.x; w < total; w += vg * kTrThreads) {
        const int c = w / wpr_out;
        const int j0 = (w - c * wpr_out) << 4;
        int t = j0 / Cout, o = j0 - t * Cout;
        uint32_t word = 0;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (j0 + e < cols_out) {
                const int src = t * Cin + c;
                const uint32_t f = (__ldg(in + (size_t)o * wpr_in + (src >> 4)) >> field_pos(src & 15)) & 3u;
                word |= f << field_pos(e);
            }
            if (++o == Cout) { o = 0; ++t; }
        }
        out[w] = word;
    }
}

// The same re-layout for filter banks whose taps start on word boundaries on both sides (Cin % 16 == 0, and
// Cout % 16 == 0 or a single tap): a thread transposes one 16 x 16 block of codes, from words of 16 rows into words of
// 16 rows, in registers.  A warp takes 4 blocks along the input channels and 8 along the output channels of a tap, so
// that its loads cover 16-byte and its stores 32-byte runs.  What bounds it is latency (a bank has a few thousand
// blocks): one round of loads per thread and a transpose in four exchange steps, 96 instructions; with four blocks per
// thread, one after the other, and 768 instructions each, 192 -> 384 channels 3x3 took 10 us.
__host__ __device__ __forceinline__ bool transpose_fast_ok(int Cout, int Cin, int taps)
{
    return Cin % 16 == 0 && (Cout % 16 == 0 || taps == 1);
}
__host__ __device__ __forceinline__ int transpose_fast_warps(int Cout, int Cin, int taps)
{
    return taps * (((Cin >> 4) + 3) / 4) * (((Cout + 15) / 16 + 7) / 8);
}
// 16 words of 16 two-bit fields each, transposed.  Row e of the block and element e of a word sit at position
// field_pos(e) / 2, for rows and elements alike, so in the order of positions this is a plain bit-matrix transpose.
__device__ __forceinline__ void transpose16(uint32_t (&w)[16])
{
    auto at = [](int k) { return k < 8 ? 2 * (7 - k) : 2 * (15 - k) + 1; };      // the row at position k
#pragma unroll
    for (int k = 0; k < 8; ++k) {
        uint32_t &a = w[at(k)], &b = w[at(k + 8)];
        const uint32_t x = __byte_perm(a, b, 0x5410), y = __byte_perm(a, b, 0x7632);
        a = x; b = y;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 4)) {
            uint32_t &a = w[at(k)], &b = w[at(k + 4)];
            const uint32_t x = __byte_perm(a, b, 0x6240), y = __byte_perm(a, b, 0x7351);
            a = x; b = y;
        }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 2)) {
            uint32_t &a = w[at(k)], &b = w[at(k + 2)];
            const uint32_t t = ((a >> 4) ^ b) & 0x0F0F0F0Fu;
            b ^= t; a ^= t << 4;
        }
#pragma unroll
    for (int k = 0; k < 16; ++k)
        if (!(k & 1)) {
            uint32_t &a = w[at(k)], &b = w[at(k + 1)];
            const uint32_t t = ((a >> 2) ^ b) & 0x33333333u;
            b ^= t; a ^= t << 2;
        }
}
__device__ __forceinline__ void transpose_codes_fast_body(const uint32_t *__restrict__ in, int ld_in, int Cout, int Cin,
                                                          int taps, uint32_t *__restrict__ out, int ld_out,
                                                          unsigned int vb, unsigned int vg)
{
    const int wpr_out = ld_out >> 4, wpr_in = ld_in >> 4;
    const int cgs = Cin >> 4, ogs = (Cout + 15) / 16;
    const int cts = (cgs + 3) / 4, ots = (ogs + 7) / 8, total = taps * cts * ots;
    const int lane = threadIdx.x & 31;
    for (int u = vb * (kTrThreads / 32) + (threadIdx.x >> 5); u < total; u += vg * (kTrThreads / 32)) {
        const int ct = u % cts, ot = (u / cts) % ots, t = u / (cts * ots);
        const int cg = ct * 4 + (lane & 3), og = ot * 8 + (lane >> 2);
        if (cg >= cgs || og >= ogs) continue;
        const int c0 = cg << 4, o0 = og << 4;
        const uint32_t *src = in + (size_t)o0 * wpr_in + ((t * Cin + c0) >> 4);
        // rows past Cout (the last block of a bank whose Cout is no multiple of 16) read as zero codes
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = o0 + i < Cout ? __ldg(src + (size_t)i * wpr_in) : 0u;
        transpose16(w);
        uint32_t *dst = out + (size_t)c0 * wpr_out + ((t * Cout + o0) >> 4);
#pragma unroll
        for (int j = 0; j < 16; ++j) dst[(size_t)j * wpr_out] = w[j];
    }
    // columns past the last tap (a row pitch larger than taps * Cout) read as zero codes
    const int used = (taps * Cout + 15) >> 4;
    if (used < wpr_out) {
        const int pad = wpr_out - used;
        for (int i = vb * kTrThreads + threadIdx.x; i < Cin * pad; i += vg * kTrThreads)
            out[(size_t)(i / pad) * wpr_out + used + i % pad] = 0u;
    }
}

__global__ void __launch_bounds__(kTrThreads)
transpose_codes_kernel(const uint32_t *__restrict__ in, int ld_in, int Cout, int Cin,
                       int taps, uint32_t *__restrict__ out, int ld_out)
{
    pdl_begin();
    if (transpose_fast_ok(Cout, Cin, taps)) transpose_codes_fast_body(in, ld_in, Cout, Cin, taps, out, ld_out, blockIdx.x, gridDim.x);
    else transpose_codes_body(in, ld_in, Cout, Cin, taps, out, ld_out, blockIdx.x, gridDim.x);
}

// The filter banks of a whole network in one launch (the backward pass of a step needs them all).
struct TransposeItem {
    const uint32_t *in;
    uint32_t *out;
    int ld_in, ld_out, Cout, Cin, taps;
};
struct TransposeBatch {
    int count;
    unsigned int first_block[kMaxBatch + 1];
    TransposeItem item[kMaxBatch];
};

__global__ void __launch_bounds__(kTrThreads)
transpose_codes_batch_kernel(const __grid_constant__ TransposeBatch P)
{
    int t = 0;
    while (t + 1 < P.count && blockIdx.x >= P.first_block[t + 1]) ++t;
    const TransposeItem &it = P.item[t];
    if (transpose_fast_ok(it.Cout, it.Cin, it.taps))
        transpose_codes_fast_body(it.in, it.ld_in, it.Cout, it.Cin, it.taps, it.out, it.ld_out,
                                  blockIdx.x - P.first_block[t], P.first_block[t + 1] - P.first_block[t]);
    else
        transpose_codes_body(it.in, it.ld_in, it.Cout, it.Cin, it.taps, it.out, it.ld_out,
                             blockIdx.x - P.first_block[t], P.first_block[t + 1] - P.first_block[t]);
}

// Codes of a stride-2 layer re-ordered for the folded input: folded row r' holds 64 columns,
// column s'*16 + (dy*2 + dx)*Cin + c  <-  tap (2r' + dy, 2s' + dx), channel c; columns without a
// tap (past kh or kw, or past 4*Cin inside a 16-group) are 0.
__global__ void __launch_bounds__(kThreads)
fold_codes_kernel(const uint32_t *__restrict__ in, int ld_in, int Cout, int Cin, int kh, int kw,
                  uint32_t *__restrict__ out, int ld_out)
{
    const int wpr_out = ld_out >> 4, wpr_in = ld_in >> 4;
    const int total = Cout * wpr_out;
    for (int w = blockIdx.x * kThreads + threadIdx.x; w < total; w += gridDim.x * kThreads) {
        const int o = w / wpr_out;
        const int j0 = (w - o * wpr_out) << 4;      // a word is one (r', s') group of 16 columns
        const int rf = j0 >> 6, sf = (j0 >> 4) & 3;
        uint32_t word = 0;
        for (int e = 0; e < 4 * Cin; ++e) {
            const int blk = e / Cin, c = e - blk * Cin;
            const int r = 2 * rf + (blk >> 1), sx = 2 * sf + (blk & 1);
            if (r < kh && sx < kw) {
                const int src = (r * kw + sx) * Cin + c;
                const uint32_t f = (__ldg(in + (size_t)o * wpr_in + (src >> 4)) >> field_pos(src & 15)) & 3u;
                word |= f << field_pos(e);
            }
        }
        out[w] = word;
    }
}

int grid_for(long long items_per_thread_units, int sm_count)
{
    long long blocks = (items_per_thread_units + kThreads - 1) / kThreads;
    const long long cap = (long long)sm_count * 8;
    if (blocks > cap) blocks = cap;
    if (blocks < 1) blocks = 1;
    return (int)blocks;
}

// What phase 1 reads last and phase 2 first is marked to stay in L2, the rest of a tensor larger than this to go first:
// of 134 MB (8192 x 4096 weights, three tensors in turn) 53.4 us without marks, 50.3 / 49.3 / 50.0 / 50.7 / 51.4 us with 1 /
// 40 / 60 / 80 / 100 MB kept; of 403 MB 136.9 us without, 131.4 us with 40 MB.  (Tensors of these sizes are read once now, at the
// usual factors.  What goes this way are tensors of 40 to 67 MB, the coding sweep alone, and what read_once leaves here:
// 44, 52 and 66 MB, three in turn, 21.6, 24.5 and 27.7 us without marks, 19.8, 22.8 and 26.5 with; the coding sweep of 134 MB 30.1 and
// 28.3.  One tensor again and again is no faster with them, 66 MB 21.2 and 22.1; 864 MB neither.)
constexpr unsigned long long kKeptBytes = 40000000ull;

int transpose_blocks(int Cout, int Cin, int taps, long long words, int sm_count)
{
    const long long threads = transpose_fast_ok(Cout, Cin, taps) ? 32ll * transpose_fast_warps(Cout, Cin, taps) : words;
    return (int)std::max(1ll, std::min((threads + kTrThreads - 1) / kTrThreads, (long long)sm_count * 16));
}

// A tensor as the sweeps see it; false if an argument is not acceptable (*rc says why).
bool make_item(const float *W, int64_t rows, int64_t cols, twn_stats_t *stats, uint32_t *packed, int64_t ld_codes,
               int8_t *codes_i8, Item *it, int *rc)
{
    const long long n = (long long)rows * cols;
    *rc = TWN_ERR_INVALID_ARG;
    if (rows < 0 || cols < 0 || !stats || ld_codes < cols || ld_codes % 64 != 0) return false;
    if (n != 0 && (!W || !packed)) return false;
    *rc = TWN_ERR_MISALIGNED;
    if (!twn_aligned(W, 16) || !twn_aligned(packed, 16) || !twn_aligned(stats, 8) || !twn_aligned(codes_i8, 16)) return false;
    it->W = W; it->stats = stats; it->packed = packed; it->codes_i8 = codes_i8;
    it->rows = rows; it->cols = cols; it->wpr = ld_codes / 16;
    it->n = (unsigned long long)n;
    const unsigned long long used = (unsigned long long)(cols + 15) / 16;
    it->words = (unsigned long long)rows * used;
    // One part per block of a full grid, of at least 8192 weights: below that the fixed cost of a part (its
    // reduction) would show in a batch.  Small tensors: at most eight parts, of whole quarter-word rounds.
    it->small = it->words <= kSmallWords;
    const unsigned long long most = it->small ? kSmallParts : kMaxParts, step = it->small ? kQuarterWords : 512;
    unsigned long long part = (it->words + most - 1) / most;
    part = std::max(1ull, (part + step - 1) / step) * step;
    *rc = TWN_ERR_TOO_LARGE;
    if (used > 0xFFFFFFFFull || part > 0x08000000ull) return false;
    it->wpr_used = (unsigned int)used;
    it->wpr_magic = used > 1 ? (unsigned int)((1ull << 32) / used + 1) : 0;
    it->last_valid = used > 0 ? (unsigned int)(cols - 16 * (used - 1)) : 0;
    it->part_words = (unsigned int)part;
    it->parts = (unsigned int)std::max(1ull, (it->words + part - 1) / part);
    it->vec4 = rows == 1 || cols % 4 == 0;
    it->dense = rows == 1 || ld_codes == cols;
    it->linear = rows == 1 || cols % 16 == 0;
    it->first_pass = 4ull * n > kKeptBytes ? (unsigned int)(16 * part - 16 * part * kKeptBytes / (4ull * n)) : 0;
    it->first_part = 0;
    *rc = TWN_OK;
    return true;
}

// Whether a tensor's codes and sums come from one read (ternarize_once_kernel): it is large enough for that to pay, every
// block has one part, the marks of a part fit, and the kept sum is exact.  Alone and in a batch alike, so that the sums are the
// same bits.
// Exact: the sweep adds up what lies above the estimate and the corrections take it to the threshold, another order than that of
// the coding sweep, which twn_ternarize_codes would put in its place for the same weights.  With the threshold in [2^e, 2^(e+1))
// every fp32 magnitude above it, and above an estimate no more than a binade below, is a multiple of 2^(e-24), and no partial sum
// exceeds sum |W| = n * threshold / factor <= 2^(e+1) * n / factor.  So for n <= 2^28 * factor all partial sums are whole
// multiples of 2^(e-24) below 2^53 of them: fp64 holds each without rounding, and every order gives the same bits.  (Factor 0.7:
// 188 million weights, factor 0.0625: 2^24.)  An estimate further below than that is a miss, whatever its window.
bool read_once(const Item &it, double factor, const twn_device_info &dev)
{
    return it.n >= kOnceWeights && (double)it.n <= 0x1p28 * factor && it.parts <= (unsigned int)(dev.sm_count * kSweepBlocksPerSm) &&
           it.part_words <= kOnceGroups * 512;
}

int launch_once(Launch<1> &P, double factor, void *ws, const twn_device_info &dev, cudaStream_t s)
{
    P.factor = factor;
    P.parts = P.item[0].parts;
    P.item[0].first_part = 0;
    static bool attr_set[64] = {false};
    if (!attr_set[dev.ordinal]) {
        TWN_CUDA_OK(cudaFuncSetAttribute(ternarize_once_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)once_smem(kOnceGroups)));
        attr_set[dev.ordinal] = true;
    }
    return launch_cooperative(ternarize_once_kernel, P.parts, s, once_smem(P.item[0].part_words >> 9), P, ws);
}

template <int N, bool SUMS>
int launch_sweeps(Launch<N> &P, double factor, void *ws, cudaStream_t s)
{
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    P.factor = factor;
    P.parts = 0;
    for (int t = 0; t < P.count; ++t) {
        P.item[t].first_part = P.parts;
        P.parts += P.item[t].parts;
    }
    if constexpr (N == 1) {
        if (P.item[0].small) {
            unsigned int grid = 1;
            while (grid < P.parts) grid *= 2;
            const unsigned int q = P.item[0].part_words / kQuarterWords;
            auto kernel = q <= 1 ? ternarize_small_kernel<1, SUMS> : q <= 2 ? ternarize_small_kernel<2, SUMS>
                        : q <= 4 ? ternarize_small_kernel<4, SUMS> : ternarize_small_kernel<8, SUMS>;
            return launch_cluster(kernel, grid, s, P);
        }
        if (SUMS && read_once(P.item[0], factor, dev)) return launch_once(P, factor, ws, dev, s);
    }
    const unsigned int grid = std::min(P.parts, (unsigned int)(dev.sm_count * kSweepBlocksPerSm));
    if (SUMS) TWN_CUDA_OK(twn_launch_pdl(true, sums_kernel<N>, (int)grid, kSweepThreads, 0, s, P, ws));
    if (SUMS && N > 1) TWN_CUDA_OK(twn_launch_pdl(true, sums_fold_kernel<N>, P.count, kSweepThreads, 0, s, P, ws));
    TWN_CUDA_OK(twn_launch_pdl(true, codes_kernel<N, SUMS && N == 1>, (int)grid, kSweepThreads, 0, s, P, ws));
    TWN_CUDA_OK(twn_launch_pdl(true, codes_fold_kernel<N>, P.count, kSweepThreads, 0, s, P, ws));
    return TWN_OK;
}

bool batch_items(const twn_ternarize_item_t *items, int count, Launch<kMaxBatch> &P, int *rc)
{
    P.count = count;
    for (int t = 0; t < count; ++t) {
        const twn_ternarize_item_t &it = items[t];
        if (!make_item(it.W, it.rows, it.cols, it.stats, it.packed, it.ld_codes, it.codes_i8, &P.item[t], rc)) return false;
    }
    return true;
}

template <int N>
int launch_sgd(SgdLaunch<N> &P, void *ws, cudaStream_t s)
{
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    // per tensor, as many blocks as run at once or fewer: the same number alone and in a batch, so the same sums
    P.blocks = 0;
    for (int t = 0; t < P.count; ++t) {
        const long long want = (P.item[t].n / 4 + kSweepThreads - 1) / kSweepThreads;
        P.item[t].first_block = P.blocks;
        P.blocks += (unsigned int)std::max(1ll, std::min((long long)kMaxParts, want));
    }
    if constexpr (N == 1) {
        if (P.blocks <= kSmallParts) {
            unsigned int grid = 1;
            while (grid < P.blocks) grid *= 2;
            return launch_cluster(sgd_update_kernel<N, true>, grid, s, P, ws);
        }
    }
    TWN_CUDA_OK(twn_launch_pdl(true, sgd_update_kernel<N, false>, (int)std::min(P.blocks, (unsigned int)(dev.sm_count * kSweepBlocksPerSm)),
                               kSweepThreads, 0, s, P, ws));
    TWN_CUDA_OK(twn_launch_pdl(true, sgd_fold_kernel<N>, P.count, kSweepThreads, 0, s, P, ws));
    return TWN_OK;
}

}  // namespace

extern "C" size_t twn_ternarize_workspace_bytes(void) { return kWorkspaceBytes; }

extern "C" size_t twn_ternarize_batch_workspace_bytes(int count) { return count > 0 ? (size_t)count * kWorkspaceBytes : 0; }

extern "C" int twn_ternarize(const float *W, int64_t rows, int64_t cols, double delta_factor,
                             twn_stats_t *stats, uint32_t *packed, int64_t ld_codes,
                             int8_t *codes_i8, void *workspace, size_t workspace_bytes,
                             twn_stream_t stream)
{
    int rc;
    Launch<1> P;
    P.count = 1;
    TWN_REQUIRE(workspace != nullptr && delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    if (!make_item(W, rows, cols, stats, packed, ld_codes, codes_i8, &P.item[0], &rc)) return rc;
    TWN_REQUIRE(workspace_bytes >= kWorkspaceBytes, TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    return launch_sweeps<1, true>(P, delta_factor, workspace, twn_cu(stream));
}

extern "C" int twn_ternarize_codes(const float *W, int64_t rows, int64_t cols, twn_stats_t *stats, uint32_t *packed,
                                   int64_t ld_codes, int8_t *codes_i8, void *workspace, size_t workspace_bytes,
                                   twn_stream_t stream)
{
    int rc;
    Launch<1> P;
    P.count = 1;
    TWN_REQUIRE(workspace != nullptr, TWN_ERR_INVALID_ARG);
    if (!make_item(W, rows, cols, stats, packed, ld_codes, codes_i8, &P.item[0], &rc)) return rc;
    TWN_REQUIRE(workspace_bytes >= kWorkspaceBytes, TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    return launch_sweeps<1, false>(P, 0.0, workspace, twn_cu(stream));
}

extern "C" int twn_ternarize_batch(const twn_ternarize_item_t *items, int count, double delta_factor,
                                   void *workspace, size_t workspace_bytes, twn_stream_t stream)
{
    TWN_REQUIRE(count >= 0 && count <= kMaxBatch, TWN_ERR_INVALID_ARG);
    if (count == 0) return TWN_OK;
    TWN_REQUIRE(items != nullptr && workspace != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace_bytes >= twn_ternarize_batch_workspace_bytes(count), TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    int rc;
    Launch<kMaxBatch> P;
    if (!batch_items(items, count, P, &rc)) return rc;
    twn_device_info dev;
    rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    // tensors that are read once have launches of their own
    int rest = 0;
    for (int t = 0; t < count; ++t) {
        if (!read_once(P.item[t], delta_factor, dev)) {
            if (rest != t) P.item[rest] = P.item[t];
            ++rest;
            continue;
        }
        Launch<1> one;
        one.count = 1;
        one.item[0] = P.item[t];
        rc = launch_once(one, delta_factor, static_cast<char *>(workspace) + (size_t)t * kWorkspaceBytes, dev, twn_cu(stream));
        if (rc != TWN_OK) return rc;
    }
    if (rest == 0) return TWN_OK;
    P.count = rest;
    return launch_sweeps<kMaxBatch, true>(P, delta_factor, workspace, twn_cu(stream));
}

extern "C" int twn_ternarize_codes_batch(const twn_ternarize_item_t *items, int count, void *workspace,
                                         size_t workspace_bytes, twn_stream_t stream)
{
    TWN_REQUIRE(count >= 0 && count <= kMaxBatch, TWN_ERR_INVALID_ARG);
    if (count == 0) return TWN_OK;
    TWN_REQUIRE(items != nullptr && workspace != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace_bytes >= twn_ternarize_batch_workspace_bytes(count), TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    int rc;
    Launch<kMaxBatch> P;
    if (!batch_items(items, count, P, &rc)) return rc;
    return launch_sweeps<kMaxBatch, false>(P, 0.0, workspace, twn_cu(stream));
}

extern "C" int twn_sgd_update(float *W, const float *dW, float *V, int64_t n, float lr, float momentum,
                              float weight_decay, double delta_factor, twn_stats_t *stats_next, void *workspace,
                              size_t workspace_bytes, twn_stream_t stream)
{
    TWN_REQUIRE(n >= 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(n == 0 || (W != nullptr && dW != nullptr && V != nullptr), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(lr == lr && momentum == momentum && weight_decay == weight_decay, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace_bytes >= kWorkspaceBytes, TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(W, 16) && twn_aligned(dW, 16) && twn_aligned(V, 16) && twn_aligned(stats_next, 8) &&
                    twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    SgdLaunch<1> P;
    P.count = 1;
    P.lr = lr; P.mu = momentum; P.wd = weight_decay; P.factor = delta_factor;
    P.item[0] = SgdItem{W, dW, V, n, stats_next, 0};
    return launch_sgd(P, workspace, twn_cu(stream));
}

extern "C" int twn_sgd_update_batch(const twn_sgd_item_t *items, int count, float lr, float momentum,
                                    float weight_decay, double delta_factor, void *workspace, size_t workspace_bytes,
                                    twn_stream_t stream)
{
    TWN_REQUIRE(count >= 0 && count <= kMaxBatch, TWN_ERR_INVALID_ARG);
    if (count == 0) return TWN_OK;
    TWN_REQUIRE(items != nullptr && workspace != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(lr == lr && momentum == momentum && weight_decay == weight_decay, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(workspace_bytes >= twn_ternarize_batch_workspace_bytes(count), TWN_ERR_WORKSPACE);
    TWN_REQUIRE(twn_aligned(workspace, 256), TWN_ERR_MISALIGNED);
    SgdLaunch<kMaxBatch> P;
    P.count = count;
    P.lr = lr; P.mu = momentum; P.wd = weight_decay; P.factor = delta_factor;
    for (int t = 0; t < count; ++t) {
        const twn_sgd_item_t &it = items[t];
        TWN_REQUIRE(it.n >= 0 && (it.n == 0 || (it.W && it.dW && it.V)), TWN_ERR_INVALID_ARG);
        TWN_REQUIRE(twn_aligned(it.W, 16) && twn_aligned(it.dW, 16) && twn_aligned(it.V, 16) &&
                        twn_aligned(it.stats_next, 8), TWN_ERR_MISALIGNED);
        P.item[t] = SgdItem{it.W, it.dW, it.V, it.n, it.stats_next, 0};
    }
    return launch_sgd(P, workspace, twn_cu(stream));
}

// ---- the variant that allocates nothing ------------------------------------------------
// Scratch for twn_ternarize_static: tickets and per-block partials, same layout as a caller's
// workspace.  File-scope device storage, one copy per GPU that loads the library.  In host
// code the name `g_static_scratch` is only a handle for cudaGetSymbolAddress, never a pointer
// a kernel may be given.
static __device__ __align__(256) unsigned char g_static_scratch[TWN_TERNARIZE_STATIC_SCRATCH_BYTES];
static_assert(TWN_TERNARIZE_STATIC_SCRATCH_BYTES >= kWorkspaceBytes, "static scratch too small");

// Device address of g_static_scratch on the current device, looked up once per device.
static int static_scratch_ptr(int ordinal, void **out)
{
    static void *cached[64] = {nullptr};
    if (ordinal < 0 || ordinal >= 64) return TWN_ERR_CUDA;
    if (cached[ordinal] == nullptr) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || p == nullptr) return TWN_ERR_CUDA;
        cached[ordinal] = p;
    }
    *out = cached[ordinal];
    return TWN_OK;
}

extern "C" int twn_ternarize_static(const float *W, int64_t rows, int64_t cols, double delta_factor,
                                    twn_stats_t *stats, uint32_t *packed, int64_t ld_codes,
                                    int8_t *codes_i8, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(cols == 0 || rows <= TWN_TERNARIZE_STATIC_MAX_WEIGHTS / cols, TWN_ERR_TOO_LARGE);
    int rc;
    Launch<1> P;
    P.count = 1;
    if (!make_item(W, rows, cols, stats, packed, ld_codes, codes_i8, &P.item[0], &rc)) return rc;
    twn_device_info dev;
    rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    void *scratch = nullptr;
    rc = static_scratch_ptr(dev.ordinal, &scratch);
    if (rc != TWN_OK) return rc;
    return launch_sweeps<1, true>(P, delta_factor, scratch, twn_cu(stream));
}

extern "C" int twn_pack(const int8_t *codes, int64_t rows, int64_t cols, uint32_t *packed,
                        int64_t ld_codes, twn_stats_t *counts, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ld_codes >= cols && ld_codes % 64 == 0, TWN_ERR_INVALID_ARG);
    const long long n = (long long)rows * cols;
    TWN_REQUIRE(n == 0 || (codes != nullptr && packed != nullptr), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed, 16) && twn_aligned(counts, 8), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    const long long words = (long long)rows * (ld_codes / 16);
    if (words == 0) {
        if (counts) TWN_CUDA_OK(cudaMemsetAsync(counts, 0, sizeof(twn_stats_t), twn_cu(stream)));
        return TWN_OK;
    }
    const int vec_ok = twn_aligned(codes, 16) && (cols % 16 == 0);
    if (counts) TWN_CUDA_OK(cudaMemsetAsync(counts, 0, sizeof(twn_stats_t), twn_cu(stream)));
    pack_kernel<<<grid_for(words, dev.sm_count), kThreads, 0, twn_cu(stream)>>>(
        codes, rows, cols, ld_codes, vec_ok, packed, counts);
    if (counts) finish_counts_kernel<<<1, 1, 0, twn_cu(stream)>>>(counts, (unsigned long long)n);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

extern "C" int twn_unpack(const uint32_t *packed, int64_t rows, int64_t cols, int64_t ld_codes,
                          int8_t *codes, int32_t *dev_status, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ld_codes >= cols && ld_codes % 64 == 0, TWN_ERR_INVALID_ARG);
    const long long n = (long long)rows * cols;
    TWN_REQUIRE(n == 0 || (codes != nullptr && packed != nullptr), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed, 16) && twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    if (n == 0) return TWN_OK;
    const int vec_ok = twn_aligned(codes, 16) && (cols % 16 == 0);
    const long long items = (long long)rows * ((cols + 15) / 16);
    unpack_kernel<<<grid_for(items, dev.sm_count), kThreads, 0, twn_cu(stream)>>>(
        packed, rows, cols, ld_codes, vec_ok, codes, dev_status);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

extern "C" int twn_transpose_codes(const uint32_t *packed_fwd, int64_t ld_fwd,
                                   const twn_conv_desc_t *d, uint32_t *packed_bwd, int64_t ld_bwd,
                                   twn_stream_t stream)
{
    TWN_REQUIRE(d != nullptr && packed_fwd != nullptr && packed_bwd != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(d->Cin > 0 && d->Cout > 0 && d->kh > 0 && d->kw > 0, TWN_ERR_INVALID_ARG);
    const long long taps = (long long)d->kh * d->kw;
    TWN_REQUIRE(ld_fwd % 64 == 0 && ld_fwd >= taps * d->Cin, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ld_bwd % 64 == 0 && ld_bwd >= taps * d->Cout, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed_fwd, 16) && twn_aligned(packed_bwd, 16), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    const long long words = d->Cin * (ld_bwd / 16);
    TWN_REQUIRE(words < 0x7fffffffLL && d->Cout * (ld_fwd / 16) < 0x7fffffffLL && ld_fwd < 0x7fffffffLL &&
                    ld_bwd < 0x7fffffffLL, TWN_ERR_INVALID_ARG);
    TWN_CUDA_OK(twn_launch_small(transpose_codes_kernel, transpose_blocks((int)d->Cout, (int)d->Cin, (int)taps, words, dev.sm_count),
                                 kTrThreads, 0, twn_cu(stream), packed_fwd, (int)ld_fwd, (int)d->Cout, (int)d->Cin, (int)taps,
                                 packed_bwd, (int)ld_bwd));
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

extern "C" int twn_transpose_codes_batch(const twn_transpose_item_t *items, int count, twn_stream_t stream)
{
    TWN_REQUIRE(count >= 0 && count <= kMaxBatch, TWN_ERR_INVALID_ARG);
    if (count == 0) return TWN_OK;
    TWN_REQUIRE(items != nullptr, TWN_ERR_INVALID_ARG);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    TransposeBatch P;
    P.count = count;
    unsigned int g = 0;
    for (int t = 0; t < count; ++t) {
        const twn_transpose_item_t &it = items[t];
        const twn_conv_desc_t *d = &it.desc;
        TWN_REQUIRE(it.packed_fwd && it.packed_bwd, TWN_ERR_INVALID_ARG);
        TWN_REQUIRE(d->Cin > 0 && d->Cout > 0 && d->kh > 0 && d->kw > 0, TWN_ERR_INVALID_ARG);
        const long long taps = (long long)d->kh * d->kw;
        TWN_REQUIRE(it.ld_fwd % 64 == 0 && it.ld_bwd % 64 == 0 && it.ld_fwd >= taps * d->Cin && it.ld_bwd >= taps * d->Cout,
                    TWN_ERR_INVALID_ARG);
        TWN_REQUIRE(twn_aligned(it.packed_fwd, 16) && twn_aligned(it.packed_bwd, 16), TWN_ERR_MISALIGNED);
        const long long words = d->Cin * (it.ld_bwd / 16);
        TWN_REQUIRE(words < 0x7fffffffLL && d->Cout * (it.ld_fwd / 16) < 0x7fffffffLL && it.ld_fwd < 0x7fffffffLL &&
                        it.ld_bwd < 0x7fffffffLL, TWN_ERR_INVALID_ARG);
        TransposeItem ti;
        ti.in = it.packed_fwd; ti.out = it.packed_bwd; ti.ld_in = (int)it.ld_fwd; ti.ld_out = (int)it.ld_bwd;
        ti.Cout = (int)d->Cout; ti.Cin = (int)d->Cin; ti.taps = (int)taps;
        P.item[t] = ti;
        P.first_block[t] = g;
        g += (unsigned int)transpose_blocks(ti.Cout, ti.Cin, ti.taps, words, dev.sm_count);
    }
    P.first_block[count] = g;
    transpose_codes_batch_kernel<<<g, kTrThreads, 0, twn_cu(stream)>>>(P);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}

extern "C" int twn_fold_codes(const twn_conv_desc_t *d, const uint32_t *packed, int64_t ld_codes,
                              uint32_t *packed_folded, int64_t ld_folded, twn_stream_t stream)
{
    int64_t ldf = 0;
    int rc = twn_fold_dims(d, nullptr, nullptr, &ldf);
    if (rc != TWN_OK) return rc;
    TWN_REQUIRE(packed && packed_folded, TWN_ERR_INVALID_ARG);
    const long long K = (long long)d->kh * d->kw * d->Cin;
    TWN_REQUIRE(ld_codes % 64 == 0 && ld_codes >= K && ld_folded == ldf, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(packed, 16) && twn_aligned(packed_folded, 16), TWN_ERR_MISALIGNED);
    TWN_REQUIRE(d->Cout * (ldf / 16) < 0x7fffffffLL && d->Cout * (ld_codes / 16) < 0x7fffffffLL, TWN_ERR_INVALID_ARG);
    twn_device_info dev;
    rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    fold_codes_kernel<<<grid_for(d->Cout * (ldf / 16), dev.sm_count), kThreads, 0, twn_cu(stream)>>>(
        packed, (int)ld_codes, (int)d->Cout, (int)d->Cin, d->kh, d->kw, packed_folded, (int)ldf);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}
