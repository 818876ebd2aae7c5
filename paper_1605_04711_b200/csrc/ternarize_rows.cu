// Per-filter threshold ternarization fused with 2-bit packing: Algorithm 1 as printed, whose
// first loop runs over the filters of a layer.  Filter r (row r of the fp32 master weights)
// gets its own threshold delta_r = factor * mean |W_r| (Sec. 2.3), its own codes (Eq. 3) and
// its own scale alpha_r = mean of |W_r,i| over |W_r,i| > delta_r (Eq. 5).
//
// A team of threads per filter: a warp for filters of up to 1024 weights (12000 filters of 64 weights took 31 us with a
// block each, most of it blocks starting and joining), a block of 128 or 256 threads beyond.  What a block adds to its filter's
// work is its start, its barriers and the sums across its warps, so smaller teams are faster where they hold a filter in few
// enough registers (blocks of 256 before and of 128 now, us: 20000 filters of 1152 weights 73.1 and 39.0, 6000 of 2304 26.2 and
// 18.2, 3000 of 4608 20.6 and 14.4, 4000 of 6912 29.8 and 26.9); few long filters want the more threads (592 of 6912: 5.4, 7.1
// with 128).  The threshold needs the whole filter before any
// code can be written, but a filter is small (25 ... 8192 weights in the networks of the paper), so the team keeps it in
// registers between the two steps, up to sixteen 16-byte vectors per thread: each weight crosses HBM once (4 bytes read,
// 0.25 bytes written), against two reads for the per-layer rule.  Longer filters are read a second time, back to front
// (from L2, as a rule).  Filters that start off the 16-byte boundaries are read by two aligned vectors and shifted (with
// 4-byte loads, twice over, 4000 filters of 5001 weights took 62 us).  Both sums are fp64 with a fixed order (per-thread
// sums, shuffle tree, warps in order): same inputs, same bits.  No scratch memory.
#include <type_traits>

#include "sweep.cuh"

namespace {

constexpr int kThreads = 256;

// T threads per filter (32, 128 or kThreads), R vectors of four weights per thread and chunk.
template <int T> __host__ __device__ constexpr int block_threads() { return T == 32 ? kThreads : T; }
template <int T, int R> __host__ __device__ constexpr int blocks_per_sm()
{
    return T == 128 ? (R > 10 ? 6 : R > 8 ? 7 : R > 4 ? 8 : 10) : R >= 12 ? 2 : R >= 5 ? 4 : 5;
}
template <int T, int R>
__global__ void __launch_bounds__(block_threads<T>(), blocks_per_sm<T, R>())
ternarize_rows_kernel(const float *__restrict__ W, long long rows, long long cols, double factor,
                      twn_stats_t *__restrict__ stats, uint32_t *__restrict__ packed, long long wpr,
                      int8_t *__restrict__ codes_i8, int vec4)
{
    constexpr int kTeams = block_threads<T>() / T, kV = (R + 3) / 4 * 4, kWarps = T / 32;
    __shared__ double part_a[T == 32 ? 1 : kWarps], part_b[T == 32 ? 1 : kWarps];
    __shared__ uint2 part_c[T == 32 ? 1 : kWarps];
    const int t = threadIdx.x % T, lane = threadIdx.x & 31, warp = t >> 5;
    const long long row = (long long)blockIdx.x * kTeams + threadIdx.x / T;
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");      // as pdl_begin, at any grid: the launch stands alone
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (row >= rows) return;             // a whole team
    const long long f_row = row * cols, n = rows * cols;
    const float *Wr = W + f_row;
    const int n4 = (int)((cols + 3) >> 2), words = (int)((cols + 15) >> 4);
    const int chunks = (n4 + T * R - 1) / (T * R);
    const unsigned int mis = (unsigned int)(reinterpret_cast<uintptr_t>(Wr) >> 2) & 3u;      // of every quarter of the filter
    // the vectors that its quarters reach into lie inside the matrix
    const bool shifted = f_row + (long long)n4 * 4 + 4 <= n && f_row >= (long long)mis;

    float4 v[kV];
#pragma unroll
    for (int k = R; k < kV; ++k) v[k] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    auto load = [&](int chunk) {
        const int q0 = chunk * (T * R) + t;
        if (vec4) {
#pragma unroll
            for (int k = 0; k < R; ++k)
                v[k] = q0 + k * T < n4 ? __ldg(reinterpret_cast<const float4 *>(Wr) + q0 + k * T) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            return;
        }
#pragma unroll
        for (int k = 0; k < R; ++k) {
            const int q = q0 + k * T;
            const long long e = 4ll * q;
            const int left = q < n4 ? (cols - e < 4 ? (int)(cols - e) : 4) : 0;
            float4 x = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (shifted) {
                const float4 *p = reinterpret_cast<const float4 *>(Wr + (left ? e : 0) - mis);
                const float4 a = __ldg(p), b = __ldg(p + 1);
                const bool one = mis & 1, two = mis & 2;
                const float s0 = one ? a.y : a.x, s1 = one ? a.z : a.y, s2 = one ? a.w : a.z, s3 = one ? b.x : a.w,
                            s4 = one ? b.y : b.x, s5 = one ? b.z : b.y;
                x = make_float4(two ? s2 : s0, two ? s3 : s1, two ? s4 : s2, two ? s5 : s3);
                if (left < 1) x.x = 0.0f;
                if (left < 2) x.y = 0.0f;
                if (left < 3) x.z = 0.0f;
                if (left < 4) x.w = 0.0f;
            } else {
                if (left > 0) x.x = __ldg(Wr + e);
                if (left > 1) x.y = __ldg(Wr + e + 1);
                if (left > 2) x.z = __ldg(Wr + e + 2);
                if (left > 3) x.w = __ldg(Wr + e + 3);
            }
            v[k] = x;
        }
    };
    // sums over the team, the same in all its threads
    auto team_sum = [&](double x, double *part) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (T == 32) return x;
        if (lane == 0) part[warp] = x;
        __syncthreads();
        x = 0.0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) x += part[w];
        return x;
    };

    // ---- step 1: S = sum |W_r,i|  ->  delta_r
    double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
    for (int c = 0; c < chunks; ++c) {
        load(c);
#pragma unroll
        for (int k = 0; k < R; ++k) {
            a0 += (double)fabsf(v[k].x); a1 += (double)fabsf(v[k].y); a2 += (double)fabsf(v[k].z); a3 += (double)fabsf(v[k].w);
        }
    }
    const double S = team_sum((a0 + a1) + (a2 + a3), part_a);
    const double delta = cols > 0 ? factor * (S / (double)cols) : 0.0;
    // a float w satisfies |w| > delta exactly when |w| > the largest float <= delta
    const float thr = __double2float_rd(delta);

    // ---- step 2: codes, packed 16 per word; sum and counts of the kept set
    uint32_t *Pr = packed + row * wpr;
    double kept[4] = {0.0, 0.0, 0.0, 0.0};
    unsigned int pos = 0, neg = 0;
    for (int c = chunks - 1; c >= 0; --c) {
        if (c < chunks - 1) load(c);     // the last chunk is still in registers
#pragma unroll
        for (int g = 0; g < kV / 4; ++g) {
            const float4 four[4] = {v[4 * g], v[4 * g + 1], v[4 * g + 2], v[4 * g + 3]};
            const uint32_t bytes = code_quarters(four, thr, kept, pos, neg);
            const int q0 = c * (T * R) + 4 * g * T;          // first quarter of these four rounds
            if (codes_i8) {
#pragma unroll 1
                for (int k = 0; k < 4; ++k) {
                    const long long e = 4ll * (q0 + k * T + t);
                    const uint32_t c4 = fields_to_i8x4((bytes >> (8 * k)) & 0xFFu);
                    if (4 * g + k < R)
                        for (int x = 0; x < 4 && e + x < cols; ++x) codes_i8[f_row + e + x] = (int8_t)(c4 >> (8 * x));
                }
            }
            const uint32_t word = exchange_quarters(bytes);
            const int w = q0 / 4 + (lane & 3) * (T / 4) + (t >> 2);
            if (w < words && 4 * g + (lane & 3) < R) Pr[w] = word;
        }
    }
    // padding words of the row
    for (long long j = words + t; j < wpr; j += T) Pr[j] = 0u;

    const double K = team_sum((kept[0] + kept[1]) + (kept[2] + kept[3]), part_b);
    unsigned int p = __reduce_add_sync(0xffffffffu, pos), q = __reduce_add_sync(0xffffffffu, neg);
    if (T > 32) {
        if (lane == 0) part_c[warp] = make_uint2(p, q);
        __syncthreads();
        p = q = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) { p += part_c[w].x; q += part_c[w].y; }
    }
    if (t == 0) {
        twn_stats_t st;
        st.delta = delta;
        st.alpha = (p | q) ? K / (double)((unsigned long long)p + q) : 0.0;
        st.sum_abs = S;
        st.sum_abs_kept = K;
        st.n_neg = q;
        st.n_pos = p;
        st.n_zero = (unsigned long long)cols - p - q;
        st.status = isfinite(S) ? TWN_OK : TWN_ERR_NONFINITE;
        st.reserved = 0;
        stats[row] = st;
    }
}

// scale_out[r] = alpha_r * scale_in[r]; the worst status of the filters goes to *dev_status.
__global__ void __launch_bounds__(kThreads)
rows_scale_kernel(const twn_stats_t *__restrict__ stats, long long rows, const float *__restrict__ scale_in,
                  float *__restrict__ scale_out, int32_t *dev_status)
{
    const long long r = (long long)blockIdx.x * kThreads + threadIdx.x;
    if (r >= rows) return;
    const float a = (float)stats[r].alpha;
    scale_out[r] = scale_in ? a * scale_in[r] : a;
    if (dev_status && stats[r].status != TWN_OK) atomicMin(dev_status, stats[r].status);
}

}  // namespace

extern "C" int twn_ternarize_rows(const float *W, int64_t rows, int64_t cols, double delta_factor,
                                  twn_stats_t *stats, uint32_t *packed, int64_t ld_codes,
                                  int8_t *codes_i8, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0 && cols >= 0 && cols <= 0x7fffffffLL, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(delta_factor >= 0.0 && delta_factor == delta_factor, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(ld_codes >= cols && ld_codes % 64 == 0, TWN_ERR_INVALID_ARG);
    if (rows == 0) return TWN_OK;
    TWN_REQUIRE(stats != nullptr && packed != nullptr && (cols == 0 || W != nullptr), TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(W, 4) && twn_aligned(packed, 16) && twn_aligned(stats, 8), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    // the smallest team and vector count that hold a filter; longer ones go round in chunks of 8192 weights
    const bool vec = twn_aligned(W, 16) && cols % 4 == 0;
    auto launch = [&](auto team, auto vectors) -> int {
        constexpr int T = decltype(team)::value, R = decltype(vectors)::value, kTeams = block_threads<T>() / T;
        const long long grid = (rows + kTeams - 1) / kTeams;
        TWN_REQUIRE(grid < 0x7fffffffLL, TWN_ERR_TOO_LARGE);
        TWN_CUDA_OK(twn_launch_pdl(true, ternarize_rows_kernel<T, R>, (int)grid, block_threads<T>(), 0, twn_cu(stream), W, (long long)rows,
                                   (long long)cols, delta_factor, stats, packed, (long long)(ld_codes / 16), codes_i8, (int)vec));
        return TWN_OK;
    };
#define TWN_TEAM(t, r) return launch(std::integral_constant<int, t>(), std::integral_constant<int, r>())
    if (cols <= 1024) switch ((cols + 127) / 128) {
        case 0: case 1: TWN_TEAM(32, 1);
        case 2: TWN_TEAM(32, 2);
        case 3: TWN_TEAM(32, 3);
        case 4: TWN_TEAM(32, 4);
        case 5: TWN_TEAM(32, 5);
        case 6: TWN_TEAM(32, 6);
        case 7: TWN_TEAM(32, 7);
        default: TWN_TEAM(32, 8);
    }
    // Blocks of 128: up to ten vectors a thread, and with up to fourteen once every SM has ten filters.  Filters off the 16-byte
    // boundaries, which cost a thread more, from two on an SM on (100 of 1537: 2.8 us, 3.0 with 128; 3000 of 5001 34.3 and 29.0), and
    // not beyond ten (3000 of 7001: 42.7 and 47.9).
    if (cols <= 5120 ? vec || rows >= 2LL * dev.sm_count : cols <= 7168 && vec && rows >= 10LL * dev.sm_count) switch ((cols + 511) / 512) {
        case 3: TWN_TEAM(128, 3);
        case 4: TWN_TEAM(128, 4);
        case 5: TWN_TEAM(128, 5);
        case 6: TWN_TEAM(128, 6);
        case 7: TWN_TEAM(128, 7);
        case 8: TWN_TEAM(128, 8);
        case 9: TWN_TEAM(128, 9);
        case 10: TWN_TEAM(128, 10);
        case 11: case 12: TWN_TEAM(128, 12);
        default: TWN_TEAM(128, 14);
    }
    if (cols <= 2048) TWN_TEAM(kThreads, 2);
    if (cols <= 3072) TWN_TEAM(kThreads, 3);
    if (cols <= 4096) TWN_TEAM(kThreads, 4);
    if (cols <= 6144) TWN_TEAM(kThreads, 6);
    if (cols <= 7168) TWN_TEAM(kThreads, 7);
    if (cols <= 8192 || cols > 16384) TWN_TEAM(kThreads, 8);      // fewer registers: more blocks on an SM
    if (cols <= 12288) TWN_TEAM(kThreads, 12);
    TWN_TEAM(kThreads, 16);
#undef TWN_TEAM
}

extern "C" int twn_rows_scale(const twn_stats_t *stats, int64_t rows, const float *scale_in, float *scale_out,
                              int32_t *dev_status, twn_stream_t stream)
{
    TWN_REQUIRE(rows >= 0, TWN_ERR_INVALID_ARG);
    if (rows == 0) return TWN_OK;
    TWN_REQUIRE(stats != nullptr && scale_out != nullptr, TWN_ERR_INVALID_ARG);
    TWN_REQUIRE(twn_aligned(stats, 8) && twn_aligned(scale_in, 4) && twn_aligned(scale_out, 4) &&
                    twn_aligned(dev_status, 4), TWN_ERR_MISALIGNED);
    twn_device_info dev;
    const int rc = twn_current_device(&dev);
    if (rc != TWN_OK) return rc;
    const int grid = (int)((rows + kThreads - 1) / kThreads);
    rows_scale_kernel<<<grid, kThreads, 0, twn_cu(stream)>>>(stats, rows, scale_in, scale_out, dev_status);
    TWN_CUDA_OK(cudaGetLastError());
    return TWN_OK;
}
