// Single-pulse search kernels for sm_103a (arXiv:1912.07704 Sec. 1: boxcar
// filters and peak finding on every dedispersed series, on the GPU).
//
//   stats   : per series exact integer moments (sum y, sum y^2 in 128 bits),
//             mu, sigma (population) and the per-width factors
//             r_w = 1/(sigma sqrt w), c_w = w (mu - m0) r_w  (FP64 -> FP32).
//   boxcar  : for every start t, B(t) = max_{w<=min(W,L-t)} SNR_w(t) with
//             SNR_w = (S'_w - w (mu - m0)) / (sigma sqrt w) = S'_w r_w - c_w,
//             S'_w = sum_{k<w} (y[t+k] - m0) summed exactly (FP32 when every
//             partial sum of the tile fits in 2^24, int64 otherwise); then
//             thresholded local maxima are appended to the candidate list,
//             one atomic per CTA (the CTA's run is contiguous and ordered by t,
//             and is described by a chunk header).
//             The CTA then resolves each of its candidates' width (the
//             smallest maximising w) from the series it staged, with the same
//             arithmetic bit for bit.
#include <algorithm>
#include <cfloat>
#include <climits>
#include <cstdint>

#include "aa_internal.h"

namespace aa {
namespace {

constexpr float kSentinel = -1.2676506002282294e30f;  // -2^100: marks t outside [0, L)
constexpr float kSentinelTest = -1e29f;

__device__ __forceinline__ float max3f(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

__global__ void rsqrt_table_kernel(double* t, int wpad) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < wpad) t[i] = 1.0 / sqrt((double)(i + 1));
}

// 128-bit warp reduction on (hi, lo) halves.
__device__ __forceinline__ void add128(unsigned long long& hi, unsigned long long& lo,
                                       unsigned long long h2, unsigned long long l2) {
    const unsigned long long n = lo + l2;
    hi += h2 + (n < lo ? 1ull : 0ull);
    lo = n;
}

constexpr int kStatsThreads = 512;

// Sparse width ladder: width chunk c (widths 16c+1 .. 16c+16) takes part iff
// its bit is set.  Chunks 0-3 always; then c_0 = 4 and
// c_{n+1} = max(c_n + 1, ceil(c_n * g16 / 16)).  Whole CTA; words past
// nchunks are cleared.
__host__ __device__ constexpr int ladder_words(int wpad) { return (wpad / kSpsSlots + 31) / 32; }
__device__ __forceinline__ void fill_ladder(uint32_t* mask, int nchunks, int g16) {
    for (int i = threadIdx.x; i < (nchunks + 31) / 32; i += blockDim.x) mask[i] = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c = 0; c < min(4, nchunks); ++c) mask[c >> 5] |= 1u << (c & 31);
        for (int c = 4; c < nchunks; c = max(c + 1, (c * g16 + 15) / 16)) mask[c >> 5] |= 1u << (c & 31);
    }
}
__device__ __forceinline__ bool ladder_has(const uint32_t* mask, int w) {  // width w >= 1
    const int c = (w - 1) / kSpsSlots;
    return (mask[c >> 5] >> (c & 31)) & 1u;
}

// Statistics of one series (row) and its width table; whole CTA.
//
// Exact integer sums N, S1 = sum y, S2 = sum y^2 (128-bit) over the kept
// samples; pass 0 keeps every sample.  With k-sigma clipping (k = c16/16),
// each further pass keeps the samples with |y - mu| <= k sigma of the previous
// set, i.e. (times 16N, squared) 256 (N y - S1)^2 <= c16^2 (N S2 - S1^2).
// That set is an interval of integers; thread 0 finds its ends exactly (an
// FP64 estimate corrected by the 128-bit test), so each sample needs two
// compares.  Stops after clip_iters passes, at a pass keeping nothing
// (dropped) or at a fixed point (same N, S1, S2).

// 256 (N v - S1)^2 <= R, exactly (|N v - S1| < 2^57 for |v| <= 2^25, N < 2^31)
__device__ __forceinline__ bool clip_keeps(long long N, long long S1, unsigned __int128 R, long long v) {
    const long long d = N * v - S1;
    const unsigned long long ad = (unsigned long long)(d < 0 ? -d : d);
    return (((unsigned __int128)ad * ad) << 8) <= R;
}

// Ends [lo, hi] of the kept interval, clamped to +-2^25 (every sample lies
// within +-2^24); lo > hi when no integer is kept.
__device__ void clip_interval(long long N, long long S1, unsigned __int128 R, long long& lo, long long& hi) {
    constexpr long long kLim = 1ll << 25;
    const double half = sqrt((double)R) / 16.0;  // |N v - S1| <= half
    const double c = (double)S1 / (double)N, h = half / (double)N;
    lo = (long long)fmax(fmin(ceil(c - h), (double)kLim), (double)-kLim);
    hi = (long long)fmax(fmin(floor(c + h), (double)kLim), (double)-kLim);
    // the estimate is within a few units; move each end onto the exact boundary
    for (int k = 0; k < 64 && lo <= hi && !clip_keeps(N, S1, R, lo); ++k) ++lo;
    for (int k = 0; k < 64 && lo > -kLim && clip_keeps(N, S1, R, lo - 1); ++k) --lo;
    for (int k = 0; k < 64 && hi >= lo && !clip_keeps(N, S1, R, hi); ++k) --hi;
    for (int k = 0; k < 64 && hi < kLim && clip_keeps(N, S1, R, hi + 1); ++k) ++hi;
}

__device__ __forceinline__ void stats_accumulate(float yf, bool clip, float lo, float hi, long long& cnt,
                                                 long long& s1, long long& s2) {
    if (clip && !(yf >= lo && yf <= hi)) return;
    const int v = (int)yf;  // exact: |y| < 2^24
    ++cnt;
    s1 += v;
    s2 += (long long)v * v;
}

// Statistics of a series from the exact sums of its N samples, S1 = sum y
// and S2 = H:Lo = sum y^2 (128 bits); f receives mu - m0.
__device__ RowStats row_stats_from_sums(long long N, long long S1, unsigned long long H, unsigned long long Lo,
                                        double& f) {
    RowStats st{};
    if (N > 0) {
        // N^2 var = N * sum y^2 - (sum y)^2, exact in 128 bits
        const unsigned __int128 S2 = ((unsigned __int128)H << 64) | Lo;
        const __int128 num = (__int128)N * (__int128)S2 - (__int128)S1 * (__int128)S1;
        const unsigned __int128 un = num > 0 ? (unsigned __int128)num : 0;
        const double numd = (double)(unsigned long long)(un >> 64) * 18446744073709551616.0 +
                            (double)(unsigned long long)un;
        st.mu = (double)S1 / (double)N;
        st.sigma = sqrt(numd) / (double)N;
        const long long m0 = llround(st.mu);
        st.m0 = (float)m0;
        st.inv_sigma = st.sigma > 0 ? 1.0 / st.sigma : 0.0;
        st.zero_sigma = st.sigma > 0 ? 0 : 1;
        f = (double)(S1 - m0 * N) / (double)N;  // mu - m0
    } else {
        st.zero_sigma = 1;
        f = 0.0;
    }
    return st;
}

// Width table of one row, whole CTA: r_w = 1/(sigma sqrt w), c_w = w f r_w
// (FP64, stored FP32 as (r_w, -c_w)); widths past max_width never win.
__device__ void write_width_table(const SpsArgs& a, const double* rsw, int row, double f, double inv) {
    float2* tab = a.table + (int64_t)row * a.wpad;
    for (int i = threadIdx.x; i < a.wpad; i += blockDim.x) {
        const int w = i + 1;
        if (w <= a.max_width) {
            const double r = inv * rsw[i];
            const double c = (double)w * f * r;
            tab[i] = make_float2((float)r, (float)(-c));
        } else {
            tab[i] = make_float2(0.0f, -FLT_MAX);
        }
    }
}

__device__ __forceinline__ void stats_row(const SpsArgs& a, const double* rsw, int row) {
    constexpr int NW = kStatsThreads / 32;
    constexpr int64_t kFlush = 4096;  // float4 steps per 128-bit flush: 2^14 samples, s2 < 2^14 * 2^48
    __shared__ long long s1w[NW], cw[NW];
    __shared__ unsigned long long hiw[NW], low[NW];
    __shared__ long long sh_N, sh_S1;           // sums of the accepted set
    __shared__ unsigned long long sh_H, sh_L;   // its S2 (high, low words)
    __shared__ float sh_lo, sh_hi;              // kept interval of the next pass
    __shared__ int sh_go;
    __shared__ double sh_f, sh_inv;
    const float* y = a.dd + (int64_t)row * a.pitch;  // 16-byte aligned rows
    const int64_t n = a.length;
    const int64_t n4 = n >> 2;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int iters = a.clip_iters;
    for (int pass = 0; pass <= iters; ++pass) {
        const bool clip = pass > 0;
        const float lo_f = clip ? sh_lo : 0.f, hi_f = clip ? sh_hi : 0.f;
        long long cnt = 0, s1 = 0;
        unsigned long long hi = 0, lo = 0;
        const float4* y4 = reinterpret_cast<const float4*>(y);
        for (int64_t b = threadIdx.x; b < n4; b += (int64_t)kStatsThreads * kFlush) {
            const int64_t e = min(n4, b + (int64_t)kStatsThreads * kFlush);
            long long s2 = 0;
            for (int64_t j = b; j < e; j += kStatsThreads) {
                const float4 q = y4[j];
                stats_accumulate(q.x, clip, lo_f, hi_f, cnt, s1, s2);
                stats_accumulate(q.y, clip, lo_f, hi_f, cnt, s1, s2);
                stats_accumulate(q.z, clip, lo_f, hi_f, cnt, s1, s2);
                stats_accumulate(q.w, clip, lo_f, hi_f, cnt, s1, s2);
            }
            add128(hi, lo, 0ull, (unsigned long long)s2);
        }
        if (threadIdx.x < (int)(n - 4 * n4)) {
            long long s2 = 0;
            stats_accumulate(y[4 * n4 + threadIdx.x], clip, lo_f, hi_f, cnt, s1, s2);
            add128(hi, lo, 0ull, (unsigned long long)s2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            const unsigned long long h2 = __shfl_xor_sync(0xffffffffu, hi, o);
            const unsigned long long l2 = __shfl_xor_sync(0xffffffffu, lo, o);
            add128(hi, lo, h2, l2);
        }
        if (lane == 0) {
            cw[warp] = cnt;
            s1w[warp] = s1;
            hiw[warp] = hi;
            low[warp] = lo;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            long long C = 0, S1 = 0;
            unsigned long long H = 0, Lo = 0;
            for (int w = 0; w < NW; ++w) {
                C += cw[w];
                S1 += s1w[w];
                add128(H, Lo, hiw[w], low[w]);
            }
            int go;
            if (clip && C == 0) {
                go = 0;  // nothing kept: keep the previous set
            } else {
                const bool same = clip && C == sh_N && S1 == sh_S1 && H == sh_H && Lo == sh_L;
                sh_N = C;
                sh_S1 = S1;
                sh_H = H;
                sh_L = Lo;
                go = pass < iters && !same;
            }
            if (go) {
                const unsigned __int128 S2 = ((unsigned __int128)sh_H << 64) | sh_L;
                const __int128 V = (__int128)sh_N * (__int128)S2 - (__int128)sh_S1 * (__int128)sh_S1;
                const unsigned __int128 R =
                    (unsigned __int128)(a.clip_c16 * a.clip_c16) * (V > 0 ? (unsigned __int128)V : 0);
                long long vlo, vhi;
                clip_interval(sh_N, sh_S1, R, vlo, vhi);
                sh_lo = (float)vlo;  // exact: |v| <= 2^25
                sh_hi = (float)vhi;
            }
            sh_go = go;
        }
        __syncthreads();
        if (!sh_go) break;
    }
    if (threadIdx.x == 0) {
        const RowStats st = row_stats_from_sums(sh_N, sh_S1, sh_H, sh_L, sh_f);
        sh_inv = st.inv_sigma;
        a.stats[row] = st;
    }
    __syncthreads();
    write_width_table(a, rsw, row, sh_f, sh_inv);
}

// Fused statistics (the dedispersion kernels summed each row exactly into
// acc[3 r .. 3 r + 2] = (sum y, sum y^2 low, high)): mu, sigma and the width
// table of every row of a range, with the arithmetic of stats_row's plain
// pass (bit for bit the same results).  One CTA per row.
__global__ void __launch_bounds__(256) sps_finalize_kernel(SpsArgs a, const double* rsw,
                                                          const unsigned long long* acc) {
    __shared__ double sh_f, sh_inv;
    const int row = blockIdx.x;
    if (threadIdx.x == 0) {
        const unsigned long long* r = acc + 3 * (int64_t)row;
        const RowStats st = row_stats_from_sums(a.length, (long long)r[0], r[2], r[1], sh_f);
        sh_inv = st.inv_sigma;
        a.stats[row] = st;
    }
    __syncthreads();
    write_width_table(a, rsw, row, sh_f, sh_inv);
}

__global__ void __launch_bounds__(kStatsThreads) sps_stats_kernel(SpsArgs a, const double* rsw) {
    stats_row(a, rsw, blockIdx.x);
}

// Block-wide exclusive scan of one int64 per thread.
template <int NT>
__device__ long long block_exclusive_scan(long long v, long long* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    if (lane == 31) scratch[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        long long t = lane < NT / 32 ? scratch[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long u = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += u;
        }
        if (lane < NT / 32) scratch[lane] = t;  // inclusive warp totals
    }
    __syncthreads();
    const long long before = warp > 0 ? scratch[warp - 1] : 0;
    return before + inc - v;
}

// Exclusive scan that also returns the block total.
template <int NT>
__device__ long long block_exclusive_scan_total(long long v, long long* scratch, long long& total) {
    const long long ex = block_exclusive_scan<NT>(v, scratch);
    total = scratch[NT / 32 - 1];
    __syncthreads();  // scratch may be reused after this
    return ex;
}

// Block-wide exclusive scan of one `run` per thread, together with the block
// total and the smallest and largest prefix value before + mn / before + mx (mn
// <= 0 <= mx relative to the thread's own start), in one barrier; a second use
// needs one between.  Values are clamped on the way so that 32 bits hold every
// sum (a thread's at 2^25 and 2^26, a warp's at 2^27 and 2^28): results whose
// range stays within 2^24 are exact, and any clamp shows as a range beyond it.
// scratch: 3 * NT / 32 entries.
template <int NT>
__device__ __forceinline__ void block_scan_minmax(int run, int mn, int mx, int* scratch, int& before, int& total, int& gmn,
                                                  int& gmx) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto clamp = [](int v, int m) { return max(-m, min(m, v)); };
    run = clamp(run, 1 << 25);
    int inc = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
    }
    const int ex = inc - run;
    const int lmn = __reduce_min_sync(0xffffffffu, ex + clamp(mn, 1 << 26));
    const int lmx = __reduce_max_sync(0xffffffffu, ex + clamp(mx, 1 << 26));
    if (lane == 31) {
        scratch[warp] = clamp(inc, 1 << 27);
        scratch[NW + warp] = clamp(lmn, 1 << 28);
        scratch[2 * NW + warp] = clamp(lmx, 1 << 28);
    }
    __syncthreads();
    int t = 0, wbase = 0;
    gmn = INT_MAX;
    gmx = INT_MIN;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        gmn = min(gmn, t + scratch[NW + w]);
        gmx = max(gmx, t + scratch[2 * NW + w]);
        if (w == warp) wbase = t;
        t += scratch[w];
    }
    before = wbase + ex;
    total = t;
}

template <int NT>
__device__ void block_minmax(long long& mn, long long& mx, long long* scratch) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    __syncthreads();
    if (lane == 0) {
        scratch[warp] = mn;
        scratch[NT / 32 + warp] = mx;
    }
    __syncthreads();
    mn = scratch[0];
    mx = scratch[NT / 32];
    for (int w = 1; w < NT / 32; ++w) {
        mn = min(mn, scratch[w]);
        mx = max(mx, scratch[NT / 32 + w]);
    }
}

constexpr int M = kSpsSlots;
constexpr int NT = kSpsThreads;

// Exact-FP32 tiles.  P is the prefix-sum array of the staged series (index
// i <-> start time t0-1+i): P[i] = sum of y - m0 over the valid samples before
// i, -kBig once a window would run past the series end.  Every window sum
// S_w(t) = P[p+w] - P[p] is an exact FP32 integer (the caller checked that
// the prefix range of the tile is <= 2^24), so this is bit for bit the
// running sum.  Thread owns slots p = M*tid + i; base[i] = P[p] (or +kBig for
// a start outside the series).  C[i] receives w0 of the first chunk of M
// widths (w0+1 .. w0+M) whose best SNR equals B[i]: the smallest maximising
// width lies in that chunk, so the candidate's width is found by evaluating
// it alone.
constexpr float kBig = 1.2676506002282294e30f;  // 2^100

// The width search of one thread's M starts.  Widths come in chunks of M
// (chunk c: widths M c + 1 .. M c + M); chunk 0 is bounded more finely.
// Of the others a thread evaluates those that can still raise the B of one of
// its starts, each thread at its own chunk: before a bright pulse the 32
// threads of a warp need 32 different widths, each of them few.
//
// Block maxima of P decide it: Q16[j] = max P over [16 j, 16 j + 16).  A window
// of chunk c from a start p of thread t (p in [16 t, 16 t + 15]) ends in the
// blocks t + c and t + c + 1, so
//   SNR_w(p) <= (max of the two - pmin - w f) / (sigma sqrt(w)),  reaches(),
// and the largest end of block t + c + 1 gives a window to every start, of
// width M c + 1 .. M c + 31, so every start of the thread has
//   B >= (Q16[t + c + 1] - pmax - w f) / (sigma sqrt(w)),         lower().
// A first pass over the chunks takes the largest lower bound, a second one
// evaluates the chunks whose upper bound reaches max(cut, that, the smallest
// running B).  The passes go through the chunks together (the threads of a
// warp at the same c, with sliding maxima over 2, 9 and 65 blocks: S1, S8,
// S64): the first 8 chunks one by one, then groups of 8, from 64 on groups of
// 64, opened where a thread's bound reaches its floor.  Eight bounds of one
// level are computed side by side before the warp looks at them.  The chunks to
// evaluate wait in a queue of the thread, eight groups of eight as their bits,
// and are looked at again when their turn comes: a warp evaluates when a queue is
// full and at the end of the pass, so that most of its threads take part (a beam
// of 1024 channels x 48611 samples with two pulses, 2000 trials, W = 8192: 2.1 ms,
// 0.84 without the pulses; with one chunk waiting, before chunk 0 had bounds of its
// own, 3.14 against 2.23).  Evaluation and bounds are written down once, in one
// loop: with one at each place that wants them the kernel waits for instructions.
// Skipping below the running B, or below a lower bound of it, is exact for every
// start (such a chunk changes neither B nor the first chunk that reaches it; the
// chunk that the lower bound comes from is not skipped); below the threshold's cut
// it is exact for every B >= threshold and for every peak decision.
//
// FP32 with the roundings covered: P's differences are exact integers, each
// further step is within 2^-22 relative of |num| or of the drift |w f|
// (|f| <= 1/2 since m0 = round(mu)); the factor 1 + 1.02e-4 in rs and the
// margin S (1.02e-4 and the largest drift's part) bound them many times over.
// Widths whose table entries are staged in shared memory: all of them where they
// may be evaluated in turn (low), else the first 1024.
constexpr int kTabWidths = 1024;
__host__ __device__ constexpr int sps_tab_smem(int wpad, bool low) {
    return wpad < kTabWidths || (low && wpad <= kSpsEveryMost * M) ? wpad : kTabWidths;
}
// entries of Q16 and of each sliding maximum (the end padded for the longest)
__host__ __device__ constexpr int sps_q16(int wpad) { return (kSpsTile / M + wpad / M + 1 + 64 + 31) / 32 * 32; }
// entries of rs: c <= the last chunk + 65, and what a pass reads as it begins
// (chunks 64 k and the 64 after them, k < 8, whatever the last chunk)
__host__ __device__ constexpr int sps_rs(int wpad) { return ((wpad / M + 66 > 513 ? wpad / M + 66 : 513) + 3) / 4 * 4; }

// A chunk's 16 table entries are 8 16-byte blocks; in shared memory block b of
// chunk c lies at b ^ (c & 7), so that threads at neighbouring chunks read
// different banks.
__device__ __forceinline__ int tab_block(int c, int b) { return 8 * c + (b ^ (c & 7)); }

struct WidthBounds {
    const float* rs;   // rs[c] = (1 + 1.02e-4) / (sigma sqrt(M c + 1))
    float pmin, pmax;  // of P over the thread's valid starts (pmin = FLT_MAX: none)
    float f;           // mu - m0
    float S;

    // w of the smallest drift w f over chunks c .. c + n - 1, less M c
    __device__ __forceinline__ float w_first(int n) const { return f >= 0.0f ? 1.0f : (float)(M * n); }
    // can windows ending at prefix sums <= top reach F + S?  r = rs + first chunk, w = M (first chunk) + w_first;
    // where F may be negative (LOW) the widest window bounds a negative sum
    template <bool LOW>
    __device__ __forceinline__ bool reaches(float top, float w, const float* r, int n, float F) const {
        const float num = fmaf(-f, w, top - pmin);
        if (LOW && num < 0.0f) return num * (r[n] * (1.0f - 2.1e-4f)) >= F;
        return num * r[0] >= F;
    }
    // an SNR that every start reaches with an end of prefix sum q, widths M c + 1 .. M c + 31
    __device__ __forceinline__ float lower(float q, int c) const {
        const float num = fmaf(-f, (float)(f >= 0.0f ? M * c + 31 : M * c + 1), q - pmax);
        return num > 0.0f ? num * (rs[c + 2] * (1.0f - 2.1e-4f)) - S : -FLT_MAX;
    }
};

// Chunk at window base pw = P + first start + M c with its 16 table entries
// (blocks tb[b ^ x]): the best SNR of each start.
__device__ __forceinline__ void eval_chunk(const float* __restrict__ pw, const float4* tb, int x,
                                           const float (&base)[M], float (&Bc)[M]) {
    float win[2 * M];  // win[k] = P[p_thread + M c + k]
#pragma unroll
    for (int k = 0; k < 2 * M; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(pw + k);
        win[k] = v.x; win[k + 1] = v.y; win[k + 2] = v.z; win[k + 3] = v.w;
    }
#pragma unroll
    for (int s = 0; s < M; s += 2) {
        const float4 rc = tb[(s >> 1) ^ x];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const float v0 = fmaf(win[i + s + 1] - base[i], rc.x, rc.y);
            const float v1 = fmaf(win[i + s + 2] - base[i], rc.z, rc.w);
            Bc[i] = s == 0 ? fmaxf(v0, v1) : max3f(Bc[i], v0, v1);
        }
    }
}

// Can a window of width 1 to 16 reach F (> 0)?  One bound for each of the widths
// 1 | 2, 3 | 4-7 | 8-15 | 16: the largest end of its windows at each start.  In
// noise hardly a warp has to evaluate chunk 0 then (2000 series of 48611 samples,
// W = 64: 0.554 ms, 0.638 without).
__device__ __forceinline__ bool chunk0_reaches(const float* __restrict__ pb, const float (&base)[M], float f, float r, float F) {
    float win[2 * M];
#pragma unroll
    for (int k = 0; k < 2 * M; k += 4) {
        const float4 v = *reinterpret_cast<const float4*>(pb + k);
        win[k] = v.x; win[k + 1] = v.y; win[k + 2] = v.z; win[k + 3] = v.w;
    }
    // largest rise from a start to win[start + w], the drift of its widths at least w0 or at most w1
    auto reach = [&](int w, int w1, float rw) {
        float top = -FLT_MAX;
#pragma unroll
        for (int i = 0; i < M; i += 2) top = max3f(top, win[i + w] - base[i], win[i + 1 + w] - base[i + 1]);
        return fmaf(-f, (float)(f >= 0.0f ? w : w1), top) * (r * rw) >= F;
    };
    bool any = reach(1, 1, 1.0f) | reach(16, 16, 0.25f);
#pragma unroll
    for (int k = 2; k + 1 < 2 * M; ++k) win[k] = fmaxf(win[k], win[k + 1]);
    any |= reach(2, 3, 0.70710678f);
#pragma unroll
    for (int k = 4; k + 3 < 2 * M; ++k) win[k] = fmaxf(win[k], win[k + 2]);
    any |= reach(4, 7, 0.5f);
#pragma unroll
    for (int k = 8; k < M + 8; ++k) win[k] = fmaxf(win[k], win[k + 4]);
    return any | reach(8, 15, 0.35355339f);
}

constexpr unsigned kQueue = 8;
// Returns the chunks this thread evaluated.  C: the first chunk reaching B[i] in
// 16-bit halves, starts 2 k and 2 k + 1 in C[k] (16 registers of them spilled).
// Q: Q16, S1, S8 and S64, nq entries each.  queue: the thread's entries, kQueue of them NT apart.
// LOW: cut is not above zero; up to `every` chunks are simply evaluated in turn
// then.
template <bool LOW>
__device__ __forceinline__ int boxcar_search(const float* __restrict__ P, const float4* tab, const float2* __restrict__ gtab,
                                             int nch, int max_width, const float (&base)[M], const WidthBounds& bnd,
                                             const float* Q, int nq, uint16_t* queue, float cut, const uint32_t* lmask,
                                             int every, float (&B)[M], uint32_t (&C)[M / 2]) {
    const int t = threadIdx.x;
    const float* pb = P + M * t;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        B[i] = -FLT_MAX;
        C[i / 2] = 0;
    }
    if (LOW && nch <= every) {
        for (int c = 0; c < nch; ++c) {
            if (lmask && !ladder_has(lmask, M * c + 1)) continue;
            float Bc[M];
            eval_chunk(pb + M * c, tab + 8 * c, c & 7, base, Bc);
#pragma unroll
            for (int i = 0; i < M; ++i) {
                if (Bc[i] > B[i]) {
                    B[i] = Bc[i];
                    C[i / 2] = __byte_perm(C[i / 2], (uint32_t)c, i & 1 ? 0x5410 : 0x3254);
                }
            }
        }
        return nch;
    }
    const float *s1 = Q + nq + t, *s8 = s1 + nq, *s64 = s8 + nq;
    float F = cut - bnd.S;              // the floor less the bounds' margin
    const bool first0 = LOW || chunk0_reaches(P + M * t, base, bnd.f, bnd.rs[0], F);
    int evaluated = 0;
    unsigned fill = 0;                  // entries in the queue << 16 | the first one's place (mod kQueue)
    unsigned cur = 0;                   // the taken entry: chunk of its first bit << 5 | bits
    bool last = nch == 1, found = false;
    int pass = -1;
    // Groups of 64 chunks from c512, of 8 from c64, chunks from c8: a thread's
    // own (m..) and the warp's (u..) that reach the floor and are still to open.
    unsigned m64 = 0, u64 = 0, m8 = 0, u8 = 0, in = 0;
    int c512 = 0, c64 = 0, c8 = 0;
    enum { kFirst, kEval, kBounds, kChunks } step = kEval;
    int level = 1;        // chunks per bit of the next bounds
    unsigned keep = ~0u;  // bits that the level above lets through
    for (;;) {
        if (step == kEval) {
            int pend = pass < 0 && first0 ? 0 : -1;  // chunk to evaluate: first chunk 0, then the queue's
            while (pend < 0 && ((cur & 0xffu) || fill >> 16)) {
                if (!(cur & 0xffu)) {
                    cur = queue[(fill % kQueue) * NT];
                    fill -= 0xffffu;  // one entry fewer, the next place
                }
                const int c = (int)(cur >> 8) * 8 + __ffs((int)cur) - 1;
                cur &= cur - 1;
                if (bnd.reaches<LOW>(s1[c], (float)(M * c) + bnd.w_first(1), bnd.rs + c, 1, F)) pend = c;
            }
            __syncwarp();
            if (pend >= 0) {
                float Bc[M];
                const bool staged = M * pend < kTabWidths || (LOW && nch <= kSpsEveryMost);
                eval_chunk(pb + M * pend, staged ? tab + 8 * pend : reinterpret_cast<const float4*>(gtab) + 8 * pend,
                           staged ? pend & 7 : 0, base, Bc);
                float low = FLT_MAX;  // smallest B over the valid starts (none: the floor is above every bound)
#pragma unroll
                for (int i = 0; i < M; ++i) {
                    if (Bc[i] > B[i]) {  // strict: an equal later chunk keeps the earlier one
                        B[i] = Bc[i];
                        C[i / 2] = __byte_perm(C[i / 2], (uint32_t)pend, i & 1 ? 0x5410 : 0x3254);
                    }
                    low = fminf(low, base[i] < kBig ? B[i] : FLT_MAX);
                }
                F = fmaxf(F, low - bnd.S);
                ++evaluated;
            }
            if (__any_sync(0xffffffffu, last ? (cur & 0xffu) || fill >> 16 : fill >> 16 == kQueue)) continue;
            if (last) break;
            step = pass < 0 ? kFirst : kBounds;
        }
        if (step == kFirst) {  // a pass begins: chunks 1-7, groups of 8 up to 63, groups of 64 up to 511, side by side
            ++pass;
            in = m8 = m64 = 0;
            const float w1 = bnd.w_first(1), w8 = bnd.w_first(8), w64 = bnd.w_first(64);
#pragma unroll
            for (int k = 1; k < 8; ++k) in |= bnd.reaches<LOW>(s1[k], w1 + M * k, bnd.rs + k, 1, F) ? 1u << k : 0u;
            if (nch > 8) {
#pragma unroll
                for (int k = 1; k < 8; ++k) m8 |= bnd.reaches<LOW>(s8[8 * k], w8 + M * 8 * k, bnd.rs + 8 * k, 8, F) ? 1u << k : 0u;
            }
            if (nch > 64) {
#pragma unroll
                for (int k = 1; k < 8; ++k) m64 |= bnd.reaches<LOW>(s64[64 * k], w64 + M * 64 * k, bnd.rs + 64 * k, 64, F) ? 1u << k : 0u;
            }
            in &= nch < 8 ? (1u << nch) - 1 : ~0u;
            m8 &= nch < 64 ? (1u << ((nch + 7) >> 3)) - 1 : ~0u;
            m64 &= nch < 512 ? (1u << ((nch + 63) >> 6)) - 1 : ~0u;
            u8 = __reduce_or_sync(0xffffffffu, m8);
            u64 = __reduce_or_sync(0xffffffffu, m64);
            c512 = c64 = c8 = 0;
            step = kChunks;
        } else if (step == kBounds) {
            // bit k: chunks c + n k .. c + n k + n - 1 (below nch) can reach the floor
            const int c0 = level == 1 ? c8 : level == 8 ? c64 : c512;
            const float* q = (level == 1 ? s1 : level == 8 ? s8 : s64) + c0;
            const float* r = bnd.rs + c0;
            const int have = min(8, (nch - c0 + level - 1) / level);  // groups below nch
            const float w0 = (float)(M * c0) + bnd.w_first(level), dw = (float)(M * level);
            unsigned m = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int o = level * min(k, have - 1);
                m |= bnd.reaches<LOW>(q[o], fmaf(dw, (float)k, w0), r + o, level, F) ? 1u << k : 0u;
            }
            m &= keep & ((1u << have) - 1);
            if (level == 64) {
                m64 = m;
                u64 = __reduce_or_sync(0xffffffffu, m);
            } else if (level == 8) {
                m8 = m;
                u8 = __reduce_or_sync(0xffffffffu, m);
            } else {
                in = m;
                step = kChunks;
            }
        }
        if (step == kChunks) {  // chunks c8 + k of the bits set in `in`
            if (lmask) in &= lmask[c8 >> 5] >> (c8 & 31);
            if (__any_sync(0xffffffffu, in)) {
                found = true;
                if (pass == 0) {
                    if (!lmask) {  // (on the sparse ladder the window behind the bound may not take part)
#pragma unroll
                        for (int k = 0; k < 8; ++k)
                            if (((in >> k) & 1u) && M * (c8 + k) + 31 <= max_width)
                                F = fmaxf(F, bnd.lower(Q[t + c8 + k + 1], c8 + k) - bnd.S);
                    }
                } else if (in) {
                    queue[((fill + (fill >> 16)) % kQueue) * NT] = (uint16_t)(c8 << 5 | in);
                    fill += 0x10000u;
                }
            }
        }
        step = kBounds;
        if (u8) {
            const int g = __ffs((int)u8) - 1;
            u8 &= u8 - 1;
            c8 = c64 + 8 * g;
            level = 1;
            keep = (m8 >> g) & 1u ? ~0u : 0u;
        } else if (u64) {
            const int g = __ffs((int)u64) - 1;
            u64 &= u64 - 1;
            c64 = c512 + 64 * g;
            level = 8;
            keep = (m64 >> g) & 1u ? ~0u : 0u;
        } else if (c512 + 512 < nch) {
            c512 += 512;
            level = 64;
            keep = ~0u;
        } else if (pass == 0 && found) {
            step = kFirst;
        } else {
            last = true;
        }
        if (__any_sync(0xffffffffu, last || fill >> 16 == kQueue)) step = kEval;
    }
    return evaluated;
}

// Every width in order (the decimated ladder's level 0: few widths, all in
// `tab`).  C[i] receives w0 of the first chunk reaching B[i].
__device__ __forceinline__ void boxcar_prefix(const float* __restrict__ P, const float2* __restrict__ tab, int wpad,
                                              const float (&base)[M], float (&B)[M], int (&C)[M]) {
    const float* pb = P + M * threadIdx.x;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        B[i] = -FLT_MAX;
        C[i] = 0;
    }
    for (int w0 = 0; w0 < wpad; w0 += M) {
        float Bc[M];
        eval_chunk(pb + w0, reinterpret_cast<const float4*>(tab + w0), 0, base, Bc);
#pragma unroll
        for (int i = 0; i < M; ++i) {
            if (Bc[i] > B[i]) {
                B[i] = Bc[i];
                C[i] = w0;
            }
        }
    }
}

// Exact int64 running sums for slot i, for tiles whose partial sums may
// exceed 2^24.  Same SNR arithmetic as boxcar_fast (fmaf of the correctly
// rounded sum).
__device__ __noinline__ float boxcar_exact_slot(const float* __restrict__ ys,
                                                const float2* __restrict__ tab, int wpad, int i,
                                                const uint32_t* lmask) {
    const float* yb = ys + M * threadIdx.x + i;
    long long S = 0;
    float best = -FLT_MAX;
    for (int w = 1; w <= wpad; ++w) {
        const float v = yb[w - 1];
        if (v < kSentinelTest) break;  // window left [0, L): later widths invalid too
        S += (long long)v;
        if (lmask && !ladder_has(lmask, w)) continue;
        const float2 rc = tab[w - 1];
        best = fmaxf(best, fmaf(__ll2float_rn(S), rc.x, rc.y));
    }
    return best;
}

// Shared memory: the series, the table's first widths, the block maxima (in
// their place, once they are done with, B(t) where it is written out, then the
// candidate entries: at most every second start is a peak), the next tile's
// new samples, the bounds' factors, the ladder's mask.
__host__ __device__ constexpr int sps_lists_words(int wpad) {
    const int q = 4 * sps_q16(wpad) + (int)kQueue * NT / 2;  // and the search's queues
    return q > 2 * kSpsTile ? q : 2 * kSpsTile;
}

// One CTA's work: tiles [tile_lo, tile_hi) of series `row`, in order.  `sm`
// is the dynamic shared memory; the caller guarantees that every thread has
// finished any previous work.
//
// Consecutive tiles of a series overlap by ylen - kSpsOwned staged samples
// (the W-sample halo), so after the first tile the staged prefix sums are
// slid down by kSpsOwned and only the kSpsOwned new samples are staged and
// summed, continuing from the exact sum at the old end.  Prefix sums are then
// relative to the first fully staged tile; sliding is allowed while every
// staged prefix sum lies within +-2^23 (so every window sum, a difference of
// two, is an exact FP32 integer); otherwise the tile is staged afresh.  The new
// samples are copied to shared memory (cp.async) while the previous tile's
// widths are searched.
//
// With 16 warps an SM (128 registers: a thread's starts, their B, the window of
// a chunk) the tile's chain of short phases is what takes the time (issue 50 %,
// no pipe above 50 %), so the phases are kept few and their barriers fewer.  4096
// channels x 2^20 samples, W = 8192, 2.3e9 starts, 20 M candidates: 30.6 ms (bounds
// of 128-width segments for a whole warp: 80.9).
template <bool LOW>
__device__ __forceinline__ void boxcar_block(const SpsArgs& a, int row, int64_t tile_lo, int64_t tile_hi,
                                             float* sm) {
    constexpr int NW = NT / 32;
    __shared__ int scratch[3 * NW];
    __shared__ float s_edge[2 * NW];  // B of each warp's first and last start
    __shared__ int s_cnt[NW];
    __shared__ unsigned long long s_base;
    __shared__ int s_pend;  // exact prefix sum just past the staged series (while sliding)
    const int wpad = a.wpad;
    const int ylen = kSpsTile + wpad + M;
    float* ys = sm;
    const int wtab = sps_tab_smem(wpad, LOW);
    float4* tab = reinterpret_cast<float4*>(sm + ylen);
    float* lists = sm + ylen + 2 * wtab;
    float* Q = lists;  // block maxima and their sliding maxima, nq each
    const int nq = sps_q16(wpad);
    float* nbuf = lists + sps_lists_words(wpad);  // the next tile's new samples
    float* rs = nbuf + kSpsTile;
    uint32_t* s_ladder = reinterpret_cast<uint32_t*>(rs + sps_rs(wpad));
    const uint32_t* lmask = a.ladder_g16 > 0 ? s_ladder : nullptr;
    if (lmask) fill_ladder(s_ladder, wpad / M, a.ladder_g16);  // visible after the staging barrier
    const int64_t L = a.length;
    const float* y = a.dd + (int64_t)row * a.pitch;
    const RowStats st = a.stats[row];
    const float m0 = st.m0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const float2* gtab = a.table + (int64_t)row * wpad;
    // entry of width w (the candidates' widths read single ones)
    auto entry = [&](int w) {
        if (w > wtab) return __ldg(gtab + w - 1);
        const int c = (w - 1) / M, e = (w - 1) % M;
        return reinterpret_cast<const float2*>(tab + tab_block(c, e >> 1))[e & 1];
    };
    WidthBounds bnd;
    bnd.rs = rs;
    bnd.f = (float)(st.mu - (double)m0);
    {   // the table's first widths, staged once for all tiles, and the bounds' factors
        const float4* g4 = reinterpret_cast<const float4*>(gtab);
        for (int i = threadIdx.x; i < wtab / 2; i += NT) tab[tab_block(i >> 3, i & 7)] = __ldg(g4 + i);
        const float inv = (float)st.inv_sigma;
        for (int c = threadIdx.x; c < sps_rs(wpad); c += NT) rs[c] = inv * (rsqrtf((float)(M * c + 1)) * (1.0f + 1.02e-4f));
        // 1.02e-4, and 2.1e-6 of the largest drift over sigma sqrt(w) (w f r <= |f| 2 sqrt(W + 64 M) / sigma)
        bnd.S = 1.02e-4f + 2.1e-6f * inv * sqrtf((float)(wpad + 64 * M));
    }
    // B(t) of every start asked for: only the running B prunes
    const float cut = a.prune && a.threshold > 0.0f ? a.threshold - 1e-3f : -FLT_MAX;
    constexpr int kBatch = 8;
    constexpr int kSlideMax = 1 << 23;
    bool slide = false;  // ys holds the previous tile's prefix sums, all within +-2^23

    for (int64_t tile = tile_lo; tile < tile_hi; ++tile) {
        const int64_t t0 = tile * kSpsOwned;
        // valid start/sample positions: i in [va, vb]  (t = t0-1+i in [0, L))
        const int va = t0 == 0 ? 1 : 0;
        const int vb = (int)min((int64_t)ylen - 1, L - t0);
        const int nkeep = ylen - kSpsOwned;  // staged samples shared with the previous tile
        bool fast = false;
        if (slide) {
            // slide P down by kSpsOwned: rounds of NT x 16 pairs, all loads of a
            // round before its stores (a round's source and destination overlap;
            // a later round's source never meets an earlier round's destination)
            constexpr int kR = 16;
            static_assert(kSpsOwned % 2 == 0, "pairs");
            for (int r0 = 0; r0 < nkeep / 2; r0 += NT * kR) {
                float2 v[kR];
#pragma unroll
                for (int u = 0; u < kR; ++u) {
                    const int i = r0 + u * NT + threadIdx.x;
                    if (i < nkeep / 2) v[u] = *reinterpret_cast<const float2*>(ys + 2 * i + kSpsOwned);
                }
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncthreads();  // (after the last round: the new samples have arrived too)
#pragma unroll
                for (int u = 0; u < kR; ++u) {
                    const int i = r0 + u * NT + threadIdx.x;
                    if (i < nkeep / 2) *reinterpret_cast<float2*>(ys + 2 * i) = v[u];
                }
            }
            // exact sums of the new samples, continuing from the old end
            const int segn = ((kSpsOwned + NT - 1) / NT) | 1;  // odd: distinct banks
            const int j0 = min(kSpsOwned, (int)threadIdx.x * segn), j1 = min(kSpsOwned, j0 + segn);
            const int jv = vb + 1 - nkeep;  // new samples below the series' end
            int run = 0, mn = 0, mx = 0;
            for (int j = j0; j < j1; ++j) {
                const float v = nbuf[j] - m0;
                if (j < jv && v > kSentinelTest) {
                    run += (int)v;
                    mn = min(mn, run);
                    mx = max(mx, run);
                }
            }
            int tot, ex, gmn, gmx;
            const int pend = s_pend;
            block_scan_minmax<NT>(run, mn, mx, scratch, ex, tot, gmn, gmx);
            fast = (long long)gmn + pend >= -kSlideMax && (long long)gmx + pend <= kSlideMax;
            if (fast) {
                float runf = (float)(pend + ex);
                for (int j = j0; j < j1; ++j) {
                    const float v = nbuf[j] - m0;
                    ys[nkeep + j] = j > jv ? -kBig : runf;
                    if (j < jv && v > kSentinelTest) runf += v;
                }
                // (the reads of s_pend above precede the scan's barrier)
                if (threadIdx.x == 0) s_pend = pend + tot;
            }
            __syncthreads();
        }
        if (!fast) {
            // stage every sample afresh (minus m0, sentinel outside [0, L)); loads in
            // batches so that latencies overlap
            for (int i0b = threadIdx.x; i0b < ylen; i0b += NT * kBatch) {
                float v[kBatch];
#pragma unroll
                for (int u = 0; u < kBatch; ++u) {
                    const int i = i0b + u * NT;
                    const int64_t t = t0 - 1 + i;
                    v[u] = (i < ylen && t >= 0 && t < L) ? __ldg(y + t) - m0 : kSentinel;
                }
#pragma unroll
                for (int u = 0; u < kBatch; ++u)
                    if (i0b + u * NT < ylen) ys[i0b + u * NT] = v[u];
            }
            __syncthreads();

            // Largest |partial sum| of the tile = range of the prefix sums of ys over
            // its valid samples: FP32 sums are exact when it is <= 2^24.
            const int seg = ((ylen + NT - 1) / NT) | 1;  // odd: the threads' segments fall on distinct banks
            const int i0 = min(ylen, (int)threadIdx.x * seg), i1 = min(ylen, i0 + seg);
            int run = 0, mn = 0, mx = 0;
            for (int i = i0; i < i1; ++i) {
                const float v = ys[i];
                if (v > kSentinelTest) {
                    run += (int)v;
                    mn = min(mn, run);
                    mx = max(mx, run);
                }
            }
            int tot, before, gmn, gmx;
            block_scan_minmax<NT>(run, mn, mx, scratch, before, tot, gmn, gmx);
            fast = (long long)gmx - gmn <= (1 << 24);
            slide = gmn >= -kSlideMax && gmx <= kSlideMax;  // the next tile may slide
            if (fast) {
                // ys -> prefix sums P, in place (exact FP32 integers)
                float runf = (float)before;
                for (int i = i0; i < i1; ++i) {
                    const float v = ys[i];
                    ys[i] = i > vb + 1 ? -kBig : runf;
                    if (v > kSentinelTest) runf += v;
                }
                if (threadIdx.x == 0) s_pend = tot;
                __syncthreads();
            }
        }
        slide = slide && fast && (tile + 1 < tile_hi);
        if (slide) {  // the next tile's new samples, copied while this one is searched
            const int64_t tn = t0 + kSpsOwned - 1 + nkeep;
#pragma unroll 4
            for (int j = threadIdx.x; j < kSpsOwned; j += NT) {
                const int64_t t = tn + j;
                const unsigned dst = (unsigned)__cvta_generic_to_shared(nbuf + j);
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(y + min(t, L - 1)), "r"(t < L ? 4 : 0)
                             : "memory");
            }
        }

        float B[M];
        uint32_t C[M / 2];  // the first width chunk reaching B, 16 bits a slot (0 on the exact path)
        if (fast) {
            const float* P = ys;
            float base[M];
            // block maxima, a thread per block of 16 (those past the staged series
            // hold no end), and the sliding maxima over 2, 9 and 65 of them
            {
                float m = -FLT_MAX;
#pragma unroll
                for (int k = 0; k < M; k += 4) {
                    const float4 v = *reinterpret_cast<const float4*>(P + M * threadIdx.x + k);
                    base[k] = v.x; base[k + 1] = v.y; base[k + 2] = v.z; base[k + 3] = v.w;
                    m = max3f(max3f(m, v.x, v.y), v.z, v.w);
                }
                Q[threadIdx.x] = m;
                for (int j = threadIdx.x + NT; j < nq; j += NT) {
                    m = -kBig;
                    if (M * j < ylen) {  // ylen is a multiple of M
#pragma unroll
                        for (int k = 0; k < M; k += 4) {
                            const float4 v = *reinterpret_cast<const float4*>(P + M * j + k);
                            m = max3f(max3f(m, v.x, v.y), v.z, v.w);
                        }
                    }
                    Q[j] = m;
                }
            }
            float pmin = FLT_MAX, pmax = -FLT_MAX;
#pragma unroll
            for (int i = 0; i < M; ++i) {
                const int p = M * threadIdx.x + i;
                const bool valid = p >= va && p <= vb;
                if (valid) {
                    pmin = fminf(pmin, base[i]);
                    pmax = fmaxf(pmax, base[i]);
                } else {
                    base[i] = kBig;
                }
            }
            bnd.pmin = pmin;
            bnd.pmax = pmax;
            __syncthreads();
            const bool bounds = wpad > M && !(LOW && wpad <= a.every * M);  // boxcar_search looks at them
            if (bounds) {
                for (int j = threadIdx.x; j < nq; j += NT) {
                    const float a1 = fmaxf(Q[j], j + 1 < nq ? Q[j + 1] : -kBig);
                    float m = a1;
#pragma unroll
                    for (int k = 2; k < 9; ++k)
                        if (j + k < nq) m = fmaxf(m, Q[j + k]);
                    Q[nq + j] = a1;
                    Q[2 * nq + j] = m;
                }
                __syncthreads();
            }
            if (wpad > 64 * M) {
                for (int j = threadIdx.x; j < nq; j += NT) {
                    float m = Q[2 * nq + j];
#pragma unroll
                    for (int k = 8; k < 64; k += 8)
                        if (j + k < nq) m = fmaxf(m, Q[2 * nq + j + k]);
                    Q[3 * nq + j] = m;
                }
                __syncthreads();
            }
            int chunks = boxcar_search<LOW>(P, tab, gtab, wpad / M, a.max_width, base, bnd, Q, nq,
                                            reinterpret_cast<uint16_t*>(Q + 4 * nq) + threadIdx.x, cut, lmask, a.every, B, C);
            if (a.evaluated) {
                chunks = __reduce_add_sync(0xffffffffu, chunks);
                if (lane == 0) atomicAdd(a.evaluated, (unsigned long long)chunks * M * M);
            }
        } else {
#pragma unroll
            for (int i = 0; i < M; ++i) {
                B[i] = boxcar_exact_slot(ys, gtab, wpad, i, lmask);
                C[i / 2] = 0;
            }
            if (a.evaluated && threadIdx.x == 0)
                atomicAdd(a.evaluated, (unsigned long long)wpad * NT * M);
        }
        if (lane == 0) s_edge[2 * warp] = B[0];
        if (lane == 31) s_edge[2 * warp + 1] = B[M - 1];
        __syncthreads();  // edges visible; everyone done with the block maxima

        const bool zero_sigma = st.zero_sigma != 0;
        if (a.snr_out) {  // through shared memory, so that consecutive threads write consecutive starts
            float* Bs = lists;
#pragma unroll
            for (int k = 0; k < M; k += 4)
                *reinterpret_cast<float4*>(Bs + M * threadIdx.x + k) = make_float4(B[k], B[k + 1], B[k + 2], B[k + 3]);
            __syncthreads();
            float* dst = a.snr_out + (int64_t)row * a.pitch + t0 - 1;
            const int pe = (int)min((int64_t)kSpsTile - 2, L - t0);  // owned starts below the series' end
            for (int p = 1 + threadIdx.x; p <= pe; p += NT) dst[p] = zero_sigma ? 0.0f : Bs[p];
        }
        // peaks: a start's neighbours are the thread's own, the next thread's or
        // the next warp's
        float left = __shfl_up_sync(0xffffffffu, B[M - 1], 1), right = __shfl_down_sync(0xffffffffu, B[0], 1);
        if (lane == 0 && warp > 0) left = s_edge[2 * warp - 1];
        if (lane == 31 && warp + 1 < NW) right = s_edge[2 * warp + 2];
        unsigned cmask = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int p = M * threadIdx.x + i;
            const float v = B[i], l = i > 0 ? B[i - 1] : left, r = i + 1 < M ? B[i + 1] : right;
            if (p >= 1 && p <= kSpsTile - 2 && p <= vb && v >= a.threshold && v > l && v >= r) cmask |= 1u << i;
        }
        if (zero_sigma) cmask = 0;
        // One atomic per tile: the tile's candidates form one contiguous run in t order.
        const int mine = __popc(cmask);
        int inc = mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) s_cnt[warp] = inc;
        __syncthreads();  // (and Bs has been read)
        int total = 0, off = inc - mine;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            if (w < warp) off += s_cnt[w];
            total += s_cnt[w];
        }
        if (total > 0) {
            // candidate entries: slot p (bits 0-15) | first chunk (bits 16-31), and B
            uint32_t* plist = reinterpret_cast<uint32_t*>(lists);
            float* blist = lists + kSpsTile;
            const uint32_t dm_index = (uint32_t)(a.dm_offset + row);
            if (threadIdx.x == 0) {
                s_base = atomicAdd(a.count, (unsigned long long)total);
                const unsigned long long ci = atomicAdd(a.nchunks, 1ull);
                if (ci < (unsigned long long)a.chunk_cap)
                    a.chunks[ci] = CandChunk{s_base, (uint32_t)total, dm_index, (uint32_t)t0, (uint32_t)a.beam};
            }
#pragma unroll
            for (int i = 0; i < M; ++i)
                if ((cmask >> i) & 1u) {
                    plist[off] = (uint32_t)(M * threadIdx.x + i) | ((i & 1 ? C[i / 2] >> 16 : C[i / 2]) << 16);
                    blist[off] = B[i];
                    ++off;
                }
            __syncthreads();

            auto store = [&](int q, int p, int w) {
                const unsigned long long idx = s_base + (unsigned long long)q;
                if (idx < (unsigned long long)a.capacity) {
                    aa_candidate c;
                    c.dm_index = dm_index;
                    c.t = (uint32_t)(t0 - 1 + p);
                    c.width = (uint16_t)w;
                    c.range = (uint8_t)a.range;
                    c.reserved = (uint8_t)a.beam;
                    c.snr = blist[q];
                    a.cands[idx] = c;
                }
            };
            if (fast) {
                // Width of each candidate: the smallest w reaching B(t) lies in its
                // chunk: half a warp per candidate evaluates the chunk's 16 widths with
                // the search's arithmetic
                const int half = lane >> 4, e = lane & 15;
                for (int q0 = 2 * warp; q0 < total; q0 += 2 * NW) {
                    const int q = q0 + half;
                    bool hit = false;
                    int p = 0, w = 0;
                    if (q < total) {
                        p = (int)(plist[q] & 0xffffu);
                        w = (int)(plist[q] >> 16) * M + e + 1;
                        if (w <= a.max_width) {
                            const float2 rc = entry(w);
                            hit = fmaf(ys[p + w] - ys[p], rc.x, rc.y) == blist[q];
                        }
                    }
                    const unsigned hits = __ballot_sync(0xffffffffu, hit) & (0xffffu << (16 * half));
                    if (hit && lane == __ffs((int)hits) - 1) store(q, p, w);
                }
            } else {
                // exact running sums, widths interleaved over a warp's lanes
                for (int q = warp; q < total; q += NW) {
                    const int p = (int)(plist[q] & 0xffffu);
                    const int wmax = (int)min((int64_t)a.max_width, L - (t0 - 1 + p));
                    const float* yq = ys + p;  // yq[w-1] = y[t+w-1] - m0
                    const float target = blist[q];
                    int bw = 0x7fffffff;
                    long long sum = 0;
                    for (int w0 = 0; w0 < wmax; w0 += 32) {
                        const int w = w0 + lane + 1;
                        long long v = (w <= wmax) ? (long long)yq[w - 1] : 0;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const long long u = __shfl_up_sync(0xffffffffu, v, o);
                            if (lane >= o) v += u;
                        }
                        const long long S = sum + v;
                        sum += __shfl_sync(0xffffffffu, v, 31);
                        if (w <= wmax && (!lmask || ladder_has(lmask, w))) {
                            const float2 rc = entry(w);
                            if (fmaf(__ll2float_rn(S), rc.x, rc.y) == target) bw = w;
                        }
                        bw = __reduce_min_sync(0xffffffffu, bw);
                        if (bw != 0x7fffffff) break;  // widths are visited in increasing order
                    }
                    if (lane == 0) store(q, p, bw);
                }
            }
        }  // total > 0
        __syncthreads();  // the next tile overwrites the series and the lists
    }  // tiles
}

// CTA = seg_tiles consecutive tiles of one series (the last segment of a
// series may be shorter).
// LOW: sps_low.
template <bool LOW>
__global__ void __launch_bounds__(NT, 2) sps_boxcar_kernel(SpsArgs a, int ntiles, int seg_tiles) {
    extern __shared__ __align__(16) float sm[];
    const int nseg = (ntiles + seg_tiles - 1) / seg_tiles;
    const int row = (int)(blockIdx.x / (unsigned)nseg);
    const int64_t lo = (int64_t)(blockIdx.x - (unsigned)row * (unsigned)nseg) * seg_tiles;
    boxcar_block<LOW>(a, row, lo, min((int64_t)ntiles, lo + seg_tiles), sm);
}

constexpr int kMaxDecLevels = 16;

// ------------------------------------------------------------ decimated ladder
// Approximate search for wide boxcars (the cited search evaluates them on the
// series decimated by pairs, Sec. 1).  Level 0: widths 1..min(W0, W) of the
// windows starting at t, evaluated as the exhaustive search's first chunks.
// Level k >= 1 (while W0 2^(k-1) < W): widths w = m 2^k, W0/2 < m <= W0,
// w <= W, of the window starting at the level-k grid point
// s = floor(t / 2^k) 2^k <= t (m samples of the series decimated k times by
// pairs).  Every level comes from the tile's one full-rate prefix sum P:
// S = P[s + w] - P[s], exact.  B(t) = the largest SNR over level 0 at t and
// each level's window at its grid point, levels in increasing width (ties to
// the smallest width); the width of a level-k maximum is known directly, that
// of a level-0 maximum is resolved as in the exhaustive search.
//
// Shared memory: the staged series with a left halo H >= 2^K (a slot's
// level-K grid point lies up to 2^K - 1 samples before it), the compact width
// table (level 0, then W0/2 entries per level), and a region that holds the
// levels' strided prefix sums P_k and grid maxima B_k, then B(t), the
// candidate list and the direct widths.
struct DecLayout {
    int K, H, W0, W0e, wpad0, ylen4, ntab;
    int npk, nbk;             // entries of all levels' P_k and B_k (upper bounds for any tile)
    int tab_off, reg_off;     // in floats
    size_t bytes;
};
__host__ __device__ inline int dec_level_points(int k) { return ((kSpsTile - 1) >> k) + 2; }
__host__ __device__ inline DecLayout dec_layout(int W, int W0) {
    DecLayout d{};
    d.W0 = W0;
    d.K = 0;
    while ((W0 << d.K) < W) ++d.K;
    d.H = d.K > 0 ? ((1 << d.K) > 16 ? (1 << d.K) : 16) : 0;
    d.W0e = W0 < W ? W0 : W;
    d.wpad0 = (d.W0e + M - 1) / M * M;
    d.ylen4 = (d.H + kSpsTile + W + M + 3) & ~3;
    d.ntab = d.wpad0 + d.K * (W0 / 2);
    d.npk = d.nbk = 0;
    for (int k = 1; k <= d.K; ++k) {
        d.nbk += dec_level_points(k);
        d.npk += dec_level_points(k) + W0;
    }
    const int reg_a = d.npk * 4 + d.nbk * 4 + d.nbk;       // P_k, B_k (float), winning m (u8)
    const int reg_b = kSpsTile * 4 + kSpsTile * 4 + kSpsTile * 2;  // B(t), candidates, direct widths
    d.tab_off = d.ylen4;
    d.reg_off = d.tab_off + ((d.ntab * 2 + 3) & ~3);
    d.bytes = (size_t)d.reg_off * 4 + (size_t)(((reg_a > reg_b ? reg_a : reg_b) + 15) & ~15);
    return d;
}

__device__ __forceinline__ void boxcar_dec_block(const SpsArgs& a, int ntiles, int64_t bid, float* sm) {
    __shared__ long long scratch[2 * NT / 32];
    __shared__ unsigned long long s_base;
    __shared__ int s_lvl[2 * kMaxDecLevels + 2];  // per level: P_k offset, B_k offset
    const DecLayout d = dec_layout(a.max_width, a.dec_w0);
    const int W0 = d.W0, K = d.K, H = d.H, ylen = d.ylen4;
    float* ys = sm;
    float2* tab = reinterpret_cast<float2*>(sm + d.tab_off);
    float* reg = sm + d.reg_off;
    const int row = (int)(bid / ntiles);
    const int64_t tile = bid - (int64_t)row * ntiles;
    const int64_t t0 = tile * kSpsOwned;
    const int64_t L = a.length;
    const int64_t o = t0 - 1 - H;  // t of ys[0]
    const float* y = a.dd + (int64_t)row * a.pitch;
    const RowStats st = a.stats[row];
    const float m0 = st.m0;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    // stage the series (minus m0, sentinel outside [0, L)) and the table
    constexpr int kBatch = 8;
    for (int i0b = threadIdx.x; i0b < ylen; i0b += NT * kBatch) {
        float v[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = i0b + u * NT;
            const int64_t t = o + i;
            v[u] = (i < ylen && t >= 0 && t < L) ? __ldg(y + t) - m0 : kSentinel;
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
            if (i0b + u * NT < ylen) ys[i0b + u * NT] = v[u];
    }
    const float2* gtab = a.table + (int64_t)row * a.wpad;
    for (int e = threadIdx.x; e < d.ntab; e += NT) {
        int w;
        if (e < d.wpad0) {
            w = e + 1;
        } else {
            const int k = 1 + (e - d.wpad0) / (W0 / 2);
            w = (W0 / 2 + 1 + (e - d.wpad0) % (W0 / 2)) << k;
        }
        tab[e] = w <= a.max_width ? __ldg(gtab + w - 1) : make_float2(0.0f, -FLT_MAX);
    }
    if (threadIdx.x == 0) {
        int pk = 0, bk = d.npk;
        for (int k = 1; k <= K; ++k) {
            s_lvl[2 * k] = pk;
            s_lvl[2 * k + 1] = bk;
            pk += dec_level_points(k) + W0;
            bk += dec_level_points(k);
        }
    }
    __syncthreads();

    // exact FP32 prefix sums when the tile's partial sums stay within 2^24
    const int seg = ((ylen + NT - 1) / NT) | 1;  // odd: the threads' segments fall on distinct banks
    const int i0 = min(ylen, threadIdx.x * seg), i1 = min(ylen, i0 + seg);
    long long run = 0, mn = 0, mx = 0;
    for (int i = i0; i < i1; ++i) {
        const float v = ys[i];
        if (v > kSentinelTest) {
            run += (long long)(int)v;
            mn = min(mn, run);
            mx = max(mx, run);
        }
    }
    const long long before = block_exclusive_scan<NT>(run, scratch);
    long long gmn = mn + before, gmx = mx + before;
    block_minmax<NT>(gmn, gmx, scratch);
    const bool fast = (gmx - gmn) <= (1ll << 24);
    const int va = (int)max((int64_t)0, -o);                 // ys index of t = 0
    const int vb = (int)min((int64_t)ylen - 1, L - 1 - o);   // ys index of t = L - 1

    float B[M];
    int C[M];  // level 0: w0 of the first width chunk reaching B
    if (fast) {
        __syncthreads();
        float runf = (float)before;
        for (int i = i0; i < i1; ++i) {
            const float v = ys[i];
            ys[i] = i > vb + 1 ? -kBig : runf;
            if (v > kSentinelTest) runf += v;
        }
        __syncthreads();
        const float* P = ys;
        float base[M];
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int q = H + M * threadIdx.x + i;
            base[i] = (q >= va && q <= vb) ? P[q] : kBig;
        }
        boxcar_prefix(P + H, tab, d.wpad0, base, B, C);
        // the levels' strided prefix sums: P_k[i] = P at t = (jk0 + i) 2^k
        for (int k = 1; k <= K; ++k) {
            const int64_t jk0 = (t0 - 1) >> k;
            float* Pk = reg + s_lvl[2 * k];
            const int n = dec_level_points(k) + W0;
            for (int i = threadIdx.x; i < n; i += NT) {
                const int64_t q = (jk0 + i) * ((int64_t)1 << k) - o;  // jk0 may be -1
                Pk[i] = q < ylen ? P[q] : -kBig;
            }
        }
    } else {
#pragma unroll
        for (int i = 0; i < M; ++i) {
            B[i] = boxcar_exact_slot(ys + H, tab, d.wpad0, i, nullptr);
            C[i] = 0;
        }
    }
    __syncthreads();

    // B_k at every grid point of the tile: the best of the level's widths
    int nitems = 0;
    for (int k = 1; k <= K; ++k) nitems += (int)((((t0 + kSpsTile - 2) >> k) - ((t0 - 1) >> k)) + 1);
    for (int it = threadIdx.x; it < nitems; it += NT) {
        int k = 1, jj = it;
        for (;;) {
            const int nk = (int)((((t0 + kSpsTile - 2) >> k) - ((t0 - 1) >> k)) + 1);
            if (jj < nk) break;
            jj -= nk;
            ++k;
        }
        const int64_t j = ((t0 - 1) >> k) + jj;
        const float2* tk = tab + d.wpad0 + (k - 1) * (W0 / 2);
        float best = -FLT_MAX;
        int bm = 0;
        if (j >= 0) {
            if (fast) {
                const float* Pk = reg + s_lvl[2 * k] + jj;
                const float p0 = Pk[0];
                for (int u = 0; u < W0 / 2; ++u) {
                    const float2 rc = tk[u];
                    const float snr = fmaf(Pk[W0 / 2 + 1 + u] - p0, rc.x, rc.y);
                    if (snr > best) { best = snr; bm = u; }
                }
            } else {
                // exact int64 running sums over the window's samples
                const int64_t q0 = (j << k) - o;
                const int step = 1 << k;
                long long S = 0;
                bool ok = true;
                for (int m = 1; m <= W0 && ok; ++m) {
                    for (int r = 0; r < step; ++r) {
                        const int64_t q = q0 + (int64_t)(m - 1) * step + r;
                        const float v = q < ylen ? ys[q] : kSentinel;
                        if (v < kSentinelTest) { ok = false; break; }  // past the series end
                        S += (long long)v;
                    }
                    if (ok && m > W0 / 2) {
                        const float2 rc = tk[m - W0 / 2 - 1];
                        const float snr = fmaf(__ll2float_rn(S), rc.x, rc.y);
                        if (snr > best) { best = snr; bm = m - W0 / 2 - 1; }
                    }
                }
            }
        }
        reg[s_lvl[2 * k + 1] + jj] = best;
        reinterpret_cast<uint8_t*>(reg + d.npk + d.nbk)[s_lvl[2 * k + 1] - d.npk + jj] = (uint8_t)bm;
    }
    __syncthreads();

    // B(t) = max over level 0 and every level's grid point at or before t
    int wdir[M];  // width of a level maximum (0: level 0)
#pragma unroll
    for (int i = 0; i < M; ++i) wdir[i] = 0;
    const int64_t tf = t0 - 1 + M * (int64_t)threadIdx.x;
    unsigned valid = 0;  // slots with t in [0, L): B is defined there only
#pragma unroll
    for (int i = 0; i < M; ++i)
        if (tf + i >= 0 && tf + i < L) valid |= 1u << i;
    for (int k = 1; k <= K; ++k) {
        const int64_t jk0 = (t0 - 1) >> k;
        const float* Bk = reg + s_lvl[2 * k + 1];
        const uint8_t* Mk = reinterpret_cast<const uint8_t*>(reg + d.npk + d.nbk) + (s_lvl[2 * k + 1] - d.npk);
        int64_t jc = -(1ll << 62);
        float bv = -FLT_MAX;
        int wv = 0;
#pragma unroll
        for (int i = 0; i < M; ++i) {
            const int64_t j = (tf + i) >> k;
            if (j != jc) {
                jc = j;
                bv = Bk[j - jk0];
                wv = (W0 / 2 + 1 + Mk[j - jk0]) << k;
            }
            if (((valid >> i) & 1u) && bv > B[i]) {
                B[i] = bv;
                wdir[i] = wv;
            }
        }
    }
    if (a.evaluated && threadIdx.x == 0)
        atomicAdd(a.evaluated, (unsigned long long)NT * M * d.wpad0 + (unsigned long long)nitems * (W0 / 2));
    __syncthreads();  // everyone done with the level arrays

    float* Bs = reg;                                          // B(t) of every slot
    uint32_t* plist = reinterpret_cast<uint32_t*>(Bs + kSpsTile);  // slot | level-0 chunk << 16
    uint16_t* WS = reinterpret_cast<uint16_t*>(plist + kSpsTile);  // direct widths per slot
#pragma unroll
    for (int i = 0; i < M; ++i) {
        Bs[M * threadIdx.x + i] = B[i];
        WS[M * threadIdx.x + i] = (uint16_t)wdir[i];
    }
    __syncthreads();

    const bool zero_sigma = st.zero_sigma != 0;
    unsigned cmask = 0;
#pragma unroll
    for (int i = 0; i < M; ++i) {
        const int p = M * threadIdx.x + i;
        const int64_t t = t0 - 1 + p;
        if (p >= 1 && p <= kSpsTile - 2 && t < L) {
            const float v = Bs[p];
            if (a.snr_out) a.snr_out[(int64_t)row * a.pitch + t] = zero_sigma ? 0.0f : v;
            if (!zero_sigma && v >= a.threshold && v > Bs[p - 1] && v >= Bs[p + 1]) cmask |= 1u << i;
        }
    }
    long long total = 0;
    const long long my_off = block_exclusive_scan_total<NT>(__popc(cmask), scratch, total);
    if (total == 0) return;
    const uint32_t dm_index = (uint32_t)(a.dm_offset + row);
    if (threadIdx.x == 0) {
        s_base = atomicAdd(a.count, (unsigned long long)total);
        const unsigned long long ci = atomicAdd(a.nchunks, 1ull);
        if (ci < (unsigned long long)a.chunk_cap)
            a.chunks[ci] = CandChunk{s_base, (uint32_t)total, dm_index, (uint32_t)t0, (uint32_t)a.beam};
    }
    {
        int j = (int)my_off;
#pragma unroll
        for (int i = 0; i < M; ++i)
            if ((cmask >> i) & 1u)
                plist[j++] = (uint32_t)(M * threadIdx.x + i) | ((uint32_t)(C[i] / M) << 16);
    }
    __syncthreads();

    // widths: direct for a level maximum; for level 0 the smallest w reaching
    // B(t) within its first chunk, as in the exhaustive search
    for (int q = warp; q < (int)total; q += NT / 32) {
        const int p = (int)(plist[q] & 0xffffu);
        const int cw0 = (int)(plist[q] >> 16) * M;
        const int64_t t = t0 - 1 + p;
        const float target = Bs[p];
        float best = -FLT_MAX;
        int bw = 0x7fffffff;
        if (WS[p] != 0) {
            best = target;
            bw = WS[p];
        } else {
            const int wmax = (int)min((int64_t)d.W0e, L - t);
            if (fast) {
                const float* P = ys + H;
                const float b0 = P[p];
                for (int w0 = cw0; w0 < wmax; w0 += 32) {
                    const int w = w0 + lane + 1;
                    if (w <= wmax) {
                        const float2 rc = __ldg(gtab + w - 1);
                        const float snr = fmaf(P[p + w] - b0, rc.x, rc.y);
                        if (snr > best) { best = snr; bw = w; }
                    }
                    if (__any_sync(0xffffffffu, best == target)) break;
                }
            } else {
                const float* yq = ys + H + p;
                long long base = 0;
                for (int w0 = 0; w0 < wmax; w0 += 32) {
                    const int w = w0 + lane + 1;
                    long long v = (w <= wmax) ? (long long)yq[w - 1] : 0;
#pragma unroll
                    for (int s = 1; s < 32; s <<= 1) {
                        const long long u = __shfl_up_sync(0xffffffffu, v, s);
                        if (lane >= s) v += u;
                    }
                    const long long S = base + v;
                    base += __shfl_sync(0xffffffffu, v, 31);
                    if (w <= wmax) {
                        const float2 rc = __ldg(gtab + w - 1);
                        const float snr = fmaf(__ll2float_rn(S), rc.x, rc.y);
                        if (snr > best) { best = snr; bw = w; }
                    }
                    if (__any_sync(0xffffffffu, best == target)) break;
                }
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                const float ob = __shfl_xor_sync(0xffffffffu, best, s);
                const int ow = __shfl_xor_sync(0xffffffffu, bw, s);
                if (ob > best || (ob == best && ow < bw)) { best = ob; bw = ow; }
            }
        }
        const unsigned long long idx = s_base + (unsigned long long)q;
        if (lane == 0 && idx < (unsigned long long)a.capacity) {
            aa_candidate c;
            c.dm_index = dm_index;
            c.t = (uint32_t)t;
            c.width = (uint16_t)bw;
            c.range = (uint8_t)a.range;
            c.reserved = (uint8_t)a.beam;
            c.snr = best;
            a.cands[idx] = c;
        }
    }
}

__global__ void __launch_bounds__(NT, 2) sps_boxcar_dec_kernel(SpsArgs a, int ntiles) {
    extern __shared__ __align__(16) float sm[];
    boxcar_dec_block(a, ntiles, blockIdx.x, sm);
}

__device__ __forceinline__ int find_desc(const int64_t* first, int n, int64_t item) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= item) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Persistent forms over several beams/ranges (work queues).
__global__ void __launch_bounds__(kStatsThreads) sps_stats_batch_kernel(
    const SpsArgs* __restrict__ descs, const int64_t* __restrict__ first, int ndesc,
    unsigned long long* queue) {
    __shared__ long long s_item;
    const int64_t total = first[ndesc];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(queue, 1ull);
        __syncthreads();
        const int64_t item = s_item;
        if (item >= total) break;
        const int k = find_desc(first, ndesc, item);
        stats_row(descs[k], descs[k].rsqrt_w, (int)(item - first[k]));
    }
}

template <bool LOW>
__global__ void __launch_bounds__(NT, 2) sps_boxcar_batch_kernel(
    const SpsArgs* __restrict__ descs, const int64_t* __restrict__ first,
    const int* __restrict__ ntiles, int ndesc, unsigned long long* queue) {
    extern __shared__ __align__(16) float sm[];
    __shared__ long long s_item;
    const int64_t total = first[ndesc];
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) s_item = (long long)atomicAdd(queue, 1ull);
        __syncthreads();
        const int64_t item = s_item;
        if (item >= total) break;
        const int k = find_desc(first, ndesc, item);
        const int64_t bid = item - first[k];
        if (descs[k].dec_w0 > 0) {
            boxcar_dec_block(descs[k], ntiles[k], bid, sm);
        } else {
            const int row = (int)(bid / ntiles[k]);
            const int64_t tile = bid - (int64_t)row * ntiles[k];
            boxcar_block<LOW>(descs[k], row, tile, tile + 1, sm);
        }
    }
}

}  // namespace

cudaError_t launch_sps_stats(const SpsArgs& a, cudaStream_t s) {
    if (a.nrows <= 0) return cudaSuccess;
    sps_stats_kernel<<<a.nrows, kStatsThreads, 0, s>>>(a, a.rsqrt_w);
    return cudaGetLastError();
}

cudaError_t launch_sps_finalize(const SpsArgs& a, const unsigned long long* acc, cudaStream_t s) {
    if (a.nrows <= 0) return cudaSuccess;
    sps_finalize_kernel<<<a.nrows, 256, 0, s>>>(a, a.rsqrt_w, acc);
    return cudaGetLastError();
}

namespace {
// One CTA per run; 16-byte records copied as uint4.
__global__ void __launch_bounds__(256) gather_runs_kernel(const uint4* __restrict__ in,
                                                          uint4* __restrict__ out,
                                                          const RunCopy* __restrict__ runs,
                                                          int64_t nruns) {
    for (int64_t r = blockIdx.x; r < nruns; r += gridDim.x) {
        const RunCopy rc = runs[r];
        for (int64_t k = threadIdx.x; k < rc.n; k += blockDim.x) out[rc.dst + k] = in[rc.src + k];
    }
}
}  // namespace

cudaError_t launch_gather_runs(const aa_candidate* d_in, aa_candidate* d_out, const RunCopy* d_runs,
                               int64_t nruns, cudaStream_t s) {
    if (nruns <= 0) return cudaSuccess;
    static_assert(sizeof(aa_candidate) == sizeof(uint4), "candidate records are 16 bytes");
    const unsigned grid = (unsigned)std::min<int64_t>(nruns, 152 * 16);
    gather_runs_kernel<<<grid, 256, 0, s>>>(reinterpret_cast<const uint4*>(d_in),
                                            reinterpret_cast<uint4*>(d_out), d_runs, nruns);
    return cudaGetLastError();
}

cudaError_t launch_rsqrt_table(double* t, int wpad, cudaStream_t s) {
    rsqrt_table_kernel<<<(wpad + 255) / 256, 256, 0, s>>>(t, wpad);
    return cudaGetLastError();
}

size_t sps_boxcar_smem(int wpad) {
    const int ylen = kSpsTile + wpad + M;
    return ((size_t)ylen + 2 * sps_tab_smem(wpad, true) + sps_lists_words(wpad) + kSpsTile + sps_rs(wpad) + ladder_words(wpad)) * 4;
}

int g_boxcar_seg_tiles = 0;

size_t sps_boxcar_smem_for(int32_t max_width, int32_t wpad, int32_t dec_w0) {
    if (dec_w0 > 0) return dec_layout(max_width, dec_w0).bytes;
    // The exhaustive search takes the widths whose series, whole width table
    // (or B(t) and the candidate entries in its place) and 128-sample block
    // maxima fit a CTA; the kernel itself holds less.
    const size_t ylen = (size_t)kSpsTile + wpad + M;
    const size_t full = ylen * 4 + std::max((size_t)wpad * 8, (size_t)kSpsTile * 8) + ((ylen + 127) / 128 + 3) / 4 * 16 +
                        (size_t)ladder_words(wpad) * 4;
    return full > kMaxBoxcarSmem ? full : sps_boxcar_smem(wpad);
}

cudaError_t launch_sps_boxcar(const SpsArgs& a, cudaStream_t s) {
    if (a.nrows <= 0 || a.length <= 0) return cudaSuccess;
    const int64_t ntiles = (a.length + kSpsOwned - 1) / kSpsOwned;
    const int64_t nblocks = ntiles * a.nrows;
    if (nblocks >= (1ll << 31)) return cudaErrorInvalidConfiguration;
    const size_t smem = sps_boxcar_smem_for(a.max_width, a.wpad, a.dec_w0);
    if (smem > kMaxBoxcarSmem) return cudaErrorInvalidConfiguration;
    if (a.dec_w0 > 0) {
        cudaError_t e = allow_smem((const void*)sps_boxcar_dec_kernel);
        if (e != cudaSuccess) return e;
        sps_boxcar_dec_kernel<<<(unsigned)nblocks, NT, smem, s>>>(a, (int)ntiles);
        return cudaGetLastError();
    }
    // tiles per CTA: up to 16 (sharing the staged halo), keeping at least
    // 16 CTAs per resident CTA slot (2 per SM)
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 1;
    const int seg = g_boxcar_seg_tiles > 0
                        ? (int)std::min<int64_t>(g_boxcar_seg_tiles, ntiles)
                        : (int)std::max<int64_t>(1, std::min<int64_t>({16, ntiles, nblocks / (sms * 2 * 16)}));
    const int64_t ncta = (int64_t)a.nrows * ((ntiles + seg - 1) / seg);
    // Chunks up to which B(t) of every start is found by evaluating all widths in
    // turn: noise leaves over a third of them to evaluate and the bounds cost more
    // (96 series of 64006 samples, W = 256 / 1024 / 2048: in turn 220 / 752 / 1449
    // us, by bounds 307 / 802 / 1084).  With one CTA an SM or fewer the bounds'
    // chain of steps is what takes the time, and in noise more widths are faster
    // in turn (4 series of 40000 samples, W = 1100 / 2048: in turn 98 / 164 us, by
    // bounds 150 / 191; with two CTAs an SM, 96 series of 12000, W = 1100: 163 and
    // 185), short series apart, most of whose windows do not exist (16 of 3000,
    // W = 2048: 157 both, with a pulse 161 and 45).
    SpsArgs b = a;
    const bool whole = a.length >= kSpsTile + a.max_width;
    b.every = ncta > (whole ? 2 * sms : sms) ? kSpsEvery : ncta > sms ? kSpsEvery * 5 / 4 : whole ? kSpsEveryMost : kSpsEvery * 3 / 2;
    auto kern = sps_low(a) ? sps_boxcar_kernel<true> : sps_boxcar_kernel<false>;
    cudaError_t e = allow_smem((const void*)kern);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)ncta, NT, smem, s>>>(b, (int)ntiles, seg);
    return cudaGetLastError();
}


}  // namespace aa

namespace aa {

cudaError_t launch_sps_stats_batch(const SpsArgs* d_descs, const int64_t* d_first, int ndesc,
                                   unsigned long long* d_queue, int grid, cudaStream_t s) {
    if (ndesc <= 0) return cudaSuccess;
    sps_stats_batch_kernel<<<grid, kStatsThreads, 0, s>>>(d_descs, d_first, ndesc, d_queue);
    return cudaGetLastError();
}

cudaError_t launch_sps_boxcar_batch(const SpsArgs* d_descs, const int64_t* d_first,
                                    const int* d_ntiles, int ndesc, size_t smem,
                                    bool low, unsigned long long* d_queue, int grid, cudaStream_t s) {
    if (ndesc <= 0) return cudaSuccess;
    if (smem > kMaxBoxcarSmem) return cudaErrorInvalidConfiguration;
    auto kern = low ? sps_boxcar_batch_kernel<true> : sps_boxcar_batch_kernel<false>;
    cudaError_t e = allow_smem((const void*)kern);
    if (e != cudaSuccess) return e;
    kern<<<grid, NT, smem, s>>>(d_descs, d_first, d_ntiles, ndesc, d_queue);
    return cudaGetLastError();
}

int sps_boxcar_tiles(int64_t length) { return (int)((length + kSpsOwned - 1) / kSpsOwned); }

}  // namespace aa
