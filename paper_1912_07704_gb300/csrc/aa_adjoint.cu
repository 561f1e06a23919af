// Differentiable form of the dedispersion (per-channel float weights):
//   forward  y[d][t]  = sum_c w[c] x[c][t + s(c,d)]              (FP32 FMA)
//   adjoint  gx[c][u] = w[c] A[c][u],  A[c][u] = sum_d gy[d][u - s(c,d)]
//            gw[c]    = sum_u x[c][u] A[c][u]       (= sum_{d,t} gy[d][t] x[c][t+s(c,d)])
// The MSE loss against a template, mean((y - T)^2), is reduced inside the
// forward; its gradient recomputes y one chunk of DM trials at a time (the
// full DM x time residual is never stored).  Dec-1 ranges only.
//
// Both directions are the same gather: a CTA owns kOut outputs rows (trials, or
// channels) x 32 KW samples and goes through the other index (channels, or
// trials) in stages of fc source rows, whose windows arrive in shared memory by
// cp.async while the stage before is added; a warp owns two output rows where a
// lane has 16 samples of each, 32 apart, and one where it has 8.  One
// shared-memory read per multiply-add bounds it (1024 ch x 65536 x 1024 trials:
// 7.8 ms, 6.3 of them reads; half a warp per row, whose halves met in the same
// banks: 14.3).  16-byte copies where rows and base are aligned (VEC), 4-byte ones elsewhere.
#include <algorithm>
#include <cstdint>

#include "aa_internal.h"

namespace aa {
namespace {

constexpr int kOut = 16;      // output rows per CTA
constexpr int kMaxStage = 8;  // source rows per stage

enum { kWriteY = 0, kLoss = 1, kResidual = 2, kAdjoint = 3 };

struct F32Args {
    const float* src;    // source rows
    int64_t src_pitch;
    int32_t nsrc;        // source rows: row r is index src0 + r of the shift table
    int32_t src0;
    int64_t src_len;     // source samples [0, src_len) count, others are zero
    const int32_t* shifts;  // [ndm][nchans] of the range
    int32_t nchans;
    int32_t out_begin, out_end;  // output rows (trials, or channels)
    int64_t out_len;
    int32_t rowlen;      // staged floats per source row (multiple of 4)
    int32_t fc;          // source rows per stage
    const float* w;      // [nchans]
    float* y;            // mode kWriteY: row d at y + d*pitch
    int64_t pitch;
    const float* tmpl;   // template, same layout as y (modes kLoss, kResidual)
    double* loss_sum;    // modes kLoss, kResidual
    float* resid;        // mode kResidual: row (d - out_begin) at resid + (d-out_begin)*rpitch
    int64_t rpitch;
    float scale;         // residual scale (2/N)
    const float* x;      // mode kAdjoint: the forward's input, for gw
    int64_t x_pitch;
    float* gx;           // [nchans][x_pitch], accumulated
    float* gw_part;      // [nchans][ntiles], overwritten
};

__device__ __forceinline__ void cp_async16(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async4(float* dst, const float* src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}

// With 8 samples a lane CTAs are few: a warp per output row instead of one per
// two (twice the warps to hide a stage's chain of short steps behind), and more
// stages in flight.
__host__ __device__ constexpr int f32_stages(int kw) { return kw == 16 ? 2 : 4; }
__host__ __device__ constexpr int f32_rows(int kw) { return kw == 16 ? 2 : 1; }  // output rows per warp
__host__ __device__ constexpr int f32_threads(int kw) { return 32 * kOut / f32_rows(kw); }

template <int MODE, int KW, bool VEC>
__global__ void __launch_bounds__(f32_threads(KW)) f32_gather_kernel(F32Args a, int ntiles) {
    constexpr bool ADJ = MODE == kAdjoint;
    constexpr int T = 32 * KW, NS = f32_stages(KW), NO = NS + 1, R = f32_rows(KW), NTH = f32_threads(KW);
    extern __shared__ __align__(16) float fsm[];  // [NS][fc][rowlen]
    // of stage k in [k % NO]: k + NS - 1 is written while a slow warp still adds k - 1
    __shared__ int64_t s_base[NO][kMaxStage];        // first staged sample of each source row (multiple of 4 when VEC)
    __shared__ __align__(8) int s_off[NO][kMaxStage][kOut];  // word of each output row's first sample
    __shared__ float s_w[NO][kMaxStage];
    __shared__ double red[NTH / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tile = blockIdx.x % ntiles;
    const int o0 = a.out_begin + (int)(blockIdx.x / ntiles) * kOut;
    const int olast = min(a.out_end, o0 + kOut) - 1;
    const int64_t t0 = (int64_t)tile * T;
    const int fc = a.fc, nstage = (a.nsrc + fc - 1) / fc;

    // Thread (o, f) < 16 fc holds the delays of output row o0 + o and source row
    // f of the stage to come: its own, and the one that the row's window starts
    // at (forward: the first trial's, the smallest; adjoint: the larger of the
    // CTA's first and last channels', delays being monotone in the channel).
    const int po = tid / fc, pf = tid - po * fc;
    const bool owner = tid < kOut * fc;
    int own = 0, ref = 0;
    float pw = 0.0f;
    auto delay = [&](int o, int r) {
        const int64_t d = ADJ ? a.src0 + r : o, c = ADJ ? o : a.src0 + r;
        return __ldg(&a.shifts[d * a.nchans + c]);
    };
    auto prefetch = [&](int k) {
        const int r = k * fc + pf;
        own = ref = 0;
        pw = 0.0f;
        if (owner && r < a.nsrc) {
            own = delay(min(o0 + po, olast), r);
            ref = ADJ ? max(delay(o0, r), delay(olast, r)) : delay(o0, r);
            if (!ADJ) pw = __ldg(&a.w[a.src0 + r]);
        }
    };
    auto publish = [&](int k) {
        const int b = k % NO;
        if (owner) {
            const int64_t first = ADJ ? t0 - ref : t0 + ref;
            const int64_t base = VEC ? first & ~(int64_t)3 : first;  // (also below zero: rounds down)
            const int off = (int)((ADJ ? t0 - own : t0 + own) - base);
            s_off[b][pf][po] = off;
            if (po == 0) {
                s_base[b][pf] = base;
                if (!ADJ) s_w[b][pf] = pw;
            }
        }
    };
    // the windows of stage k into its buffer, one or more warps a row; what lies
    // outside [0, src_len) is zero
    const int parts = NTH / 32 / fc, cf = warp % fc, cpart = warp / fc;
    auto copy = [&](int k) {
        const int r = k * fc + cf;
        const int64_t base = s_base[k % NO][cf];
        const float* row = a.src + (int64_t)min(r, a.nsrc - 1) * a.src_pitch;
        const int64_t len = r < a.nsrc ? a.src_len : 0;
        float* dst = fsm + ((size_t)(k % NS) * fc + cf) * a.rowlen;
        if constexpr (VEC) {
            for (int j = 4 * (lane + 32 * cpart); j < a.rowlen; j += 128 * parts) {
                const int64_t u = base + j;
                const int n = u < 0 ? 0 : (int)max((int64_t)0, min((int64_t)4, len - u));
                cp_async16(dst + j, n ? row + u : row, 4 * n);
            }
        } else {
            for (int j = lane + 32 * cpart; j < a.rowlen; j += 32 * parts) {
                const int64_t u = base + j;
                const bool in = u >= 0 && u < len;
                cp_async4(dst + j, in ? row + u : row, in ? 4 : 0);
            }
        }
    };

    float acc[R][KW];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
        for (int q = 0; q < KW; ++q) acc[i][q] = 0.0f;
    for (int k = 0; k < NS - 1 && k < nstage; ++k) {
        prefetch(k);
        publish(k);
    }
    if (NS - 1 < nstage) prefetch(NS - 1);
    __syncthreads();
    for (int k = 0; k < NS - 1; ++k) {  // (a group per stage, empty past the last)
        if (k < nstage) copy(k);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int k = 0; k < nstage; ++k) {
        const int kn = k + NS - 1;
        if (kn < nstage) {
            publish(kn);
            if (kn + 1 < nstage) prefetch(kn + 1);
        }
        __syncthreads();  // offsets of stage kn visible; stage k - 1 added by every warp
        if (kn < nstage) copy(kn);
        asm volatile("cp.async.commit_group;" ::: "memory");
        asm volatile("cp.async.wait_group %0;" ::"n"(NS - 1) : "memory");
        __syncthreads();  // stage k complete
        const float* buf = fsm + (size_t)(k % NS) * fc * a.rowlen + lane;
        const int b = k % NO;
#pragma unroll 2
        for (int f = 0; f < fc; ++f) {
            const float wc = ADJ ? 0.0f : s_w[b][f];
            int off[R];
            if constexpr (R == 2) {
                const int2 v = *reinterpret_cast<const int2*>(&s_off[b][f][2 * warp]);
                off[0] = v.x;
                off[1] = v.y;
            } else {
                off[0] = s_off[b][f][warp];
            }
#pragma unroll
            for (int i = 0; i < R; ++i) {
                const float* r = buf + f * a.rowlen + off[i];
#pragma unroll
                for (int q = 0; q < KW; ++q) acc[i][q] = ADJ ? acc[i][q] + r[32 * q] : fmaf(wc, r[32 * q], acc[i][q]);
            }
        }
    }

    double local = 0.0;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int o = o0 + R * warp + i;
        if (o > olast) continue;
        if constexpr (ADJ) {
            const float wc = __ldg(&a.w[o]);
            const float* xr = a.x + (int64_t)o * a.x_pitch;
            float* gr = a.gx + (int64_t)o * a.x_pitch;
            float part = 0.0f;
#pragma unroll
            for (int q = 0; q < KW; ++q) {
                const int64_t u = t0 + lane + 32 * q;
                if (u < a.out_len) {
                    gr[u] += wc * acc[i][q];
                    part = fmaf(__ldg(xr + u), acc[i][q], part);
                }
            }
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) part += __shfl_xor_sync(0xffffffffu, part, s);
            if (lane == 0) a.gw_part[(int64_t)o * ntiles + tile] = part;
        } else {
#pragma unroll
            for (int q = 0; q < KW; ++q) {
                const int64_t t = t0 + lane + 32 * q;
                if (t >= a.out_len) continue;
                if constexpr (MODE == kWriteY) {
                    a.y[(int64_t)o * a.pitch + t] = acc[i][q];
                } else {
                    const float r = acc[i][q] - __ldg(&a.tmpl[(int64_t)o * a.pitch + t]);
                    local += (double)r * (double)r;
                    if constexpr (MODE == kResidual) a.resid[(int64_t)(o - a.out_begin) * a.rpitch + t] = a.scale * r;
                }
            }
        }
    }
    if constexpr (MODE == kLoss || MODE == kResidual) {
#pragma unroll
        for (int s = 16; s > 0; s >>= 1) local += __shfl_xor_sync(0xffffffffu, local, s);
        if (lane == 0) red[warp] = local;
        __syncthreads();
        if (tid == 0) {
            double sum = 0.0;
            for (int i = 0; i < NTH / 32; ++i) sum += red[i];
            atomicAdd(a.loss_sum, sum);
        }
    }
}

// gw[c] += sum over time tiles of the partials (fixed order: deterministic), a warp per channel
__global__ void gw_reduce_kernel(const float* part, int32_t nchans, int ntiles, float* gw) {
    const int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (c >= nchans) return;
    float s = 0.0f;
    for (int i = lane; i < ntiles; i += 32) s += part[(int64_t)c * ntiles + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) gw[c] += s;
}

__global__ void finish_loss_kernel(const double* sum, double n, double* loss) {
    if (threadIdx.x == 0 && blockIdx.x == 0) *loss = n > 0 ? *sum / n : 0.0;
}

// Samples per lane and row: 16, or 8 where 16 would leave the SMs without two
// CTAs each (256 ch x 4096 x 256 trials: 128 CTAs of 16, 256 of 8).
constexpr int kSmallTile = 32 * 8;

template <int MODE>
cudaError_t launch_gather(F32Args a, int32_t span, int64_t out_len, cudaStream_t s, int* ntiles_out) {
    if (64 * (257 + (int64_t)span) > 227 * 1024) return cudaErrorInvalidValue;  // delay spreads this form has never taken
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 1;
    const int64_t nout = (a.out_end - a.out_begin + kOut - 1) / kOut;
    int kw = 16;
    if ((out_len + 2 * kSmallTile - 1) / (2 * kSmallTile) * nout < 2 * sms) kw = 8;
    // source rows per stage: 8, fewer where the stages of wide windows would not
    // leave room for two CTAs (at least for one)
    auto smem_of = [&](int w, int fc) { return (size_t)f32_stages(w) * fc * (round_up(32 * w + span + 4, 4)) * 4; };
    int fc = kMaxStage;
    while (fc > 2 && smem_of(kw, fc) > 100 * 1024) fc /= 2;
    while (fc > 1 && smem_of(kw, fc) > 200 * 1024) fc /= 2;
    a.fc = fc;
    a.rowlen = (int32_t)round_up(32 * kw + span + 4, 4);
    const size_t smem = smem_of(kw, fc);
    const int64_t ntiles = (out_len + 32 * kw - 1) / (32 * kw);
    const int64_t nblocks = ntiles * nout;
    if (nblocks >= (1ll << 31)) return cudaErrorInvalidConfiguration;
    *ntiles_out = (int)ntiles;
    const bool vec = a.src_pitch % 4 == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0;
    auto kern = kw == 16 ? (vec ? f32_gather_kernel<MODE, 16, true> : f32_gather_kernel<MODE, 16, false>)
                         : (vec ? f32_gather_kernel<MODE, 8, true> : f32_gather_kernel<MODE, 8, false>);
    const cudaError_t e = allow_smem((const void*)kern);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)nblocks, f32_threads(kw), smem, s>>>(a, (int)ntiles);
    return cudaGetLastError();
}

}  // namespace

int f32_adj_tiles(int64_t nsamp) { return (int)((nsamp + kSmallTile - 1) / kSmallTile); }

cudaError_t launch_f32_forward(int mode, const F32FwdArgs& p, cudaStream_t s) {
    if (p.d_end <= p.d_begin || p.length <= 0) return cudaSuccess;
    F32Args a{};
    a.src = p.x;
    a.src_pitch = p.x_pitch;
    a.nsrc = p.nchans;
    a.src_len = p.nsamp;
    a.shifts = p.shifts;
    a.nchans = p.nchans;
    a.out_begin = p.d_begin;
    a.out_end = p.d_end;
    a.out_len = p.length;
    a.w = p.w;
    a.y = p.y;
    a.pitch = p.pitch;
    a.tmpl = p.tmpl;
    a.loss_sum = p.loss_sum;
    a.resid = p.resid;
    a.rpitch = p.rpitch;
    a.scale = p.scale;
    int ntiles;
    switch (mode) {
        case kWriteY: return launch_gather<kWriteY>(a, p.span, p.length, s, &ntiles);
        case kLoss: return launch_gather<kLoss>(a, p.span, p.length, s, &ntiles);
        default: return launch_gather<kResidual>(a, p.span, p.length, s, &ntiles);
    }
}

cudaError_t launch_f32_adjoint(const F32AdjArgs& p, cudaStream_t s) {
    if (p.d_end <= p.d_begin || p.length <= 0) return cudaSuccess;
    F32Args a{};
    a.src = p.gy;
    a.src_pitch = p.gpitch;
    a.nsrc = p.d_end - p.d_begin;
    a.src0 = p.d_begin;
    a.src_len = p.length;
    a.shifts = p.shifts;
    a.nchans = p.nchans;
    a.out_begin = 0;
    a.out_end = p.nchans;
    a.out_len = p.nsamp;
    a.w = p.w;
    a.x = p.x;
    a.x_pitch = p.x_pitch;
    a.gx = p.gx;
    a.gw_part = p.gw_part;
    int ntiles = 0;
    const cudaError_t e = launch_gather<kAdjoint>(a, p.span, p.nsamp, s, &ntiles);
    if (e != cudaSuccess) return e;
    gw_reduce_kernel<<<(p.nchans + 7) / 8, 256, 0, s>>>(p.gw_part, p.nchans, ntiles, p.gw);
    return cudaGetLastError();
}

cudaError_t launch_finish_loss(const double* sum, double n, double* loss, cudaStream_t s) {
    finish_loss_kernel<<<1, 32, 0, s>>>(sum, n, loss);
    return cudaGetLastError();
}

}  // namespace aa
