// Corner turn of a time-major filterbank block into the channel-major layout
// the dedispersion reads: cm[c * pitch + t] = tm[t * stride + c].
// HBM-bound (one byte read and one written per sample): 128 x 128-byte tiles
// through shared memory, 16-byte global accesses where aligned.  A thread loads
// four 16-byte pieces of time samples (eight threads a sample's 128 bytes),
// then turns 16 time samples x 4 channels with byte permutes (4 x 4 bytes each)
// into four 16-byte stores (eight threads 128 bytes of a channel).  Word w of
// time sample t lies at w ^ 4 (t / 16 mod 8) of its row, so that neither side
// meets a bank twice.  4096 channels x 2^20 samples: 1.48 ms, 5.8 TB/s (64 x 64 tiles
// gathered byte by byte 2.28 ms).  Rows that do not begin at 16 bytes are read by
// words and shifted into place: 4095 channels x 2^18, 0.41 ms (by bytes, in the
// small tiles, 1.34; 1000 x 300001: 0.13, 0.36).
#include <cstdint>

#include "aa_internal.h"

namespace aa {
namespace {

constexpr int kTile = 128;

__global__ void __launch_bounds__(256) corner_turn_kernel(const uint8_t* __restrict__ tm,
                                                          int64_t nsamp, int nchans, int64_t stride,
                                                          uint8_t* __restrict__ cm, int64_t pitch,
                                                          int64_t ntile_c, int64_t ntiles) {
    __shared__ __align__(16) uint32_t tile[kTile][kTile / 4];  // [t][4 c]
    const uint8_t* end = tm + (nsamp - 1) * stride + nchans;
    for (int64_t it = blockIdx.x; it < ntiles; it += gridDim.x) {
        const int64_t t0 = (it / ntile_c) * kTile;
        const int c0 = (int)(it % ntile_c) * kTile;
        // load: time samples t0 + row + 32 k, channels c0 + 16 seg .. + 15
        {
            const int row = threadIdx.x >> 3, seg = threadIdx.x & 7;
            const int c = c0 + 16 * seg;
            uint4 v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int64_t t = t0 + row + 32 * k;
                const uint8_t* src = tm + t * stride + c;
                v[k] = make_uint4(0, 0, 0, 0);
                if (t < nsamp && c < nchans) {
                    const uintptr_t at = reinterpret_cast<uintptr_t>(src);
                    if ((at & 15) == 0 && src + 16 <= end) {  // (channels from nchans on are read, not stored)
                        v[k] = __ldcs(reinterpret_cast<const uint4*>(src));
                    } else if (src - (at & 3) >= tm && src - (at & 3) + 20 <= end) {
                        const uint32_t* s4 = reinterpret_cast<const uint32_t*>(at & ~(uintptr_t)3);
                        const int sh = 8 * (int)(at & 3);
                        const uint32_t w0 = __ldg(s4), w1 = __ldg(s4 + 1), w2 = __ldg(s4 + 2), w3 = __ldg(s4 + 3),
                                       w4 = __ldg(s4 + 4);
                        v[k] = make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh),
                                          __funnelshift_r(w2, w3, sh), __funnelshift_r(w3, w4, sh));
                    } else {  // the block's first and last bytes
                        uint32_t w[4] = {0, 0, 0, 0};
                        for (int b = 0; b < 16 && c + b < nchans; ++b) w[b >> 2] |= (uint32_t)src[b] << (8 * (b & 3));
                        v[k] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int t = row + 32 * k;
                *reinterpret_cast<uint4*>(&tile[t][4 * (seg ^ ((t >> 4) & 7))]) = v[k];
            }
        }
        __syncthreads();
        // store: channels c0 + 4 quad .. + 3, time samples t0 + 16 tb .. + 15
        {
            const int tb = threadIdx.x & 7, quad = threadIdx.x >> 3;
            const int64_t t = t0 + 16 * tb;
            uint32_t o[4][4];  // [channel][4 time samples]
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                uint32_t r[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) r[k] = tile[16 * tb + 4 * q + k][quad ^ (4 * tb)];
                const uint32_t a = __byte_perm(r[0], r[1], 0x5140), b = __byte_perm(r[2], r[3], 0x5140);
                const uint32_t c = __byte_perm(r[0], r[1], 0x7362), d = __byte_perm(r[2], r[3], 0x7362);
                o[0][q] = __byte_perm(a, b, 0x5410);
                o[1][q] = __byte_perm(a, b, 0x7632);
                o[2][q] = __byte_perm(c, d, 0x5410);
                o[3][q] = __byte_perm(c, d, 0x7632);
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int c = c0 + 4 * quad + u;
                if (c >= nchans || t >= nsamp) continue;
                uint8_t* dst = cm + (int64_t)c * pitch + t;
                if (t + 16 <= nsamp && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
                    __stcs(reinterpret_cast<uint4*>(dst), make_uint4(o[u][0], o[u][1], o[u][2], o[u][3]));
                } else {
#pragma unroll
                    for (int k = 0; k < 16; ++k)
                        if (t + k < nsamp) dst[k] = (uint8_t)(o[u][k >> 2] >> (8 * (k & 3)));
                }
            }
        }
        __syncthreads();
    }
}

}  // namespace
}  // namespace aa

using namespace aa;

extern "C" aa_status aa_corner_turn_device(const uint8_t* d_tm, int64_t nsamp, int32_t nchans,
                                           int64_t tm_stride, uint8_t* d_cm, int64_t cm_pitch,
                                           aa_stream_t stream) {
    clear_error();
    if (!d_tm || !d_cm) { set_error("device pointer is NULL"); return AA_ERR_ARG; }
    if (nsamp < 0 || nchans < 1 || tm_stride < nchans || cm_pitch < nsamp) {
        set_error("bad sizes (nsamp %lld, nchans %d, stride %lld, pitch %lld)", (long long)nsamp,
                  nchans, (long long)tm_stride, (long long)cm_pitch);
        return AA_ERR_ARG;
    }
    if (nsamp == 0) return AA_OK;
    // channels fastest: consecutive CTAs read consecutive pieces of the same samples
    const int64_t ntile_c = (nchans + kTile - 1) / kTile;
    const int64_t ntiles = ntile_c * ((nsamp + kTile - 1) / kTile);
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t grid = std::min<int64_t>(ntiles, (int64_t)std::max(sms, 1) * 8);
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    {
        ProfScope prof(kKCornerTurn, s);
        corner_turn_kernel<<<(unsigned)grid, 256, 0, s>>>(d_tm, nsamp, nchans, tm_stride, d_cm, cm_pitch,
                                                           ntile_c, ntiles);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        set_error("corner turn launch: %s", cudaGetErrorString(e));
        return AA_ERR_CUDA;
    }
    return AA_OK;
}
