// FDMT-style tree dedispersion (arXiv:1912.07704 Sec. 1, the dedispersion
// module's cited work).  Row r of a depth of the channel tree holds a
// subband's series at one delay:
//   out[r][t] = U[t] + Lo[t + gap],   t < nsamp - delta_r,
// where U and Lo are rows of the next-deeper depth (32-bit) or input channel
// rows (8- or 16-bit leaves).  The root depth writes one FP32 row per trial
// of the range (t < the range's output length).  Sums are exact integers.
//
// A launch merges a group of up to five depths: a CTA takes one block (some
// consecutive rows of the group's top depth) x one tile of samples, loads the
// windows it needs into slots of shared memory and merges depth after depth
// there; only the top depth's rows go to memory.  With one launch per depth every
// sum read two samples and wrote one: 75 GB and 15.2 ms for 2^17 samples of 4096
// channels under the four ranges of the SKA plan; in groups of 4-3-5 depths it
// is 10 GB and 5.4 ms (5.9 with one tile a CTA, its tables read again for each,
// 5.5 with a warp per channel row instead of all rows' pieces dealt out together).
// Shared memory bounds it (its pipe is 61-68 % busy; two CTAs of an SM hide the
// loads of each other).  A lane sums four consecutive
// samples: with one sample a lane (12 wavefronts for 128 sums instead of 16, but
// twice the instructions) it was 7.0 ms; blocks of 52 and 71 KB, four and three to
// an SM, 8.2 and 6.9 ms (more of their windows is overlap).
#include <algorithm>
#include <cstdint>

#include "aa_internal.h"

namespace aa {
namespace {

constexpr int kFdmtThreads = 512;
constexpr int kFdmtWarps = kFdmtThreads / 32;

struct FdmtArgs {
    const FdmtBlock* blocks;
    const FdmtLoad* loads;
    const FdmtOp* ops;
    const void* leaf;  // channel rows
    int64_t leaf_pitch;
    const uint32_t* prev;
    uint32_t* out;
    int64_t pitch;
    int64_t nsamp;
    float* fout;
    int64_t fpitch, flen;
    int32_t nblocks, tile, levels;
    int32_t op_words, load_words;  // words of the ops, and of the loads behind them, before the slots
    int32_t per;       // consecutive tiles of a CTA
    int32_t leaves;    // blocks load channels
    int32_t quads;     // pieces of four samples of the widest window
    uint32_t quad_inv;  // 2^22 / quads, up: exact for fewer than 2^15 pieces of 128 at most
    int64_t ntiles;
};

__device__ __forceinline__ void cp_async16(uint32_t* dst, const uint32_t* src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src),
                 "r"(bytes)
                 : "memory");
}

// Sums of one op, four consecutive samples a lane: the upper series starts at a
// multiple of four words, the lower one anywhere (its place within four words
// is the same for all lanes).
template <class Put>
__device__ __forceinline__ void merge(const uint32_t* slots, const int4& op, int lane, Put put) {
    const uint32_t* u = slots + (op.x & 0xffff);
    const uint32_t lo = (uint32_t)op.x >> 16;
    const uint32_t* l = slots + (lo & ~3u);
    const int r = lo & 3;
    auto run = [&](auto pick) {
#pragma unroll 2
        for (int i = 4 * lane; i < op.z; i += 128) {
            const uint4 a = *reinterpret_cast<const uint4*>(u + i);
            const uint4 b = pick(i);
            put(i, make_uint4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w));
        }
    };
    auto at = [&](int i) { return *reinterpret_cast<const uint4*>(l + i); };
    if (r == 0) run([&](int i) { return at(i); });
    else if (r == 1) run([&](int i) { const uint4 p = at(i); return make_uint4(p.y, p.z, p.w, l[i + 4]); });
    else if (r == 2) run([&](int i) { const uint4 p = at(i); const uint2 q = *reinterpret_cast<const uint2*>(l + i + 4); return make_uint4(p.z, p.w, q.x, q.y); });
    else run([&](int i) { const uint4 p = at(i), q = at(i + 4); return make_uint4(p.w, q.x, q.y, q.z); });
}

template <int EB, bool FINAL>
__global__ void __launch_bounds__(kFdmtThreads, 2) fdmt_group_kernel(FdmtArgs a) {
    extern __shared__ __align__(16) uint32_t fdmt_smem[];
    const int4* ops = reinterpret_cast<const int4*>(fdmt_smem);                  // src, dst, n, delta
    const int4* loads = reinterpret_cast<const int4*>(fdmt_smem + a.op_words);  // ref, lo, dst, n
    uint32_t* slots = fdmt_smem + a.op_words + a.load_words;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const FdmtBlock& b = a.blocks[blockIdx.x % a.nblocks];  // neighbouring blocks share rows: side by side
    const int load0 = __ldg(&b.load0), nload = __ldg(&b.nload), op0 = __ldg(&b.op0), nops = __ldg(&b.end[a.levels - 1]);
    for (int i = threadIdx.x; i < nops + nload; i += kFdmtThreads) {
        if (i < nops) reinterpret_cast<int4*>(fdmt_smem)[i] = __ldg(reinterpret_cast<const int4*>(a.ops + op0) + i);
        else reinterpret_cast<int4*>(fdmt_smem + a.op_words)[i - nops] = __ldg(reinterpret_cast<const int4*>(a.loads + load0) + i - nops);
    }
    const int64_t tile0 = (int64_t)(blockIdx.x / a.nblocks) * a.per, tile1 = min(a.ntiles, tile0 + a.per);
#pragma unroll 1
    for (int64_t tile = tile0; tile < tile1; ++tile) {
        const int64_t t0 = tile * a.tile;
        __syncthreads();  // tables in place; the tile before is done with the slots
        for (int i = warp; i < nload; i += kFdmtWarps) {
            const int4 l = loads[i];
            const int64_t t = t0 + l.y;
            uint32_t* dst = slots + l.z;
            if (l.x < 0) continue;
            const uint32_t* src = a.prev + (int64_t)l.x * a.pitch;
            for (int j = 4 * lane; j < l.w; j += 128) {
                const bool in = t + j < a.pitch;  // beyond the row: zeros, which no valid output reads
                cp_async16(dst + j, in ? src + t + j : a.prev, in ? 16 : 0);
            }
        }
        // channels, four samples a thread, four such pieces at a time over all of them
        for (int p0 = threadIdx.x; p0 < (a.leaves ? nload * a.quads : 0); p0 += 4 * kFdmtThreads) {
            uint2 w[4];
            uint32_t* dst[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int p = p0 + u * kFdmtThreads;
                const int i = (int)(((uint32_t)p * a.quad_inv) >> 22);  // p / quads
                dst[u] = nullptr;
                if (i >= nload) continue;
                const int4 l = loads[i];
                const int j = 4 * (p - i * a.quads);
                if (l.x >= 0 || j >= l.w) continue;
                dst[u] = slots + l.z + j;
                const int64_t t = t0 + l.y + j, at = (int64_t)(-(l.x + 1)) * a.leaf_pitch + t;
                w[u] = make_uint2(0, 0);
                if (t < a.nsamp) {  // the pitch is a multiple of four samples
                    if constexpr (EB == 1) w[u].x = __ldg(reinterpret_cast<const uint32_t*>(static_cast<const uint8_t*>(a.leaf) + at));
                    else w[u] = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(a.leaf) + at));
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (!dst[u]) continue;
                *reinterpret_cast<uint4*>(dst[u]) = EB == 1
                    ? make_uint4(w[u].x & 0xff, (w[u].x >> 8) & 0xff, (w[u].x >> 16) & 0xff, w[u].x >> 24)
                    : make_uint4(w[u].x & 0xffff, w[u].x >> 16, w[u].y & 0xffff, w[u].y >> 16);
            }
        }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        int begin = 0;
#pragma unroll 1
        for (int lev = 0; lev < a.levels - 1; ++lev) {
            const int end = __ldg(&b.end[lev]);
            for (int o = begin + warp; o < end; o += kFdmtWarps) {
                const int4 op = ops[o];
                uint32_t* d = slots + op.y;
                merge(slots, op, lane, [&](int i, uint4 v) { *reinterpret_cast<uint4*>(d + i) = v; });
            }
            begin = end;
            __syncthreads();
        }
        for (int o = begin + warp; o < nops; o += kFdmtWarps) {
            const int4 op = ops[o];
            const int64_t left = (FINAL ? a.flen : a.nsamp - op.w) - t0;
            const int n = left < op.z ? (int)left : op.z;  // op.z: the tile
            merge(slots, op, lane, [&](int i, uint4 v) {
                if constexpr (FINAL) {
                    float* row = a.fout + (int64_t)op.y * a.fpitch + t0 + i;
                    if (i + 4 <= n) *reinterpret_cast<float4*>(row) = make_float4((float)v.x, (float)v.y, (float)v.z, (float)v.w);
                    else {
                        if (i < n) row[0] = (float)v.x;
                        if (i + 1 < n) row[1] = (float)v.y;
                        if (i + 2 < n) row[2] = (float)v.z;
                    }
                } else if (i < n) {  // the pitch is a multiple of four samples; beyond a row's valid part nothing is read
                    *reinterpret_cast<uint4*>(a.out + (int64_t)op.y * a.pitch + t0 + i) = v;
                }
            });
        }
    }
}

}  // namespace

cudaError_t launch_fdmt_group(const FdmtPlan& fd, const FdmtGroup& g, int leaf_elem, const void* leaves,
                              int64_t leaf_pitch, const uint32_t* prev, uint32_t* out, int64_t pitch,
                              int64_t nsamp, float* fout, int64_t fpitch, int64_t flen, cudaStream_t s) {
    const bool fin = fout != nullptr;
    const int64_t n = fin ? flen : nsamp;
    if (n <= 0 || g.nblocks <= 0) return cudaSuccess;
    const int64_t ntiles = (n + g.tile - 1) / g.tile;
    // Up to eight tiles a CTA, which then reads its block's tables once, while
    // eight CTAs are left for each of the SMs' places.
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 1;
    const int64_t per = std::max<int64_t>(1, std::min<int64_t>(8, ntiles * g.nblocks / (sms * 2 * 8)));
    const int64_t grid = (ntiles + per - 1) / per * g.nblocks;
    if (grid >= (1ll << 31)) return cudaErrorInvalidConfiguration;
    FdmtArgs a{};
    a.blocks = fd.d_blocks + g.block0;
    a.loads = fd.d_loads;
    a.ops = fd.d_ops;
    a.leaf = leaves;
    a.leaf_pitch = leaf_pitch;
    a.prev = prev;
    a.out = out;
    a.pitch = pitch;
    a.nsamp = nsamp;
    a.fout = fout;
    a.fpitch = fpitch;
    a.flen = flen;
    a.nblocks = g.nblocks;
    a.tile = g.tile;
    a.levels = g.bottom - g.top + 1;
    a.op_words = g.max_ops * 4;
    a.load_words = g.max_loads * 4;
    a.per = (int32_t)per;
    a.leaves = g.leaves;
    a.quads = g.width / 4;
    a.quad_inv = ((1u << 22) + a.quads - 1) / a.quads;
    a.ntiles = ntiles;
    const size_t smem = ((size_t)a.op_words + (size_t)a.load_words + (size_t)g.words) * 4;
    auto kern = leaf_elem == 1 ? (fin ? fdmt_group_kernel<1, true> : fdmt_group_kernel<1, false>)
                               : (fin ? fdmt_group_kernel<2, true> : fdmt_group_kernel<2, false>);
    const cudaError_t e = allow_smem((const void*)kern);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, kFdmtThreads, smem, s>>>(a);
    return cudaGetLastError();
}

}  // namespace aa
