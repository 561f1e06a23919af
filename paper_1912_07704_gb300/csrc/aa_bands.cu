// Band rows of a slab, and the trials' sums over them (see aa_bands.h).
//
//   band_rows_kernel  one CTA per (band, tile of words): the band's channels
//                     in shared memory as words of two samples hw apart, its
//                     quads (sums of up to four channels at their delays) in
//                     shared memory, and every row = one or two quads written
//                     to the row buffer.
//   band_sum_kernel   one CTA per (block of 64 trials, tile of 256 words = 512
//                     samples): each band's row windows arrive by bulk copies
//                     in a ring of shared-memory slots (two mbarriers a slot);
//                     16 warps of 4 trials add one row per band and trial, 8
//                     words a lane.
//
// What bounds them (4096 channels, 1500 trials, 2^20 samples: 61.4 ms, 51 of them
// sums; the grouped kernel takes 180):
//   sums  shared memory (its pipe 85 % busy): 64 trials x 8 word reads a lane and
//         band are 512 wavefronts, the ring's fill 74 more, of 645 cycles.  Two
//         pairs of bands are added per round where their rows fit 16 bits (one
//         pair: 712 cycles a band), their sum's two 16-bit lanes go straight into
//         32-bit totals by dot products (16-bit accumulators flushed every 32
//         bands hold loads back by the registers they take), and a place of the
//         ring is refilled three pairs after its own (one pair after, every pair
//         waits for the slowest warp: 1.7 times the time, measured on the form
//         that adds one pair a round).
//   rows  latency and shared memory (71 % of its pipe): 2 reads a word and row
//         plus the quads, 6 CTAs an SM (tiles of 256 words; two CTAs of 1024 took
//         1.18 times the time).
// Segments of 256 / 512 / 1024 / 1536 trials, the same range: 86.0 / 71.4 /
// 66.4 / 61.5 ms (rows shared by more trials are written once; the blocks of a
// tile still find them in L2: 2.4 GB read for 2.1 written a slab).
#include <algorithm>
#include <cstdint>

#include "aa_internal.h"
#include "aa_row_sums.cuh"

namespace aa {
namespace {

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}
// the clock in units of 1.024 us
__device__ __forceinline__ uint32_t ticks() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return (uint32_t)(t >> 10);
}
// Wait for a phase; false if it did not complete within `limit` ticks, or the CTA
// gave up.  Only the first try is inline (2^18 samples of 4096 channels, four ranges:
// 24.04 ms, 24.30 with the clock's loop in line).
__device__ __noinline__ bool mbar_wait_on(uint64_t* bar, uint32_t parity, uint32_t limit, const volatile int* gave_up) {
    const uint32_t start = ticks();
    while (!mbar_try(bar, parity))
        if (*gave_up || ticks() - start > limit) return false;
    return true;
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit, const volatile int* gave_up) {
    if (mbar_try(bar, parity)) return true;
    return mbar_wait_on(bar, parity, limit, gave_up);
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(smem_addr(bar))
                 : "memory");
}

// ------------------------------------------------------------------ rows --

struct RowArgs {
    const void* in;
    int64_t in_pitch;  // samples
    int64_t t0;        // first sample of the slab (multiple of 16)
    int32_t hw;        // words per row beyond its span = samples from a word's low to its high lane
    int32_t blk_lo, blk_hi;  // rows that only other blocks use are left out
    const BandInfo* infos;   // of the segment
    const BandRow* rows;     // of the range
    const BandQuad* quads;
    uint32_t* out;     // where place 0 would lie (the buffer may begin with a later one)
    int32_t k, tile, raw_words, quad_words, max_quads, nbands;
    int32_t dec;  // EB = 0: samples summed as they are read
};

constexpr int kRowThreads = 256;
constexpr int kRowWarps = kRowThreads / 32;

// Sums of dec samples of an 8-bit row, words lo .. lo + 3 of the decimated
// row, as two words of 16-bit lanes.  dec = 2, 4, 8, 16: aligned vector loads
// (lo is a multiple of 4, rows are 16-byte aligned and a multiple of 16 bytes
// long, so a load that starts inside the row ends inside it).
__device__ __forceinline__ uint32_t pair_sums(uint32_t v) { return (v & 0x00ff00ffu) + ((v >> 8) & 0x00ff00ffu); }
__device__ __forceinline__ uint32_t sum4(uint32_t v) {
    const uint32_t p = pair_sums(v);
    return (p & 0xffffu) + (p >> 16);
}
__device__ __forceinline__ uint2 load_decimated(const uint8_t* row, int64_t lo, int dec, int64_t pitch) {
    const int64_t at = lo * dec;
    if (at >= pitch) return make_uint2(0, 0);
    if (dec == 2) {
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(row + at));
        return make_uint2(pair_sums(v.x), pair_sums(v.y));
    }
    uint32_t s[4] = {0, 0, 0, 0};
    if (dec == 4) {
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + at));
        s[0] = sum4(v.x), s[1] = sum4(v.y), s[2] = sum4(v.z), s[3] = sum4(v.w);
    } else if (dec == 8 || dec == 16) {
        for (int b = 0; b < 4 * dec; b += 16)
            if (at + b < pitch) {
                const uint4 v = __ldg(reinterpret_cast<const uint4*>(row + at + b));
                if (dec == 8) {
                    s[b / 8] = sum4(v.x) + sum4(v.y);
                    s[b / 8 + 1] = sum4(v.z) + sum4(v.w);
                } else {
                    s[b / 16] = sum4(v.x) + sum4(v.y) + sum4(v.z) + sum4(v.w);
                }
            }
    } else {
        for (int w = 0; w < 4; ++w)
            for (int b = w * dec; b < (w + 1) * dec; ++b)
                if (at + b < pitch) s[w] += __ldg(row + at + b);
    }
    return make_uint2(s[0] | (s[1] << 16), s[2] | (s[3] << 16));
}

// EB: bytes per sample of the input; 0: the 8-bit input, decimated as it is read
template <int EB>
__global__ void __launch_bounds__(kRowThreads, 6) band_rows_kernel(RowArgs a) {
    extern __shared__ __align__(16) uint32_t rsm[];
    const BandInfo info = a.infos[blockIdx.x % a.nbands];
    const int64_t ua0 = (a.t0 + info.umin) & ~(int64_t)15;  // first sample of the band's first tile
    const int64_t at = ua0 + (int64_t)(blockIdx.x / a.nbands) * a.tile;
    const int32_t ua = (int32_t)(at - a.t0);  // the tile's first word, relative to the slab
    if (ua >= info.umin + info.ulen + a.hw) return;
    uint32_t* raw = rsm;
    uint32_t* qs = rsm + a.k * a.raw_words;
    const int nquads = info.nqa + info.nqb;
    uint32_t* s_quads = qs + a.max_quads * a.quad_words;  // descriptors: 3 words a quad, then 7 a row
    uint32_t* s_rows = s_quads + 3 * a.max_quads;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

    {
        const uint32_t* gq = reinterpret_cast<const uint32_t*>(a.quads + info.quad0);
        const uint32_t* gr = reinterpret_cast<const uint32_t*>(a.rows + info.row0);
        static_assert(sizeof(BandQuad) == 12 && sizeof(BandRow) == 28, "descriptor words");
        for (int i = threadIdx.x; i < 3 * nquads; i += kRowThreads) s_quads[i] = __ldg(gq + i);
        for (int i = threadIdx.x; i < 7 * info.nrows; i += kRowThreads) s_rows[i] = __ldg(gr + i);
    }
    // channels, one or more warps each: word i = samples at + i and at + hw + i;
    // samples past the row's pitch are zero (no valid output reads them)
    const int per = kRowWarps / a.k;  // warps per channel
    const int j = warp / per;
    if (j < info.nch) {
        const int64_t pitch = a.in_pitch;
        uint32_t* dst = raw + j * a.raw_words;
#pragma unroll 4
        for (int i = 4 * (lane + 32 * (warp - j * per)); i < a.raw_words; i += 128 * per) {
            const int64_t lo = at + i, hi = lo + a.hw;
            uint4 w;
            if constexpr (EB == 1) {
                const uint8_t* src = static_cast<const uint8_t*>(a.in) + (int64_t)(info.c0 + j) * pitch;
                const uint32_t l = lo < pitch ? __ldg(reinterpret_cast<const uint32_t*>(src + lo)) : 0u;
                const uint32_t h = hi < pitch ? __ldg(reinterpret_cast<const uint32_t*>(src + hi)) : 0u;
                const uint32_t x = __byte_perm(l, h, 0x5140), y = __byte_perm(l, h, 0x7362);  // l0 h0 l1 h1, l2 h2 l3 h3
                w = make_uint4(__byte_perm(x, 0, 0x4140), __byte_perm(x, 0, 0x4342), __byte_perm(y, 0, 0x4140),
                               __byte_perm(y, 0, 0x4342));
            } else {
                uint2 l = make_uint2(0, 0), h = make_uint2(0, 0);
                if constexpr (EB == 0) {
                    const uint8_t* src = static_cast<const uint8_t*>(a.in) + (int64_t)(info.c0 + j) * pitch;
                    l = load_decimated(src, lo, a.dec, pitch);
                    h = load_decimated(src, hi, a.dec, pitch);
                } else {
                    const uint16_t* src = static_cast<const uint16_t*>(a.in) + (int64_t)(info.c0 + j) * pitch;
                    if (lo < pitch) l = __ldg(reinterpret_cast<const uint2*>(src + lo));
                    if (hi < pitch) h = __ldg(reinterpret_cast<const uint2*>(src + hi));
                }
                w = make_uint4(__byte_perm(l.x, h.x, 0x5410), __byte_perm(l.x, h.x, 0x7632),
                               __byte_perm(l.y, h.y, 0x5410), __byte_perm(l.y, h.y, 0x7632));
            }
            *reinterpret_cast<uint4*>(dst + i) = w;
        }
    }
    __syncthreads();

    for (int q = warp; q < nquads; q += kRowWarps) {
        const uint32_t r01 = s_quads[3 * q], r23 = s_quads[3 * q + 1], blks = s_quads[3 * q + 2];
        if ((int)(blks >> 16) < a.blk_lo || (int)(blks & 0xffffu) > a.blk_hi) continue;
        const int r1 = (int)(r01 >> 16), r2 = (int)(r23 & 0xffffu), r3 = (int)(r23 >> 16);
        const uint32_t* src = raw + (q < info.nqa ? 0 : 4) * a.raw_words + lane;
        const uint32_t* s0 = src + (r01 & 0xffffu);  // every quad has its first channel
        const uint32_t* s1 = src + a.raw_words + r1;
        const uint32_t* s2 = src + 2 * a.raw_words + r2;
        const uint32_t* s3 = src + 3 * a.raw_words + r3;
        uint32_t* dst = qs + q * a.quad_words + lane;
        const int n = a.quad_words - lane;
        if (r3 != 0xffff) {
#pragma unroll 4
            for (int i = 0; i < n; i += 32) dst[i] = s0[i] + s1[i] + s2[i] + s3[i];
        } else {
            for (int i = 0; i < n; i += 32) {
                uint32_t v = s0[i];
                if (r1 != 0xffff) v += s1[i];
                if (r2 != 0xffff) v += s2[i];
                dst[i] = v;
            }
        }
    }
    __syncthreads();

    for (int p = warp; p < info.nrows; p += kRowWarps) {
        const uint32_t* d = s_rows + 7 * p;
        const uint32_t blks = d[5];
        if ((int)(blks >> 16) < a.blk_lo || (int)(blks & 0xffffu) > a.blk_hi) continue;
        const int32_t smin = (int32_t)d[2];
        const int32_t i0 = max(0, smin - ua), n = min(a.tile, smin + (int32_t)d[3] + a.hw - ua) - i0 - lane;
        uint32_t* dst = a.out + ((int64_t)d[6] * a.hw + d[4]) + (ua - smin) + i0 + lane;
        const uint32_t* qa = qs + (d[0] & 0xffffu) * a.quad_words + (d[1] & 0xffffu) + i0 + lane;
        if ((d[0] >> 16) == 0xffffu) {
            for (int i = 0; i < n; i += 32) dst[i] = qa[i];
        } else {
            const uint32_t* qb = qs + (d[0] >> 16) * a.quad_words + (d[1] >> 16) + i0 + lane;
#pragma unroll 4
            for (int i = 0; i < n; i += 32) dst[i] = qa[i] + qb[i];
        }
    }
}

// ------------------------------------------------------------------ sums --

struct SumArgs {
    const uint32_t* rows;  // where place 0 would lie
    int32_t hw;
    const BandCopy* copies;
    const BandHead* heads;  // of the launch's first block
    const uint16_t* offs;
    int32_t nbands, nblk;
    int32_t trial0;      // first trial of the launch's first block, in the range
    int32_t d_lo, d_hi;  // trials written: row d - d_lo of out
    int64_t t0, length;
    float* out;
    int64_t pitch;
    unsigned long long* st_acc;
    unsigned* err;
    uint32_t wait;      // limit of each wait, ticks of 1.024 us
    int32_t skip_band;  // test hook: this band's copies are never issued (-1: none)
};

constexpr int kSumWarps = 16;
constexpr int kSumThreads = kSumWarps * 32;
constexpr int kTrialsPerWarp = kBandTrials / kSumWarps;

// G: pairs added in a round (2: their four rows in 16 bits before the totals)
// Q: words a lane and trial (8, or 4 with CTAs of half the tile and windows).
template <int G, int Q>
__global__ void __launch_bounds__(kSumThreads, 1) band_sum_kernel(SumArgs a) {
    extern __shared__ __align__(128) uint32_t ring[];
    __shared__ uint64_t full[kBandBars], empty[kBandBars];  // pair p: p % kBandBars
    __shared__ int gave_up;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int blk = blockIdx.x % a.nblk;
    constexpr int kLess = kBandWords - 32 * Q;           // words that the tables' windows are longer
    const int tw = (blockIdx.x / a.nblk) * (32 * Q);     // first word of the tile
    if (threadIdx.x == 0) {
        gave_up = 0;
        for (int s = 0; s < kBandBars; ++s) {
            mbar_init(&full[s], 2);  // a pair's two bands
            mbar_init(&empty[s], kSumWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    // Filling the ring is shared by the warps: warp w copies bands w, w + 16, ...
    // (one lane per row window), each when the pair its head names is added.
    // Heads and copy descriptors are loaded a band (of the warp's own) ahead.
    const int npairs = (a.nbands + 1) / 2;
    const BandHead* heads = a.heads + (int64_t)blk * 2 * npairs;
    const uint16_t* offs = a.offs + (int64_t)blk * 2 * npairs * kBandTrials;
    const uint32_t* rows = a.rows + tw;
    int nb = warp;  // next band this warp copies (of 2 npairs; the last may be empty)
    uint4 h = make_uint4(0, 0, 0, 0x7fff0000u), h_next = h;  // BandHead; at = 0x7fff: none
    uint4 c = make_uint4(0, 0, 0, 0);
    auto fetch = [&]() {  // head and copies of band nb; head of the one after
        h = h_next;
        c = lane < (int)(h.y & 0xffffu) ? __ldg(reinterpret_cast<const uint4*>(a.copies + h.x + lane)) : make_uint4(0, 0, 0, 0);
        h_next = nb + kSumWarps < 2 * npairs ? __ldg(reinterpret_cast<const uint4*>(heads + nb + kSumWarps))
                                             : make_uint4(0, 0, 0, 0x7fff0000u);
    };
    if (nb < 2 * npairs) h_next = __ldg(reinterpret_cast<const uint4*>(heads + nb));
    fetch();

    uint32_t tot[kTrialsPerWarp][2 * Q];
#pragma unroll
    for (int i = 0; i < kTrialsPerWarp; ++i)
#pragma unroll
        for (int q = 0; q < Q; ++q) tot[i][2 * q] = tot[i][2 * q + 1] = 0;
    // both 16-bit lanes of a word into their totals, one dot product each
    auto add = [&](int i, int q, uint32_t w) {
        tot[i][2 * q] = __dp2a_lo(w, 0x00000001u, tot[i][2 * q]);
        tot[i][2 * q + 1] = __dp2a_lo(w, 0x00000100u, tot[i][2 * q + 1]);
    };
    int place[G];
    auto places = [&](int pr) {  // of pairs pr .. pr + G - 1, known to every warp from the heads (read a round ahead)
#pragma unroll
        for (int u = 0; u < G; ++u) place[u] = pr + u < npairs ? (int)__ldg(&heads[2 * (pr + u)].place) : 0;
    };
    places(0);
    bool ok = true;
    for (int pr = 0; pr < npairs; pr += G) {
        while ((int)h.w >> 16 <= pr) {  // at
            const int after = (int16_t)(h.w & 0xffffu);
            if (after >= 0 && !__all_sync(0xffffffffu, mbar_wait(&empty[after % kBandBars], (uint32_t)(after / kBandBars) & 1u, a.wait, &gave_up))) {
                ok = false;
                break;
            }
            uint64_t* bar = &full[(nb >> 1) % kBandBars];
            const uint32_t dst = smem_addr(ring + h.z);
            const bool issue = nb != a.skip_band;
            if (lane == 0 && issue) {  // the pair's first band's offsets, then the second's
                mbar_expect(bar, ((h.y >> 16) - (h.y & 0xffffu) * kLess) * 4u + kBandTrials * 2u);
                bulk_g2s(dst + (nb & 1) * kBandTrials * 2u, offs + (int64_t)nb * kBandTrials, kBandTrials * 2u, bar);
            }
            __syncwarp();
            if (c.w && issue) bulk_g2s(dst + (kBandTrials + c.z) * 4u, rows + (int64_t)c.x * a.hw + c.y, (c.w - kLess) * 4u, bar);
            nb += kSumWarps;
            fetch();
        }
        if (!ok) break;
        const uint32_t* sp[G];
#pragma unroll
        for (int u = 0; u < G; ++u) sp[u] = ring + place[u];
        places(pr + G);
#pragma unroll
        for (int u = 0; u < G; ++u)
            if (pr + u < npairs)
                ok = ok && __all_sync(0xffffffffu, mbar_wait(&full[(pr + u) % kBandBars], (uint32_t)((pr + u) / kBandBars) & 1u, a.wait, &gave_up));
        if (!ok) break;
        // this warp's trials' words of the first and the second band of a pair
        auto first = [&](int u) { return *reinterpret_cast<const uint2*>(sp[u] + 2 * warp); };
        auto second = [&](int u) { return *reinterpret_cast<const uint2*>(sp[u] + kBandTrials / 2 + 2 * warp); };
        auto word = [](uint2 o, int i) { return i == 0 ? o.x & 0xffffu : i == 1 ? o.x >> 16 : i == 2 ? o.y & 0xffffu : o.y >> 16; };
        if (G == 2 && 2 * pr + 3 < a.nbands) {
            const uint2 o0 = first(0), o1 = second(0), o2 = first(G - 1), o3 = second(G - 1);
            const uint32_t *z0 = sp[0] + kBandTrials + lane, *z1 = sp[G - 1] + kBandTrials + lane;
#pragma unroll
            for (int i = 0; i < kTrialsPerWarp; ++i) {
                const uint32_t *p0 = z0 + word(o0, i), *p1 = z0 + word(o1, i), *p2 = z1 + word(o2, i), *p3 = z1 + word(o3, i);
#pragma unroll
                for (int q = 0; q < Q; ++q) add(i, q, p0[32 * q] + p1[32 * q] + (p2[32 * q] + p3[32 * q]));
            }
        } else {
#pragma unroll
            for (int u = 0; u < G; ++u) {
                if (pr + u >= npairs) continue;
                const uint32_t* z = sp[u] + kBandTrials + lane;
                const uint2 o = first(u);
                if (2 * (pr + u) + 1 < a.nbands) {
                    const uint2 v = second(u);
#pragma unroll
                    for (int i = 0; i < kTrialsPerWarp; ++i) {
                        const uint32_t *p0 = z + word(o, i), *p1 = z + word(v, i);
#pragma unroll
                        for (int q = 0; q < Q; ++q) add(i, q, p0[32 * q] + p1[32 * q]);
                    }
                } else {
#pragma unroll
                    for (int i = 0; i < kTrialsPerWarp; ++i) {
                        const uint32_t* p0 = z + word(o, i);
#pragma unroll
                        for (int q = 0; q < Q; ++q) add(i, q, p0[32 * q]);
                    }
                }
            }
        }
        __syncwarp();
        if (lane < G && pr + lane < npairs) mbar_arrive(&empty[(pr + lane) % kBandBars]);
    }
    if (!ok && lane == 0) {
        gave_up = 1;
        atomicOr(a.err, 1u);
    }
    __syncthreads();
    if (gave_up) {  // this warp's copies in flight land before the CTA leaves, one limit for all of them
        const uint32_t start = ticks();
        for (int i = max(warp, nb - 2 * kBandBars); i < nb; i += kSumWarps)
            while (!mbar_try(&full[(i >> 1) % kBandBars], (uint32_t)((i >> 1) / kBandBars) & 1u))
                if (ticks() - start > a.wait) break;
        __syncthreads();
        return;
    }
    // word j of the tile: samples t0 + tw + j and t0 + hw + tw + j
    const int64_t tl = a.t0 + tw + lane, th = tl + a.hw;
#pragma unroll
    for (int i = 0; i < kTrialsPerWarp; ++i) {
        const int d = a.trial0 + blk * kBandTrials + warp * kTrialsPerWarp + i;
        if (d < a.d_lo || d >= a.d_hi) continue;
        float* row = a.out + (int64_t)(d - a.d_lo) * a.pitch;
        unsigned long long s1 = 0, s2 = 0;
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const uint32_t vl = tot[i][2 * q], vh = tot[i][2 * q + 1];
            if (tl + 32 * q < a.length) {
                row[tl + 32 * q] = (float)vl;
                s1 += vl;
                s2 += (unsigned long long)vl * vl;
            }
            if (th + 32 * q < a.length) {
                row[th + 32 * q] = (float)vh;
                s1 += vh;
                s2 += (unsigned long long)vh * vh;
            }
        }
        if (a.st_acc) add_row_sums(a.st_acc + 3 * (int64_t)(d - a.d_lo), s1, s2);
    }
}

}  // namespace

bool bands_fit(const DedispArgs& a) {
    if (!a.bands || !a.band_rows || a.length <= 0) return false;
    const int64_t need = (a.length + 2 * kBandWords - 1) / (2 * kBandWords);
    const int64_t least = std::min<int64_t>(need, kBandLeastTiles);
    for (const BandSegment& s : a.bands->segs) {
        const int d0 = std::max(a.trial0, s.trial0), d1 = std::min(a.trial0 + a.ndm, s.trial0 + s.ntrials);
        if (d0 >= d1) continue;
        int64_t id, pre, nrows, words;
        band_window(s, (d0 - s.trial0) / kBandTrials, (d1 - 1 - s.trial0) / kBandTrials, id, pre, nrows, words);
        if (nrows * least * kBandWords + words > a.band_bytes / 4) return false;
    }
    return true;
}

cudaError_t launch_bands(const DedispArgs& a, cudaStream_t s) {
    const BandPlan& bp = *a.bands;
    auto rows_kern = a.row_dec > 1 ? band_rows_kernel<0> : a.elem == 1 ? band_rows_kernel<1> : band_rows_kernel<2>;
    cudaError_t e = allow_smem((const void*)rows_kern);
    if (e != cudaSuccess) return e;
    auto sum_kern = bp.by_two_pairs ? band_sum_kernel<2, 8> : band_sum_kernel<1, 8>;
    auto half_kern = bp.by_two_pairs ? band_sum_kernel<2, 4> : band_sum_kernel<1, 4>;
    for (auto kern : {sum_kern, half_kern}) {
        e = allow_smem((const void*)kern);
        if (e != cudaSuccess) return e;
    }
    int dev = 0, sms = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) sms = 1;
    const int64_t all_tiles = (a.length + 2 * kBandWords - 1) / (2 * kBandWords);
    for (size_t q = 0; q < bp.segs.size(); ++q) {
        const BandSegment& seg = bp.segs[q];
        const int d0 = std::max(a.trial0, seg.trial0), d1 = std::min(a.trial0 + a.ndm, seg.trial0 + seg.ntrials);
        if (d0 >= d1) continue;
        const int g0 = (d0 - seg.trial0) / kBandTrials, g1 = (d1 - 1 - seg.trial0) / kBandTrials;
        const int nblk = g1 - g0 + 1;
        // tiles per slab: as many as the row buffer holds, and of the upper half
        // of those counts the one whose CTAs leave the fewest SMs idle in the
        // slabs' last waves
        int64_t id, pre, nrows, words;
        band_window(seg, g0, g1, id, pre, nrows, words);
        const int64_t most = std::min<int64_t>(all_tiles, (a.band_bytes / 4 - words) / (nrows * kBandWords));
        int64_t per = most, best = INT64_MAX;
        for (int64_t n = most; n >= std::max<int64_t>(1, most / 2); --n) {
            const int64_t full = all_tiles / n, rem = all_tiles % n;
            const int64_t waves = full * ((n * nblk + sms - 1) / sms) + (rem * nblk + sms - 1) / sms;
            if (waves < best) {
                best = waves;
                per = n;
            }
        }
        for (int64_t tile = 0; tile < all_tiles; tile += per) {
            const int64_t nt = std::min(per, all_tiles - tile);
            const int32_t hw = (int32_t)(nt * kBandWords);
            RowArgs ra{};
            ra.in = a.in;
            ra.in_pitch = a.in_pitch;
            ra.t0 = tile * 2 * kBandWords;
            ra.hw = hw;
            ra.blk_lo = g0;
            ra.blk_hi = g1;
            ra.infos = bp.d_infos + q * bp.nbands;
            ra.rows = bp.d_rows;
            ra.quads = bp.d_quads;
            ra.out = reinterpret_cast<uint32_t*>(reinterpret_cast<uintptr_t>(a.band_rows) - (uintptr_t)(id * hw + pre) * 4);
            ra.k = bp.k;
            ra.tile = bp.tile;
            ra.raw_words = bp.raw_words;
            ra.quad_words = bp.quad_words;
            ra.max_quads = bp.max_quads;
            ra.nbands = bp.nbands;
            ra.dec = a.row_dec;
            const int64_t row_tiles = (hw + bp.max_ulen + 15 + bp.tile - 1) / bp.tile;
            rows_kern<<<(unsigned)(row_tiles * bp.nbands), kRowThreads, bp.smem_rows, s>>>(ra);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
            SumArgs sa{};
            sa.rows = ra.out;
            sa.hw = hw;
            sa.copies = bp.d_copies;
            sa.heads = bp.d_heads + (int64_t)(seg.blk0 + g0) * ((bp.nbands + 1) & ~1);
            sa.offs = bp.d_offs + (int64_t)(seg.blk0 + g0) * ((bp.nbands + 1) & ~1) * kBandTrials;
            sa.nbands = bp.nbands;
            sa.nblk = nblk;
            sa.trial0 = seg.trial0 + g0 * kBandTrials;
            sa.d_lo = d0;
            sa.d_hi = d1;
            sa.t0 = ra.t0;
            sa.length = a.length;
            sa.out = a.out + (int64_t)(d0 - a.trial0) * a.out_pitch;
            sa.pitch = a.out_pitch;
            sa.st_acc = a.st_acc ? a.st_acc + 3 * (int64_t)(d0 - a.trial0) : nullptr;
            sa.err = a.err;
            sa.wait = (uint32_t)std::min<uint64_t>((g_wait_limit_ns + 1023) >> 10, UINT32_MAX);
            sa.skip_band = g_fault_skip_chunk;
            // Half tiles take three quarters of a whole one's time (123 us against 167, a
            // wave of 512 bands): worth it where twice the CTAs take as many waves.
            const int64_t waves = (nt * nblk + sms - 1) / sms, half = (2 * nt * nblk + sms - 1) / sms;
            if (half <= waves) half_kern<<<(unsigned)(2 * nt * nblk), kSumThreads, bp.smem_sum, s>>>(sa);
            else sum_kern<<<(unsigned)(nt * nblk), kSumThreads, bp.smem_sum, s>>>(sa);
            e = cudaGetLastError();
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

}  // namespace aa
