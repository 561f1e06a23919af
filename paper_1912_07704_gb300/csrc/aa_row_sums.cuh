// Device code shared by the dedispersion kernels' epilogues.
#pragma once

namespace aa {

// Fused statistics of the single-pulse search: the warp's exact sums of one
// output row's samples (s1 = sum y, s2 = sum y^2 per lane; y < 2^24, at most
// 16 samples a lane, so every partial fits in 64 bits) are added to the row's
// accumulators acc = (sum y, sum y^2 low, sum y^2 high); a wrap of the low
// word is carried into the high one, so the 128-bit total is exact.
__device__ __forceinline__ void add_row_sums(unsigned long long* acc, unsigned long long s1,
                                             unsigned long long s2) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicAdd(&acc[0], s1);
        const unsigned long long old = atomicAdd(&acc[1], s2);
        if (old + s2 < old) atomicAdd(&acc[2], 1ull);
    }
}

}  // namespace aa
