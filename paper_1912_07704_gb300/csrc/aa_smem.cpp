// Dynamic shared memory of the kernels.
#include <mutex>

#include "aa_internal.h"

namespace aa {

// The limit is a property of the kernel on a device and not of a launch: were
// each launch to set its own size, a launch on another host thread could lower
// the limit between this one's set and its launch, which is then refused.  So
// every launch sets the same value, all that the kernel can have.  (Set on each
// launch and not once: a device that was reset has forgotten it.)  The static
// part of a kernel is looked up once; it is the same on every device.
cudaError_t allow_smem(const void* kernel) {
    struct Known {
        const void* kernel;
        int most;
    };
    constexpr int kMax = 64;  // kernels that take dynamic shared memory: 44
    static std::mutex mu;
    static Known known[kMax];
    static int n = 0;
    int most = -1;
    {
        std::lock_guard<std::mutex> lock(mu);
        for (int i = 0; i < n; ++i)
            if (known[i].kernel == kernel) most = known[i].most;
    }
    if (most < 0) {
        cudaFuncAttributes attr{};
        const cudaError_t e = cudaFuncGetAttributes(&attr, kernel);
        if (e != cudaSuccess) return e;
        most = kMaxSmem - (int)attr.sharedSizeBytes;
        std::lock_guard<std::mutex> lock(mu);
        if (n < kMax) known[n++] = Known{kernel, most};
    }
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
}

}  // namespace aa
