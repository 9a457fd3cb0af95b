// osd_host.hpp -- host-side helpers shared by the launchers: status mapping,
// argument checks and cluster launches through cudaLaunchKernelEx.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cmath>
#include <cstdint>
#include <mutex>

#include "osd.h"

namespace osd {

inline osd_status from_cuda(cudaError_t e) { return e == cudaSuccess ? OSD_OK : OSD_ERR_CUDA; }

inline bool aligned_to(const void* p, size_t a) {
    return (reinterpret_cast<uintptr_t>(p) % a) == 0;
}

inline size_t dtype_size(osd_dtype d) { return d == OSD_BF16 ? 2 : 4; }

// exp(x / T) = 2^(x * c) with c = log2(e) / T, carried as c_hi + c_lo where both
// halves are positive floats: the pair removes the rounding of c from every
// exponent argument, and positive halves keep -inf inputs at -inf.
inline void split_scale(float temperature, float* c_hi, float* c_lo) {
    const double c = 1.4426950408889634074 / static_cast<double>(temperature);
    float hi = static_cast<float>(c);
    if (static_cast<double>(hi) > c) hi = std::nextafter(hi, 0.0f);
    float lo = static_cast<float>(c - static_cast<double>(hi));
    if (!(lo > 0.0f)) lo = 1e-30f;
    *c_hi = hi;
    *c_lo = lo;
}

// Streaming multiprocessors of the current device, looked up once per device
// (0 when the query fails).
inline int device_sms() {
    static std::atomic<int> sms[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int n = sms[dev].load(std::memory_order_relaxed);
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
        sms[dev].store(n, std::memory_order_relaxed);
    return n;
}

// Opt in for `smem` bytes of dynamic shared memory and ask how many CTAs an SM then
// holds (0 when a query fails).  Kept per device for the last size asked, so repeated
// calls (and calls under stream capture) make no runtime query.
template <auto kern, int kThreads>
static int ctas_per_sm(size_t smem) {
    static std::mutex mu;
    static size_t allowed[64] = {};
    static size_t last_smem[64] = {};
    static int last_occ[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    std::lock_guard<std::mutex> lock(mu);
    if (last_smem[dev] == smem && last_occ[dev] > 0) return last_occ[dev];
    if (allowed[dev] < smem) {
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) !=
            cudaSuccess)
            return 0;
        allowed[dev] = smem;
    }
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kThreads, smem) != cudaSuccess) return 0;
    last_smem[dev] = smem;
    last_occ[dev] = occ;
    return occ;
}

// The largest cluster size of 1 .. `most` of which `clusters` run at the same time when each
// CTA takes `smem` bytes of dynamic shared memory (a fixed figure per kern), 0 if none: the
// SMs of a cluster lie in one GPC, so fewer fit than the SMs' own count says.  `spare`: of
// sizes above 2, with a 32nd of the slots to spare.  Kept per device.
template <auto kern, int kThreads>
static int widest_cluster(long long clusters, int most, size_t smem, bool spare) {
    constexpr int kMost = 8;
    static std::atomic<int> fit[64][kMost + 1];  // clusters of a size that run at once, plus 1
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    for (int c = most < kMost ? most : kMost; c >= 1; --c) {
        int n = fit[dev][c].load(std::memory_order_relaxed) - 1;
        if (n < 0) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(static_cast<unsigned>(c));
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = smem;
            cudaLaunchAttribute attr = {};
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = static_cast<unsigned>(c);
            attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            if (ctas_per_sm<kern, kThreads>(smem) < 1 || cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) return 0;
            fit[dev][c].store(n + 1, std::memory_order_relaxed);
        }
        if (clusters + (spare && c > 2 ? clusters / 31 : 0) <= n) return c;
    }
    return 0;
}

// Launch `kernel` with an optional thread-block cluster of `cluster` CTAs
// along x (cluster == 1 launches without the attribute); launch_ex can also
// mark it a programmatic dependent of the previous kernel on the stream.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_ex(bool dependent, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                             cudaStream_t stream, int cluster, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    unsigned n = 0;
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = static_cast<unsigned>(cluster);
        attr[n].val.clusterDim.y = 1;
        attr[n].val.clusterDim.z = 1;
        ++n;
    }
    if (dependent) {  // may start before the previous kernel on the stream ends (it waits in-kernel)
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n].val.programmaticStreamSerializationAllowed = 1;
        ++n;
    }
    cfg.attrs = n ? attr : nullptr;
    cfg.numAttrs = n;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                          int cluster, Args&&... args) {
    return launch_ex(false, kernel, grid, block, smem, stream, cluster, static_cast<Args&&>(args)...);
}

}  // namespace osd
