// Launch helpers shared by the translation units.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>

namespace lddmm {

// The dynamic shared-memory limit of a kernel is process-wide: every site that
// raises it sets the device's opt-in maximum, so that a handle (or call) for a
// smaller grid never lowers the limit under a concurrent launch of a larger one.
inline int smem_optin_max() {
    int dev = 0, v = 48 * 1024;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
}
template <class K>
inline bool raise_smem_limit(K kernel, size_t need) {
    const int mx = smem_optin_max();
    if ((size_t)mx < need) return false;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, mx) == cudaSuccess) return true;
    cudaGetLastError();  // a refusal must not stay pending: the caller falls back to another kernel
    return false;
}

// Ask for the smallest shared-memory carveout that holds `blocks` resident
// blocks of `bytes` dynamic shared memory each, so that the rest of the SM's
// unified L1/shared storage stays L1 (a hint: the driver rounds it up to a
// split it supports).
template <class K>
inline void prefer_l1(K kernel, size_t bytes, int blocks) {
    int dev = 0, per_sm = 0, resv = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&resv, cudaDevAttrReservedSharedMemoryPerBlock, dev) != cudaSuccess || per_sm <= 0) {
        cudaGetLastError();
        return;
    }
    const size_t need = (size_t)blocks * (bytes + (size_t)resv);
    const int pct = (int)std::min<size_t>(100, (need * 100 + (size_t)per_sm - 1) / (size_t)per_sm);
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct) != cudaSuccess)
        cudaGetLastError();  // a hint only
}

// Grid of a persistent pass: `per_sm` resident blocks per SM, never more
// blocks than work items.
inline int persistent_grid(int items, int per_sm = 3) {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (sms <= 0) sms = 152;
    }
    return std::max(1, std::min(items, per_sm * sms));
}

}  // namespace lddmm
