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

// Launch that may begin before the kernel in front of it on the stream has
// ended (programmatic dependent launch): the kernel's prologue overlaps the
// other's last blocks.  Every kernel launched this way calls after_previous()
// before its first access to memory that another kernel of the stream writes
// or reads, reads what the kernel in front of it wrote by plain loads (not
// __ldg: that memory is not read-only while this kernel runs), and calls
// dependents_may_launch() when it is about to write its last results: at that point the launch latency and the prologue are hidden and
// the dependents take no room from its own blocks.  Hessian-vector product at
// 64^3: 1.52 ms without, 1.42 ms so, 1.64 ms with the call at every kernel's
// start; at 128^3 7.11, 6.97 and 6.91 ms.  k_spec_step alone calls it first: it
// has no prologue worth the name and its blocks no shared memory, and the place
// makes no difference there (1,417 us at 64^3 and 6,973 us at 128^3 either way).
template <class A>
inline void launch_dependent(void (*kernel)(A), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, const A& a) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, a);
}
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dependents_may_launch() { asm volatile("griddepcontrol.launch_dependents;"); }

}  // namespace lddmm
