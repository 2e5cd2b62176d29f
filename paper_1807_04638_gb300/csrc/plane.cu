// The plane kernels (plane_kernels.cuh) of one number type: compiled once per
// type with -DLDDMM_T=<type>.  In FP32 they serve the lengths without compiled
// line kernels (line.cuh), one axis per launch.
#include "launch_util.cuh"
#include "plane_kernels.cuh"

namespace lddmm {

template <class K>
static bool go(K kernel, const PlaneArgs<LDDMM_T>& a, dim3 grid, int threads, size_t smem, cudaStream_t st,
               bool set_attr) {
    if (set_attr) return raise_smem_limit(kernel, smem);
    kernel<<<grid, threads, smem, st>>>(a);
    return true;
}

template <>
bool plane_kernel<LDDMM_T>(bool inverse, int ph, const PlaneArgs<LDDMM_T>& a, dim3 grid, int threads, size_t smem,
                           cudaStream_t st, bool set_attr) {
    using T = LDDMM_T;
    if constexpr (sizeof(T) == 8)
        if (ph == 3)
            return inverse ? go(k_plane_inv<T, 3>, a, grid, threads, smem, st, set_attr)
                           : go(k_plane_fwd<T, 3>, a, grid, threads, smem, st, set_attr);
    if (ph == 1)
        return inverse ? go(k_plane_inv<T, 1>, a, grid, threads, smem, st, set_attr)
                       : go(k_plane_fwd<T, 1>, a, grid, threads, smem, st, set_attr);
    if (ph == 2)
        return inverse ? go(k_plane_inv<T, 2>, a, grid, threads, smem, st, set_attr)
                       : go(k_plane_fwd<T, 2>, a, grid, threads, smem, st, set_attr);
    return false;
}

}  // namespace lddmm
