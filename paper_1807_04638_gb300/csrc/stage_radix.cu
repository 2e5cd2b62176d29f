// The stage kernels (stage.cuh) of one number type and last radix:
// compiled once per pair with -DLDDMM_STAGE_T=<type> -DLDDMM_STAGE_P=<radix>.
#include "stage.cuh"

namespace lddmm {

template <int P, int KIND>
static bool go_kind(const StageArgs<double>& a, int grid, int threads, size_t smem, cudaStream_t st, bool set_attr) {
    return stage_go(k_stage<double, P, KIND>, a, grid, threads, smem, st, set_attr);
}
template <int P, int KIND>
static bool go_kind(const StageArgs<float>& a, int grid, int threads, size_t smem, cudaStream_t st, bool set_attr) {
    return stage_go(k_stage2<0, 0, 0, P, KIND, false>, a, grid, threads, smem, st, set_attr);
}

template <>
bool stage_launch_p<LDDMM_STAGE_T, LDDMM_STAGE_P>(int kind, const StageArgs<LDDMM_STAGE_T>& a, int grid, int threads,
                                                  size_t smem, cudaStream_t st, bool set_attr) {
    switch (kind) {
        case 0: return go_kind<LDDMM_STAGE_P, 0>(a, grid, threads, smem, st, set_attr);
        case 1: return go_kind<LDDMM_STAGE_P, 1>(a, grid, threads, smem, st, set_attr);
        default: return go_kind<LDDMM_STAGE_P, 2>(a, grid, threads, smem, st, set_attr);
    }
}

}  // namespace lddmm
