// Choice of the kernels of the band form for a line length.
#pragma once
#include "line.cuh"
#include "stage.cuh"

namespace lddmm {

inline bool stage_launch(int kind, const StageArgs<float>& a, int grid, int threads, size_t smem, cudaStream_t st,
                         bool set_attr = false) {
    if (a.rows % 2 == 0) switch (a.n2) {
#define LDDMM_X(N, A, B, C) \
    case N: return stage_launch_n<N>(kind, a, grid, threads, smem, st, set_attr);
            LDDMM_STAGE_LENGTHS(LDDMM_X)
#undef LDDMM_X
            default: break;
        }
    switch (a.pl.c) {
        case 3: return stage_launch_p<float, 3>(kind, a, grid, threads, smem, st, set_attr);
        case 4: return stage_launch_p<float, 4>(kind, a, grid, threads, smem, st, set_attr);
        case 5: return stage_launch_p<float, 5>(kind, a, grid, threads, smem, st, set_attr);
        case 6: return stage_launch_p<float, 6>(kind, a, grid, threads, smem, st, set_attr);
        default: return false;
    }
}
inline bool stage_launch(int kind, const StageArgs<double>& a, int grid, int threads, size_t smem, cudaStream_t st,
                         bool set_attr = false) {
    switch (a.pl.c) {
        case 4: return stage_launch_p<double, 4>(kind, a, grid, threads, smem, st, set_attr);
        case 5: return stage_launch_p<double, 5>(kind, a, grid, threads, smem, st, set_attr);
        case 6: return stage_launch_p<double, 6>(kind, a, grid, threads, smem, st, set_attr);
        case 8: return stage_launch_p<double, 8>(kind, a, grid, threads, smem, st, set_attr);
        case 9: return stage_launch_p<double, 9>(kind, a, grid, threads, smem, st, set_attr);
        case 10: return stage_launch_p<double, 10>(kind, a, grid, threads, smem, st, set_attr);
        default: return false;
    }
}
// FP32 line transforms of a compiled length (false: the length is not)
inline bool line_launch(int n, int mode, const PlaneArgs<float>& a, dim3 grid, cudaStream_t st, bool set_attr = false) {
    switch (n) {
#define LDDMM_X(N, A, B, C) \
    case N: return line_launch_n<N>(mode, a, grid, st, set_attr);
        LDDMM_STAGE_LENGTHS(LDDMM_X)
#undef LDDMM_X
        default: return false;
    }
}

}  // namespace lddmm
