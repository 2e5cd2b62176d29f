// The FP32 kernels of one compiled line length, the stages (stage.cuh) and the
// axis-0 and axis-1 transforms (line.cuh): compiled once per length with
// -DLDDMM_STAGE_N=<length>.
#include "line.cuh"
#include "stage.cuh"

namespace lddmm {

template <int N> struct StageRadices;
#define LDDMM_X(N, A, B, C) \
    template <> struct StageRadices<N> { static constexpr int a = A, b = B, c = C; };
LDDMM_STAGE_LENGTHS(LDDMM_X)
#undef LDDMM_X

template <>
bool stage_launch_n<LDDMM_STAGE_N>(int kind, const StageArgs<float>& a, int grid, int threads, size_t smem,
                                   cudaStream_t st, bool set_attr) {
    constexpr int N = LDDMM_STAGE_N;
    using R = StageRadices<N>;
    static_assert(R::a * R::b * R::c == N, "radices of the length");
    switch (kind) {
        case 0: return stage_go(k_stage2<N, R::a, R::b, R::c, 0, true>, a, grid, threads, smem, st, set_attr);
        case 1: return stage_go(k_stage2<N, R::a, R::b, R::c, 1, true>, a, grid, threads, smem, st, set_attr);
        default: return stage_go(k_stage2<N, R::a, R::b, R::c, 2, true>, a, grid, threads, smem, st, set_attr);
    }
}

// radices of the line transforms: two stages where the length allows
constexpr int line_radix(int which) {
    constexpr int firsts[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
    int ba = 0, bb = 0, bc = 0, score = 1 << 30;
    for (int a : firsts)
        for (int c : firsts) {
            if (LDDMM_STAGE_N % (a * c)) continue;
            const int b = LDDMM_STAGE_N / (a * c);
            bool ok = b == 1;
            for (int q : firsts) ok = ok || (q == b && b <= 10);
            if (!ok) continue;
            // few stages, then a small largest radix, then the larger one first
            const int s = (b > 1 ? 1000 : 0) + 10 * (a > c ? (a > b ? a : b) : (c > b ? c : b)) + (a < c ? 1 : 0);
            if (s < score) score = s, ba = a, bb = b, bc = c;
        }
    return which == 0 ? ba : (which == 1 ? bb : bc);
}

template <int MODE> static bool line_go(const PlaneArgs<float>& a, dim3 grid, cudaStream_t st, bool set_attr) {
    constexpr int N = LDDMM_STAGE_N;
    auto* k = k_line<N, line_radix(0), line_radix(1), line_radix(2), MODE>;
    if (set_attr) {
        if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)line_smem(N)) == cudaSuccess)
            return true;
        cudaGetLastError();
        return false;
    }
    launch_dependent(k, grid, line_threads(N), line_smem(N), st, a);
    return true;
}
template <>
bool line_launch_n<LDDMM_STAGE_N>(int mode, const PlaneArgs<float>& a, dim3 grid, cudaStream_t st, bool set_attr) {
    switch (mode) {
        case 0: return line_go<0>(a, grid, st, set_attr);
        case 1: return line_go<1>(a, grid, st, set_attr);
        case 2: return line_go<2>(a, grid, st, set_attr);
        default: return line_go<3>(a, grid, st, set_attr);
    }
}

}  // namespace lddmm
