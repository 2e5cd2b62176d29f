// Launch of the register-blocked passes for the compiled line lengths.
#pragma once
#include "common.cuh"

namespace lddmm {

// defined in fast_pass.cu, one translation unit per number type
template <class T> struct FastPass {
    // n: the line length of this axis.  Returns false when no plan exists.
    static bool launch(int n, int axis, int sign, PassParams<T>& pp, int nj, size_t rows, int n0, int n1, int n2h,
                       cudaStream_t st, bool set_attr = false);
    static bool has(int n) { return n == 32 || n == 64 || n == 96 || n == 128 || n == 160 || n == 192 || n == 256; }
};

}  // namespace lddmm
