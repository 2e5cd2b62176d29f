// Launch of the C2C passes with run-time radices (gen_pass.cuh).
#pragma once
#include "radix.cuh"

namespace lddmm {

// defined in gen_pass.cu, one translation unit per number type
template <class T> struct GenPass {
    static bool prepare(int axis, const RPlan& pl);
    static void launch(int axis, int sign, const PassParams<T>& q, int nj, const RPlan& pl, cudaStream_t st);
};

}  // namespace lddmm
