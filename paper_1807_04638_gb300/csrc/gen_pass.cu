// The C2C passes with run-time radices (gen_pass.cuh) of one number type:
// compiled once per type with -DLDDMM_T=<type>.
#include "gen_pass.cuh"
#include "gen_launch.cuh"
#include "launch_util.cuh"

namespace lddmm {

template <> bool GenPass<LDDMM_T>::prepare(int axis, const RPlan& pl) {
    using T = LDDMM_T;
    const size_t one = gen_pass_smem<T>(pl.n, false), two = gen_pass_smem<T>(pl.n, true);
    return axis == 0 ? raise_smem_limit(k_gen_c2c<T, 0, 1>, one) && raise_smem_limit(k_gen_c2c<T, 0, -1>, two)
                     : raise_smem_limit(k_gen_c2c<T, 1, 1>, one) && raise_smem_limit(k_gen_c2c<T, 1, -1>, two);
}

template <>
void GenPass<LDDMM_T>::launch(int axis, int sign, const PassParams<LDDMM_T>& q, int nj, const RPlan& pl,
                              cudaStream_t st) {
    using T = LDDMM_T;
    bool acc = false;
    for (int j = 0; j < nj; ++j) acc = acc || q.jobs[j].nin > 1;
    const size_t sm = gen_pass_smem<T>(pl.n, sign < 0 && acc);
    const int tA = (q.c1 + GP_LINES - 1) / GP_LINES, tpk = tA + (q.n1 - q.s1 + GP_LINES - 1) / GP_LINES;
    const unsigned tiles = axis == 0 ? (unsigned)(q.nb2 * tpk)
                                     : (unsigned)(((size_t)q.nb2 * q.n0 + GP_LINES - 1) / GP_LINES);
    const dim3 g(tiles, nj);
    if (axis == 0 && sign > 0) k_gen_c2c<T, 0, 1><<<g, GP_THREADS, sm, st>>>(q, pl, tA, tpk);
    else if (axis == 0) k_gen_c2c<T, 0, -1><<<g, GP_THREADS, sm, st>>>(q, pl, tA, tpk);
    else if (sign > 0) k_gen_c2c<T, 1, 1><<<g, GP_THREADS, sm, st>>>(q, pl, tA, tpk);
    else k_gen_c2c<T, 1, -1><<<g, GP_THREADS, sm, st>>>(q, pl, tA, tpk);
}

}  // namespace lddmm
