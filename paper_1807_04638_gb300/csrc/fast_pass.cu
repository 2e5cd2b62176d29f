// The register-blocked passes (fft_fast.cuh) of one number type: compiled once
// per type with -DLDDMM_T=<type>.
#include "fast_pass.cuh"
#include "fft_fast.cuh"
#include "launch_util.cuh"

namespace lddmm {

// Launch of the register-blocked passes for the compiled line lengths.
template <class T> struct FastPassImpl {
    // the persistent axis-2 kernel's shared-memory limit is raised (per N)
    template <int N> static bool& a2p_ready() {
        static bool v = false;
        return v;
    }
    // The persistent axis-2 kernel takes full tiles of r2 rows, one input per
    // inverse job, and 16-byte aligned inputs (its copies are 16-byte
    // cp.async of whole rows or plane segments).
    static bool axis2p_fits(const PassParams<T>& pp, int nj, size_t rows, int r2) {
        if (rows % (size_t)r2 != 0 || (rows / r2) * (size_t)nj >= (1u << 24)) return false;
        for (int j = 0; j < nj; ++j) {
            const PassJobT<T>& jb = pp.jobs[j];
            if (pp.sign > 0 && jb.nin != 1) return false;
            for (int i = 0; i < jb.nin; ++i)
                if ((uintptr_t)jb.in[i] % 16 != 0) return false;
        }
        return true;
    }
    template <int N>
    static bool go(int axis, int sign, PassParams<T>& pp, int nj, size_t rows, int n0, int n1, int n2h,
                   cudaStream_t st, bool set_attr) {
        (void)sign;
        constexpr int TL = FAST_THREADS / (N / FastPlan<N>::E);
        if (axis == 2) {
            const size_t sm = fast_axis2_smem<T, N>();
            constexpr bool PERS = sizeof(T) == 4 && FastPlan<N>::E <= 12;
            if (set_attr) {
                if constexpr (PERS) a2p_ready<N>() = raise_smem_limit(k_fast_axis2p<T, N>, fast_axis2p_smem<T, N>());
                return raise_smem_limit(k_fast_axis2<T, N>, sm);
            }
            if constexpr (PERS) {
                if (a2p_ready<N>() && axis2p_fits(pp, nj, rows, 2 * TL)) {
                    const int ntiles = (int)(rows / (2 * TL));
                    pp.fd_tiles = FastDiv((unsigned)ntiles);
                    k_fast_axis2p<T, N><<<persistent_grid(ntiles * nj, A2P_BLOCKS), FAST_THREADS, fast_axis2p_smem<T, N>(),
                                          st>>>(pp, ntiles);
                    return true;
                }
            }
            const int gx = (int)((rows + 2 * TL - 1) / (2 * TL));
            k_fast_axis2<T, N><<<dim3(gx, nj), FAST_THREADS, sm, st>>>(pp);
        } else if (axis == 1) {
            const size_t sm = fast_c2c_smem<T, N>(1);
            if (set_attr) {
                if (!raise_smem_limit(k_fast_c2c<T, N, 1>, sm)) return false;
                prefer_l1(k_fast_c2c<T, N, 1>, sm, FastOccC2C<T, N>::value);
                return true;
            }
            (void)n2h;
            const int ntiles = (int)(((size_t)pp.nb2 * n0 + TL - 1) / TL);
            pp.fd_tiles = FastDiv((unsigned)ntiles);
            pp.fd_n0 = FastDiv((unsigned)n0);
            k_fast_c2c<T, N, 1><<<persistent_grid(ntiles * nj), FAST_THREADS, sm, st>>>(pp, ntiles);
        } else {
            const size_t sm = fast_c2c_smem<T, N>(0);
            if (set_attr) {
                if (!raise_smem_limit(k_fast_c2c<T, N, 0>, sm)) return false;
                prefer_l1(k_fast_c2c<T, N, 0>, sm, FastOccC2C<T, N>::value);
                return true;
            }
            const int tpk = (pp.c1 + TL - 1) / TL + (n1 - pp.s1 + TL - 1) / TL;
            const int ntiles = pp.nb2 * tpk;
            pp.fd_tiles = FastDiv((unsigned)ntiles);
            pp.fd_tpk = FastDiv((unsigned)tpk);
            k_fast_c2c<T, N, 0><<<persistent_grid(ntiles * nj), FAST_THREADS, sm, st>>>(pp, ntiles);
        }
        return true;
    }
    // n: the line length of this axis.  Returns false when no plan exists.
    static bool launch(int n, int axis, int sign, PassParams<T>& pp, int nj, size_t rows, int n0, int n1, int n2h,
                       cudaStream_t st, bool set_attr = false) {
        switch (n) {
            case 32: return go<32>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 64: return go<64>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 128: return go<128>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 256: return go<256>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 96: return go<96>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 160: return go<160>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            case 192: return go<192>(axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
            default: return false;
        }
    }
};

template <>
bool FastPass<LDDMM_T>::launch(int n, int axis, int sign, PassParams<LDDMM_T>& pp, int nj, size_t rows, int n0, int n1,
                               int n2h, cudaStream_t st, bool set_attr) {
    return FastPassImpl<LDDMM_T>::launch(n, axis, sign, pp, nj, rows, n0, n1, n2h, st, set_attr);
}

}  // namespace lddmm
