// C2C passes (the jobs of fft_kernels.cuh) for line lengths without a
// register-blocked plan in fft_fast.cuh: run-time radices of up to 16
// (radix.cuh), one butterfly per item in registers, 16 lines per block with
// the lines as lanes.  Axis 0 reads and writes 16 neighbouring columns; axis 1
// reads rows, where the four items of a warp's lanes cover a row's
// neighbouring entries, whole 32-byte sectors.  Inputs of an inverse job are
// read again for each of its outputs (they come from L2); a forward job adds
// its inputs' transforms up in a second tile.  Band-limited as the
// register-blocked passes are.  The passes that these replace walked radices
// of at most 5 through shared memory with a division per element: 2.48 ms
// against 0.66 ms per launch at 256 x 300 x 256, axis 1.  Bound by the latency of one 16-line tile per block: two
// blocks of 256 threads an SM.
#pragma once
#include "radix.cuh"

namespace lddmm {

constexpr int GP_LINES = 16, GP_THREADS = 256;
template <class T> inline size_t gen_pass_smem(int n, bool acc) {
    return ((size_t)n * GP_LINES * (acc ? 2 : 1) + n) * sizeof(cpx<T>);
}

template <class T, int AXIS, int DIR>
__global__ void __launch_bounds__(GP_THREADS, sizeof(T) == 4 ? 2 : 1)
    k_gen_c2c(const __grid_constant__ PassParams<T> pp, const __grid_constant__ RPlan pl, int tA, int tpk) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    constexpr int TH = GP_THREADS / GP_LINES;  // item slots
    const int N = pl.n, n0 = pp.n0, n1 = pp.n1;
    cpx<T>* const S = (cpx<T>*)smem_raw;
    cpx<T>* const tws = S + N * GP_LINES;
    cpx<T>* const acc = tws + N;  // forward jobs of several inputs
    for (int i = threadIdx.x; i < N; i += GP_THREADS) tws[i] = ldg((const cpx<T>*)pp.ax.tw + i);
    const PassJobT<T>& job = pp.jobs[blockIdx.y];
    const int c = threadIdx.x % GP_LINES, m = threadIdx.x / GP_LINES;
    // this thread's line: first element g, element step gs, fixed frequencies
    int g, gs, kf, k2;
    bool on;
    if (AXIS == 1) {
        const int line = blockIdx.x * GP_LINES + c, lines = pp.nb2 * n0;
        on = line < lines;
        k2 = min(line, lines - 1) / n0;
        kf = min(line, lines - 1) - k2 * n0;
        g = min(line, lines - 1) * n1;
        gs = 1;
    } else {
        k2 = blockIdx.x / tpk;
        const int r = blockIdx.x - k2 * tpk;
        const int kb = r < tA ? r * GP_LINES : pp.s1 + (r - tA) * GP_LINES, ke = r < tA ? pp.c1 : n1;
        on = kb + c < ke;
        kf = min(kb + c, ke - 1);
        g = k2 * n0 * n1 + kf;
        gs = n1;
    }
    auto out_of_band = [&](int p) { return AXIS == 1 && p >= pp.c1 && p < pp.s1; };
    auto apply = [&](const SymT<T>& sy, int p, cpx<T> v) {
        return AXIS == 0 ? sym_apply(sy, pp.tabs, p, kf, k2, v) : sym_apply(sy, pp.tabs, kf, p, k2, v);
    };
    cpx<T>* const Sc = S + c;
    __syncthreads();
    // stages after the first, up to the last one's butterflies: out(k, value)
    auto rest = [&](auto out) {
        __syncthreads();
        if (pl.b > 1) {
            LDDMM_MID(pl.b, {
                for (int i = m; i < N / R; i += TH) {
                    const int j2 = (int)pl.fa.div((unsigned)i), q0 = i - j2 * pl.a;
                    cpx<T>* s = Sc + (q0 + pl.a * R * j2) * GP_LINES;
                    const int st = pl.a * GP_LINES;
                    cpx<T> v[R];
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, DIR>(v);
                    twiddles<R, DIR>(v, tws, pl.a * j2);
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        LDDMM_LAST(pl.c, {
            const int M = N / R;
            for (int i = m; i < M; i += TH) {
                cpx<T> v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = Sc[(i + r * M) * GP_LINES];
                dft<R, DIR>(v);
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) out(i + r * M, v[r]);
            }
        })
    };
    auto first = [&](auto load) {
        LDDMM_FIRST(pl.a, {
            const int M = N / R;
            for (int j = m; j < M; j += TH) {
                cpx<T> v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = load(j + r * M);
                dft<R, DIR>(v);
                twiddles<R, DIR>(v, tws, j);
                const int r1 = (int)pl.fc.div((unsigned)j), j2 = j - r1 * pl.c;
                cpx<T>* s = Sc + (R * (r1 + pl.b * j2)) * GP_LINES;
                LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * GP_LINES] = v[q];
            }
        })
    };
    if (DIR > 0) {
        for (int o = 0; o < job.nout; ++o) {
            const SymT<T> sy = job.osym[o];
            first([&](int p) {
                cpx<T> x = mk((T)0, (T)0);
                if (!out_of_band(p)) {
                    const int e = g + p * gs;
                    x = job.isym[0].scale * ((const cpx<T>*)job.in[0])[e];
                    for (int b = 1; b < job.nin; ++b) x = x + job.isym[b].scale * ((const cpx<T>*)job.in[b])[e];
                    x = apply(sy, p, x);
                }
                return x;
            });
            cpx<T>* const ob = (cpx<T>*)job.out[o] + g;
            rest([&](int p, cpx<T> v) {
                if (on) ob[p * gs] = v;
            });
            __syncthreads();
        }
    } else {
        for (int q = 0; q < job.nin; ++q) {
            const cpx<T>* const in = (const cpx<T>*)job.in[q] + g;
            const SymT<T> sy = job.isym[q];
            first([&](int p) { return in[p * gs]; });
            const bool last = q == job.nin - 1;
            cpx<T>* const ob = (cpx<T>*)job.out[0] + g;
            rest([&](int p, cpx<T> v) {
                if (out_of_band(p)) return;
                v = apply(sy, p, v);
                cpx<T>& a = acc[p * GP_LINES + c];
                if (q > 0) v = v + a;
                if (!last) {
                    a = v;
                    return;
                }
                for (int b = 0; b < job.nb; ++b) v = v + job.bcoef[b] * ((const cpx<T>*)job.base[b])[g + p * gs];
                if (on) ob[p * gs] = v;
            });
            __syncthreads();
        }
    }
}

}  // namespace lddmm
