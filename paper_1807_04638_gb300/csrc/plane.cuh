// Axis-0 and axis-1 transforms of the band, one plane k2 at a time, and the
// spectral step between two stages (the band form of the path: 2/3-rule
// projector on, states kept in the compute type).
//
// Spectra of this path are stored on the band only, [k2 < nb2][k1c][k0c] with
// k0c fastest (rows padded to an even pitch): k0c counts k0 = 0..kc0 and then k0 = n0 - kc0..n0 - 1.  The
// axis-2 side holds [k2 < nb2][row], row = i0 n1 + i1, as everywhere else.
//   k_plane_inv: spectra -> (k1 -> i1, lanes k0c) -> shared plane [i1][k0]
//                -> (k0 -> i0, lanes i1) -> [row], coalesced at both ends;
//   k_plane_fwd: the same backwards.
// A field of the inverse is a symbol applied to up to three spectra while
// they are loaded (a component, a divergence, or a component of a curl, times
// L, K or 1).  PH = 3 runs both axes on one plane in shared memory, which
// saves the trip of the half-transformed plane through L2 and its addressing;
// FP64 takes it while a plane fits (n0 n1 up to about 14,000 points).  Larger
// FP64 planes, and all FP32 ones, run the two axes as two launches (PH = 1,
// then 2; forward 2, then 1) over column and line tiles with the
// half-transformed band [k2][i1][k0c] between them: a 128^2 FP32 plane leaves
// an SM one block, and the inverse of a stage at 128^3 took 88 us so against
// 2 x 38 us in tiles of 16.  Lengths that are compiled in take line.cuh
// instead: 2 x 23 us.  FP64 is bound by the FP64 rate: its warps wait for that
// pipe while HBM idles.
#pragma once
#include "launch_util.cuh"
#include "radix.cuh"

namespace lddmm {

// The band |k_a| <= kc_a = (n_a - 1) / 3 of the spectra: extents b_a, and the
// number p_a of non-negative wave numbers among them.
struct Band {
    int n0, n1, n2, nb2;
    int b0, p0, b1, p1;
    int b0p;  // row pitch of the spectra: b0 rounded up to even (16-byte rows of FP32 pairs)
    int kc0, kc1, kc2;
    FastDiv fb0, fn1;
    size_t size;  // nb2 b1 b0p
};
// index of a band entry on its axis, and back (-1: outside)
__device__ __forceinline__ int band_k(int kc, int p, int b, int n) { return kc < p ? kc : kc + n - b; }
__device__ __forceinline__ int band_c(int k, int p, int b, int n) { return k < p ? k : (k >= n - (b - p) ? k + b - n : -1); }
__device__ __forceinline__ bool in_cut(int k, int kc, int n) { return k <= kc || k >= n - kc; }

constexpr int PLANE_JOBS = 14;
// kinds: 0 X_0; 1 i (kappa . X); 2..4 component 0..2 of i kappa x X
template <class T> struct PlaneJob {
    const cpx<T>* in;  // component 0; the others follow at stride cs
    cpx<T>* out;
    const T* tab;      // factor table over the band, or null
    T scale;
    int kind;
};
template <class T> struct PlaneArgs {
    PlaneJob<T> jobs[PLANE_JOBS];
    Band bd;
    RPlan pl0, pl1;
    const cpx<T>*tw0, *tw1;  // e^{-2 pi i t / n} of the axes
    const T* dk[3];          // kappa tables
    size_t cs;               // component stride of the inputs
    cpx<T>* mid;             // PH 1 / 2: half-transformed band, one field after the other
    size_t mids;             // its field stride
    int tile;                // PH 1: columns per block; PH 2: lines per block
    FastDiv ft;              // division by tile
};

template <class T> __host__ __device__ inline size_t plane_smem(int ph, const Band& b, int tile) {
    const size_t pitch = (size_t)(b.n0 | 1);
    const size_t s = ph == 3 ? pitch * b.n1 : (ph == 1 ? (size_t)b.n1 * tile : pitch * tile);
    return (s + b.n0 + b.n1) * sizeof(cpx<T>);
}

// Launch of the plane kernels (plane_kernels.cuh) of a type, ph as above
// (set_attr: raise the shared-memory limit instead); defined in plane.cu.
template <class T>
bool plane_kernel(bool inverse, int ph, const PlaneArgs<T>& a, dim3 grid, int threads, size_t smem, cudaStream_t st,
                  bool set_attr = false);

// ---------------------------------------------------------------- spectral step
// What follows a stage's transforms, entry by entry over the band: the
// derivatives, L and K of the products' spectra, and the Heun step.  All
// transforms t come doubled (the stage kernels leave out the halving of the
// split of two packed rows).
//   modes 0, 1  tangent stage 1, 2:  t = (t_0..2, s, a_0..2, r_0..2),
//               p = t + i kappa s,  q = r + i kappa x a;
//               stage 1: e1 = e0 - dt K p,  x1 = x0 + dt (e0 + q);
//               stage 2: e0 <- (e0 + e1)/2 - dt/2 K p,
//                        x0 <- (x0 + x1)/2 + dt/2 (e1 + q)
//   modes 2, 3  adjoint stage 1, 2:  t = (eb_0..2, db, mb_0..2, ob_0..2, xb_0..2, dxb),
//               E = -(eb - i kappa db + L (mb + i kappa x ob)),  X = xb - i kappa dxb;
//               stage 1: e1 = dt/2 e0 + dt^2/2 (E + x0),  x1 = dt/2 x0 + dt^2/2 X;
//               stage 2: e0 <- e0/2 + e1/dt + E + x1 (+ src),  x0 <- x0/2 + x1/dt + X
//   modes 4, 5  shooting stage 1, 2:  t = (t_0..2, s):  p as above;
//               stage 1: e1 = e0 - dt K p;  stage 2: e0 <- (e0 + e1)/2 - dt/2 K p
template <class T> struct StepArgs {
    const cpx<T>* t[14];
    cpx<T>*e0, *x0, *e1, *x1;   // three components each, stride cs
    const cpx<T>* src;          // mode 3: added to e0 (nullable), stride cs
    const T *Lt, *Kt;           // L and K over the band
    const T* dk[3];
    Band bd;
    size_t cs;
    T dt;
};
// One thread an entry, no shared memory: bound by L2 and HBM (18 to 30
// band arrays, 2.5 MB each at 128^3).  Apart from the transforms because every
// output of a vector needs all its components, and a block of line transforms
// holds lines of one field.
template <class T, int MODE>
__global__ void __launch_bounds__(256) k_spec_step(const __grid_constant__ StepArgs<T> a) {
    const Band& bd = a.bd;
    dependents_may_launch();  // see launch_util.cuh
    after_previous();
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= (int)bd.size) return;
    const int q = i / bd.b0p, kc0 = min(i - q * bd.b0p, bd.b0 - 1), k2 = q / bd.b1, kc1 = q - k2 * bd.b1;
    const T kp[3] = {a.dk[0][band_k(kc0, bd.p0, bd.b0, bd.n0)], a.dk[1][band_k(kc1, bd.p1, bd.b1, bd.n1)], a.dk[2][k2]};
    const T h = (T)0.5, dt = a.dt;
    // i kappa_c z
    auto ik = [&](int c, cpx<T> z) { return mk(-kp[c] * z.y, kp[c] * z.x); };
    auto curl = [&](const cpx<T>(&z)[3], int c) {
        const int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
        const cpx<T> d = kp[c1] * z[c2] - kp[c2] * z[c1];
        return mk(-d.y, d.x);
    };
    if constexpr (MODE == 0 || MODE == 1 || MODE >= 4) {
        const T K = a.Kt[i];
        const cpx<T> s = a.t[3][i];
        constexpr bool X = MODE < 2;
        cpx<T> av[3];
        if constexpr (X) {
LDDMM_UNROLL
            for (int c = 0; c < 3; ++c) av[c] = a.t[4 + c][i];
        }
LDDMM_UNROLL
        for (int c = 0; c < 3; ++c) {
            const size_t o = c * a.cs + i;
            const cpx<T> p = a.t[c][i] + ik(c, s);
            const cpx<T> e0 = a.e0[o];
            if constexpr (MODE == 0 || MODE == 4) {
                a.e1[o] = e0 - (h * dt * K) * p;
                if constexpr (X) a.x1[o] = a.x0[o] + dt * (e0 + h * (a.t[7 + c][i] + curl(av, c)));
            } else {
                const cpx<T> e1 = a.e1[o];
                a.e0[o] = h * (e0 + e1) - (h * h * dt * K) * p;
                if constexpr (X)
                    a.x0[o] = h * (a.x0[o] + a.x1[o]) + (h * dt) * (e1 + h * (a.t[7 + c][i] + curl(av, c)));
            }
        }
    } else {
        const T L = a.Lt[i];
        const cpx<T> db = a.t[3][i], dx = a.t[13][i];
        cpx<T> ob[3];
LDDMM_UNROLL
        for (int c = 0; c < 3; ++c) ob[c] = a.t[7 + c][i];
LDDMM_UNROLL
        for (int c = 0; c < 3; ++c) {
            const size_t o = c * a.cs + i;
            const cpx<T> E = (-h) * (a.t[c][i] - ik(c, db) + L * (a.t[4 + c][i] + curl(ob, c)));
            const cpx<T> X = h * (a.t[10 + c][i] - ik(c, dx));
            const cpx<T> e0 = a.e0[o], x0 = a.x0[o];
            if constexpr (MODE == 2) {
                a.e1[o] = (h * dt) * e0 + (h * dt * dt) * (E + x0);
                a.x1[o] = (h * dt) * x0 + (h * dt * dt) * X;
            } else {
                const cpx<T> x1 = a.x1[o];
                cpx<T> e = h * e0 + ((T)1 / dt) * a.e1[o] + E + x1;
                if (a.src) e = e + a.src[o];
                a.e0[o] = e;
                a.x0[o] = h * x0 + ((T)1 / dt) * x1 + X;
            }
        }
    }
}

// L and K over the band, evaluated in double precision
template <class T>
__global__ void k_band_tables(Band bd, double l0, double l1, double l2, double alpha, int s, T* Lt, T* Kt) {
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i >= (int)bd.size) return;
    const int q = i / bd.b0p, kc0 = min(i - q * bd.b0p, bd.b0 - 1), k2 = q / bd.b1, kc1 = q - k2 * bd.b1;
    auto ksq = [](int k, int n, double l) {
        const double w = 6.283185307179586477 / l * (double)(2 * k > n ? k - n : k);
        return w * w;
    };
    const double b = 1.0 + alpha * (ksq(band_k(kc0, bd.p0, bd.b0, bd.n0), bd.n0, l0) +
                                    ksq(band_k(kc1, bd.p1, bd.b1, bd.n1), bd.n1, l1) + ksq(k2, bd.n2, l2));
    double p = 1.0;
    for (int e = 0; e < s; ++e) p *= b;
    Lt[i] = (T)p;
    Kt[i] = (T)(1.0 / p);
}

// Full half spectrum [k2][k0][k1] <-> band spectrum, per component (blockIdx.y).
// TOBAND: dst(band) = P src; else dst(full) = src inside the band, 0 elsewhere.
template <class T, bool TOBAND>
__global__ void __launch_bounds__(256) k_band_copy(Band bd, const cpx<T>* src, size_t ss, cpx<T>* dst, size_t ds) {
    const cpx<T>* s = src + blockIdx.y * ss;
    cpx<T>* d = dst + blockIdx.y * ds;
    const size_t total = TOBAND ? bd.size : (size_t)(bd.n2 / 2 + 1) * bd.n0 * bd.n1;
    for (size_t i = blockIdx.x * (size_t)256 + threadIdx.x; i < total; i += (size_t)gridDim.x * 256) {
        if (TOBAND) {
            const int q = (int)i / bd.b0p, kc0 = min((int)i - q * bd.b0p, bd.b0 - 1), k2 = q / bd.b1, kc1 = q - k2 * bd.b1;
            const int k0 = band_k(kc0, bd.p0, bd.b0, bd.n0), k1 = band_k(kc1, bd.p1, bd.b1, bd.n1);
            d[i] = s[((size_t)k2 * bd.n0 + k0) * bd.n1 + k1];
        } else {
            const size_t r = i / bd.n1;
            const int k1 = (int)(i - r * bd.n1), k2 = (int)(r / bd.n0), k0 = (int)(r - (size_t)k2 * bd.n0);
            const bool in = in_cut(k0, bd.kc0, bd.n0) && in_cut(k1, bd.kc1, bd.n1) && k2 <= bd.kc2;
            d[i] = in ? s[((size_t)k2 * bd.b1 + band_c(k1, bd.p1, bd.b1, bd.n1)) * bd.b0p +
                          band_c(k0, bd.p0, bd.b0, bd.n0)]
                      : mk((T)0, (T)0);
        }
    }
}

}  // namespace lddmm
