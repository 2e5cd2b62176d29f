// Pointwise kernels on real fields: the ad* / ad bilinear forms of the EPDiff
// equation and of the Jacobi sweeps, semi-Lagrangian transport (global-gather
// and shared-memory-staged map steps), warping, the exact transposes of the
// map step and of the warp (discrete gradient), Jacobian determinants and
// double-precision reductions.
//
// A time state holds 24 real fields, each N = n0*n1*n2 values (the band form's
// ten are in stage.cuh):
//   [0..2]   v_c          [3 + 3c + j]  D_j v_c
//   [12..14] m_c = (L v)_c [15 + 3c + j] D_j m_c
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "radix.cuh"

namespace lddmm {

constexpr int PW_THREADS = 256;

// Stored values are T or bfloat16 (the precision form's state storage); they
// are widened to the compute type on load.
template <class T> __device__ __forceinline__ T widen(T x) { return x; }
__device__ __forceinline__ float widen(__nv_bfloat16 x) { return __bfloat162float(x); }

template <class S> struct StatePtr {
    const S* p;  // 24 fields, stride N
    size_t N;
    __device__ __forceinline__ auto v(int c, size_t x) const { return widen(p[c * N + x]); }
    __device__ __forceinline__ auto Dv(int c, int j, size_t x) const { return widen(p[(3 + 3 * c + j) * N + x]); }
    __device__ __forceinline__ auto m(int c, size_t x) const { return widen(p[(12 + c) * N + x]); }
    __device__ __forceinline__ auto Dm(int c, int j, size_t x) const { return widen(p[(15 + 3 * c + j) * N + x]); }
};

// ad*_v m = (Dv)^T m + (Dm) v + m div v  (EPDiff bracket, Sec. 2.2).
// With store != nullptr the 24 input fields are also written to the state
// store in bfloat16 (precision form).
template <class T>
__global__ void k_adstar(StatePtr<T> S, T* __restrict__ out, size_t N, __nv_bfloat16* __restrict__ store) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        T v[3], m[3], Dv[3][3], Dm[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = S.v(c, x);
            m[c] = S.m(c, x);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                Dv[c][j] = S.Dv(c, j, x);
                Dm[c][j] = S.Dm(c, j, x);
            }
        }
        const T divv = Dv[0][0] + Dv[1][1] + Dv[2][2];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T a = m[i] * divv;
#pragma unroll
            for (int j = 0; j < 3; ++j) a += Dv[j][i] * m[j] + Dm[i][j] * v[j];
            out[i * N + x] = a;
        }
        if (store) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                store[c * N + x] = __float2bfloat16_rn((float)v[c]);
                store[(12 + c) * N + x] = __float2bfloat16_rn((float)m[c]);
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    store[(3 + 3 * c + j) * N + x] = __float2bfloat16_rn((float)Dv[c][j]);
                    store[(15 + 3 * c + j) * N + x] = __float2bfloat16_rn((float)Dm[c][j]);
                }
            }
        }
    }
}

// Tangent (forward Jacobi) stage, pointwise part:
//  p = ad*_eta m + ad*_v mu  (mu = L eta),   q = ad_v xi = (Dv) xi - (Dxi) v.
// E holds eta in the 24-field state layout (eta, D eta, mu, D mu);
// X holds xi (0..2) and D_j xi_c at 3 + 3c + j.
template <class T, class SS>
__global__ void k_tangent_pw(StatePtr<SS> S, StatePtr<T> E, const T* __restrict__ X, T* __restrict__ out, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        T v[3], m[3], e[3], mu[3], xi[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = S.v(c, x);
            m[c] = S.m(c, x);
            e[c] = E.v(c, x);
            mu[c] = E.m(c, x);
            xi[c] = X[c * N + x];
        }
        const T divv = S.Dv(0, 0, x) + S.Dv(1, 1, x) + S.Dv(2, 2, x);
        const T dive = E.Dv(0, 0, x) + E.Dv(1, 1, x) + E.Dv(2, 2, x);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            T p = m[i] * dive + mu[i] * divv;
            T q = 0;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                p += E.Dv(j, i, x) * m[j] + S.Dm(i, j, x) * e[j] + S.Dv(j, i, x) * mu[j] + E.Dm(i, j, x) * v[j];
                q += S.Dv(i, j, x) * xi[j] - X[(3 + 3 * i + j) * N + x] * v[j];
            }
            out[i * N + x] = p;
            out[(3 + i) * N + x] = q;
        }
    }
}

// Adjoint (transposed Jacobi) stage, pointwise part.  Inputs y = K ybar_eta
// and yx = ybar_xi (3 fields each).  Writes 9 groups of 4 fields
// [scalar s, f_0, f_1, f_2]; the forward transform of a group is
// F(s) + sum_j i kappa_j F(f_j):
//   group c     : R'^T part without L:  s = -sum_i D_c m_i y_i,  f_i = m_c y_i + delta_ic (m.y)
//   group 3 + c : R'^T part under -L:   s = sum_i D_i v_c y_i + (div v) y_c,  f_j = -v_j y_c
//   group 6 + c : ad_v^T yx:            s = sum_i D_c v_i yx_i,  f_j = v_j yx_c
template <class T, class SS>
__global__ void k_adjoint_pw(StatePtr<SS> S, const T* __restrict__ Y, T* __restrict__ out, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        T v[3], m[3], y[3], yx[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            v[c] = S.v(c, x);
            m[c] = S.m(c, x);
            y[c] = Y[c * N + x];
            yx[c] = Y[(3 + c) * N + x];
        }
        const T divv = S.Dv(0, 0, x) + S.Dv(1, 1, x) + S.Dv(2, 2, x);
        const T my = m[0] * y[0] + m[1] * y[1] + m[2] * y[2];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            T s1 = 0, s2 = divv * y[c], s3 = 0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                s1 -= S.Dm(i, c, x) * y[i];
                s2 += S.Dv(c, i, x) * y[i];
                s3 += S.Dv(i, c, x) * yx[i];
            }
            T* g1 = out + (size_t)(4 * c) * N;
            T* g2 = out + (size_t)(4 * (3 + c)) * N;
            T* g3 = out + (size_t)(4 * (6 + c)) * N;
            g1[x] = s1;
            g2[x] = s2;
            g3[x] = s3;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                g1[(1 + j) * N + x] = m[c] * y[j] + (j == c ? my : (T)0);
                g2[(1 + j) * N + x] = -v[j] * y[c];
                g3[(1 + j) * N + x] = v[j] * yx[c];
            }
        }
    }
}

// ---------------------------------------------------------------- interpolation
struct GridI {
    int n0, n1, n2;
};

__device__ __forceinline__ int wrapi(int i, int n) {
    int r = i % n;
    return r < 0 ? r + n : r;
}

template <class T> __device__ __forceinline__ void cr_weights(T t, T* w) {
    const T t2 = t * t, t3 = t2 * t;
    w[0] = (T)0.5 * (-t3 + (T)2 * t2 - t);
    w[1] = (T)0.5 * ((T)3 * t3 - (T)5 * t2 + (T)2);
    w[2] = (T)0.5 * ((T)-3 * t3 + (T)4 * t2 + t);
    w[3] = (T)0.5 * (t3 - t2);
}

// Interpolate NC fields at voxel (i0,i1,i2) + d (d in voxels); component c of
// grid point o is f[o es + c cs].  The taps of a row along axis 2 are summed
// first, then the rows (the order that the other kernels below share, so that
// they agree to the last bit).
template <class T, int NC>
__device__ __forceinline__ void interp_at(const T* __restrict__ f, size_t cs, int es, GridI g, int i0, int i1, int i2,
                                          const T d[3], int cubic, T* res) {
    int base[3];
    T w[3][4];
    const int ii[3] = {i0, i1, i2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const T fl = floor(d[a]);
        const T t = d[a] - fl;
        base[a] = ii[a] + (int)fl;
        if (cubic) {
            cr_weights(t, w[a]);
        } else {
            w[a][0] = (T)1 - t;
            w[a][1] = t;
        }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) res[c] = 0;
    const int lo = cubic ? -1 : 0, cnt = cubic ? 4 : 2;
    for (int a0 = 0; a0 < cnt; ++a0) {
        const size_t o0 = (size_t)wrapi(base[0] + lo + a0, g.n0) * g.n1;
        for (int a1 = 0; a1 < cnt; ++a1) {
            const size_t o1 = (o0 + wrapi(base[1] + lo + a1, g.n1)) * g.n2;
            T row[NC];
            for (int a2 = 0; a2 < cnt; ++a2) {
                const size_t o = (o1 + wrapi(base[2] + lo + a2, g.n2)) * es;
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const T x = __ldg(&f[c * cs + o]);
                    row[c] = a2 == 0 ? w[2][0] * x : fma(w[2][a2], x, row[c]);
                }
            }
            const T w01 = w[0][a0] * w[1][a1];
#pragma unroll
            for (int c = 0; c < NC; ++c) res[c] = fma(w01, row[c], res[c]);
        }
    }
}

// One semi-Lagrangian step of the inverse-map displacement u (psi = x + u):
//   Xt = x - dt v1(x);  X = x - dt/2 (v1(x) + v0(Xt));  u1(x) = (X - x) + u0(X).
template <class T>
__global__ void k_sl_step(GridI g, const T* __restrict__ v0, const T* __restrict__ v1, const T* __restrict__ u0,
                          T* __restrict__ u1, T dt, T ih0, T ih1, T ih2, int cubic, size_t N) {
    const T ih[3] = {ih0, ih1, ih2};
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const int i2 = (int)(x % g.n2);
        const int i1 = (int)((x / g.n2) % g.n1);
        const int i0 = (int)(x / ((size_t)g.n2 * g.n1));
        T w1[3], d[3], vt[3], ut[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            w1[c] = v1[c * N + x];
            d[c] = -dt * w1[c] * ih[c];
        }
        interp_at<T, 3>(v0, N, 1, g, i0, i1, i2, d, cubic, vt);
        T disp[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            disp[c] = (T)-0.5 * dt * (w1[c] + vt[c]);
            d[c] = disp[c] * ih[c];
        }
        interp_at<T, 3>(u0, N, 1, g, i0, i1, i2, d, cubic, ut);
#pragma unroll
        for (int c = 0; c < 3; ++c) u1[c * N + x] = disp[c] + ut[c];
    }
}

// ---------------------------------------------------------------- map step (FP32)
// The sampled fields are kept as one float4 (x, y, z, 0) per grid point; a step
// leaves u1 and v1 in that form for the next one.  A block owns 4 x 8 x 32
// points and stages the sampled field over them and a halo in shared memory,
// (x, y) and z apart: 12 bytes a point, and a tap is an 8-byte and a 4-byte
// load with constant offsets and two packed multiply-adds.  Points whose
// stencil leaves the box (more than SL_DMAX voxels in the step) gather from
// global memory in the same order.  Bound by shared memory: 128 taps of 12
// bytes a point, 87 us at 128^3.  Taps from L1 instead (16-byte loads, no
// staging) take two cycles where a quarter warp's 128 bytes straddle two
// lines: 262 us a step.
constexpr int SLT0 = 4, SLT1 = 8, SLT2 = 32;
constexpr int SL_DMAX = 1;  // staged displacement per step, voxels
template <bool CUBIC> struct SLBox {
    static constexpr int TLO = CUBIC ? -1 : 0, CNT = CUBIC ? 4 : 2;  // tap offsets TLO .. TLO + CNT - 1
    static constexpr int LO = SL_DMAX - TLO, HI = SL_DMAX + TLO + CNT - 1;
    static constexpr int B0 = SLT0 + LO + HI, B1 = SLT1 + LO + HI, B2 = SLT2 + LO + HI;
    // row pitches of whole 128 bytes, so that the lanes of a warp whose stencils
    // start in different rows still take different banks (without: 49% of the
    // wavefronts were conflicts)
    static constexpr int PXY = (B2 + 15) / 16 * 16, PZ = (B2 + 31) / 32 * 32;
    static constexpr size_t SMEM = (size_t)B0 * B1 * (PXY * 8 + PZ * 4);
};
// The stencil of a point with the wrapped offsets of the taps of each axis.
template <bool CUBIC> struct Sten {
    static constexpr int CNT = CUBIC ? 4 : 2, LO = CUBIC ? -1 : 0;
    int o[3][CNT];  // offsets (points) of the taps of each axis
    float w[3][CNT];
    // first tap of an axis, wrapped (one period off at most for moderate displacements)
    static __device__ __forceinline__ int wrap1(int i, int n) {
        if (i < -n || i >= 2 * n) return wrapi(i, n);
        return i < 0 ? i + n : (i >= n ? i - n : i);
    }
    __device__ __forceinline__ Sten(GridI g, int i0, int i1, int i2, const float d[3]) {
        const int ii[3] = {i0, i1, i2}, nn[3] = {g.n0, g.n1, g.n2}, st[3] = {g.n1 * g.n2, g.n2, 1};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const float fl = floorf(d[a]);
            const float t = d[a] - fl;
            int k = wrap1(ii[a] + (int)fl + LO, nn[a]);
#pragma unroll
            for (int q = 0; q < CNT; ++q) {
                o[a][q] = k * st[a];
                if (++k == nn[a]) k = 0;
            }
            if constexpr (CUBIC) {
                cr_weights(t, w[a]);
            } else {
                w[a][0] = 1.f - t;
                w[a][1] = t;
            }
        }
    }
};
// stage f over the box whose corner is (c0, c1, c2), periodic
template <bool CUBIC>
__device__ __forceinline__ void sl_stage(float2* sxy, float* sz, const float4* __restrict__ f, GridI g, int c0, int c1,
                                         int c2) {
    using B = SLBox<CUBIC>;
    // box coordinates lie in [-LO, n + B - LO): within one period of the grid
    // when n >= B, so one compare and add wraps them; smaller grids take the
    // general modulo
    const bool near = g.n0 >= B::B0 && g.n1 >= B::B1 && g.n2 >= B::B2;
    auto wrap = [near](int x, int n) { return near ? (x < 0 ? x + n : (x >= n ? x - n : x)) : wrapi(x, n); };
    // a thread stages the same columns (b1, b2) of every plane b0
    constexpr int COLS = B::B1 * B::B2, PT = (COLS + SLT1 * SLT2 - 1) / (SLT1 * SLT2);
    const size_t plane = (size_t)g.n1 * g.n2;
#pragma unroll
    for (int q = 0; q < PT; ++q) {
        const int e = threadIdx.x + q * SLT1 * SLT2;
        if (e >= COLS) break;
        const int b1 = e / B::B2, b2 = e - b1 * B::B2;
        const float4* const p = f + (wrap(c1 + b1, g.n1) * g.n2 + wrap(c2 + b2, g.n2));
        float4 v[B::B0];
#pragma unroll
        for (int b0 = 0; b0 < B::B0; ++b0) v[b0] = __ldg(p + wrap(c0 + b0, g.n0) * plane);
#pragma unroll
        for (int b0 = 0; b0 < B::B0; ++b0) {
            sxy[(b0 * B::B1 + b1) * B::PXY + b2] = make_float2(v[b0].x, v[b0].y);
            sz[(b0 * B::B1 + b1) * B::PZ + b2] = v[b0].z;
        }
    }
}
// the interpolant at (i0,i1,i2) + d in interp_at's order: from the staged box
// when the whole stencil lies in it
template <bool CUBIC>
__device__ __forceinline__ void sl_sample(const float2* sxy, const float* sz, const float4* __restrict__ f, GridI g, int i0,
                                          int i1, int i2, int c0, int c1, int c2, const float d[3], float res[3]) {
    using B = SLBox<CUBIC>;
    constexpr int CNT = B::CNT;
    int base[3];
    float w[3][4];
    const int ii[3] = {i0, i1, i2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float fl = floorf(d[a]);
        const float t = d[a] - fl;
        base[a] = ii[a] + (int)fl;
        if constexpr (CUBIC) {
            cr_weights(t, w[a]);
        } else {
            w[a][0] = 1.f - t;
            w[a][1] = t;
        }
    }
    const int l0 = base[0] + B::TLO - c0, l1 = base[1] + B::TLO - c1, l2 = base[2] + B::TLO - c2;
    const bool inside = l0 >= 0 && l1 >= 0 && l2 >= 0 && l0 + CNT <= B::B0 && l1 + CNT <= B::B1 && l2 + CNT <= B::B2;
    if (!inside) {
        interp_at<float, 3>((const float*)f, 1, 4, g, i0, i1, i2, d, CUBIC ? 1 : 0, res);
        return;
    }
    const int r0 = l0 * B::B1 + l1;
    const P2* const pxy = (const P2*)(sxy + r0 * B::PXY + l2);
    const float* const pz = sz + r0 * B::PZ + l2;
    P2 xy = p2(0.f, 0.f), w2[CNT];
    float z = 0.f;
#pragma unroll
    for (int q = 0; q < CNT; ++q) w2[q] = p2(w[2][q], w[2][q]);
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0)
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            P2 rxy = p2(0.f, 0.f);
            float rz = 0.f;
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const P2 vxy = pxy[(a0 * B::B1 + a1) * B::PXY + a2];
                const float vz = pz[(a0 * B::B1 + a1) * B::PZ + a2];
                rxy = a2 == 0 ? w2[0] * vxy : fma2(w2[a2], vxy, rxy);
                rz = a2 == 0 ? w[2][0] * vz : fmaf(w[2][a2], vz, rz);
            }
            const float w01 = w[0][a0] * w[1][a1];
            xy = fma2(p2(w01, w01), rxy, xy);
            z = fmaf(w01, rz, z);
        }
    res[0] = lo(xy);
    res[1] = hi(xy);
    res[2] = z;
}
// planar field -> float4 per point
static __global__ void k_pack4(const float* __restrict__ f, float4* __restrict__ out, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x)
        out[x] = make_float4(f[x], f[N + x], f[2 * N + x], 0.f);
}

constexpr int SL4_X = 32, SL4_Y = 8;
// grid (ceil(n2 / SLT2), ceil(n1 / SLT1), ceil(n0 / SLT0)), SLT1 SLT2 threads; v1
// planar; v1q (nullable): v1 in packed form; u1p: planar copy of u1 (nullable).
// PLAIN: the loops of interp_at alone (cross-check).
template <bool CUBIC, bool PLAIN>
__global__ void __launch_bounds__(SLT1* SLT2, 3) k_sl_step4(GridI g, const float4* __restrict__ v0,
                                                            const float* __restrict__ v1,
                                                            const float4* __restrict__ u0, float4* __restrict__ u1,
                                                            float4* __restrict__ v1q, float* __restrict__ u1p, float dt,
                                                            float ih0, float ih1, float ih2, size_t N) {
    using B = SLBox<CUBIC>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2* const sxy = (float2*)smem_raw;
    float* const sz = (float*)(sxy + B::B0 * B::B1 * B::PXY);
    const float ih[3] = {ih0, ih1, ih2};
    const int o0 = blockIdx.z * SLT0, o1 = blockIdx.y * SLT1, o2 = blockIdx.x * SLT2;
    const int i1 = o1 + threadIdx.x / SLT2, i2 = o2 + threadIdx.x % SLT2;
    const int c0 = o0 - B::LO, c1 = o1 - B::LO, c2 = o2 - B::LO;  // box corner
    const bool col = i1 < g.n1 && i2 < g.n2;
    float disp[SLT0][3];
    if (!PLAIN) sl_stage<CUBIC>(sxy, sz, v0, g, c0, c1, c2);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < SLT0; ++p) {
        const int i0 = o0 + p;
        if (!col || i0 >= g.n0) continue;
        const size_t x = ((size_t)i0 * g.n1 + i1) * g.n2 + i2;
        float w1[3], d[3], s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            w1[c] = __ldg(v1 + c * N + x);
            d[c] = -dt * w1[c] * ih[c];
        }
        if (v1q) v1q[x] = make_float4(w1[0], w1[1], w1[2], 0.f);
        if constexpr (PLAIN) interp_at<float, 3>((const float*)v0, 1, 4, g, i0, i1, i2, d, CUBIC ? 1 : 0, s);
        else sl_sample<CUBIC>(sxy, sz, v0, g, i0, i1, i2, c0, c1, c2, d, s);
#pragma unroll
        for (int c = 0; c < 3; ++c) disp[p][c] = -0.5f * dt * (w1[c] + s[c]);
    }
    __syncthreads();
    if (!PLAIN) sl_stage<CUBIC>(sxy, sz, u0, g, c0, c1, c2);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < SLT0; ++p) {
        const int i0 = o0 + p;
        if (!col || i0 >= g.n0) continue;
        const size_t x = ((size_t)i0 * g.n1 + i1) * g.n2 + i2;
        float d[3], s[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = disp[p][c] * ih[c];
        if constexpr (PLAIN) interp_at<float, 3>((const float*)u0, 1, 4, g, i0, i1, i2, d, CUBIC ? 1 : 0, s);
        else sl_sample<CUBIC>(sxy, sz, u0, g, i0, i1, i2, c0, c1, c2, d, s);
#pragma unroll
        for (int c = 0; c < 3; ++c) s[c] = disp[p][c] + s[c];
        u1[x] = make_float4(s[0], s[1], s[2], 0.f);
        if (u1p) {
#pragma unroll
            for (int c = 0; c < 3; ++c) u1p[c * N + x] = s[c];
        }
    }
}

// m(x) = I(x + u(x))
template <class T>
__global__ void k_warp(GridI g, const T* __restrict__ img, const T* __restrict__ u, T* __restrict__ out, T ih0, T ih1,
                       T ih2, int cubic, size_t N) {
    const T ih[3] = {ih0, ih1, ih2};
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const int i2 = (int)(x % g.n2);
        const int i1 = (int)((x / g.n2) % g.n1);
        const int i0 = (int)(x / ((size_t)g.n2 * g.n1));
        T d[3], r[1];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = u[c * N + x] * ih[c];
        interp_at<T, 1>(img, 0, 1, g, i0, i1, i2, d, cubic, r);
        out[x] = r[0];
    }
}
// the same in FP32, with the stencil's offsets formed once and its loops
// unrolled (100 -> 54 us at 128^3); grid (ceil(n2 / 32), ceil(n1 / 8), n0)
template <bool CUBIC>
__global__ void __launch_bounds__(SL4_X* SL4_Y) k_warp4(GridI g, const float* __restrict__ img, const float* __restrict__ u,
                                                        float* __restrict__ out, float ih0, float ih1, float ih2,
                                                        size_t N) {
    constexpr int CNT = Sten<CUBIC>::CNT;
    const int i2 = blockIdx.x * SL4_X + threadIdx.x % SL4_X, i1 = blockIdx.y * SL4_Y + threadIdx.x / SL4_X;
    const int i0 = blockIdx.z;
    if (i1 >= g.n1 || i2 >= g.n2) return;
    const size_t x = ((size_t)i0 * g.n1 + i1) * g.n2 + i2;
    const float d[3] = {__ldg(u + x) * ih0, __ldg(u + N + x) * ih1, __ldg(u + 2 * N + x) * ih2};
    const Sten<CUBIC> s(g, i0, i1, i2, d);
    float r = 0.f;
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0)
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            const float* const row = img + (s.o[0][a0] + s.o[1][a1]);
            float q = 0.f;
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const float v = __ldg(row + s.o[2][a2]);
                q = a2 == 0 ? s.w[2][0] * v : fmaf(s.w[2][a2], v, q);
            }
            r = fmaf(s.w[0][a0] * s.w[1][a1], q, r);
        }
    out[x] = r;
}

// ---------------------------------------------------------------- exact adjoint of the transport
// Interpolation weights w and their coordinate derivatives dw for one point.
template <class T> __device__ __forceinline__ void cr_dweights(T t, T* dw) {
    const T t2 = t * t;
    dw[0] = (T)0.5 * ((T)-3 * t2 + (T)4 * t - (T)1);
    dw[1] = (T)0.5 * ((T)9 * t2 - (T)10 * t);
    dw[2] = (T)0.5 * ((T)-9 * t2 + (T)8 * t + (T)1);
    dw[3] = (T)0.5 * ((T)3 * t2 - (T)2 * t);
}
// Taps of one point for the Catmull-Rom (CUBIC) or trilinear interpolant,
// with the tap count known at compile time (the weight arrays stay in
// registers).
template <class T, bool CUBIC> struct Taps {
    static constexpr int CNT = CUBIC ? 4 : 2;
    static constexpr int LO = CUBIC ? -1 : 0;
    int base[3];
    T w[3][CNT], dw[3][CNT];
    __device__ __forceinline__ Taps(int i0, int i1, int i2, const T d[3]) {
        const int ii[3] = {i0, i1, i2};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const T fl = floor(d[a]);
            const T t = d[a] - fl;
            base[a] = ii[a] + (int)fl;
            if constexpr (CUBIC) {
                cr_weights(t, w[a]);
                cr_dweights(t, dw[a]);
            } else {
                w[a][0] = (T)1 - t;
                w[a][1] = t;
                dw[a][0] = (T)-1;
                dw[a][1] = (T)1;
            }
        }
    }
};

// d/dp_b of the interpolant of NC fields at the point: G[b][c]
template <class T, bool CUBIC, int NC>
__device__ __forceinline__ void interp_grad_at(const T* __restrict__ f, size_t N, GridI g, const Taps<T, CUBIC>& tp,
                                               T (&G)[3][NC]) {
    constexpr int CNT = Taps<T, CUBIC>::CNT, LO = Taps<T, CUBIC>::LO;
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < NC; ++c) G[b][c] = 0;
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0) {
        const size_t o0 = (size_t)wrapi(tp.base[0] + LO + a0, g.n0) * g.n1;
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            const size_t o1 = (o0 + wrapi(tp.base[1] + LO + a1, g.n1)) * g.n2;
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const size_t o = o1 + wrapi(tp.base[2] + LO + a2, g.n2);
                const T g0 = tp.dw[0][a0] * tp.w[1][a1] * tp.w[2][a2];
                const T g1 = tp.w[0][a0] * tp.dw[1][a1] * tp.w[2][a2];
                const T g2 = tp.w[0][a0] * tp.w[1][a1] * tp.dw[2][a2];
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const T val = __ldg(&f[c * N + o]);
                    G[0][c] += g0 * val;
                    G[1][c] += g1 * val;
                    G[2][c] += g2 * val;
                }
            }
        }
    }
}

// Transpose of the interpolation at the point: fb[taps] += w * vals (atomic)
template <class T, bool CUBIC, int NC>
__device__ __forceinline__ void interp_scatter_at(T* fb, size_t N, GridI g, const Taps<T, CUBIC>& tp,
                                                  const T (&vals)[NC]) {
    constexpr int CNT = Taps<T, CUBIC>::CNT, LO = Taps<T, CUBIC>::LO;
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0) {
        const size_t o0 = (size_t)wrapi(tp.base[0] + LO + a0, g.n0) * g.n1;
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            const size_t o1 = (o0 + wrapi(tp.base[1] + LO + a1, g.n1)) * g.n2;
            const T w01 = tp.w[0][a0] * tp.w[1][a1];
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const size_t o = o1 + wrapi(tp.base[2] + LO + a2, g.n2);
                const T ww = w01 * tp.w[2][a2];
#pragma unroll
                for (int c = 0; c < NC; ++c) atomicAdd(&fb[c * N + o], ww * vals[c]);
            }
        }
    }
}

// Cotangent of the final warp m1 = I0(x + u/h) with respect to u, for
// E_data = ||m1 - I1||^2:  ub(x) = 2 (m1 - I1)(x) dI0/dp(x + u/h) / h.
template <class T, bool CUBIC>
__global__ void k_warp_adj(GridI g, const T* __restrict__ img, const T* __restrict__ u, const T* __restrict__ m1,
                           const T* __restrict__ I1, T* __restrict__ ub, T ih0, T ih1, T ih2, size_t N) {
    const T ih[3] = {ih0, ih1, ih2};
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const int i2 = (int)(x % g.n2);
        const int i1 = (int)((x / g.n2) % g.n1);
        const int i0 = (int)(x / ((size_t)g.n2 * g.n1));
        T d[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) d[c] = u[c * N + x] * ih[c];
        const Taps<T, CUBIC> tp(i0, i1, i2, d);
        T G[3][1];
        interp_grad_at<T, CUBIC, 1>(img, N, g, tp, G);
        const T r2 = (T)2 * (m1[x] - I1[x]);
#pragma unroll
        for (int b = 0; b < 3; ++b) ub[b * N + x] = r2 * G[b][0] * ih[b];
    }
}

// Transpose of one map step (k_sl_step) u_{k+1} = disp + u_k(X),
// X = x + disp/h, disp = -dt/2 (v1 + v0(p1)), p1 = x - dt v1/h:
// from ub1 = dE/du_{k+1}, scatter dE/du_k into ub0 and the v0(p1) part of
// dE/dv_k into vb0 (both atomic), and add the v1 part of dE/dv_{k+1} to vb1.
// (FP64; FP32 runs k_sl_adj4.)
template <class T, bool CUBIC>
__global__ void k_sl_adj(GridI g, const T* __restrict__ v0, const T* __restrict__ v1, const T* __restrict__ u0,
                         const T* __restrict__ ub1, T* ub0, T* vb0, T* __restrict__ vb1, T dt, T ih0, T ih1, T ih2,
                         size_t N) {
    const T ih[3] = {ih0, ih1, ih2};
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const int i2 = (int)(x % g.n2);
        const int i1 = (int)((x / g.n2) % g.n1);
        const int i0 = (int)(x / ((size_t)g.n2 * g.n1));
        T w1[3], d1[3], vt[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            w1[c] = v1[c * N + x];
            d1[c] = -dt * w1[c] * ih[c];
        }
        interp_at<T, 3>(v0, N, 1, g, i0, i1, i2, d1, CUBIC ? 1 : 0, vt);
        T dX[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) dX[c] = (T)-0.5 * dt * (w1[c] + vt[c]) * ih[c];
        const Taps<T, CUBIC> tX(i0, i1, i2, dX);
        T Gu[3][3];
        interp_grad_at<T, CUBIC, 3>(u0, N, g, tX, Gu);
        T ub[3], dispb[3], vtb[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) ub[c] = ub1[c * N + x];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            dispb[b] = ub[b] + ih[b] * (Gu[b][0] * ub[0] + Gu[b][1] * ub[1] + Gu[b][2] * ub[2]);
            vtb[b] = (T)-0.5 * dt * dispb[b];
        }
        interp_scatter_at<T, CUBIC, 3>(ub0, N, g, tX, ub);
        const Taps<T, CUBIC> t1(i0, i1, i2, d1);
        interp_scatter_at<T, CUBIC, 3>(vb0, N, g, t1, vtb);
        T Gv[3][3];
        interp_grad_at<T, CUBIC, 3>(v0, N, g, t1, Gv);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const T p1b = Gv[b][0] * vtb[0] + Gv[b][1] * vtb[1] + Gv[b][2] * vtb[2];
            vb1[b * N + x] += (T)-0.5 * dt * dispb[b] - dt * ih[b] * p1b;
        }
    }
}

// float4 per point -> planar field
static __global__ void k_unpack4(const float4* __restrict__ f, float* __restrict__ out, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const float4 v = f[x];
        out[x] = v.x;
        out[N + x] = v.y;
        out[2 * N + x] = v.z;
    }
}
// weights' derivatives of a stencil
template <bool CUBIC> struct StenD : Sten<CUBIC> {
    float dw[3][Sten<CUBIC>::CNT];
    __device__ __forceinline__ StenD(GridI g, int i0, int i1, int i2, const float d[3]) : Sten<CUBIC>(g, i0, i1, i2, d) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            if constexpr (CUBIC) {
                cr_dweights(d[a] - floorf(d[a]), dw[a]);
            } else {
                dw[a][0] = -1.f;
                dw[a][1] = 1.f;
            }
        }
    }
};
// value r[c] and coordinate derivatives G[b][c] of the interpolant of a packed
// field, the row sums along axis 2 shared between them
template <bool CUBIC>
__device__ __forceinline__ void sample4_grad(const float4* __restrict__ f, const StenD<CUBIC>& s, float r[3],
                                             float (&G)[3][3]) {
    constexpr int CNT = Sten<CUBIC>::CNT;
#pragma unroll
    for (int c = 0; c < 3; ++c) r[c] = G[0][c] = G[1][c] = G[2][c] = 0.f;
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0)
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            const float4* const row = f + (s.o[0][a0] + s.o[1][a1]);
            float q[3] = {0.f, 0.f, 0.f}, p[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const float4 v = __ldg(row + s.o[2][a2]);
                const float x[3] = {v.x, v.y, v.z};
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    q[c] = fmaf(s.w[2][a2], x[c], q[c]);
                    p[c] = fmaf(s.dw[2][a2], x[c], p[c]);
                }
            }
            const float w01 = s.w[0][a0] * s.w[1][a1], d01 = s.dw[0][a0] * s.w[1][a1], w0d = s.w[0][a0] * s.dw[1][a1];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                r[c] = fmaf(w01, q[c], r[c]);
                G[0][c] = fmaf(d01, q[c], G[0][c]);
                G[1][c] = fmaf(w0d, q[c], G[1][c]);
                G[2][c] = fmaf(w01, p[c], G[2][c]);
            }
        }
}
// f[taps] += w x (atomic, 16 bytes a tap)
template <bool CUBIC>
__device__ __forceinline__ void scatter4(float4* f, const Sten<CUBIC>& s, const float x[3]) {
    constexpr int CNT = Sten<CUBIC>::CNT;
#pragma unroll
    for (int a0 = 0; a0 < CNT; ++a0)
#pragma unroll
        for (int a1 = 0; a1 < CNT; ++a1) {
            float4* const row = f + (s.o[0][a0] + s.o[1][a1]);
            const float w01 = s.w[0][a0] * s.w[1][a1];
#pragma unroll
            for (int a2 = 0; a2 < CNT; ++a2) {
                const float w = w01 * s.w[2][a2];
                atomicAdd(row + s.o[2][a2], make_float4(w * x[0], w * x[1], w * x[2], 0.f));
            }
        }
}
// k_sl_adj in FP32 on packed fields: a tap is one 16-byte load or atomic instead
// of three scalar ones, and v0's value and gradient at p1 share their taps.
// Bound by the atomics: 128 of 16 bytes a point.  Grid as k_warp4.
template <bool CUBIC>
__global__ void __launch_bounds__(SL4_X* SL4_Y) k_sl_adj4(GridI g, const float4* __restrict__ v0,
                                                          const float* __restrict__ v1, const float4* __restrict__ u0,
                                                          const float4* __restrict__ ub1, float4* ub0, float4* vb0,
                                                          float4* __restrict__ vb1, float dt, float ih0, float ih1,
                                                          float ih2, size_t N) {
    const int i2 = blockIdx.x * SL4_X + threadIdx.x % SL4_X, i1 = blockIdx.y * SL4_Y + threadIdx.x / SL4_X;
    const int i0 = blockIdx.z;
    if (i1 >= g.n1 || i2 >= g.n2) return;
    const size_t x = ((size_t)i0 * g.n1 + i1) * g.n2 + i2;
    const float ih[3] = {ih0, ih1, ih2};
    float w1[3], d1[3], vt[3], dX[3], Gv[3][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        w1[c] = __ldg(v1 + c * N + x);
        d1[c] = -dt * w1[c] * ih[c];
    }
    sample4_grad<CUBIC>(v0, StenD<CUBIC>(g, i0, i1, i2, d1), vt, Gv);
#pragma unroll
    for (int c = 0; c < 3; ++c) dX[c] = -0.5f * dt * (w1[c] + vt[c]) * ih[c];
    const float4 ubq = ub1[x];
    const float ub[3] = {ubq.x, ubq.y, ubq.z};
    float dispb[3], vtb[3];
    {
        const StenD<CUBIC> tX(g, i0, i1, i2, dX);
        float ut[3], Gu[3][3];
        sample4_grad<CUBIC>(u0, tX, ut, Gu);
        scatter4<CUBIC>(ub0, tX, ub);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            dispb[b] = ub[b] + ih[b] * (Gu[b][0] * ub[0] + Gu[b][1] * ub[1] + Gu[b][2] * ub[2]);
            vtb[b] = -0.5f * dt * dispb[b];
        }
    }
    scatter4<CUBIC>(vb0, Sten<CUBIC>(g, i0, i1, i2, d1), vtb);
    float4 o = vb1[x];
    float add[3];
#pragma unroll
    for (int b = 0; b < 3; ++b)
        add[b] = -0.5f * dt * dispb[b] - dt * ih[b] * (Gv[b][0] * vtb[0] + Gv[b][1] * vtb[1] + Gv[b][2] * vtb[2]);
    o.x += add[0];
    o.y += add[1];
    o.z += add[2];
    vb1[x] = o;
}

// ---------------------------------------------------------------- reductions
// Deterministic two-phase double reductions: block partials, then one block.
constexpr int RED_THREADS = 256;
constexpr int RED_BLOCKS = 592;  // 4 x 148..152 SMs; partial buffer size

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// op: 0 sum, 1 max, 2 min
__device__ __forceinline__ double block_reduce(double v, int op) {
    __shared__ double sh[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    v = op == 0 ? warp_sum(v) : (op == 1 ? warp_max(v) : warp_min(v));
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    const int nw = blockDim.x >> 5;
    const double id = op == 0 ? 0.0 : (op == 1 ? -1.0e300 : 1.0e300);
    v = threadIdx.x < nw ? sh[threadIdx.x] : id;
    if (wid == 0) v = op == 0 ? warp_sum(v) : (op == 1 ? warp_max(v) : warp_min(v));
    __syncthreads();
    return v;
}

// 16-byte loads of an array that may start anywhere: V elements at a time from
// its first 16-byte boundary, the few before and after it one by one.  A
// reduction that reads one element per thread and step is bound by the latency
// of its loads (0.9 TB/s at 3 x 128^3 FP32); four 16-byte loads in flight per
// thread bring it to the rate of its FP64 adds or of memory.
template <class T> struct Vec16 {
    static constexpr int V = 16 / (int)sizeof(T);
    T v[V];
};
__device__ __forceinline__ Vec16<float> ld16(const float* p) {
    const float4 q = __ldg((const float4*)p);
    return {{q.x, q.y, q.z, q.w}};
}
__device__ __forceinline__ Vec16<double> ld16(const double* p) {
    const double2 q = __ldg((const double2*)p);
    return {{q.x, q.y}};
}
// elements of a before its first 16-byte boundary (at most n)
template <class T> __device__ __forceinline__ size_t head16(const T* a, size_t n) {
    const size_t h = ((16 - ((size_t)a & 15)) & 15) / sizeof(T);
    return h < n ? h : n;
}

// what a dot product sums: a b, a^2, or (a - b)^2
enum { DOT_AB = 0, DOT_AA = 1, DOT_DIFF = 2 };
template <class T, int KIND> __device__ __forceinline__ double dot_term(T a, T b) {
    if (KIND == DOT_AB) return (double)a * (double)b;
    const double x = KIND == DOT_AA ? (double)a : (double)(a - b);
    return x * x;
}
// partial[block] = sum over this block's share of the terms
template <class T, int KIND>
__global__ void k_dot_partial(const T* __restrict__ a, const T* __restrict__ b, size_t n, double* __restrict__ partial) {
    constexpr int V = Vec16<T>::V, U = 4;
    const size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    double acc[U] = {0.0, 0.0, 0.0, 0.0};
    size_t done = 0;
    if (KIND == DOT_AA || (((size_t)a ^ (size_t)b) & 15) == 0) {
        const size_t h = head16(a, n), nv = (n - h) / V;
        if (id < h) acc[0] += dot_term<T, KIND>(a[id], KIND == DOT_AA ? (T)0 : b[id]);
        for (size_t q = id; q < nv; q += U * step) {
            Vec16<T> x[U], y[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const size_t i = q + u * step;
                if (i < nv) {
                    x[u] = ld16(a + h + i * V);
                    if (KIND != DOT_AA) y[u] = ld16(b + h + i * V);
                }
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (q + u * step < nv) {
#pragma unroll
                    for (int e = 0; e < V; ++e) acc[u] += dot_term<T, KIND>(x[u].v[e], KIND == DOT_AA ? (T)0 : y[u].v[e]);
                }
        }
        done = h + nv * V;
    }
    for (size_t x = done + id; x < n; x += step) acc[0] += dot_term<T, KIND>(a[x], KIND == DOT_AA ? (T)0 : b[x]);
    const double s = block_reduce((acc[0] + acc[1]) + (acc[2] + acc[3]), 0);
    if (threadIdx.x == 0) partial[blockIdx.x] = s;
}

// partial[block] = sum over the half spectrum F(v) [k2][k0][k1] of three
// components (stride cs) of L |F(v)|^2, entries with a conjugate partner
// twice: N <L v, v> by Parseval's identity
template <class T>
__global__ void k_spec_energy(const cpx<T>* __restrict__ vh, size_t cs, SpecTabs<T> tb, int n0, int n1, int n2h,
                              double* __restrict__ partial) {
    double acc = 0.0;
    const int rows = n0 * n2h;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int k2 = r / n0, k0 = r - k2 * n0;
        const double w = k2 == 0 || 2 * k2 == tb.n[2] ? 1.0 : 2.0;
        const T q = tb.ksq[0][k0] + tb.ksq[2][k2];
        for (int k1 = threadIdx.x; k1 < n1; k1 += blockDim.x) {
            const T base = (T)1 + tb.alpha * (q + tb.ksq[1][k1]);
            T L = (T)1;
            for (int e = 0; e < tb.s; ++e) L *= base;
            const size_t x = (size_t)r * n1 + k1;
            double m = 0.0;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const cpx<T> z = vh[c * cs + x];
                m += (double)z.x * (double)z.x + (double)z.y * (double)z.y;
            }
            acc += w * (double)L * m;
        }
    }
    acc = block_reduce(acc, 0);
    if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// partial[3*b + {0,1,2}] = {max|a|, max a, min a}
template <class T>
__global__ void k_absmax_partial(const T* __restrict__ a, size_t n, double* __restrict__ partial) {
    double am = 0.0, mx = -1.0e300, mn = 1.0e300;
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < n; x += (size_t)gridDim.x * blockDim.x) {
        const double v = (double)a[x];
        am = fmax(am, fabs(v));
        mx = fmax(mx, v);
        mn = fmin(mn, v);
        if (v != v) am = 1.0e308;  // NaN poisons max|a|
    }
    am = block_reduce(am, 1);
    mx = block_reduce(mx, 1);
    mn = block_reduce(mn, 2);
    if (threadIdx.x == 0) {
        partial[3 * blockIdx.x] = am;
        partial[3 * blockIdx.x + 1] = mx;
        partial[3 * blockIdx.x + 2] = mn;
    }
}

// Non-finite scan of up to SCAN_MAX arrays: *flag = 1 when any entry is a
// NaN or an infinity (the flag is never cleared; the caller's status is
// sticky).  The result does not depend on the launch shape.
constexpr int SCAN_MAX = 4;
template <class T> struct ScanArgs {
    const T* p[SCAN_MAX];
    size_t n[SCAN_MAX];
    int cnt;
};
template <class T>
__global__ void k_nonfinite_scan(const __grid_constant__ ScanArgs<T> a, double* __restrict__ flag) {
    bool bad = false;
    constexpr int V = Vec16<T>::V, U = 4;
    const size_t id = blockIdx.x * (size_t)blockDim.x + threadIdx.x, step = (size_t)gridDim.x * blockDim.x;
    for (int k = 0; k < a.cnt; ++k) {
        const T* const p = a.p[k];
        const size_t n = a.n[k], h = head16(p, n), nv = (n - h) / V;
        if (id < h) bad |= !isfinite(p[id]);
        for (size_t q = id; q < nv; q += U * step) {
            Vec16<T> x[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const size_t i = q + u * step;
                if (i < nv) x[u] = ld16(p + h + i * V);
                else x[u] = Vec16<T>{};
            }
#pragma unroll
            for (int u = 0; u < U; ++u)
#pragma unroll
                for (int e = 0; e < V; ++e) bad |= !isfinite(x[u].v[e]);
        }
        for (size_t x = h + nv * V + id; x < n; x += step) bad |= !isfinite(p[x]);
    }
    if (__syncthreads_or(bad) && threadIdx.x == 0) *flag = 1.0;
}

// out[slot] = scale * reduce(partial[0..nb*stride) with the given stride/offset)
static __global__ void k_finish(const double* __restrict__ partial, int nb, int stride, int off, int op, double scale,
                         double* __restrict__ out) {
    const double id = op == 0 ? 0.0 : (op == 1 ? -1.0e300 : 1.0e300);
    double v = id;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        const double p = partial[i * stride + off];
        v = op == 0 ? v + p : (op == 1 ? fmax(v, p) : fmin(v, p));
    }
    v = block_reduce(v, op);
    if (threadIdx.x == 0) *out = scale * v;
}

// ---------------------------------------------------------------- small pointwise ops
// y = a*x + b*y  over n values
template <class T>
__global__ void k_axpby(T a, const T* __restrict__ x, T b, T* __restrict__ y, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        y[i] = a * x[i] + b * y[i];
}
// z = a*x + b*y
template <class T>
__global__ void k_lincomb2(T a, const T* __restrict__ x, T b, const T* __restrict__ y, T* __restrict__ z, size_t n) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        z[i] = a * x[i] + b * y[i];
}

// Final-time sources.  mode 0 (gradient):  out_c = -2 (m1 - I1) grad_c m1
//                      mode 1 (Gauss-Newton): out_c = 2 (grad m1 . xi) grad_c m1
template <class T>
__global__ void k_final_source(const T* __restrict__ m1, const T* __restrict__ I1, const T* __restrict__ gm,
                               const T* __restrict__ xi, T* __restrict__ out, int mode, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const T g0 = gm[x], g1 = gm[N + x], g2 = gm[2 * N + x];
        T f;
        if (mode == 0) f = (T)-2 * (m1[x] - I1[x]);
        else f = (T)2 * (g0 * xi[x] + g1 * xi[N + x] + g2 * xi[2 * N + x]);
        out[x] = f * g0;
        out[N + x] = f * g1;
        out[2 * N + x] = f * g2;
    }
}

// Source of the shooting vector-Jacobian product: out_c = -G grad_c m1
template <class T>
__global__ void k_vjp_source(const T* __restrict__ G, const T* __restrict__ gm, T* __restrict__ out, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        const T g = -G[x];
        out[x] = g * gm[x];
        out[N + x] = g * gm[N + x];
        out[2 * N + x] = g * gm[2 * N + x];
    }
}

// det(I + Du), Du[c][j] = D_j u_c at field 3c + j
template <class T>
__global__ void k_jacdet(const T* __restrict__ Du, T* __restrict__ J, size_t N) {
    for (size_t x = blockIdx.x * (size_t)blockDim.x + threadIdx.x; x < N; x += (size_t)gridDim.x * blockDim.x) {
        T a[3][3];
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int j = 0; j < 3; ++j) a[c][j] = Du[(3 * c + j) * N + x] + (c == j ? (T)1 : (T)0);
        J[x] = a[0][0] * (a[1][1] * a[2][2] - a[1][2] * a[2][1]) - a[0][1] * (a[1][0] * a[2][2] - a[1][2] * a[2][0]) +
               a[0][2] * (a[1][0] * a[2][1] - a[1][1] * a[2][0]);
    }
}

// Spectral-space combination on [k2][k0][k1] arrays: out = sum_b sym_b . in_b
template <class T> struct SpecComb {
    const cpx<T>* in[MAXI];
    SymT<T> sym[MAXI];
    int nin;
};
// A block walks (k2, k0) rows of n1 entries; its threads take the k1 of a
// row, so that the frequency indices cost one division per row.
template <class T>
__global__ void k_spec_comb(SpecComb<T> sc, SpecTabs<T> tb, int n0, int n1, int n2h, cpx<T>* __restrict__ out) {
    const int rows = n0 * n2h;
    for (int r = blockIdx.x; r < rows; r += gridDim.x) {
        const int k2 = r / n0, k0 = r - k2 * n0;
        const size_t base = (size_t)r * n1;
        for (int k1 = threadIdx.x; k1 < n1; k1 += blockDim.x) {
            const size_t x = base + k1;
            cpx<T> acc = mk((T)0, (T)0);
            for (int b = 0; b < sc.nin; ++b) acc = acc + sym_apply(sc.sym[b], tb, k0, k1, k2, sc.in[b][x]);
            out[x] = acc;
        }
    }
}
// launch shape of k_spec_comb: threads per block (whole warps covering a row, at most 256), blocks
inline int spec_comb_threads(int n1) { return n1 >= 256 ? 256 : ((n1 + 31) / 32) * 32; }
inline int spec_comb_blocks(int n0, int n2h) { return n0 * n2h < 152 * 16 ? n0 * n2h : 152 * 16; }

}  // namespace lddmm
