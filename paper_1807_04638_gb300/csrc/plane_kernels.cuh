// The kernels of plane.cuh: both axes of a plane (PH = 3), or one (PH = 1: axis
// 1, PH = 2: axis 0).
#pragma once
#include "plane.cuh"

namespace lddmm {

// The middle stage of a three-stage transform over `lines` lines: element p
// of line l at S[p ps + l ls]; ll line slots (fl divides by it).  NAT: natural placement, else in place.
template <class T, int DIR, bool NAT>
__device__ __forceinline__ void mid_stage(cpx<T>* S, int ps, int ls, int lines, int ll, const FastDiv& fl, const RPlan& pl,
                                          const cpx<T>* tw) {
    const int items = (pl.n / pl.b) * ll;
    LDDMM_MID(pl.b, {
        for (int i = threadIdx.x; i < items; i += blockDim.x) {
            const int it = (int)fl.div((unsigned)i), l = i - it * ll;
                if (l >= lines) continue;
            const int j2 = (int)pl.fa.div((unsigned)it), q0 = it - j2 * pl.a;  // j2 < c
            cpx<T>* s = S + l * ls + (NAT ? (q0 + pl.a * R * j2) : (q0 * R * pl.c + j2)) * ps;
            const int st = (NAT ? pl.a : pl.c) * ps;
            cpx<T> v[R];
LDDMM_UNROLL
            for (int r = 0; r < R; ++r) v[r] = s[r * st];
            dft<R, DIR>(v);
            twiddles<R, DIR>(v, tw, pl.a * j2);
LDDMM_UNROLL
            for (int r = 0; r < R; ++r) s[r * st] = v[r];
        }
    })
    __syncthreads();
}

template <class T, int PH>
__global__ void __launch_bounds__(512) k_plane_inv(const __grid_constant__ PlaneArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Band& bd = a.bd;
    const PlaneJob<T>& job = a.jobs[blockIdx.y];
    const int n0 = bd.n0, n1 = bd.n1, b0 = bd.b0;
    const int pitch = PH == 1 ? a.tile : (n0 | 1);
    const int nt_ = PH == 3 ? 1 : (PH == 1 ? (b0 + a.tile - 1) / a.tile : (n1 + a.tile - 1) / a.tile);
    const int k2 = PH == 3 ? blockIdx.x : blockIdx.x / nt_;
    const int t0 = PH == 3 ? 0 : (blockIdx.x - k2 * nt_) * a.tile;
    cpx<T>* const S = (cpx<T>*)smem_raw;
    cpx<T>* const tw0 = S + (PH == 3 ? pitch * n1 : (PH == 1 ? n1 * a.tile : pitch * a.tile));
    cpx<T>* const tw1 = tw0 + n0;
    if (PH & 2)
        for (int i = threadIdx.x; i < n0; i += blockDim.x) tw0[i] = ldg(a.tw0 + i);
    if (PH & 1) {
        for (int i = threadIdx.x; i < n1; i += blockDim.x) tw1[i] = ldg(a.tw1 + i);
        __syncthreads();
        // ---- k1 -> i1 over the columns k0c of the tile
        const RPlan& pl = a.pl1;
        const int cols = PH == 3 ? b0 : min(a.tile, b0 - t0);
        const int cl = PH == 3 ? b0 : a.tile;  // column slots of an item row
        auto divc = [&](int i) { return (int)(PH == 3 ? bd.fb0 : a.ft).div((unsigned)i); };
        const T k2v = a.dk[2][k2];
        const int ns = job.kind == 0 ? 1 : 3;
        LDDMM_FIRST(pl.a, {
            const int M = pl.n / R, items = M * cl;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int j = divc(i), cc = i - j * cl, kc = t0 + cc;
                if (cc >= cols) continue;
                const int k0 = band_k(kc, bd.p0, b0, n0);
                const T k0v = a.dk[0][k0];
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) {
                    const int k1 = j + r * M;
                    const int c1 = band_c(k1, bd.p1, bd.b1, n1);
                    cpx<T> x = mk((T)0, (T)0);
                    if (c1 >= 0) {
                        const int o = (k2 * bd.b1 + c1) * bd.b0p + kc;
                        const cpx<T>* p = job.in + o;
                        const T f = job.tab ? job.scale * job.tab[o] : job.scale;
                        if (ns == 1) {
                            x = f * p[0];
                        } else {
                            const T k1v = a.dk[1][k1];
                            // curl component c: kappa_{c+1} X_{c+2} - kappa_{c+2} X_{c+1}
                            cpx<T> s;
                            if (job.kind == 1) s = k0v * p[0] + k1v * p[a.cs] + k2v * p[2 * a.cs];
                            else if (job.kind == 2) s = k1v * p[2 * a.cs] - k2v * p[a.cs];
                            else if (job.kind == 3) s = k2v * p[0] - k0v * p[2 * a.cs];
                            else s = k0v * p[a.cs] - k1v * p[0];
                            x = mk(-f * s.y, f * s.x);
                        }
                    }
                    v[r] = x;
                }
                dft<R, 1>(v);
                twiddles<R, 1>(v, tw1, j);
                // natural placement; line slot: true k0 (both axes) or the tile column
                const int r1 = (int)pl.fc.div((unsigned)j), j2 = j - r1 * pl.c;
                cpx<T>* s = S + (R * (r1 + pl.b * j2)) * pitch + (PH == 3 ? k0 : cc);
LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * pitch] = v[q];
            }
        })
        __syncthreads();
        if (pl.b > 1) {
            const int items = (pl.n / pl.b) * cl;
            LDDMM_MID(pl.b, {
                for (int i = threadIdx.x; i < items; i += blockDim.x) {
                    const int it = divc(i), cc = i - it * cl;
                if (cc >= cols) continue;
                    const int j2 = (int)pl.fa.div((unsigned)it), q0 = it - j2 * pl.a;
                    cpx<T>* s = S + (q0 + pl.a * R * j2) * pitch + (PH == 3 ? band_k(cc, bd.p0, b0, n0) : cc);
                    const int st = pl.a * pitch;
                    cpx<T> v[R];
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, 1>(v);
                    twiddles<R, 1>(v, tw1, pl.a * j2);
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        LDDMM_LAST(pl.c, {
            const int M = pl.n / R, items = M * cl;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int it = divc(i), cc = i - it * cl;
                if (cc >= cols) continue;
                cpx<T>* s = S + it * pitch + (PH == 3 ? band_k(cc, bd.p0, b0, n0) : cc);
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r * M * pitch];
                dft<R, 1>(v);
                if (PH == 3) {
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * M * pitch] = v[r];
                } else {
                    cpx<T>* o = a.mid + blockIdx.y * a.mids + ((size_t)k2 * n1 + it) * bd.b0p + t0 + cc;
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) o[r * M * bd.b0p] = v[r];
                }
            }
        })
        __syncthreads();
    }
    if (PH & 2) {
        // ---- k0 -> i0 over the lines i1 of the tile
        const RPlan& pl = a.pl0;
        const int lines = PH == 3 ? n1 : min(a.tile, n1 - t0);
        if (PH == 2) {
            const cpx<T>* src = a.mid + blockIdx.y * a.mids + ((size_t)k2 * n1 + t0) * bd.b0p;
            for (int i = threadIdx.x; i < lines * b0; i += blockDim.x) {
                const int l = (int)bd.fb0.div((unsigned)i), kc = i - l * b0;
                S[l * pitch + band_k(kc, bd.p0, b0, n0)] = src[l * bd.b0p + kc];
            }
            __syncthreads();
        }
        const int ll = PH == 3 ? n1 : a.tile;
        auto divl = [&](int i) { return (int)(PH == 3 ? bd.fn1 : a.ft).div((unsigned)i); };
        LDDMM_FIRST(pl.a, {
            const int M = pl.n / R, items = M * ll;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int j = divl(i), l = i - j * ll;
                if (l >= lines) continue;
                cpx<T>* s = S + l * pitch + j;
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r)
                    v[r] = band_c(j + r * M, bd.p0, b0, n0) >= 0 ? s[r * M] : mk((T)0, (T)0);
                dft<R, 1>(v);
                twiddles<R, 1>(v, tw0, j);
LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * M] = v[q];
            }
        })
        __syncthreads();
        if (pl.b > 1) mid_stage<T, 1, false>(S, 1, pitch, lines, ll, PH == 3 ? bd.fn1 : a.ft, pl, tw0);
        cpx<T>* out = job.out + (size_t)k2 * n0 * n1 + t0;
        LDDMM_LAST(pl.c, {
            const int items = (pl.n / R) * ll;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int it = divl(i), l = i - it * ll;
                if (l >= lines) continue;
                const int q0 = (int)pl.fb.div((unsigned)it), q1 = it - q0 * pl.b;
                const cpx<T>* s = S + l * pitch + it * R;
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r];
                dft<R, 1>(v);
                cpx<T>* o = out + (q0 + pl.a * q1) * n1 + l;
                const int st = pl.a * pl.b * n1;
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) o[r * st] = v[r];
            }
        })
    }
}

template <class T, int PH>
__global__ void __launch_bounds__(512) k_plane_fwd(const __grid_constant__ PlaneArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const Band& bd = a.bd;
    const PlaneJob<T>& job = a.jobs[blockIdx.y];
    const int n0 = bd.n0, n1 = bd.n1, b0 = bd.b0;
    const int pitch = PH == 1 ? a.tile : (n0 | 1);
    const int nt_ = PH == 3 ? 1 : (PH == 1 ? (b0 + a.tile - 1) / a.tile : (n1 + a.tile - 1) / a.tile);
    const int k2 = PH == 3 ? blockIdx.x : blockIdx.x / nt_;
    const int t0 = PH == 3 ? 0 : (blockIdx.x - k2 * nt_) * a.tile;
    cpx<T>* const S = (cpx<T>*)smem_raw;
    cpx<T>* const tw0 = S + (PH == 3 ? pitch * n1 : (PH == 1 ? n1 * a.tile : pitch * a.tile));
    cpx<T>* const tw1 = tw0 + n0;
    if (PH & 2)
        for (int i = threadIdx.x; i < n0; i += blockDim.x) tw0[i] = ldg(a.tw0 + i);
    if (PH & 1)
        for (int i = threadIdx.x; i < n1; i += blockDim.x) tw1[i] = ldg(a.tw1 + i);
    __syncthreads();
    if (PH & 2) {
        // ---- i0 -> k0 over the lines i1 of the tile
        const RPlan& pl = a.pl0;
        const int lines = PH == 3 ? n1 : min(a.tile, n1 - t0);
        const int ll = PH == 3 ? n1 : a.tile;
        auto divl = [&](int i) { return (int)(PH == 3 ? bd.fn1 : a.ft).div((unsigned)i); };
        const cpx<T>* in = job.in + (size_t)k2 * n0 * n1 + t0;
        LDDMM_FIRST(pl.a, {
            const int M = pl.n / R, items = M * ll;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int j = divl(i), l = i - j * ll;
                if (l >= lines) continue;
                const cpx<T>* p = in + j * n1 + l;
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = p[r * M * n1];
                dft<R, -1>(v);
                twiddles<R, -1>(v, tw0, j);
                const int r1 = (int)pl.fc.div((unsigned)j), j2 = j - r1 * pl.c;
                cpx<T>* s = S + l * pitch + R * (r1 + pl.b * j2);
LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q] = v[q];
            }
        })
        __syncthreads();
        if (pl.b > 1) mid_stage<T, -1, true>(S, 1, pitch, lines, ll, PH == 3 ? bd.fn1 : a.ft, pl, tw0);
        LDDMM_LAST(pl.c, {
            const int M = pl.n / R, items = M * ll;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int it = divl(i), l = i - it * ll;
                if (l >= lines) continue;
                cpx<T>* s = S + l * pitch + it;
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r * M];
                dft<R, -1>(v);
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) s[r * M] = v[r];
            }
        })
        __syncthreads();
        if (PH == 2) {
            cpx<T>* dst = a.mid + blockIdx.y * a.mids + ((size_t)k2 * n1 + t0) * bd.b0p;
            for (int i = threadIdx.x; i < lines * b0; i += blockDim.x) {
                const int l = (int)bd.fb0.div((unsigned)i), kc = i - l * b0;
                dst[l * bd.b0p + kc] = S[l * pitch + band_k(kc, bd.p0, b0, n0)];
            }
        }
    }
    if (PH & 1) {
        // ---- i1 -> k1 over the columns k0c of the tile
        const RPlan& pl = a.pl1;
        const int cols = PH == 3 ? b0 : min(a.tile, b0 - t0);
        const int cl = PH == 3 ? b0 : a.tile;
        auto divc = [&](int i) { return (int)(PH == 3 ? bd.fb0 : a.ft).div((unsigned)i); };
        const cpx<T>* mid = PH == 1 ? a.mid + blockIdx.y * a.mids + (size_t)k2 * n1 * bd.b0p + t0 : nullptr;
        LDDMM_FIRST(pl.a, {
            const int M = pl.n / R, items = M * cl;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int j = divc(i), cc = i - j * cl;
                if (cc >= cols) continue;
                cpx<T>* s = S + j * pitch + (PH == 3 ? band_k(cc, bd.p0, b0, n0) : cc);
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = PH == 3 ? s[r * M * pitch] : mid[(j + r * M) * bd.b0p + cc];
                dft<R, -1>(v);
                twiddles<R, -1>(v, tw1, j);
LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * M * pitch] = v[q];
            }
        })
        __syncthreads();
        if (pl.b > 1) {
            const int items = (pl.n / pl.b) * cl;
            LDDMM_MID(pl.b, {
                for (int i = threadIdx.x; i < items; i += blockDim.x) {
                    const int it = divc(i), cc = i - it * cl;
                if (cc >= cols) continue;
                    const int j2 = (int)pl.fa.div((unsigned)it), q0 = it - j2 * pl.a;
                    cpx<T>* s = S + (q0 * R * pl.c + j2) * pitch + (PH == 3 ? band_k(cc, bd.p0, b0, n0) : cc);
                    const int st = pl.c * pitch;
                    cpx<T> v[R];
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, -1>(v);
                    twiddles<R, -1>(v, tw1, pl.a * j2);
LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        LDDMM_LAST(pl.c, {
            const int items = (pl.n / R) * cl;
            for (int i = threadIdx.x; i < items; i += blockDim.x) {
                const int it = divc(i), cc = i - it * cl;
                if (cc >= cols) continue;
                const int q0 = (int)pl.fb.div((unsigned)it), q1 = it - q0 * pl.b;
                const cpx<T>* s = S + it * R * pitch + (PH == 3 ? band_k(cc, bd.p0, b0, n0) : cc);
                cpx<T> v[R];
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r * pitch];
                dft<R, -1>(v);
                cpx<T>* o = job.out + (size_t)k2 * bd.b1 * bd.b0p + t0 + cc;
LDDMM_UNROLL
                for (int r = 0; r < R; ++r) {
                    const int c1 = band_c(q0 + pl.a * (q1 + pl.b * r), bd.p1, bd.b1, n1);
                    if (c1 >= 0) o[c1 * bd.b0p] = v[r];
                }
            }
        })
    }
}

}  // namespace lddmm
