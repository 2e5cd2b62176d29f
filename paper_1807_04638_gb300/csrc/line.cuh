// FP32 axis-0 and axis-1 transforms of the band (see plane.cuh for the data and
// the symbols), one axis per launch with the line length compiled in.
//
// A block of 64 or 128 threads transforms 16 lines, two per thread packed side
// by side (P2): c < 8 is the line pair (lanes), m the item of a stage.  Small
// blocks keep a barrier between two to four warps and leave many of them on an
// SM, so that loads, butterflies and stores of different lines overlap; with
// radices up to 16 most lengths need one exchange through shared memory
// ([place][pair], 16 bytes a pair: no bank conflicts, constant offsets).
//   MODE 0  inverse, axis 1: band spectra [k2][k1c][k0c], symbol applied while
//           loading, lines = columns k0c -> mid [k2][i1][k0c]
//   MODE 1  inverse, axis 0: mid, lines i1 -> [k2][i0][i1]
//   MODE 2  forward, axis 0: [k2][i0][i1] -> mid (band entries k0c)
//   MODE 3  forward, axis 1: mid -> band spectra
// The transposition between the axes is in the access to mid by the axis-0
// kernels: a warp's 8-byte accesses cover four neighbouring k0c of eight lines,
// whole 32-byte sectors.
//
// Bound by the latency of their loads (long_scoreboard; 13 warps an SM, as many
// as the registers leave room for): 4.4 TB/s of algorithmic bytes a launch
// inverse, 4.1 forward.  At 128^3 a launch takes 23 us on average inverse and 22
// forward (an inverse one 38 us with run-time radices, 35 us with the band's
// limits taken from the arguments); radices of
// at most 10 or 8 make the whole product 16 % slower (more exchanges), 10 or 12
// blocks of 64 threads an SM the launch 12 to 14 % (registers).
#pragma once
#include "plane.cuh"

namespace lddmm {

constexpr int LINE_RB = 8;  // line pairs per block
__host__ __device__ constexpr int line_slots(int n) { return n <= 128 ? 8 : 16; }  // item slots (threads / LINE_RB)
__host__ __device__ constexpr int line_threads(int n) { return LINE_RB * line_slots(n); }
__host__ __device__ constexpr size_t line_smem(int n) { return (size_t)16 * n * LINE_RB + 24 * (size_t)n; }

// The band of a line of N entries under the 2/3 rule, as the spectra store it:
// entry k -> place, or -1 (most comparisons are settled at compile time).
template <int N> struct LineBand {
    static constexpr int kc = (N - 1) / 3, p = kc + 1, b = 2 * kc + 1;
    // the place of k = j + r M, 0 <= j < M
    template <int M> static __device__ __forceinline__ int at(int j, int r) {
        if (r * M + M <= p) return j + r * M;            // every j inside, non-negative wave numbers
        if (r * M >= N - kc) return j + r * M - (N - b);  // inside, negative ones
        if (r * M >= p && r * M + M <= N - kc) return -1;
        const int k = j + r * M;
        return k < p ? k : (k >= N - kc ? k - (N - b) : -1);
    }
};

template <int N, int AA, int BB, int CC, int MODE>
__global__ void __launch_bounds__(line_threads(N), 512 / line_threads(N)) k_line(const __grid_constant__ PlaneArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    static_assert(AA * BB * CC == N, "radices of the length");
    using C2 = cpx<P2>;
    constexpr int DIR = MODE < 2 ? 1 : -1, AXIS = MODE == 0 || MODE == 3 ? 1 : 0, RB = LINE_RB, T = line_slots(N);
    C2* const bufs = (C2*)smem_raw;
    C2* const tws = bufs + N * RB;
    P2* const twn = (P2*)(tws + N);
    const cpx<float>* const tw = AXIS == 1 ? a.tw1 : a.tw0;
    for (int i = threadIdx.x; i < N; i += T * RB) {
        const cpx<float> t = ldg(tw + i);
        tws[i] = mk(p2(t.x, t.x), p2(t.y, t.y));
        twn[i] = p2(-t.y, -t.y);
    }
    const Band& bd = a.bd;
    const PlaneJob<float>& job = a.jobs[blockIdx.z];
    const int c = threadIdx.x % RB, m = threadIdx.x / RB, k2 = blockIdx.y;
    const int l0 = 2 * (blockIdx.x * RB + c);  // first line of the pair: k0c (axis 1) or i1 (axis 0)
    const int lines = AXIS == 1 ? bd.b0 : bd.n1;
    const bool on = l0 < lines;
    const int b0p = bd.b0p, n1 = AXIS == 1 ? N : bd.n1;
    C2* const buf = bufs + c;
    // What the kernel in front wrote is read by plain loads from here on: it may
    // have been written while this kernel ran, which a read-only load (__ldg)
    // rules out and may be moved in front of the wait for.
    auto one = [](const cpx<float>* p) {
        const float2 v = *(const float2*)p;
        return mk(v.x, v.y);
    };
    after_previous();
    __syncthreads();

    // ---- stage 0: element n = j + r M of the line
    constexpr int M = N / AA;
#pragma unroll 1
    for (int j = m; j < M; j += T) {
        C2 v[AA];
#pragma unroll
        for (int r = 0; r < AA; ++r) v[r] = mk(p2(0.f, 0.f), p2(0.f, 0.f));
        if (on) {
            auto pair = [](float4 q) { return mk(p2(q.x, q.z), p2(q.y, q.w)); };
            if constexpr (MODE == 0) {
                const float* const tab = job.tab;
                const int ka = band_k(l0, bd.p0, bd.b0, bd.n0), kb = min(band_k(l0 + 1, bd.p0, bd.b0, bd.n0), bd.n0 - 1);
                const P2 sc = p2(job.scale, job.scale);
                const unsigned o0 = (unsigned)k2 * (unsigned)(bd.b1 * b0p) + (unsigned)l0;
                if (job.kind == 0) {
#pragma unroll
                    for (int r = 0; r < AA; ++r) {
                        const int c1 = LineBand<N>::template at<M>(j, r);
                        if (c1 >= 0) v[r] = pair(*(const float4*)(job.in + o0 + (unsigned)(c1 * b0p)));
                    }
                } else {
                    const P2 k0v = p2(a.dk[0][ka], a.dk[0][kb]);
                    const float k2s = a.dk[2][k2];
                    const P2 k2v = p2(k2s, k2s);
                    // curl component q: kappa_{q+1} X_{q+2} - kappa_{q+2} X_{q+1}
                    const int q = job.kind - 2;
                    const cpx<float>* const pa = job.in + (q == 1 ? 0 : (q == 0 ? 2 : 1)) * a.cs;
                    const cpx<float>* const pb = job.in + (q == 2 ? 0 : (q == 0 ? 1 : 2)) * a.cs;
#pragma unroll
                    for (int r = 0; r < AA; ++r) {
                        const int k1 = j + r * M, c1 = LineBand<N>::template at<M>(j, r);
                        if (c1 < 0) continue;
                        const unsigned o = o0 + (unsigned)(c1 * b0p);
                        const float k1s = a.dk[1][k1];
                        const P2 k1v = p2(k1s, k1s);
                        C2 s;
                        if (job.kind == 1) {
                            const C2 x0 = pair(*(const float4*)(job.in + o));
                            const C2 x1 = pair(*(const float4*)(job.in + a.cs + o));
                            const C2 x2 = pair(*(const float4*)(job.in + 2 * a.cs + o));
                            s = mk(fma2(k2v, x2.x, fma2(k1v, x1.x, k0v * x0.x)), fma2(k2v, x2.y, fma2(k1v, x1.y, k0v * x0.y)));
                        } else {
                            const C2 xa = pair(*(const float4*)(pa + o)), xb = pair(*(const float4*)(pb + o));
                            const P2 ua = q == 0 ? k1v : (q == 1 ? k2v : k0v), ub = q == 0 ? k2v : (q == 1 ? k0v : k1v);
                            s = mk(fma2(ua, xa.x, -(ub * xb.x)), fma2(ua, xa.y, -(ub * xb.y)));
                        }
                        v[r] = mk(-s.y, s.x);
                    }
                }
#pragma unroll
                for (int r = 0; r < AA; ++r) {
                    const int c1 = LineBand<N>::template at<M>(j, r);
                    if (c1 < 0) continue;
                    P2 f = sc;
                    if (tab) {
                        const float2 t = __ldg((const float2*)(tab + o0 + (unsigned)(c1 * b0p)));
                        f = f * p2(t.x, t.y);
                    }
                    v[r] = mk(f * v[r].x, f * v[r].y);
                }
            } else if constexpr (MODE == 1) {
                const cpx<float>* const p0 =
                    a.mid + blockIdx.z * a.mids + (unsigned)(k2 * n1 + l0) * (unsigned)b0p;
                const cpx<float>* const p1 = p0 + (l0 + 1 < lines ? b0p : 0);
#pragma unroll
                for (int r = 0; r < AA; ++r) {
                    const int kc = LineBand<N>::template at<M>(j, r);
                    if (kc >= 0) {
                        const cpx<float> x = one(p0 + kc), y = one(p1 + kc);
                        v[r] = mk(p2(x.x, y.x), p2(x.y, y.y));
                    }
                }
            } else if constexpr (MODE == 2) {
                const cpx<float>* const p = job.in + (size_t)k2 * N * n1 + l0;
                if (n1 % 2 == 0) {
#pragma unroll
                    for (int r = 0; r < AA; ++r) v[r] = pair(*(const float4*)(p + (unsigned)((j + r * M) * n1)));
                } else {
                    const int d = l0 + 1 < lines ? 1 : 0;
#pragma unroll
                    for (int r = 0; r < AA; ++r) {
                        const cpx<float>* s = p + (unsigned)((j + r * M) * n1);
                        const cpx<float> x = one(s), y = one(s + d);
                        v[r] = mk(p2(x.x, y.x), p2(x.y, y.y));
                    }
                }
            } else {
                const cpx<float>* const p = a.mid + blockIdx.z * a.mids + (unsigned)(k2 * N) * (unsigned)b0p + l0;
#pragma unroll
                for (int r = 0; r < AA; ++r) v[r] = pair(*(const float4*)(p + (unsigned)((j + r * M) * b0p)));
            }
        }
        dft<AA, DIR>(v);
        twiddles2<AA, DIR>(v, tws, twn, j);
        const int r1 = j / CC, j2 = j - r1 * CC;
        C2* s = buf + (AA * (r1 + BB * j2)) * RB;
#pragma unroll
        for (int q = 0; q < AA; ++q) s[q * RB] = v[q];
    }
    __syncthreads();
    if constexpr (BB > 1) {
#pragma unroll 1
        for (int i = m; i < N / BB; i += T) {
            const int j2 = i / AA, q0 = i - j2 * AA;
            C2* s = buf + (q0 + AA * BB * j2) * RB;
            C2 v[BB];
#pragma unroll
            for (int r = 0; r < BB; ++r) v[r] = s[r * AA * RB];
            dft<BB, DIR>(v);
            twiddles2<BB, DIR>(v, tws, twn, AA * j2);
#pragma unroll
            for (int r = 0; r < BB; ++r) s[r * AA * RB] = v[r];
        }
        __syncthreads();
    }
    dependents_may_launch();
    // ---- last stage: output k = i + r ML
    constexpr int ML = N / CC;
    if (!on) return;
#pragma unroll 1
    for (int i = m; i < ML; i += T) {
        C2 v[CC];
#pragma unroll
        for (int r = 0; r < CC; ++r) v[r] = buf[(i + r * ML) * RB];
        dft<CC, DIR>(v);
        auto quad = [](C2 x) { return make_float4(lo(x.x), lo(x.y), hi(x.x), hi(x.y)); };
        if constexpr (MODE == 0) {
            cpx<float>* const p = a.mid + blockIdx.z * a.mids + (unsigned)(k2 * N + i) * (unsigned)b0p + l0;
#pragma unroll
            for (int r = 0; r < CC; ++r) *(float4*)(p + (unsigned)(r * ML * b0p)) = quad(v[r]);
        } else if constexpr (MODE == 1) {
            cpx<float>* const p = job.out + (size_t)k2 * N * n1 + (unsigned)(i * n1) + l0;
            if (n1 % 2 == 0) {
#pragma unroll
                for (int r = 0; r < CC; ++r) *(float4*)(p + (unsigned)(r * ML * n1)) = quad(v[r]);
            } else {
#pragma unroll
                for (int r = 0; r < CC; ++r) {
                    cpx<float>* s = p + (unsigned)(r * ML * n1);
                    s[0] = mk(lo(v[r].x), lo(v[r].y));
                    if (l0 + 1 < lines) s[1] = mk(hi(v[r].x), hi(v[r].y));
                }
            }
        } else if constexpr (MODE == 2) {
            cpx<float>* const p0 = a.mid + blockIdx.z * a.mids + (unsigned)(k2 * n1 + l0) * (unsigned)b0p;
#pragma unroll
            for (int r = 0; r < CC; ++r) {
                const int kc = LineBand<N>::template at<ML>(i, r);
                if (kc < 0) continue;
                p0[kc] = mk(lo(v[r].x), lo(v[r].y));
                if (l0 + 1 < lines) p0[b0p + kc] = mk(hi(v[r].x), hi(v[r].y));
            }
        } else {
            cpx<float>* const p = job.out + (unsigned)k2 * (unsigned)(bd.b1 * b0p) + l0;
#pragma unroll
            for (int r = 0; r < CC; ++r) {
                const int c1 = LineBand<N>::template at<ML>(i, r);
                if (c1 >= 0) *(float4*)(p + (unsigned)(c1 * b0p)) = quad(v[r]);
            }
        }
    }
}

// Launch of k_line of a mode (set_attr: raise its shared-memory limit instead);
// defined in stage_length.cu, one translation unit per length.
template <int N>
bool line_launch_n(int mode, const PlaneArgs<float>& a, dim3 grid, cudaStream_t st, bool set_attr);

}  // namespace lddmm
