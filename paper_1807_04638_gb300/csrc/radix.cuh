// Line transforms of run-time length in shared memory, from compile-time
// radices.
//
// A length n = a b c (b = 1: two stages) is transformed by decimation in
// frequency: with element index j + r n/a, r < a, stage 0 is a DFT over r
// (output q0) followed by the twiddle w_n^{q0 j}; the rest is a transform of
// length n/a over j for every q0, split the same way.  Every stage is one
// radix-R butterfly per item, held in registers, whose R elements are read
// from and written to the same R places, so that stages need one buffer and a
// barrier between them.  Two placements of the digits are used:
//   natural   stage 0 reads from elsewhere (global memory, registers) and puts
//             output (q0, j = j2 + r1 c) at q0 + a (r1 + b j2); the last stage
//             leaves element k = q0 + a (q1 + b q2) at place k;
//   in place  stage 0 too works in place; the last stage holds the outputs
//             k = q0 + a (q1 + b r), r < c, of item (q0, q1) in registers and
//             the caller stores them where they belong.
// Radices go up to 16, so that lengths up to about 160 take two stages (one
// exchange through shared memory) and all lengths up to 512 at most three;
// the batch dimension (the lines) is the lane dimension of every access, so
// that the index arithmetic and the twiddle reads are uniform along a warp's
// lanes and are spread over the elements of a butterfly.
#pragma once
#include "fft_fast.cuh"

namespace lddmm {

// ---------------------------------------------------------------- number types
// Two FP32 numbers of two lines side by side in one 64-bit register, for the
// packed add, multiply and fused multiply-add of sm_100 and later: a thread
// that transforms two lines at once spends one instruction where it would
// spend two, and shares the index arithmetic, the twiddles and the 16-byte
// shared-memory accesses between them.
struct P2 {
    unsigned long long v;
};
__device__ __forceinline__ P2 p2(float lo, float hi) {
    P2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ float lo(P2 a) { return __uint_as_float((unsigned)a.v); }
__device__ __forceinline__ float hi(P2 a) { return __uint_as_float((unsigned)(a.v >> 32)); }
__device__ __forceinline__ P2 operator+(P2 a, P2 b) {
    P2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 operator-(P2 a, P2 b) {
    P2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 operator*(P2 a, P2 b) {
    P2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ P2 operator-(P2 a) {
    P2 r;
    r.v = a.v ^ 0x8000000080000000ull;
    return r;
}
__device__ __forceinline__ P2 fma2(P2 a, P2 b, P2 c) {
    P2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
template <> struct __align__(16) cpx<P2> { P2 x, y; };

// a c and a c + b for a compile-time constant c (an immediate operand of the
// scalar instructions)
template <class T> __device__ __forceinline__ T kmul(T a, double c) { return a * (T)c; }
__device__ __forceinline__ P2 kmul(P2 a, double c) { return p2(lo(a) * (float)c, hi(a) * (float)c); }
template <class T> __device__ __forceinline__ T kfma(T a, double c, T b) { return a * (T)c + b; }
__device__ __forceinline__ P2 kfma(P2 a, double c, P2 b) {
    return p2(fmaf(lo(a), (float)c, lo(b)), fmaf(hi(a), (float)c, hi(b)));
}
// a + DIR i b, a - DIR i b
template <int DIR, class T> __device__ __forceinline__ cpx<T> addi(cpx<T> a, cpx<T> b) {
    if (DIR > 0) return mk(a.x - b.y, a.y + b.x);
    return mk(a.x + b.y, a.y - b.x);
}

// ---------------------------------------------------------------- codelets
// cos and sin of 2 pi k / 9 and 2 pi k / 16
constexpr double kC9[9] = {1.0, 0.766044443118978035202, 0.173648177666930348852, -0.5, -0.939692620785908384054,
                           -0.939692620785908384054, -0.5, 0.173648177666930348852, 0.766044443118978035202};
constexpr double kS9[9] = {0.0, 0.642787609686539326323, 0.984807753012208059367, 0.866025403784438646764,
                           0.342020143325668733044, -0.342020143325668733044, -0.866025403784438646764,
                           -0.984807753012208059367, -0.642787609686539326323};
constexpr double kC16[16] = {1.0, 0.923879532511286756128, 0.707106781186547524401, 0.382683432365089771728,
                             0.0, -0.382683432365089771728, -0.707106781186547524401, -0.923879532511286756128,
                             -1.0, -0.923879532511286756128, -0.707106781186547524401, -0.382683432365089771728,
                             0.0, 0.382683432365089771728, 0.707106781186547524401, 0.923879532511286756128};

// a e^{DIR 2 pi i K / N} for N = 8 (as 2K of 16), 9 or 16
template <int N, int K, int DIR, class T> __device__ __forceinline__ cpx<T> mul_root(cpx<T> a) {
    constexpr int k = K % N;
    constexpr double h = kC16[2];
    if constexpr (k == 0) return a;
    else if constexpr (4 * k == N) return DIR > 0 ? mk(-a.y, a.x) : mk(a.y, -a.x);
    else if constexpr (8 * k == N) return DIR > 0 ? mk(kmul(a.x - a.y, h), kmul(a.y + a.x, h))
                                                  : mk(kmul(a.x + a.y, h), kmul(a.y - a.x, h));
    else if constexpr (8 * k == 3 * N) return DIR > 0 ? mk(kmul(a.x + a.y, -h), kmul(a.x - a.y, h))
                                                      : mk(kmul(a.y - a.x, h), kmul(a.x + a.y, -h));
    else {
        constexpr double c = N == 9 ? kC9[N == 9 ? k : 0] : kC16[N == 16 ? k : 0];
        constexpr double s = DIR * (N == 9 ? kS9[N == 9 ? k : 0] : kC16[N == 16 ? (k + 12) % 16 : 0]);
        return mk(kfma(a.x, c, kmul(a.y, -s)), kfma(a.x, s, kmul(a.y, c)));
    }
}

template <int R, int DIR, class T> __device__ __forceinline__ void dft(cpx<T> (&v)[R]);

template <int DIR, class T> __device__ __forceinline__ void dft3(cpx<T> (&v)[3]) {
    constexpr double h = 0.86602540378443864676;  // sqrt(3) / 2
    const cpx<T> s = v[1] + v[2], d = v[1] - v[2];
    const cpx<T> m = mk(kfma(s.x, -0.5, v[0].x), kfma(s.y, -0.5, v[0].y));
    const cpx<T> q = mk(kmul(d.x, h), kmul(d.y, h));
    v[0] = v[0] + s;
    v[1] = addi<DIR>(m, q);
    v[2] = addi<-DIR>(m, q);
}
template <int DIR, class T> __device__ __forceinline__ void dft4(cpx<T> (&v)[4]) {
    const cpx<T> t0 = v[0] + v[2], t1 = v[0] - v[2], t2 = v[1] + v[3], t3 = v[1] - v[3];
    v[0] = t0 + t2;
    v[2] = t0 - t2;
    v[1] = addi<DIR>(t1, t3);
    v[3] = addi<-DIR>(t1, t3);
}
template <int DIR, class T> __device__ __forceinline__ void dft5(cpx<T> (&v)[5]) {
    constexpr double c1 = 0.30901699437494742410, c2 = -0.80901699437494742410;
    constexpr double s1 = 0.95105651629515357212, s2 = 0.58778525229247312917;
    const cpx<T> a1 = v[1] + v[4], b1 = v[1] - v[4], a2 = v[2] + v[3], b2 = v[2] - v[3];
    const cpx<T> p1 = mk(kfma(a2.x, c2, kfma(a1.x, c1, v[0].x)), kfma(a2.y, c2, kfma(a1.y, c1, v[0].y)));
    const cpx<T> p2_ = mk(kfma(a2.x, c1, kfma(a1.x, c2, v[0].x)), kfma(a2.y, c1, kfma(a1.y, c2, v[0].y)));
    const cpx<T> q1 = mk(kfma(b2.x, s2, kmul(b1.x, s1)), kfma(b2.y, s2, kmul(b1.y, s1)));
    const cpx<T> q2 = mk(kfma(b2.x, -s1, kmul(b1.x, s2)), kfma(b2.y, -s1, kmul(b1.y, s2)));
    v[0] = v[0] + a1 + a2;
    v[1] = addi<DIR>(p1, q1);
    v[4] = addi<-DIR>(p1, q1);
    v[2] = addi<DIR>(p2_, q2);
    v[3] = addi<-DIR>(p2_, q2);
}
template <int DIR, class T> __device__ __forceinline__ void dft8(cpx<T> (&v)[8]) {
    cpx<T> e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    dft4<DIR>(e);
    dft4<DIR>(o);
    const cpx<T> o1 = mul_root<16, 2, DIR>(o[1]), o3 = mul_root<16, 6, DIR>(o[3]);
    v[0] = e[0] + o[0];
    v[4] = e[0] - o[0];
    v[1] = e[1] + o1;
    v[5] = e[1] - o1;
    v[2] = addi<DIR>(e[2], o[2]);
    v[6] = addi<-DIR>(e[2], o[2]);
    v[3] = e[3] + o3;
    v[7] = e[3] - o3;
}

// R = N1 N2 with coprime factors (Good-Thomas: no twiddles)
template <int N1, int N2, int DIR, class T> __device__ __forceinline__ void dft_coprime(cpx<T> (&v)[N1 * N2]) {
    constexpr int N = N1 * N2;
    cpx<T> y[N2][N1];
#pragma unroll
    for (int n2 = 0; n2 < N2; ++n2) {
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) y[n2][n1] = v[(N2 * n1 + N1 * n2) % N];
        dft<N1, DIR>(y[n2]);
    }
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) {
        cpx<T> z[N2];
#pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) z[n2] = y[n2][k1];
        dft<N2, DIR>(z);
#pragma unroll
        for (int k = 0; k < N; ++k)
            if (k % N1 == k1) v[k] = z[k % N2];
    }
}

// R = M^2 (Cooley-Tukey with constant roots)
template <int M, int DIR, int N2, int K1, class T> __device__ __forceinline__ void root_rows(cpx<T> (&y)[M][M]) {
    y[N2][K1] = mul_root<M * M, N2 * K1, DIR>(y[N2][K1]);
    if constexpr (K1 + 1 < M) root_rows<M, DIR, N2, K1 + 1>(y);
    else if constexpr (N2 + 1 < M) root_rows<M, DIR, N2 + 1, 0>(y);
}
template <int M, int DIR, class T> __device__ __forceinline__ void dft_square(cpx<T> (&v)[M * M]) {
    cpx<T> y[M][M];
#pragma unroll
    for (int n2 = 0; n2 < M; ++n2) {
#pragma unroll
        for (int n1 = 0; n1 < M; ++n1) y[n2][n1] = v[n2 + M * n1];
        dft<M, DIR>(y[n2]);
    }
    root_rows<M, DIR, 0, 0>(y);
#pragma unroll
    for (int k1 = 0; k1 < M; ++k1) {
        cpx<T> z[M];
#pragma unroll
        for (int n2 = 0; n2 < M; ++n2) z[n2] = y[n2][k1];
        dft<M, DIR>(z);
#pragma unroll
        for (int k2 = 0; k2 < M; ++k2) v[k1 + M * k2] = z[k2];
    }
}

// y_k = sum_r v_r e^{DIR 2 pi i r k / R}
template <int R, int DIR, class T> __device__ __forceinline__ void dft(cpx<T> (&v)[R]) {
    if constexpr (R == 2) {
        const cpx<T> a = v[0], b = v[1];
        v[0] = a + b;
        v[1] = a - b;
    } else if constexpr (R == 3) dft3<DIR>(v);
    else if constexpr (R == 4) dft4<DIR>(v);
    else if constexpr (R == 5) dft5<DIR>(v);
    else if constexpr (R == 6) dft_coprime<2, 3, DIR>(v);
    else if constexpr (R == 8) dft8<DIR>(v);
    else if constexpr (R == 9) dft_square<3, DIR>(v);
    else if constexpr (R == 10) dft_coprime<2, 5, DIR>(v);
    else if constexpr (R == 12) dft_coprime<4, 3, DIR>(v);
    else if constexpr (R == 15) dft_coprime<3, 5, DIR>(v);
    else dft_square<4, DIR>(v);
}

// The radices of a length: n = a b c with b = 1 for two stages.
struct RPlan {
    int n, a, b, c;
    FastDiv fa, fb, fc;
    __host__ RPlan() : n(0), a(0), b(1), c(0) {}
    __host__ RPlan(int aa, int bb, int cc) : n(aa * bb * cc), a(aa), b(bb), c(cc), fa(aa), fb(bb), fc(cc) {}
};
constexpr int RP_FIRST[] = {2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16};  // radices of stage 0
constexpr int RP_MID[] = {2, 3, 4, 5, 6, 8, 9, 10};                // of the middle stage

// The plan with the fewest stages and, among those, the smallest largest
// radix (registers); n = 0 when there is none.  Every length up to 512 with
// factors 2, 3 and 5 has one but those below 8, and 9.  few: last radix 3 to 6,
// the others at most 10 (the FP32 stage kernels); none for 375 and 512 either.
inline RPlan radix_plan3(int n, bool few = false) {
    RPlan best;
    int score = 1 << 30;
    for (int c : {3, 4, 5, 6, 8, 9, 10}) {
        if (few ? c > 6 : c == 3) continue;
        for (int a : RP_FIRST) {
            if (n % (a * c) || (few && a > 10)) continue;
            const int b = n / (a * c);
            int s = a > c ? a : c;
            bool ok = b == 1;
            if (!ok)
                for (int m : RP_MID)
                    if (m == b) {
                        ok = true;
                        s = 1000 + 16 * (s > b ? s : b) + c;
                    }
            if (ok && s < score) score = s, best = RPlan(a, b, c);
        }
    }
    return best;
}

#define LDDMM_UNROLL _Pragma("unroll")
#define LDDMM_RCASE(RR, ...) \
    case RR: {               \
        constexpr int R = RR; \
        __VA_ARGS__          \
    } break;
#define LDDMM_FIRST(r, ...)                                                                                           \
    switch (r) {                                                                                                      \
        LDDMM_RCASE(2, __VA_ARGS__) LDDMM_RCASE(3, __VA_ARGS__) LDDMM_RCASE(4, __VA_ARGS__) LDDMM_RCASE(5, __VA_ARGS__)   \
        LDDMM_RCASE(6, __VA_ARGS__) LDDMM_RCASE(8, __VA_ARGS__) LDDMM_RCASE(9, __VA_ARGS__) LDDMM_RCASE(10, __VA_ARGS__)  \
        LDDMM_RCASE(12, __VA_ARGS__) LDDMM_RCASE(15, __VA_ARGS__) LDDMM_RCASE(16, __VA_ARGS__) default: break;            \
    }
#define LDDMM_FIRST10(r, ...)                                                                                         \
    switch (r) {                                                                                                      \
        LDDMM_RCASE(2, __VA_ARGS__) LDDMM_RCASE(3, __VA_ARGS__) LDDMM_RCASE(4, __VA_ARGS__) LDDMM_RCASE(5, __VA_ARGS__)   \
        LDDMM_RCASE(6, __VA_ARGS__) LDDMM_RCASE(8, __VA_ARGS__) LDDMM_RCASE(9, __VA_ARGS__) LDDMM_RCASE(10, __VA_ARGS__)  \
        default: break;                                                                                               \
    }
#define LDDMM_MID(r, ...)                                                                                             \
    switch (r) {                                                                                                      \
        LDDMM_RCASE(2, __VA_ARGS__) LDDMM_RCASE(3, __VA_ARGS__) LDDMM_RCASE(4, __VA_ARGS__) LDDMM_RCASE(5, __VA_ARGS__)   \
        LDDMM_RCASE(6, __VA_ARGS__) LDDMM_RCASE(8, __VA_ARGS__) LDDMM_RCASE(9, __VA_ARGS__) LDDMM_RCASE(10, __VA_ARGS__)  \
        default: break;                                                                                               \
    }
#define LDDMM_LAST(r, ...)                                                                                            \
    switch (r) {                                                                                                      \
        LDDMM_RCASE(4, __VA_ARGS__) LDDMM_RCASE(5, __VA_ARGS__) LDDMM_RCASE(6, __VA_ARGS__) LDDMM_RCASE(8, __VA_ARGS__)   \
        LDDMM_RCASE(9, __VA_ARGS__) LDDMM_RCASE(10, __VA_ARGS__) default: break;                                        \
    }

// v w with w = e^{-2 pi i e / n} from the table, conjugated for DIR = +1
template <int DIR, class T> __device__ __forceinline__ cpx<T> twiddle(cpx<T> v, cpx<T> w) {
    if (DIR > 0) w.y = -w.y;
    return v * w;
}
// stage outputs q = 1..R-1 times w^{q e}
template <int R, int DIR, class T, class W>
__device__ __forceinline__ void twiddles(cpx<T> (&v)[R], const cpx<W>* tw, int e) {
#pragma unroll
    for (int q = 1; q < R; ++q) v[q] = twiddle<DIR>(v[q], tw[q * e]);
}

// the same with the root's parts held twice (w) and -Im w twice (n)
template <int R, int DIR>
__device__ __forceinline__ void twiddles2(cpx<P2> (&v)[R], const cpx<P2>* w, const P2* n, int e) {
#pragma unroll
    for (int q = 1; q < R; ++q) {
        const cpx<P2> t = w[q * e];
        const P2 s = n[q * e];
        const P2 yp = DIR > 0 ? s : t.y, yn = DIR > 0 ? t.y : s;  // Im and -Im of the root
        v[q] = mk(fma2(v[q].x, t.x, v[q].y * yn), fma2(v[q].x, yp, v[q].y * t.x));
    }
}

}  // namespace lddmm
