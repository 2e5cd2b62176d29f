// Stages of the band form of the path: the axis-2 inverse transforms of a
// stage's spectra, the pointwise products and the axis-2 forward transforms,
// in one kernel, so that the real fields of a stage never leave the SM.
//
// With the 2/3-rule projector on, every product here is of two band-limited
// fields and is read through the projector, which removes all that aliasing
// adds; so the product rule holds exactly between band entries, and
//     ad*_v m  = grad(v . m) - v x curl m + m div v,
//     ad_v xi  = curl(v x xi) - v div xi + xi div v
// need far fewer transforms than the sums over Dv and Dm: a tangent stage 14
// inverse and 10 forward (36 and 6 otherwise), its transpose 10 and 14, a
// shooting stage 10 and 4.  A stored state is ten fields:
//     0..2 v, 3..5 m = L v, 6..8 w = curl m, 9 d = div v.
//   KIND 0 tangent: in eta_0..2, div eta, mu_0..2, curl mu_0..2, xi_0..2, div xi
//       out t_0..2, s, a_0..2, r_0..2 with s = eta.m + v.mu,
//       t = m div eta + mu d - eta x w - v x curl mu, a = v x xi,
//       r = xi d - v div xi
//   KIND 1 adjoint: in y_0..2, sb = -div y, yx_0..2, ab_0..2 = curl yx
//       out eb = sb m - w x y, db = m.y, mb = sb v + d y, ob = v x y,
//       xb = d yx + ab x v, dxb = -v.yx
//   KIND 2 shooting: in v, d, m, w (order v_0..2, d, m_0..2, w_0..2), stored as
//       the state; out t = m d - v x w, s = v.m
//
// Layout: a block owns RB consecutive grid rows (lane c, fastest) and all N
// points of each; thread (c, m), m < W = N / P, holds the points m + r W, r < P,
// of its row for the whole kernel: they are the outputs of the last radix-P
// stage of an inverse line and the inputs of the first radix-P stage of a
// forward line.  Rows are the fastest index of the band planes [k2][row] and
// of the stored state [field][i2][row], so every access is a segment of RB
// entries, and the exchange buffer [p][c] has no bank conflicts.
//
// A complex line transform packs two neighbouring rows of one field (two
// fields can differ in size by a factor that L or kappa then multiplies, and
// the smaller would keep the rounding of the larger): of a pair of fields
// (f, f + 1), the even lane transforms f on rows (2i, 2i + 1) and the odd lane
// f + 1 on the same rows, and one shuffle per point hands each row its own.
#pragma once
#include "launch_util.cuh"
#include "radix.cuh"

namespace lddmm {

constexpr int ST_FIELDS = 10;
template <class T> struct StageArgs {
    const cpx<T>* in[14];
    cpx<T>* out[14];
    T* state;             // ten fields, stride npts (KIND 2: written; may be null there)
    const cpx<T>* tw;     // e^{-2 pi i t / n2}
    size_t npts;
    int n2, rows, nb2, lrb;  // lrb: log2 of the rows per block
    RPlan pl;                // of n2, last radix P
};

constexpr int STAGE_THREADS = 256;  // at most (FP64)
constexpr int STAGE2_THREADS = 512; // at most (FP32; 128 registers)
// row pairs of a block (FP32): 8 (128-byte segments of a plane) while that is at
// most 256 threads, else 4, so that two blocks and more share an SM
__host__ __device__ constexpr int stage_rb(int n, int p) { return n / p * 8 <= 256 ? 8 : 4; }
// blocks per SM that leave a thread 128 registers (three blocks at 80 registers:
// 112 us an adjoint stage at 128^3 against 92)
__host__ __device__ constexpr int stage_blocks(int n, int p) {
    return 512 / ((n / p * stage_rb(n, p) + 31) / 32 * 32);
}
// shared memory: FP64, 2^lrb rows: two exchange buffers and the twiddles; FP32:
// one exchange buffer, the twiddles three times, and the staged planes
inline size_t stage_smem(bool f64, int n2, int lrb) {
    if (f64) return 16 * (((size_t)2 * n2 << lrb) + n2);
    const size_t rb = (size_t)1 << lrb;
    return 16 * (n2 * rb + n2 + 4 * (n2 / 2 + 2) * rb) + 8 * (size_t)n2;
}

__device__ __forceinline__ double shfl_x1(double v) { return __shfl_xor_sync(0xffffffffu, v, 1); }

template <class T, int P, int KIND>
__global__ void __launch_bounds__(STAGE_THREADS) k_stage(const __grid_constant__ StageArgs<T> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int rb = 1 << a.lrb, N = a.n2, rows = a.rows, nb2 = a.nb2;
    const RPlan& pl = a.pl;
    const int W = N / P;
    cpx<T>* const buf0 = (cpx<T>*)smem_raw;
    cpx<T>* const tws = buf0 + 2 * N * rb;
    for (int i = threadIdx.x; i < N; i += blockDim.x) tws[i] = ldg(a.tw + i);
    // threads beyond W rb (the block is whole warps) only take part in barriers and shuffles
    const int c = threadIdx.x & (rb - 1), mt = threadIdx.x >> a.lrb;
    const bool act = mt < W;
    const int m = act ? mt : 0, mj = act ? mt : N;  // mj: first item of a strided loop
    const int row0 = blockIdx.x * rb + c;
    const bool valid = act && row0 < rows;
    const int row = min(row0, rows - 1);
    const bool odd = c & 1;
    const int rA = min((int)blockIdx.x * rb + (c & ~1), (rows - 1) & ~1), dB = rA + 1 < rows ? 1 : 0;
    int sel = 0;  // exchange buffer of the next line
    __syncthreads();

    // inverse transform of the fields (f, f + 1): u, w at this thread's points
    auto inv = [&](int f, T(&u)[P], T(&w)[P]) {
        const cpx<T>* const in = a.in[f + (odd ? 1 : 0)] + rA;
        cpx<T>* const buf = buf0 + sel * N * rb + c;
        LDDMM_FIRST(pl.a, {
            const int M = N / R;
            for (int j = mj; j < M; j += W) {
                cpx<T> v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) {
                    const int k = j + r * M, kn = N - k;
                    // which half k lies in is known from r but for the middle of an odd radix
                    const bool hi = 2 * r + 1 == R ? kn < k : 2 * r >= R;
                    const int kk = hi ? kn : k;
                    cpx<T> p = mk((T)0, (T)0), q = p;
                    if (kk < nb2) {
                        const cpx<T>* s = in + kk * rows;
                        p = ldg(s);
                        q = ldg(s + dB);
                    }
                    if ((r == 0 && j == 0) || k == kn) p.y = q.y = (T)0;
                    if (hi) {
                        p.y = -p.y;
                        q.y = -q.y;
                    }
                    v[r] = mk(p.x - q.y, p.y + q.x);
                }
                dft<R, 1>(v);
                twiddles<R, 1>(v, tws, j);
                const int r1 = j / P, j2 = j - r1 * P;
                cpx<T>* s = buf + (R * (r1 + pl.b * j2)) * rb;
                LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * rb] = v[q];
            }
        })
        __syncthreads();
        if (pl.b > 1) {
            LDDMM_MID(pl.b, {
                for (int i = mj; i < N / R; i += W) {
                    const int j2 = (int)pl.fa.div((unsigned)i), q0 = i - j2 * pl.a;
                    cpx<T>* s = buf + (q0 + pl.a * R * j2) * rb;
                    const int st = pl.a * rb;
                    cpx<T> v[R];
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, 1>(v);
                    twiddles<R, 1>(v, tws, pl.a * j2);
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        cpx<T> x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = buf[(m + r * W) * rb];
        dft<P, 1>(x);
#pragma unroll
        for (int r = 0; r < P; ++r) {
            const T got = shfl_x1(odd ? x[r].x : x[r].y);
            u[r] = odd ? got : x[r].x;
            w[r] = odd ? x[r].y : got;
        }
        sel ^= 1;
    };
    // forward transform of two fields given at this thread's points, into the
    // planes out[f], out[f + 1] (doubled)
    auto fwd = [&](int f, const T(&u)[P], const T(&w)[P]) {
        cpx<T>* const buf = buf0 + sel * N * rb + c;
        cpx<T> x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) {
            const T got = shfl_x1(odd ? u[r] : w[r]);
            x[r] = odd ? mk(got, w[r]) : mk(u[r], got);
        }
        dft<P, -1>(x);
        twiddles<P, -1>(x, tws, m);
        {
            const int r1 = (int)pl.fa.div((unsigned)m), j2 = m - r1 * pl.a;
            cpx<T>* s = buf + (P * (r1 + pl.b * j2)) * rb;
            if (act) {
#pragma unroll
                for (int q = 0; q < P; ++q) s[q * rb] = x[q];
            }
        }
        __syncthreads();
        if (pl.b > 1) {
            LDDMM_MID(pl.b, {
                for (int i = mj; i < N / R; i += W) {
                    const int j2 = i / P, q0 = i - j2 * P;
                    cpx<T>* s = buf + (q0 + P * R * j2) * rb;
                    const int st = P * rb;
                    cpx<T> v[R];
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, -1>(v);
                    twiddles<R, -1>(v, tws, P * j2);
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        LDDMM_FIRST(pl.a, {
            const int M = N / R;
            for (int i = mj; i < M; i += W) {
                cpx<T>* s = buf + i * rb;
                cpx<T> v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r * M * rb];
                dft<R, -1>(v);
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) s[r * M * rb] = v[r];
            }
        })
        __syncthreads();
        cpx<T>* const o0 = a.out[f] + row0;
        cpx<T>* const o1 = a.out[f + 1] + row0;
        for (int kb = 0; kb < nb2; kb += W) {
            const int k = kb + m;
            const int kk = min(k, nb2 - 1);
            const cpx<T> zk = buf[kk * rb];
            const cpx<T> zn = cj(buf[(kk == 0 ? 0 : N - kk) * rb]);
            const cpx<T> A = zk + zn, B = rot(zk - zn, -1);  // rows 2i and 2i + 1 of this lane's field
            const cpx<T> snd = odd ? A : B;
            const cpx<T> got = mk(shfl_x1(snd.x), shfl_x1(snd.y));
            if (valid && k < nb2) {
                o0[k * rows] = odd ? got : A;
                o1[k * rows] = odd ? B : got;
            }
        }
        sel ^= 1;
    };

    T* const st0 = a.state ? a.state + (size_t)m * rows + row : nullptr;
    auto S = [&](int f, int r) { return __ldg(st0 + f * a.npts + (unsigned)(r * W) * (unsigned)rows); };

    // A: the fields held across the lines of a phase; V (shooting): v and d
    T A[4][P], V[KIND == 2 ? 4 : 1][P], u[P], w[P];
    constexpr int PHASES = KIND == 2 ? 1 : 2;
#pragma unroll 1
    for (int ph = 0; ph < PHASES; ++ph) {
        const int l0 = KIND == 0 ? (ph == 0 ? 5 : 0) : (KIND == 1 ? (ph == 0 ? 0 : 2) : 0);
        const int l1 = KIND == 0 ? (ph == 0 ? 7 : 5) : (KIND == 1 ? (ph == 0 ? 2 : 5) : 5);
#pragma unroll 1
        for (int l = l0; l < l1; ++l) {
            inv(2 * l, u, w);
            if constexpr (KIND == 0) {
                switch (l) {
                    case 0:  // eta_0, eta_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T w2 = S(8, r);
                            A[0][r] = -w[r] * w2;
                            A[1][r] = u[r] * w2;
                            A[2][r] = w[r] * S(6, r) - u[r] * S(7, r);
                            A[3][r] = u[r] * S(3, r) + w[r] * S(4, r);
                        }
                        break;
                    case 1:  // eta_2, div eta
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T m2 = S(5, r);
                            A[0][r] += u[r] * S(7, r) + w[r] * S(3, r);
                            A[1][r] += w[r] * S(4, r) - u[r] * S(6, r);
                            A[2][r] += w[r] * m2;
                            A[3][r] += u[r] * m2;
                        }
                        break;
                    case 2:  // mu_0, mu_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T d = S(9, r);
                            A[0][r] += u[r] * d;
                            A[1][r] += w[r] * d;
                            A[3][r] += u[r] * S(0, r) + w[r] * S(1, r);
                        }
                        break;
                    case 3:  // mu_2, (curl mu)_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T v2 = S(2, r);
                            A[1][r] -= v2 * w[r];
                            A[2][r] += u[r] * S(9, r) + S(1, r) * w[r];
                            A[3][r] += u[r] * v2;
                        }
                        break;
                    case 4:  // (curl mu)_1, (curl mu)_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T v0 = S(0, r);
                            A[0][r] += S(2, r) * u[r] - S(1, r) * w[r];
                            A[1][r] += v0 * w[r];
                            A[2][r] -= v0 * u[r];
                        }
                        break;
                    case 5:  // xi_0, xi_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[0][r] = u[r];
                            A[1][r] = w[r];
                        }
                        break;
                    default:  // xi_2, div xi
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[2][r] = u[r];
                            A[3][r] = w[r];
                        }
                }
            } else if constexpr (KIND == 1) {
                switch (l) {
                    case 0:  // y_0, y_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[0][r] = u[r];
                            A[1][r] = w[r];
                        }
                        break;
                    case 1:  // y_2, sb
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[2][r] = u[r];
                            A[3][r] = w[r];
                        }
                        break;
                    case 2:  // yx_0, yx_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T d = S(9, r);
                            A[0][r] = d * u[r];
                            A[1][r] = d * w[r];
                            A[3][r] = -(S(0, r) * u[r] + S(1, r) * w[r]);
                        }
                        break;
                    case 3:  // yx_2, ab_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T v2 = S(2, r);
                            A[1][r] -= w[r] * v2;
                            A[2][r] = S(9, r) * u[r] + w[r] * S(1, r);
                            A[3][r] -= v2 * u[r];
                        }
                        break;
                    default:  // ab_1, ab_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const T v0 = S(0, r);
                            A[0][r] += u[r] * S(2, r) - w[r] * S(1, r);
                            A[1][r] += w[r] * v0;
                            A[2][r] -= u[r] * v0;
                        }
                }
            } else {
                const bool keep = a.state && valid;
                auto put = [&](int f, int r, T x) {
                    if (keep) st0[f * a.npts + (unsigned)(r * W) * (unsigned)rows] = x;
                };
                switch (l) {
                    case 0:  // v_0, v_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            V[0][r] = u[r];
                            V[1][r] = w[r];
                            put(0, r, u[r]);
                            put(1, r, w[r]);
                        }
                        break;
                    case 1:  // v_2, d
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            V[2][r] = u[r];
                            V[3][r] = w[r];
                            put(2, r, u[r]);
                            put(9, r, w[r]);
                        }
                        break;
                    case 2:  // m_0, m_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(3, r, u[r]);
                            put(4, r, w[r]);
                            A[0][r] = u[r] * V[3][r];
                            A[1][r] = w[r] * V[3][r];
                            A[3][r] = V[0][r] * u[r] + V[1][r] * w[r];
                        }
                        break;
                    case 3:  // m_2, w_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(5, r, u[r]);
                            put(6, r, w[r]);
                            A[1][r] -= V[2][r] * w[r];
                            A[2][r] = u[r] * V[3][r] + V[1][r] * w[r];
                            A[3][r] += V[2][r] * u[r];
                        }
                        break;
                    default:  // w_1, w_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(7, r, u[r]);
                            put(8, r, w[r]);
                            A[0][r] += V[2][r] * u[r] - V[1][r] * w[r];
                            A[1][r] += V[0][r] * w[r];
                            A[2][r] -= V[0][r] * u[r];
                        }
                }
            }
        }
        const int o0 = KIND == 0 ? (ph == 0 ? 2 : 0) : (KIND == 1 ? (ph == 0 ? 0 : 5) : 0);
        const int o1 = KIND == 0 ? (ph == 0 ? 5 : 2) : (KIND == 1 ? (ph == 0 ? 5 : 7) : 2);
#pragma unroll 1
        for (int o = o0; o < o1; ++o) {
            if (ph == PHASES - 1 && o == o1 - 1) dependents_may_launch();
            int which = o;  // 0 / 1: (A_0, A_1) / (A_2, A_3)
            if constexpr (KIND == 1) which = o >= 5 ? o - 5 : o + 2;
            switch (which) {
                case 0:
#pragma unroll
                    for (int r = 0; r < P; ++r) {
                        u[r] = A[0][r];
                        w[r] = A[1][r];
                    }
                    break;
                case 1:
#pragma unroll
                    for (int r = 0; r < P; ++r) {
                        u[r] = A[2][r];
                        w[r] = A[3][r];
                    }
                    break;
                default:
                    if constexpr (KIND == 0) {
                        if (o == 2) {  // a_0, a_1 (A = xi_0..2, div xi)
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T v2 = S(2, r);
                                u[r] = S(1, r) * A[2][r] - v2 * A[1][r];
                                w[r] = v2 * A[0][r] - S(0, r) * A[2][r];
                            }
                        } else if (o == 3) {  // a_2, r_0
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T v0 = S(0, r);
                                u[r] = v0 * A[1][r] - S(1, r) * A[0][r];
                                w[r] = S(9, r) * A[0][r] - v0 * A[3][r];
                            }
                        } else {  // r_1, r_2
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T d = S(9, r);
                                u[r] = d * A[1][r] - S(1, r) * A[3][r];
                                w[r] = d * A[2][r] - S(2, r) * A[3][r];
                            }
                        }
                    } else if constexpr (KIND == 1) {
                        // A = y_0..2, sb
                        if (o == 0) {  // eb_0, eb_1
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T w2 = S(8, r);
                                u[r] = A[3][r] * S(3, r) - (S(7, r) * A[2][r] - w2 * A[1][r]);
                                w[r] = A[3][r] * S(4, r) - (w2 * A[0][r] - S(6, r) * A[2][r]);
                            }
                        } else if (o == 1) {  // eb_2, db
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T m2 = S(5, r);
                                u[r] = A[3][r] * m2 - (S(6, r) * A[1][r] - S(7, r) * A[0][r]);
                                w[r] = S(3, r) * A[0][r] + S(4, r) * A[1][r] + m2 * A[2][r];
                            }
                        } else if (o == 2) {  // mb_0, mb_1
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T d = S(9, r);
                                u[r] = A[3][r] * S(0, r) + d * A[0][r];
                                w[r] = A[3][r] * S(1, r) + d * A[1][r];
                            }
                        } else if (o == 3) {  // mb_2, ob_0
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T v2 = S(2, r);
                                u[r] = A[3][r] * v2 + S(9, r) * A[2][r];
                                w[r] = S(1, r) * A[2][r] - v2 * A[1][r];
                            }
                        } else {  // ob_1, ob_2
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const T v0 = S(0, r);
                                u[r] = S(2, r) * A[0][r] - v0 * A[2][r];
                                w[r] = v0 * A[1][r] - S(1, r) * A[0][r];
                            }
                        }
                    }
            }
            fwd(2 * o, u, w);
        }
    }
}

// ---------------------------------------------------------------- FP32
// The same stages with two rows and two fields per thread: a thread packs the
// row pair (2i, 2i + 1) of the fields f and f + 1 into two complex lines side
// by side (P2), so that a packed instruction, a 16-byte exchange and an
// address serve both, and no shuffle is needed; the products run packed over
// the two rows.  Lanes are row pairs.  The band planes of the next inverse
// line are copied (cp.async) into the other half of a double buffer while the
// current line is transformed, and the state fields of a line's products are
// prefetched into L1 when the line begins, so that neither load stands in the
// chain of a line's barriers.  Bound by shared memory (the LSU is 60% busy) and
// by the barriers between a line's short steps; DRAM moves 229 MB in the
// adjoint stage at 128^3, 241 MB in the tangent stage.  Adjoint and tangent stage there: 131 us each with
// one line per thread as in FP64, 107 and 102 packed with run-time radices, 92
// and 90 compiled; 106 and 102 with four row pairs a block, 112 and 99 with
// three blocks an SM (80 registers).  The last radix is small (3 to 6: the points a
// thread holds), which leaves registers for several blocks per SM.
__device__ __forceinline__ void put2(float* p, P2 x) { *(float2*)p = make_float2(lo(x), hi(x)); }
__device__ __forceinline__ P2 get2(const float* p) {
    const float2 q = __ldg((const float2*)p);
    return p2(q.x, q.y);
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem) {
    const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(s), "l"(gmem) : "memory");
}
// state fields to prefetch when inverse line l begins, one bit per field
template <int KIND> __device__ __forceinline__ unsigned line_states(int l) {
    if (KIND == 0) return l == 5 ? 0x207u : (l == 0 ? 0x1d8u : (l == 1 ? 0x20u : 0u));
    if (KIND == 1) return l == 0 ? 0x1f8u : (l == 1 ? 0x207u : 0u);
    return 0u;
}

// NN, AA, BB: the length and its first two radices where they are compiled in
// (every address of the shared buffers is then a constant offset); NN = 0: the
// radices come from the arguments.
template <int NN, int AA, int BB, int P, int KIND, bool EVEN>
__global__ void __launch_bounds__(NN ? (NN / P * stage_rb(NN, P) + 31) / 32 * 32 : STAGE2_THREADS,
                                  NN ? stage_blocks(NN, P) : 1) k_stage2(const __grid_constant__ StageArgs<float> a) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using C2 = cpx<P2>;
    // EVEN: the row count is even, so that every row pair is there and aligned;
    // otherwise a pair is two accesses, and the last one reads its row twice
    const int rb = NN ? stage_rb(NN ? NN : 1, P) : 1 << a.lrb;
    const int N = NN ? NN : a.n2, rows = a.rows, nb2 = NN ? (NN - 1) / 3 + 1 : a.nb2;
    const int pa = NN ? AA : a.pl.a, pb = NN ? BB : a.pl.b;
    const int W = N / P;
    auto div_a = [&](int i) { return NN ? i / (AA ? AA : 1) : (int)a.pl.fa.div((unsigned)i); };
    C2* const bufs = (C2*)smem_raw;
    C2* const tws = bufs + N * rb;
    // staged planes: two halves of two fields; planes above the band are zeros
    // (all of them, or one that every index above the band is clamped to)
    const int fp = NN ? NN / 2 + 1 : nb2 + 1, fs = fp * rb;  // planes and entries of a field
    float4* const ring = (float4*)(tws + N);
    P2* const twn = (P2*)(ring + 4 * fs);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const cpx<float> t = ldg(a.tw + i);
        tws[i] = mk(p2(t.x, t.x), p2(t.y, t.y));
        twn[i] = p2(-t.y, -t.y);
    }
    for (int f = 0; f < 4; ++f)
        for (int i = nb2 * rb + threadIdx.x; i < fs; i += blockDim.x) ring[f * fs + i] = make_float4(0.f, 0.f, 0.f, 0.f);
    // threads beyond W rb (the block is whole warps) only copy and take part in barriers
    const int c = threadIdx.x % rb, mt = threadIdx.x / rb;
    const bool act = (NN && NN / P * rb % 32 == 0) || mt < W;
    const int m = act ? mt : 0, mj = act ? mt : N;
    const int base = 2 * (int)blockIdx.x * rb;  // first row of the block
    const int row0 = base + 2 * c;
    const bool valid = act && row0 < rows;
    const int row = min(row0, (rows - 1) & ~1), dB = EVEN || row + 1 < rows ? 1 : 0;
    int half = 0;
    C2* const buf = bufs + c;

    // copies of the planes of inverse line l into half h of the ring
    auto issue = [&](int l, int h) {
        float4* const dst = ring + h * 2 * fs + c;
        const cpx<float>* const p0 = a.in[2 * l] + row;
        const cpx<float>* const p1 = a.in[2 * l + 1] + row;
        const int step = NN ? (NN / P * rb + 31) / 32 * 32 / rb : (int)blockDim.x / rb;
        for (int k = mt; k < nb2; k += step) {
            const unsigned o = (unsigned)k * (unsigned)rows;
            if constexpr (EVEN) {
                cp_async16(dst + k * rb, p0 + o);
                cp_async16(dst + fs + k * rb, p1 + o);
            } else {
                cp_async8(dst + k * rb, p0 + o);
                cp_async8((float2*)(dst + k * rb) + 1, p0 + o + dB);
                cp_async8(dst + fs + k * rb, p1 + o);
                cp_async8((float2*)(dst + fs + k * rb) + 1, p1 + o + dB);
            }
        }
        cp_async_commit();
    };
    // the next inverse line of the block after l (-1: none)
    auto next_line = [&](int l) { return KIND == 0 ? (l == 6 ? 0 : (l == 4 ? -1 : l + 1)) : (l == 4 ? -1 : l + 1); };
    after_previous();
    issue(KIND == 0 ? 5 : 0, 0);

    auto inv = [&](int l, P2(&u)[P], P2(&w)[P]) {
        cp_async_wait<0>();
        __syncthreads();  // the line's planes are in; the exchange buffer and the other half are free
        const int nl = next_line(l);
        if (nl >= 0) issue(nl, half ^ 1);
        if constexpr (KIND != 2) {
            // the block's rows of a field at one point are 8 rb bytes: one prefetch each
            const unsigned want = line_states<KIND>(l);
            if (want) {
                for (int f = 0; f < ST_FIELDS; ++f)
                    if (want >> f & 1) {
                        const float* p = a.state + (size_t)f * a.npts + base;
                        for (int i = threadIdx.x; i < N; i += blockDim.x)
                            asm volatile("prefetch.global.L1 [%0];" ::"l"(p + (size_t)i * rows));
                    }
            }
        }
        const float4* const rf = ring + half * 2 * fs + c;
        LDDMM_FIRST10(pa, {
            const int M = N / R;
            for (int j = mj; j < M; j += W) {
                C2 v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) {
                    const int k = j + r * M, kn = N - k;
                    // which half k lies in is known from r but for the middle of an odd radix
                    const bool hh = 2 * r + 1 == R ? kn < k : 2 * r >= R;
                    // entries above the band: zero for every j, or a plane of zeros
                    if (NN && (2 * r < R ? r * M >= nb2 : N - r * M - M >= nb2)) {
                        v[r] = mk(p2(0.f, 0.f), p2(0.f, 0.f));
                        continue;
                    }
                    const int kk = NN ? (hh ? kn : k) : min(hh ? kn : k, nb2);
                    float4 fv = rf[kk * rb], gv = rf[fs + kk * rb];
                    // the imaginary parts of the real entries k = 0 and N / 2 do not count
                    if ((r == 0 && j == 0) || ((r == R / 2) && k == kn)) fv.y = fv.w = gv.y = gv.w = 0.f;
                    if (2 * r + 1 == R ? !hh : 2 * r < R)
                        v[r] = mk(p2(fv.x - fv.w, gv.x - gv.w), p2(fv.y + fv.z, gv.y + gv.z));
                    else
                        v[r] = mk(p2(fv.x + fv.w, gv.x + gv.w), p2(fv.z - fv.y, gv.z - gv.y));
                }
                dft<R, 1>(v);
                twiddles2<R, 1>(v, tws, twn, j);
                const int r1 = j / P, j2 = j - r1 * P;
                C2* s = buf + (R * (r1 + pb * j2)) * rb;
                LDDMM_UNROLL
                for (int q = 0; q < R; ++q) s[q * rb] = v[q];
            }
        })
        __syncthreads();
        if (pb > 1) {
            LDDMM_MID(pb, {
                for (int i = mj; i < N / R; i += W) {
                    const int j2 = div_a(i), q0 = i - j2 * pa;
                    C2* s = buf + (q0 + pa * R * j2) * rb;
                    const int st = pa * rb;
                    C2 v[R];
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, 1>(v);
                    twiddles2<R, 1>(v, tws, twn, pa * j2);
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        C2 x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = buf[(m + r * W) * rb];
        dft<P, 1>(x);
        // x.x = (f, f + 1) on row 2i, x.y on row 2i + 1
#pragma unroll
        for (int r = 0; r < P; ++r) {
            u[r] = p2(lo(x[r].x), lo(x[r].y));
            w[r] = p2(hi(x[r].x), hi(x[r].y));
        }
        half ^= 1;
    };
    auto fwd = [&](int f, const P2(&u)[P], const P2(&w)[P]) {
        C2 x[P];
#pragma unroll
        for (int r = 0; r < P; ++r) x[r] = mk(p2(lo(u[r]), lo(w[r])), p2(hi(u[r]), hi(w[r])));
        dft<P, -1>(x);
        twiddles2<P, -1>(x, tws, twn, m);
        __syncthreads();  // the exchange buffer is free
        {
            const int r1 = div_a(m), j2 = m - r1 * pa;
            C2* s = buf + (P * (r1 + pb * j2)) * rb;
            if (act) {
#pragma unroll
                for (int q = 0; q < P; ++q) s[q * rb] = x[q];
            }
        }
        __syncthreads();
        if (pb > 1) {
            LDDMM_MID(pb, {
                for (int i = mj; i < N / R; i += W) {
                    const int j2 = i / P, q0 = i - j2 * P;
                    C2* s = buf + (q0 + P * R * j2) * rb;
                    const int st = P * rb;
                    C2 v[R];
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) v[r] = s[r * st];
                    dft<R, -1>(v);
                    twiddles2<R, -1>(v, tws, twn, P * j2);
                    LDDMM_UNROLL
                    for (int r = 0; r < R; ++r) s[r * st] = v[r];
                }
            })
            __syncthreads();
        }
        LDDMM_FIRST10(pa, {
            const int M = N / R;
            for (int i = mj; i < M; i += W) {
                C2* s = buf + i * rb;
                C2 v[R];
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) v[r] = s[r * M * rb];
                dft<R, -1>(v);
                LDDMM_UNROLL
                for (int r = 0; r < R; ++r) s[r * M * rb] = v[r];
            }
        })
        __syncthreads();
        if (valid) {
            cpx<float>* const of = a.out[f] + row;
            cpx<float>* const og = a.out[f + 1] + row;
            for (int k = m; k < nb2; k += W) {
                const C2 zk = buf[k * rb], zn = buf[(k == 0 ? 0 : N - k) * rb];
                const unsigned o = (unsigned)k * (unsigned)rows;
                // 2 F(row 2i) = Z_k + conj Z_{N-k}, 2 F(row 2i + 1) = -i (Z_k - conj Z_{N-k})
                const float4 qf = make_float4(lo(zk.x) + lo(zn.x), lo(zk.y) - lo(zn.y), lo(zk.y) + lo(zn.y),
                                              lo(zn.x) - lo(zk.x));
                const float4 qg = make_float4(hi(zk.x) + hi(zn.x), hi(zk.y) - hi(zn.y), hi(zk.y) + hi(zn.y),
                                              hi(zn.x) - hi(zk.x));
                if constexpr (EVEN) {
                    *(float4*)(of + o) = qf;
                    *(float4*)(og + o) = qg;
                } else {
                    of[o] = mk(qf.x, qf.y);
                    og[o] = mk(qg.x, qg.y);
                    if (dB) {
                        of[o + 1] = mk(qf.z, qf.w);
                        og[o + 1] = mk(qg.z, qg.w);
                    }
                }
            }
        }
    };

    float* const st0 = a.state ? a.state + (size_t)m * rows + row : nullptr;
    // read-only loads: no kernel that may still run when this one starts writes
    // the state (a shooting's last stage is two launches and their waits earlier)
    auto S = [&](int f, int r) {
        const float* p = st0 + f * a.npts + (unsigned)(r * W) * (unsigned)rows;
        if constexpr (EVEN) return get2(p);
        else return p2(__ldg(p), __ldg(p + dB));
    };

    // A: the fields held across the lines of a phase; V (shooting): v and d
    P2 A[4][P], V[KIND == 2 ? 4 : 1][P], u[P], w[P];
    constexpr int PHASES = KIND == 2 ? 1 : 2;
#pragma unroll 1
    for (int ph = 0; ph < PHASES; ++ph) {
        const int l0 = KIND == 0 ? (ph == 0 ? 5 : 0) : (KIND == 1 ? (ph == 0 ? 0 : 2) : 0);
        const int l1 = KIND == 0 ? (ph == 0 ? 7 : 5) : (KIND == 1 ? (ph == 0 ? 2 : 5) : 5);
#pragma unroll 1
        for (int l = l0; l < l1; ++l) {
            inv(l, u, w);
            if constexpr (KIND == 0) {
                switch (l) {
                    case 0:  // eta_0, eta_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 w2 = S(8, r);
                            A[0][r] = -(w[r] * w2);
                            A[1][r] = u[r] * w2;
                            A[2][r] = fma2(w[r], S(6, r), -(u[r] * S(7, r)));
                            A[3][r] = fma2(u[r], S(3, r), w[r] * S(4, r));
                        }
                        break;
                    case 1:  // eta_2, div eta
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 m2 = S(5, r);
                            A[0][r] = fma2(u[r], S(7, r), fma2(w[r], S(3, r), A[0][r]));
                            A[1][r] = fma2(w[r], S(4, r), A[1][r] - u[r] * S(6, r));
                            A[2][r] = fma2(w[r], m2, A[2][r]);
                            A[3][r] = fma2(u[r], m2, A[3][r]);
                        }
                        break;
                    case 2:  // mu_0, mu_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 d = S(9, r);
                            A[0][r] = fma2(u[r], d, A[0][r]);
                            A[1][r] = fma2(w[r], d, A[1][r]);
                            A[3][r] = fma2(u[r], S(0, r), fma2(w[r], S(1, r), A[3][r]));
                        }
                        break;
                    case 3:  // mu_2, (curl mu)_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 v2 = S(2, r);
                            A[1][r] = A[1][r] - v2 * w[r];
                            A[2][r] = fma2(u[r], S(9, r), fma2(S(1, r), w[r], A[2][r]));
                            A[3][r] = fma2(u[r], v2, A[3][r]);
                        }
                        break;
                    case 4:  // (curl mu)_1, (curl mu)_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 v0 = S(0, r);
                            A[0][r] = fma2(S(2, r), u[r], A[0][r] - S(1, r) * w[r]);
                            A[1][r] = fma2(v0, w[r], A[1][r]);
                            A[2][r] = A[2][r] - v0 * u[r];
                        }
                        break;
                    case 5:  // xi_0, xi_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[0][r] = u[r];
                            A[1][r] = w[r];
                        }
                        break;
                    default:  // xi_2, div xi
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[2][r] = u[r];
                            A[3][r] = w[r];
                        }
                }
            } else if constexpr (KIND == 1) {
                switch (l) {
                    case 0:  // y_0, y_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[0][r] = u[r];
                            A[1][r] = w[r];
                        }
                        break;
                    case 1:  // y_2, sb
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            A[2][r] = u[r];
                            A[3][r] = w[r];
                        }
                        break;
                    case 2:  // yx_0, yx_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 d = S(9, r);
                            A[0][r] = d * u[r];
                            A[1][r] = d * w[r];
                            A[3][r] = -fma2(S(0, r), u[r], S(1, r) * w[r]);
                        }
                        break;
                    case 3:  // yx_2, ab_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 v2 = S(2, r);
                            A[1][r] = A[1][r] - w[r] * v2;
                            A[2][r] = fma2(S(9, r), u[r], w[r] * S(1, r));
                            A[3][r] = A[3][r] - v2 * u[r];
                        }
                        break;
                    default:  // ab_1, ab_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            const P2 v0 = S(0, r);
                            A[0][r] = fma2(u[r], S(2, r), A[0][r] - w[r] * S(1, r));
                            A[1][r] = fma2(w[r], v0, A[1][r]);
                            A[2][r] = A[2][r] - u[r] * v0;
                        }
                }
            } else {
                const bool keep = a.state && valid;
                auto put = [&](int f, int r, P2 x) {
                    if (!keep) return;
                    float* p = st0 + f * a.npts + (unsigned)(r * W) * (unsigned)rows;
                    if constexpr (EVEN) {
                        put2(p, x);
                    } else {
                        p[0] = lo(x);
                        if (dB) p[1] = hi(x);
                    }
                };
                switch (l) {
                    case 0:  // v_0, v_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            V[0][r] = u[r];
                            V[1][r] = w[r];
                            put(0, r, u[r]);
                            put(1, r, w[r]);
                        }
                        break;
                    case 1:  // v_2, d
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            V[2][r] = u[r];
                            V[3][r] = w[r];
                            put(2, r, u[r]);
                            put(9, r, w[r]);
                        }
                        break;
                    case 2:  // m_0, m_1
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(3, r, u[r]);
                            put(4, r, w[r]);
                            A[0][r] = u[r] * V[3][r];
                            A[1][r] = w[r] * V[3][r];
                            A[3][r] = fma2(V[0][r], u[r], V[1][r] * w[r]);
                        }
                        break;
                    case 3:  // m_2, w_0
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(5, r, u[r]);
                            put(6, r, w[r]);
                            A[1][r] = A[1][r] - V[2][r] * w[r];
                            A[2][r] = fma2(u[r], V[3][r], V[1][r] * w[r]);
                            A[3][r] = fma2(V[2][r], u[r], A[3][r]);
                        }
                        break;
                    default:  // w_1, w_2
#pragma unroll
                        for (int r = 0; r < P; ++r) {
                            put(7, r, u[r]);
                            put(8, r, w[r]);
                            A[0][r] = fma2(V[2][r], u[r], A[0][r] - V[1][r] * w[r]);
                            A[1][r] = fma2(V[0][r], w[r], A[1][r]);
                            A[2][r] = A[2][r] - V[0][r] * u[r];
                        }
                }
            }
        }
        const int o0 = KIND == 0 ? (ph == 0 ? 2 : 0) : (KIND == 1 ? (ph == 0 ? 0 : 5) : 0);
        const int o1 = KIND == 0 ? (ph == 0 ? 5 : 2) : (KIND == 1 ? (ph == 0 ? 5 : 7) : 2);
#pragma unroll 1
        for (int o = o0; o < o1; ++o) {
            if (ph == PHASES - 1 && o == o1 - 1) dependents_may_launch();
            int which = o;  // 0 / 1: (A_0, A_1) / (A_2, A_3)
            if constexpr (KIND == 1) which = o >= 5 ? o - 5 : o + 2;
            switch (which) {
                case 0:
#pragma unroll
                    for (int r = 0; r < P; ++r) {
                        u[r] = A[0][r];
                        w[r] = A[1][r];
                    }
                    break;
                case 1:
#pragma unroll
                    for (int r = 0; r < P; ++r) {
                        u[r] = A[2][r];
                        w[r] = A[3][r];
                    }
                    break;
                default:
                    if constexpr (KIND == 0) {
                        if (o == 2) {  // a_0, a_1 (A = xi_0..2, div xi)
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 v2 = S(2, r);
                                u[r] = fma2(S(1, r), A[2][r], -(v2 * A[1][r]));
                                w[r] = fma2(v2, A[0][r], -(S(0, r) * A[2][r]));
                            }
                        } else if (o == 3) {  // a_2, r_0
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 v0 = S(0, r);
                                u[r] = fma2(v0, A[1][r], -(S(1, r) * A[0][r]));
                                w[r] = fma2(S(9, r), A[0][r], -(v0 * A[3][r]));
                            }
                        } else {  // r_1, r_2
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 d = S(9, r);
                                u[r] = fma2(d, A[1][r], -(S(1, r) * A[3][r]));
                                w[r] = fma2(d, A[2][r], -(S(2, r) * A[3][r]));
                            }
                        }
                    } else if constexpr (KIND == 1) {
                        // A = y_0..2, sb
                        if (o == 0) {  // eb_0, eb_1
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 w2 = S(8, r);
                                u[r] = fma2(A[3][r], S(3, r), fma2(w2, A[1][r], -(S(7, r) * A[2][r])));
                                w[r] = fma2(A[3][r], S(4, r), fma2(S(6, r), A[2][r], -(w2 * A[0][r])));
                            }
                        } else if (o == 1) {  // eb_2, db
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 m2 = S(5, r);
                                u[r] = fma2(A[3][r], m2, fma2(S(7, r), A[0][r], -(S(6, r) * A[1][r])));
                                w[r] = fma2(S(3, r), A[0][r], fma2(S(4, r), A[1][r], m2 * A[2][r]));
                            }
                        } else if (o == 2) {  // mb_0, mb_1
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 d = S(9, r);
                                u[r] = fma2(A[3][r], S(0, r), d * A[0][r]);
                                w[r] = fma2(A[3][r], S(1, r), d * A[1][r]);
                            }
                        } else if (o == 3) {  // mb_2, ob_0
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 v2 = S(2, r);
                                u[r] = fma2(A[3][r], v2, S(9, r) * A[2][r]);
                                w[r] = fma2(S(1, r), A[2][r], -(v2 * A[1][r]));
                            }
                        } else {  // ob_1, ob_2
#pragma unroll
                            for (int r = 0; r < P; ++r) {
                                const P2 v0 = S(0, r);
                                u[r] = fma2(S(2, r), A[0][r], -(v0 * A[2][r]));
                                w[r] = fma2(v0, A[1][r], -(S(1, r) * A[0][r]));
                            }
                        }
                    }
            }
            fwd(2 * o, u, w);
        }
    }
}

template <class K, class A>
inline bool stage_go(K kernel, const A& a, int grid, int threads, size_t smem, cudaStream_t st, bool set_attr) {
    if (set_attr) {
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess) return true;
        cudaGetLastError();
        return false;
    }
    if constexpr (sizeof(a.tw->x) == 4) launch_dependent(kernel, dim3(grid), threads, smem, st, a);
    else kernel<<<grid, threads, smem, st>>>(a);
    return true;
}

// Line lengths whose FP32 kernels are compiled with the length and its stage
// radices (length, first, middle, last radix): every 5-smooth length from 16 to
// 320, and 384.  Fewest stages, then the smallest largest radix, then the larger
// last one (fewer threads a row).  Other lengths and odd row counts take the
// kernels with run-time radices.  The build compiles one unit per entry.
#define LDDMM_STAGE_LENGTHS(X) \
    X(16, 4, 1, 4) X(18, 3, 1, 6) X(20, 4, 1, 5) X(24, 4, 1, 6) X(25, 5, 1, 5) X(27, 9, 1, 3) X(30, 5, 1, 6) \
    X(32, 8, 1, 4) X(36, 6, 1, 6) X(40, 8, 1, 5) X(45, 9, 1, 5) X(48, 8, 1, 6) X(50, 10, 1, 5) X(54, 9, 1, 6) \
    X(60, 10, 1, 6) X(64, 4, 4, 4) X(72, 6, 2, 6) X(75, 5, 3, 5) X(80, 4, 4, 5) X(81, 9, 3, 3) X(90, 5, 3, 6) \
    X(96, 4, 4, 6) X(100, 5, 4, 5) X(108, 6, 3, 6) X(120, 5, 4, 6) X(125, 5, 5, 5) X(128, 8, 4, 4) X(135, 9, 3, 5) \
    X(144, 6, 4, 6) X(150, 5, 5, 6) X(160, 8, 4, 5) X(162, 9, 3, 6) X(180, 6, 5, 6) X(192, 8, 4, 6) X(200, 8, 5, 5) \
    X(216, 6, 6, 6) X(225, 9, 5, 5) X(240, 8, 5, 6) X(243, 9, 9, 3) X(250, 10, 5, 5) X(256, 8, 8, 4) \
    X(270, 9, 5, 6) X(288, 8, 6, 6) X(300, 10, 5, 6) X(320, 8, 8, 5) X(384, 8, 8, 6)

// Launch of the stage kernel of a kind with last radix P (set_attr: raise its
// shared-memory limit to smem bytes instead); defined in stage_radix.cu and
// stage_length.cu, one translation unit per number type and radix, or length.
template <class T, int P>
bool stage_launch_p(int kind, const StageArgs<T>& a, int grid, int threads, size_t smem, cudaStream_t st,
                    bool set_attr);
template <int N>
bool stage_launch_n(int kind, const StageArgs<float>& a, int grid, int threads, size_t smem, cudaStream_t st,
                    bool set_attr);
// the last radix of a length's FP32 plan: the compiled one, else by rule
inline RPlan stage_plan(bool f64, int n) {
#define LDDMM_X(N, A, B, C) \
    if (!f64 && n == N) return RPlan(A, B, C);
    LDDMM_STAGE_LENGTHS(LDDMM_X)
#undef LDDMM_X
    return radix_plan3(n, !f64);
}

}  // namespace lddmm
