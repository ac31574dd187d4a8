// wcc2d_scheme.cuh -- device arithmetic of the 2D WCC half-step (Sec. 3.1,
// Sec. 3.2, Sec. 4 and Appendix B of arXiv 2104.04347), in the compute type
// T (double or float).
//
// DOFs are Taylor coefficients e_kl = u_{kx,ly} / (k! l!), u_{kx,ly} = dx^k dy^l
// d^k_x d^l_y u the paper's scaled derivatives at the cell centre (Eq.
// 2DPolynomial_Space), k + l <= P, at position q = (k+l)(k+l+1)/2 + l of a
// variable's block.  Space-time series are kept as cubes X[k][l][m] of Taylor
// coefficients (dx^k dy^l dt^m d^k_x d^l_y d^m_t u / (k! l! m!)), of which only
// the entries with k + l + m <= P are ever touched: products of series are plain
// Cauchy products, without the binomial weights of the derivative form (a
// multiplication in one term of four at P = 3).  Every loop is unrolled so that each
// entry is a register and each coefficient a compile-time constant.
//
// R is float or d3 (FP64 in three-register DFMAs, wcc_d3.cuh).
#pragma once

#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>
#include <utility>

#include "wcc_d3.cuh"
#include "wcc_ff.cuh"

namespace wcc2d {

enum { ADVECTION = 0, BURGERS = 1, EULER = 2 };
enum { PERIODIC = 0, TRANSMISSIVE = 1 };
enum : unsigned { ERR_NONFINITE = 1u, ERR_POSITIVITY = 2u, ERR_BOUNDS = 4u /* checked build only */ };

__host__ __device__ constexpr int nvars(int sys) { return sys == EULER ? 4 : 1; }
__host__ __device__ constexpr int nq(int P) { return (P + 1) * (P + 2) / 2; }
__host__ __device__ constexpr int qidx(int k, int l) { return (k + l) * (k + l + 1) / 2 + l; }
// total degree d and the pair (k, l) stored at position q
__host__ __device__ constexpr int qdeg(int q) {
    int d = 0;
    while ((d + 1) * (d + 2) / 2 <= q) ++d;
    return d;
}
__host__ __device__ constexpr int ql_of(int q) { return q - qdeg(q) * (qdeg(q) + 1) / 2; }
__host__ __device__ constexpr int qk_of(int q) { return qdeg(q) - ql_of(q); }
__host__ __device__ constexpr double factd(int n) { return n <= 1 ? 1.0 : n * factd(n - 1); }
__host__ __device__ constexpr double binomd(int n, int k) { return factd(n) / (factd(k) * factd(n - k)); }
__host__ __device__ constexpr double pow2m(int n) { return n <= 0 ? 1.0 : 0.5 * pow2m(n - 1); }  // 2^-n

// mean of xi^e over [-1/2, 1/2]
__host__ __device__ constexpr double moment(int e) { return (e & 1) ? 0.0 : pow2m(e) / (e + 1); }

// j (j-1) ... (j-k+1)
__host__ __device__ constexpr double falling(int j, int k) { return factd(j) / factd(j - k); }

// Coefficient of e_ab e_a2b2 in the smoothness indicator of Eq.
// 2DSmoothIndicator (scaled form: the mean over the cell of the squared
// xi/eta-derivatives of every order 1..P).
__host__ __device__ constexpr double beta_coef(int P, int a, int b, int a2, int b2) {
    double s = 0.0;
    for (int k = 0; k <= P; ++k)
        for (int l = 0; k + l <= P; ++l) {
            if (k + l == 0 || a < k || b < l || a2 < k || b2 < l) continue;
            s += falling(a, k) * falling(a2, k) * moment(a + a2 - 2 * k) * falling(b, l) * falling(b2, l) *
                 moment(b + b2 - 2 * l);
        }
    return s;
}

// Physical constants and options a kernel needs; the float copies spare the
// FP32 kernels conversions, which run on the FP64 pipe.
struct Law2D {
    double ax, ay;     // advection velocity
    double gamma;      // Euler
    double alpha, eps; // limiter weights
    int limiter;
    int alpha_is_two;
    double g1;         // gamma - 1
    float ax_f, ay_f, gamma_f, g1_f, g1_lo_f, ax_lo_f, ay_lo_f, alpha_f, eps_f;
};

inline Law2D make_law2d(double ax, double ay, double gamma, double alpha, double eps, int limiter) {
    Law2D w{};
    w.ax = ax;
    w.ay = ay;
    w.gamma = gamma;
    w.alpha = alpha;
    w.eps = eps;
    w.limiter = limiter;
    w.alpha_is_two = alpha == 2.0;
    w.g1 = gamma - 1.0;
    w.ax_f = (float)ax;
    w.ay_f = (float)ay;
    w.gamma_f = (float)gamma;
    w.g1_f = (float)w.g1;
    w.g1_lo_f = (float)(w.g1 - (double)w.g1_f);
    w.ax_lo_f = (float)(ax - (double)w.ax_f);
    w.ay_lo_f = (float)(ay - (double)w.ay_f);
    w.alpha_f = (float)alpha;
    w.eps_f = (float)eps;
    return w;
}

using ::fabs;
using ::fma;
using wcc::d3;
using wcc::fabs;
using wcc::fma;

template <class R>
constexpr bool is_f32 = std::is_same<R, float>::value;
template <class R>
__device__ __forceinline__ R cst(double c) { return (R)c; }
// x times a constant, without the multiplication when it is 1
template <class R>
__device__ __forceinline__ R scale_by(R x, std::integral_constant<int, 1>, double) { return x; }
template <class R>
__device__ __forceinline__ R scale_by(R x, std::integral_constant<int, 0>, double c) { return x * cst<R>(c); }
#define WCC2D_TIMES(x, c) scale_by((x), std::integral_constant<int, ((c) == 1.0 ? 1 : 0)>{}, (c))

template <class R>
__device__ __forceinline__ R pick(double d, float f) {
    if constexpr (is_f32<R>) return f;
    else return (R)d;
}
__device__ __forceinline__ bool positive(float x) { return x > 0.f; }
__device__ __forceinline__ bool positive(d3 x) { return wcc::all_pos(x); }
__device__ __forceinline__ bool is_nan(float x) { return x != x; }
__device__ __forceinline__ bool is_nan(d3 x) { return x.v != x.v; }

// 1/x for a positive normal x: FP32 from the hardware estimate refined by one
// Newton step (within an ulp or two).
__device__ __forceinline__ float recip_t(float x) {
    const float r = __fdividef(1.f, x);
    return fmaf(r, fmaf(-x, r, 1.f), r);
}
__device__ __forceinline__ d3 recip_t(d3 x) { return wcc::recip(x); }
// sqrt(x) and 1/sqrt(x) of a positive x
__device__ __forceinline__ float sqrt_t(float x, float& inv) {
    const float c = x * rsqrtf(x);
    inv = recip_t(c);
    return c;
}
__device__ __forceinline__ d3 sqrt_t(d3 x, d3& inv) { return wcc::sqrt_and_recip(x, inv); }
// (a, b) / sqrt(x) for a direction
__device__ __forceinline__ void over_root(float a, float b, float x, float& oa, float& ob) {
    const float rn = rsqrtf(x);
    oa = a * rn;
    ob = b * rn;
}
__device__ __forceinline__ void over_root(d3 a, d3 b, d3 x, d3& oa, d3& ob) {
    d3 ic;
    const d3 c = sqrt_t(x, ic);
    oa = wcc::quotient(a, c, ic);
    ob = wcc::quotient(b, c, ic);
}
// a / b from rb = 1/b: FP64 rounded once
__device__ __forceinline__ float over(float a, float, float rb) { return a * rb; }
__device__ __forceinline__ d3 over(d3 a, d3 b, d3 rb) { return wcc::quotient(a, b, rb); }

__device__ __forceinline__ float weight_pow(float x, const Law2D& law) {
    return law.alpha_is_two ? x * x : exp2f(law.alpha_f * log2f(x));
}
__device__ __forceinline__ d3 weight_pow(d3 x, const Law2D& law) {
    return law.alpha_is_two ? x * x : wcc::pow_any(x, law.alpha);
}

// FP32 ratio a / b of the limiter weights for 0 < a <= b: one approximate
// reciprocal (no division sequence, no branch).  b is kept at or above the
// smallest normal float, which only changes denominators below 1.2e-38,
// where the candidate is flat to rounding.
__device__ __forceinline__ float weight_ratio(float a, float b) { return __fdividef(a, fmaxf(b, 0x1p-126f)); }

// ------------------------------------------------------------------ parent

// What an old cell contributes to the four new cells it touches, per
// variable v:
//   c[v][r]: its share of the cell average of Eq. 2DIntegral in the new cell
//            of which it is vertex r (0: lower left, 1: lower right, 2: upper
//            right, 3: upper left), i.e. a quarter of the quarter average
//            (Eqs. SubEq:2DCellAVGRU ... LD) plus lamx/2 and lamy/2 times its
//            time-averaged edge fluxes (Eqs. SubEq:2DFluxFU ... GL) with the
//            signs of Eq. 2DIntegral;
//   V[v][q]: Taylor coefficients at the centre at t^{n+1/2}, k + l <= P - 1
//            (the entries Eqs. SubEq:2DUx, SubEq:2DUy read; q = 0 is the
//            vertex value of the limiter), Eq. SubEq:2DUij.
// The shares are a +- p +- q +- r with the signs of the four quadrants: a the
// even part (a quarter of the average), p the part odd along x, q along y, r
// along both.  FP32-mixed (MX): p, q, r without the leading flux terms
// hx f(u_00) in p and hy g(u_00) in q (added in float-float), no a, and V[v][0]
// without the point value u_00 itself.
template <int SYS, int P, class R, bool MX = false>
struct Parent {
    static constexpr int NV = nvars(SYS);
    static constexpr int NQ1 = nq(P - 1);
    R c[NV][4];
    R V[NV][NQ1];
    R p[NV], q[NV], r[NV];
};

// Compile-time loop: f(std::integral_constant<int, I>{}) for I = 0 .. N-1, so
// that every index the body forms is a constant (loops whose bounds depend on
// an outer index are not reliably unrolled by #pragma unroll, and a run-time
// index into a register array sends it to local memory).
template <class F, int... I>
__device__ __forceinline__ void unroll_seq(F&& f, std::integer_sequence<int, I...>) {
    (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void unroll(F&& f) {
    unroll_seq(f, std::make_integer_sequence<int, (N > 0 ? N : 0)>{});
}

// How a stage and a new cell hold coefficient (k, l): e_kl times this.  FP64 holds the
// derivatives u_3x and u_3y themselves: 6 is the one k! l! that is not a power of two, and
// a value multiplied by it and divided again does not always come back, whereas a
// stage read back to the host has to load again bit for bit.  (FP32 coefficients
// times 6 are exact in the host's doubles.)
template <class R>
__host__ __device__ constexpr double kept(int k, int l) {
    return std::is_same<R, d3>::value && (k == 3 || l == 3) ? 6.0 : 1.0;
}
template <class R>
__host__ __device__ constexpr double kept(int q) { return kept<R>(qk_of(q), ql_of(q)); }

// mean of xi^k over [0, 1/2]
__host__ __device__ constexpr double half_mean(int k) { return pow2m(k) / (k + 1); }

// Cauchy-Kovalewski procedure in 2D (Sec. 3.1; Sec. 4 for systems):
// X_{k,l,m+1} = -(lamx (k+1) F_{k+1,l,m} + lamy (l+1) G_{k,l+1,m}) / (m+1), with
// Cauchy products for the products and quotients of series (Dyson /
// Dumbser-Munz).  Each flux entry is used as soon as it is formed: for the
// next time level of X and for the edge-flux integrals of Appendix B.
template <int SYS, int P, class R, bool MX = false>
__device__ __forceinline__ void parent_terms(const R (&q)[nvars(SYS)][nq(P)], R lamx, R lamy, const Law2D& law,
                                             Parent<SYS, P, R, MX>& out) {
    constexpr int NV = nvars(SYS);
    R X[NV][P + 1][P + 1][P + 1];
    unroll<NV>([&](auto vc) {
        unroll<P + 1>([&](auto kc) {
            unroll<P + 1 - kc>([&](auto lc) {
                constexpr double c = 1.0 / kept<R>(kc, lc);
                X[vc][kc][lc][0] = WCC2D_TIMES(q[vc][qidx(kc, lc)], c);
            });
        });
    });
    // time-averaged fluxes on the half lines through the centre, along x the
    // even (FE) and odd (FO) parts in eta, along y those in xi
    R FE[NV], FO[NV], GE[NV], GO[NV];
    if constexpr (MX) {
        unroll<NV>([&](auto vc) { FE[vc] = FO[vc] = GE[vc] = GO[vc] = 0.f; });
    }
    R w1[P + 1][P + 1][P + 1], w2[P + 1][P + 1][P + 1], H[P + 1][P + 1][P + 1];
    float2 W[P + 1][P + 1][P + 1];  // plain FP32: the velocities (w1, w2) as pairs
    R inv_rho;
    if constexpr (SYS == EULER) inv_rho = recip_t(X[0][0][0][0]);

    unroll<P + 1>([&](auto mc) {
        constexpr int m = mc;
        unroll<P + 1 - m>([&](auto kc) {
            constexpr int k = kc;
            unroll<P + 1 - m - k>([&](auto lc) {
                constexpr int l = lc;
                R F[NV], G[NV];
                if constexpr (SYS == ADVECTION) {
                    F[0] = pick<R>(law.ax, law.ax_f) * X[0][k][l][m];
                    G[0] = pick<R>(law.ay, law.ay_f) * X[0][k][l][m];
                } else if constexpr (SYS == BURGERS) {
                    R s;
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                if constexpr (i + j + n == 0) s = X[0][i][j][n] * X[0][k - i][l - j][m - n];
                                else s = fma(X[0][i][j][n], X[0][k - i][l - j][m - n], s);
                            });
                        });
                    });
                    F[0] = cst<R>(0.5) * s;
                    G[0] = F[0];
                } else if constexpr (is_f32<R> && !MX) {
                    // plain FP32: the two velocities, (q_xx, q_xy) and the two
                    // energy fluxes two at a time in paired FP32 instructions
                    // (FFMA2); the same operations as the scalar form below.
                    // The FP32-mixed kernel keeps the scalar form: there the
                    // pairs cost registers (spills) and it ran slower.
                    float2 s12 = make_float2(X[1][k][l][m], X[2][k][l][m]);
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                if constexpr (i + j + n != 0) {
                                    const float c = X[0][i][j][n];
                                    s12 = __ffma2_rn(make_float2(-c, -c), W[k - i][l - j][m - n], s12);
                                }
                            });
                        });
                    });
                    W[k][l][m] = __fmul2_rn(s12, make_float2(inv_rho, inv_rho));
                    float2 qx = make_float2(0.f, 0.f);
                    float qyy = 0.f;
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                const float a1 = X[1][i][j][n], a2 = X[2][i][j][n];
                                qx = __ffma2_rn(make_float2(a1, a1), W[k - i][l - j][m - n], qx);
                                qyy = fmaf(a2, W[k - i][l - j][m - n].y, qyy);
                            });
                        });
                    });
                    const float p = law.g1_f * (X[3][k][l][m] - 0.5f * (qx.x + qyy));
                    H[k][l][m] = X[3][k][l][m] + p;
                    float2 e12 = make_float2(0.f, 0.f);
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                const float c = H[i][j][n];
                                e12 = __ffma2_rn(make_float2(c, c), W[k - i][l - j][m - n], e12);
                            });
                        });
                    });
                    F[0] = X[1][k][l][m];
                    F[1] = qx.x + p;
                    F[2] = qx.y;
                    F[3] = e12.x;
                    G[0] = X[2][k][l][m];
                    G[1] = qx.y;
                    G[2] = qyy + p;
                    G[3] = e12.y;
                } else {
                    // velocities from rho w = momentum, solved entry by entry
                    R s1 = X[1][k][l][m], s2 = X[2][k][l][m];
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                if constexpr (i + j + n != 0) {
                                    s1 = fma(-X[0][i][j][n], w1[k - i][l - j][m - n], s1);
                                    s2 = fma(-X[0][i][j][n], w2[k - i][l - j][m - n], s2);
                                }
                            });
                        });
                    });
                    w1[k][l][m] = s1 * inv_rho;
                    w2[k][l][m] = s2 * inv_rho;
                    R qxx, qxy, qyy;
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                if constexpr (i + j + n == 0) {
                                    qxx = X[1][i][j][n] * w1[k - i][l - j][m - n];
                                    qxy = X[1][i][j][n] * w2[k - i][l - j][m - n];
                                    qyy = X[2][i][j][n] * w2[k - i][l - j][m - n];
                                } else {
                                    qxx = fma(X[1][i][j][n], w1[k - i][l - j][m - n], qxx);
                                    qxy = fma(X[1][i][j][n], w2[k - i][l - j][m - n], qxy);
                                    qyy = fma(X[2][i][j][n], w2[k - i][l - j][m - n], qyy);
                                }
                            });
                        });
                    });
                    const R p = pick<R>(law.g1, law.g1_f) * fma(cst<R>(-0.5), qxx + qyy, X[3][k][l][m]);
                    H[k][l][m] = X[3][k][l][m] + p;
                    R e1, e2;
                    unroll<k + 1>([&](auto i) {
                        unroll<l + 1>([&](auto j) {
                            unroll<m + 1>([&](auto n) {
                                if constexpr (i + j + n == 0) {
                                    e1 = H[i][j][n] * w1[k - i][l - j][m - n];
                                    e2 = H[i][j][n] * w2[k - i][l - j][m - n];
                                } else {
                                    e1 = fma(H[i][j][n], w1[k - i][l - j][m - n], e1);
                                    e2 = fma(H[i][j][n], w2[k - i][l - j][m - n], e2);
                                }
                            });
                        });
                    });
                    F[0] = X[1][k][l][m];
                    F[1] = qxx + p;
                    F[2] = qxy;
                    F[3] = e1;
                    G[0] = X[2][k][l][m];
                    G[1] = qxy;
                    G[2] = qyy + p;
                    G[3] = e2;
                }
                // (k + l >= 1 implies m + 1 <= P; an entry's y term comes first)
                if constexpr (l >= 1) {
                    const R lw = WCC2D_TIMES(lamy, (double)l / (m + 1));
                    unroll<NV>([&](auto vc) { X[vc][k][l - 1][m + 1] = -lw * G[vc]; });
                }
                if constexpr (k >= 1) {
                    const R lw = WCC2D_TIMES(lamx, (double)k / (m + 1));
                    unroll<NV>([&](auto vc) { X[vc][k - 1][l][m + 1] = fma(-lw, F[vc], X[vc][k - 1][l][m + 1]); });
                }
                // Eqs. SubEq:2DFluxFU ... GL: one space direction along the edge, and time
                if constexpr (k == 0 && (!MX || l + m > 0)) {
                    constexpr double c = half_mean(l) / (m + 1);
                    unroll<NV>([&](auto vc) {
                        if constexpr (!MX && l + m == 0) FE[vc] = F[vc];
                        else if constexpr (!MX && l == 1 && m == 0) FO[vc] = cst<R>(c) * F[vc];
                        else if constexpr ((l & 1) == 0) FE[vc] = fma(cst<R>(c), F[vc], FE[vc]);
                        else FO[vc] = fma(cst<R>(c), F[vc], FO[vc]);
                    });
                }
                if constexpr (l == 0 && (!MX || k + m > 0)) {
                    constexpr double c = half_mean(k) / (m + 1);
                    unroll<NV>([&](auto vc) {
                        if constexpr (!MX && k + m == 0) GE[vc] = G[vc];
                        else if constexpr (!MX && k == 1 && m == 0) GO[vc] = cst<R>(c) * G[vc];
                        else if constexpr ((k & 1) == 0) GE[vc] = fma(cst<R>(c), G[vc], GE[vc]);
                        else GO[vc] = fma(cst<R>(c), G[vc], GO[vc]);
                    });
                }
            });
        });
    });
    // shares of the new cell averages (Eq. 2DIntegral): quarter of the quarter
    // averages by parity, with the edge fluxes of the same parity
    const R hx = cst<R>(0.5) * lamx, hy = cst<R>(0.5) * lamy;
    unroll<NV>([&](auto vc) {
        constexpr int v = vc;
        R a = cst<R>(0.25) * q[v][0], p = cst<R>(0.25 * half_mean(1)) * q[v][qidx(1, 0)],
          s = cst<R>(0.25 * half_mean(1)) * q[v][qidx(0, 1)], r;
        if constexpr (P >= 2) r = cst<R>(0.25 * half_mean(1) * half_mean(1)) * q[v][qidx(1, 1)];
        unroll<P + 1>([&](auto kc) {
            unroll<P + 1 - kc>([&](auto lc) {
                constexpr int k = kc, l = lc;
                if constexpr (k + l >= 2 && !(k == 1 && l == 1)) {
                    const R w = cst<R>(0.25 * half_mean(k) * half_mean(l) / kept<R>(k, l));
                    if constexpr (!(k & 1) && !(l & 1)) a = fma(w, q[v][qidx(k, l)], a);
                    else if constexpr (!(l & 1)) p = fma(w, q[v][qidx(k, l)], p);
                    else if constexpr (!(k & 1)) s = fma(w, q[v][qidx(k, l)], s);
                    else r = fma(w, q[v][qidx(k, l)], r);
                }
            });
        });
        p = fma(hx, FE[v], p);
        s = fma(hy, GE[v], s);
        if constexpr (P >= 2) r = fma(hx, FO[v], fma(hy, GO[v], r));
        else r = fma(hx, FO[v], hy * GO[v]);
        if constexpr (MX) {
            out.p[v] = p;
            out.q[v] = s;
            out.r[v] = r;
        } else {
            const R ap = a + s, am = a - s, pp = p + r, pm = p - r;
            out.c[v][0] = ap + pp;
            out.c[v][1] = ap - pp;
            out.c[v][2] = am - pm;
            out.c[v][3] = am + pm;
        }
    });
    // Eq. SubEq:2DUij
    unroll<NV>([&](auto vc) {
        unroll<P>([&](auto kc) {
            unroll<P - kc>([&](auto lc) {
                constexpr int k = kc, l = lc, m0 = (MX && k + l == 0) ? 1 : 0;
                R s = X[vc][k][l][m0];
                unroll<P - k - l - m0>([&](auto mc) { s = s + X[vc][k][l][mc + m0 + 1]; });
                out.V[vc][qidx(k, l)] = s;
            });
        });
    });
}

// ---------------------------------------------------------------- new cell

// Derivatives of the unlimited new cell from the highest degree down to degree
// LOW (Eqs. SubEq:2DUx, SubEq:2DUy, mixed ones as the mean of both), in Taylor
// coefficients: with the parents' vertex coefficients T at the four vertices
// (1 lower left, 2 lower right, 3 upper right, 4 upper left),
//   (k+1) e_{k+1,l} = ((T_2 + T_3) - (T_1 + T_4))_{kl} / 2
//       - sum_{s odd, t even, s+t >= 3} 2^{1-s-t} C(k+s, s) C(l+t, t) e_{k+s,l+t}
// and the same along y, each as a new cell keeps it (kept).  dxy(k, l, dx, dy) gives
// the two differences.
template <int P, int LOW, class R, class Diff>
__device__ __forceinline__ void derivatives2d(Diff&& dxy, R (&D)[nq(P)]) {
    unroll<P + 1 - LOW>([&](auto dd) {
        constexpr int d = P - 1 - dd;  // degree of the vertex coefficients used: gives degree d + 1
        // contributions to e_{k+1,l} (x) and e_{k,l+1} (y) of every (k, l) of degree d
        unroll<d + 1>([&](auto lc) {
            constexpr int l = lc, k = d - l, r = P - d;
            R dx, dy;
            dxy(std::integral_constant<int, qidx(k, l)>{}, dx, dy);
            // mixed derivatives are the mean of the two formulas
            constexpr double wx = (l > 0 ? 0.5 : 1.0) / (k + 1) * kept<R>(k + 1, l),
                             wy = (k > 0 ? 0.5 : 1.0) / (l + 1) * kept<R>(k, l + 1);
            R ex = WCC2D_TIMES(dx, 0.5 * wx), ey = WCC2D_TIMES(dy, 0.5 * wy);
            unroll<r + 1>([&](auto sc) {
                unroll<r + 1>([&](auto tc) {
                    constexpr int s = sc, t = tc;
                    if constexpr ((s & 1) && !(t & 1) && s + t >= 3 && s + t <= r) {
                        ex = fma(cst<R>(-wx * 2.0 * pow2m(s + t) * binomd(k + s, s) * binomd(l + t, t) / kept<R>(k + s, l + t)),
                                 D[qidx(k + s, l + t)], ex);
                        ey = fma(cst<R>(-wy * 2.0 * pow2m(s + t) * binomd(l + s, s) * binomd(k + t, t) / kept<R>(k + t, l + s)),
                                 D[qidx(k + t, l + s)], ey);
                    }
                });
            });
            if constexpr (l == 0) D[qidx(k + 1, 0)] = ex;
            else D[qidx(k + 1, l)] = D[qidx(k + 1, l)] + ex;  // its y term came with (k + 1, l - 1)
            D[qidx(k, l + 1)] = ey;
        });
    });
}

// Mean over the cell of the even terms (k, l) != (0, 0): the cell average is
// e_00 plus this (Eq. SubEq:2DCellAVG).
template <int P, class R>
__device__ __forceinline__ R even_correction(const R (&d)[nq(P)]) {
    if constexpr (P < 2) return cst<R>(0.0);
    else return cst<R>(1.0 / 12.0) * (d[qidx(2, 0)] + d[qidx(0, 2)]);
}
static_assert(moment(2) == 1.0 / 12.0, "the even terms of degree 2");

// The linear part of a new cell (Sec. 3.1): the cell average (Eq. 2DIntegral)
// and the derivatives of degree >= LOW.  rd.c(r, v) and rd.V(r, v, q) read the
// terms of parent r (struct Parent).
template <int SYS, int P, int LOW, class R, class Rd>
__device__ __forceinline__ void linear_cell(const Rd& rd, R (&D)[nvars(SYS)][nq(P)], R (&ubar)[nvars(SYS)]) {
    unroll<nvars(SYS)>([&](auto vc) {
        constexpr int v = vc;
        ubar[v] = (rd.c(0, v) + rd.c(1, v)) + (rd.c(2, v) + rd.c(3, v));
        derivatives2d<P, LOW, R>(
            [&](auto qc, R& dx, R& dy) {
                const R A = rd.V(2, v, qc) - rd.V(0, v, qc), B = rd.V(1, v, qc) - rd.V(3, v, qc);
                dx = A + B;
                dy = A - B;
            },
            D[v]);
    });
}

// The first derivatives from the vertex values less the average.
template <int P, class R>
__device__ __forceinline__ void first_derivatives(R (&d)[nq(P)], const R (&vv)[4]) {
    const R A = vv[2] - vv[0], B = vv[1] - vv[3];
    R ex = cst<R>(0.5) * (A + B), ey = cst<R>(0.5) * (A - B);
    if constexpr (P >= 3) {
        if constexpr (is_f32<R>) {
            ex = fma(cst<R>(-0.25), d[qidx(3, 0)] + d[qidx(1, 2)], ex);
            ey = fma(cst<R>(-0.25), d[qidx(0, 3)] + d[qidx(2, 1)], ey);
        } else {
            constexpr double c = -0.25 / kept<R>(3, 0);
            ex = fma(cst<R>(c), d[qidx(3, 0)], fma(cst<R>(-0.25), d[qidx(1, 2)], ex));
            ey = fma(cst<R>(c), d[qidx(0, 3)], fma(cst<R>(-0.25), d[qidx(2, 1)], ey));
        }
    }
    d[1] = ex;
    d[2] = ey;
}

// ----------------------------------------------------------------- limiter

// Limiter of Sec. 3.2 for one scalar component in deviation form: d[1..] the
// Taylor coefficients of u_0 as kept (replaced by those of u_*) and the vertex
// values vv[0..3] at vertices 1..4 less the cell average ub, which the limiter
// keeps (only the rounding of FP64's residuals depends on it).  FP64 follows the printed weights; in
// FP32 the same weights are formed from ratios (every term divided by the
// largest) so that the tiny epsilon cannot overflow them.
//
// The residuals of u_0 at opposite vertices are equal: by construction of the
// first derivatives u_0's differences across the cell are those of the vertex
// values along x and along y, so r_1 + r_2 = r_0 + r_3 and r_3 + r_2 = r_0 + r_1.
// The odd terms drop out of their means:
//   r_0 = r_2 = a + e_11 / 4 - (v_0 + v_2) / 2,  r_1 = r_3 = a - e_11 / 4 - (v_1 + v_3) / 2,
// a = (e_20 + e_02) (1/4 - 1/12) the even part at a vertex less the average.
//
// Returns false, with d as it was, where the limiter does not act: FP64 with
// sigma tau below 2^-31 of every denominator (compared on the exponents), FP32
// below 2^-15 of them (the side weights, squares of the ratios, are then below
// 2^-62 and 2^-30: w_0 is 1).
template <int P, class R>
__device__ __forceinline__ bool limit_scalar(R (&d)[nq(P)], const R (&vv)[4], const Law2D& law, R ub) {
    constexpr int NQ = nq(P);
    R sx[5], sy[5];
    sx[1] = -(vv[0] + vv[3]);
    sy[1] = vv[3] - vv[0];
    sx[2] = vv[1] - vv[0];
    sy[2] = -(vv[0] + vv[1]);
    sx[3] = vv[1] + vv[2];
    sy[3] = vv[2] - vv[1];
    sx[4] = vv[2] - vv[3];
    sy[4] = vv[3] + vv[2];
    R beta[5];
    // the quadratic form of Eq. 2DSmoothIndicator over pairs q1 <= q2, as sum
    // over q1 of d[q1] times an inner sum over q2 (independent chains)
    unroll<NQ - 1>([&](auto q1c) {
        constexpr int q1 = q1c + 1;
        constexpr double c1 = beta_coef(P, qk_of(q1), ql_of(q1), qk_of(q1), ql_of(q1)) / (kept<R>(q1) * kept<R>(q1));
        R inner = WCC2D_TIMES(d[q1], c1);
        unroll<NQ>([&](auto q2) {
            if constexpr (q2 > q1) {
                constexpr double c = 2.0 * beta_coef(P, qk_of(q1), ql_of(q1), qk_of(q2), ql_of(q2)) / (kept<R>(q1) * kept<R>(q2));
                if constexpr (c != 0.0) inner = fma(cst<R>(c), d[q2], inner);
            }
        });
        if constexpr (q1 == 1) beta[0] = d[q1] * inner;
        else beta[0] = fma(d[q1], inner, beta[0]);
    });
#pragma unroll
    for (int m = 1; m <= 4; ++m) beta[m] = fma(sx[m], sx[m], sy[m] * sy[m]);
    const R eps = pick<R>(law.eps, law.eps_f);
    R w[5];
    if constexpr (P == 1) {
        // Eq. 2D2ndOrderWeights
        if constexpr (!is_f32<R>) {
#pragma unroll
            for (int m = 0; m < 5; ++m) w[m] = weight_pow(recip_t(beta[m] + eps), law);
            const R sum = ((w[0] + w[1]) + (w[2] + w[3])) + w[4], is = recip_t(sum);
#pragma unroll
            for (int m = 1; m < 5; ++m) w[m] = over(w[m], sum, is);
            w[0] = cst<R>(1.0) - ((w[1] + w[2]) + (w[3] + w[4]));
        } else {
            // every weight divided by that of the smallest denominator
            R bmin = beta[0] + eps;
#pragma unroll
            for (int m = 1; m < 5; ++m) bmin = fminf(bmin, beta[m] + eps);
            R s = 0;
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                w[m] = weight_pow(weight_ratio(bmin, beta[m] + eps), law);
                s += w[m];
            }
            const R is = recip_t(s);  // s >= 1
#pragma unroll
            for (int m = 0; m < 5; ++m) w[m] *= is;
        }
    } else {
        // Eq. 1DHighOrderWeights in the 2D form of Sec. 3.2: sigma from the
        // vertex residuals, tau from the degree-P derivatives
        const R a = cst<R>(0.25 - 1.0 / 12.0) * (d[qidx(2, 0)] + d[qidx(0, 2)]), c11 = d[qidx(1, 1)];
        const R a0 = fma(cst<R>(0.25), c11, a), a1 = fma(cst<R>(-0.25), c11, a);
        R r0, r1;
        if constexpr (is_f32<R>) {
            r0 = fma(cst<R>(-0.5), vv[0] + vv[2], a0);
            r1 = fma(cst<R>(-0.5), vv[1] + vv[3], a1);
        } else {
            // differences of the values themselves: their rounding is part of
            // the printed weights where the flow is uniform to rounding
            r0 = (ub + a0) - fma(cst<R>(0.5), vv[0] + vv[2], ub);
            r1 = (ub + a1) - fma(cst<R>(0.5), vv[1] + vv[3], ub);
        }
        const R half_sigma = fma(r0, r0, r1 * r1);
        // tau in the derivatives u_{kx,ly} = k! l! e_kl
        R tau;
        if constexpr (P == 2) {
            tau = fma(c11, c11, cst<R>(4.0) * fma(d[qidx(2, 0)], d[qidx(2, 0)], d[qidx(0, 2)] * d[qidx(0, 2)]));
        } else {
            const R t0 = fma(d[qidx(3, 0)], d[qidx(3, 0)], d[qidx(0, 3)] * d[qidx(0, 3)]);
            const R t1 = fma(d[qidx(2, 1)], d[qidx(2, 1)], d[qidx(1, 2)] * d[qidx(1, 2)]);
            constexpr double c = 36.0 / (kept<R>(3, 0) * kept<R>(3, 0));
            if constexpr (c == 1.0) tau = fma(cst<R>(4.0), t1, t0);
            else tau = fma(cst<R>(c), t0, cst<R>(4.0) * t1);
        }
        const R st = (half_sigma + half_sigma) * tau;
        if constexpr (!is_f32<R>) {
            R den[5];
            int least = 2047;
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                den[m] = fma(beta[m], beta[m], eps);
                least = min(least, wcc::exponent_of(den[m]));
            }
            if (law.alpha_is_two && wcc::exponent_of(st) + 32 <= least) return false;
#pragma unroll
            for (int m = 0; m < 5; ++m) w[m] = weight_pow(wcc::quotient(st, den[m]), law);
            const R rest = (w[1] + w[2]) + (w[3] + w[4]);
            const R sum = (w[0] + cst<R>(1.0)) + rest, is = recip_t(sum);
#pragma unroll
            for (int m = 1; m < 5; ++m) w[m] = over(w[m], sum, is);
            w[0] = cst<R>(1.0) - ((w[1] + w[2]) + (w[3] + w[4]));  // 1 when the others vanish
        } else {
            // divide every weight by (st / dmin)^alpha, dmin the smallest denominator
            R den[5];
            R dmin = INFINITY;
#pragma unroll
            for (int m = 0; m < 5; ++m) {
                den[m] = fmaf(beta[m], beta[m], eps);
                dmin = fminf(dmin, den[m]);
            }
            if (law.alpha_is_two && !(st * 0x1p15f >= dmin)) return false;
            // the "1 +" of w_0, rescaled.  dmin and st both scaled by 2^64
            // (exact), so that a subnormal st (its dmin can be subnormal too:
            // eps = 1e-40) is a normal number for the reciprocal; st above
            // 2^62 gives lead = 0, its value to rounding
            const R lead = weight_pow((dmin * 0x1p64f) * recip_t(st * 0x1p64f), law);
            // lead above 2^30 puts the other weights below 5 2^-30 of the
            // sum: w_0 rounds to 1 (this also keeps the sum, and so the
            // reciprocal below, in range)
            if (!(st > 0.f) || !(lead < 0x1p30f)) {
                w[0] = 1;
                w[1] = w[2] = w[3] = w[4] = 0;
            } else {
                R s = 0;
#pragma unroll
                for (int m = 0; m < 5; ++m) {
                    w[m] = weight_pow(weight_ratio(dmin, den[m]), law);
                    if (m == 0) w[m] += lead;
                    s += w[m];
                }
                const R is = recip_t(s);  // s >= 1
#pragma unroll
                for (int m = 0; m < 5; ++m) w[m] *= is;
            }
        }
    }
    // Eq. 2DLimitedPolynomial
    R l1 = w[0] * d[1], l2 = w[0] * d[2];
#pragma unroll
    for (int m = 1; m <= 4; ++m) {
        l1 = fma(w[m], sx[m], l1);
        l2 = fma(w[m], sy[m], l2);
    }
    d[1] = l1;
    d[2] = l2;
#pragma unroll
    for (int i = 3; i < NQ; ++i) d[i] = w[0] * d[i];
    return true;
}

// Rotated characteristic limiting for the 2D Euler equations (Sec. 4):
// direction n from the central-difference gradient of rho e (Eq.
// RotatedNormal), eigenvectors of cos(theta) dF/dU + sin(theta) dG/dU at the
// cell average ub in closed form, the scalar limiter on each characteristic
// component, and back.  vv: the vertex values less the average.  FP64 takes
// D's coefficients of degree >= 2 and forms the first derivatives after the
// projection.  Returns false if the average has non-positive density or
// pressure.
template <int P, class R>
__device__ __forceinline__ bool limit_euler(R (&D)[4][nq(P)], const R (&ub)[4], const R (&vv)[4][4], R lamx, R lamy,
                                            const Law2D& law) {
    constexpr int NQ = nq(P);
    const R gA = vv[3][2] - vv[3][0], gB = vv[3][1] - vv[3][3];
    R gx = (gA + gB) * lamx, gy = (gA - gB) * lamy;  // (twice the gradient: only its direction counts)
    const R g2 = fma(gx, gx, gy * gy);
    R nx = cst<R>(1.0), ny = cst<R>(0.0);
    if (positive(g2)) over_root(gx, gy, g2, nx, ny);
    const R gm1 = pick<R>(law.g1, law.g1_f), gamma = pick<R>(law.gamma, law.gamma_f);
    const R rho = ub[0];
    const R irho = recip_t(rho);
    const R u = over(ub[1], rho, irho), v = over(ub[2], rho, irho);
    const R hq2 = cst<R>(0.5) * fma(u, u, v * v);
    const R p = gm1 * fma(-rho, hq2, ub[3]);
    if (!positive(rho) || !positive(p)) return false;
    R ic;
    // c and 1/c within an ulp of each other, so that the left and right
    // eigenvectors stay inverse to rounding (the projection and the
    // back-projection then cancel where the weights are linear)
    const R c = sqrt_t(over(gamma * p, rho, irho), ic);
    const R H = over(ub[3] + p, rho, irho);
    const R un = fma(u, nx, v * ny), ut = fma(v, nx, -(u * ny));
    if constexpr (!is_f32<R>) {
        // With X = (b_1/2) (q^2/2 d_0 - u d_1 - v d_2 + d_3), b_1 = (gamma - 1)/c^2, and
        // Y = (n . (d_1, d_2) - u_n d_0) / (2 c):
        //   L d = (X - Y, d_0 - 2 X, n x (d_1, d_2) - u_t d_0, X + Y),
        //   R w = (s + w_1, u (s + w_1) + n_x m - n_y w_2, v (s + w_1) + n_y m + n_x w_2,
        //          H s + q^2/2 w_1 + u_t w_2 + u_n m),  s = w_0 + w_3, m = c (w_3 - w_0).
        const R cc = c * c, hic = cst<R>(0.5) * ic, b1h = cst<R>(0.5) * over(gm1, cc, recip_t(cc)), kx = nx * hic, ky = ny * hic, ku = un * hic;
        auto left = [&](R d0, R d1, R d2, R d3_, R (&w)[4]) {
            const R Xc = b1h * fma(-u, d1, fma(-v, d2, fma(hq2, d0, d3_)));
            const R Y = fma(kx, d1, fma(ky, d2, -(ku * d0)));
            w[0] = Xc - Y;
            w[1] = fma(cst<R>(-2.0), Xc, d0);
            w[2] = fma(nx, d2, fma(-ny, d1, -(ut * d0)));
            w[3] = Xc + Y;
        };
        R cd[4][NQ], cvv[4][4], cub[4];
        left(ub[0], ub[1], ub[2], ub[3], cub);
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            R w[4];
            left(vv[0][r], vv[1][r], vv[2][r], vv[3][r], w);
#pragma unroll
            for (int i = 0; i < 4; ++i) cvv[i][r] = w[i];
        }
#pragma unroll
        for (int qq = 3; qq < NQ; ++qq) {
            R w[4];
            left(D[0][qq], D[1][qq], D[2][qq], D[3][qq], w);
#pragma unroll
            for (int i = 0; i < 4; ++i) cd[i][qq] = w[i];
        }
        bool limited = false;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            first_derivatives<P>(cd[i], cvv[i]);
            limited |= limit_scalar<P>(cd[i], cvv[i], law, cub[i]);
        }
        if (!limited) {  // nothing to map back
#pragma unroll
            for (int j = 0; j < 4; ++j) first_derivatives<P>(D[j], vv[j]);
            return true;
        }
#pragma unroll
        for (int qq = 1; qq < NQ; ++qq) {
            const R w0 = cd[0][qq], w1 = cd[1][qq], w2 = cd[2][qq], w3 = cd[3][qq];
            const R s = w0 + w3, m = c * (w3 - w0);
            const R d0 = s + w1;
            D[0][qq] = d0;
            D[1][qq] = fma(u, d0, fma(nx, m, -(ny * w2)));
            D[2][qq] = fma(v, d0, fma(ny, m, nx * w2));
            D[3][qq] = fma(H, s, fma(hq2, w1, fma(ut, w2, un * m)));
        }
    } else {
        const R b1 = gm1 * ic * ic;
        const R b2 = b1 * hq2;
        const R Rm[4][4] = {{1, 1, 0, 1},
                            {u - c * nx, u, -ny, u + c * nx},
                            {v - c * ny, v, nx, v + c * ny},
                            {H - c * un, hq2, ut, H + c * un}};
        const R L[4][4] = {{0.5f * (b2 + un * ic), -0.5f * (b1 * u + nx * ic), -0.5f * (b1 * v + ny * ic), 0.5f * b1},
                           {1 - b2, b1 * u, b1 * v, -b1},
                           {-ut, -ny, nx, 0},
                           {0.5f * (b2 - un * ic), -0.5f * (b1 * u - nx * ic), -0.5f * (b1 * v - ny * ic), 0.5f * b1}};
        // the projections two DOFs (two vertices) at a time in paired FP32
        // instructions (FFMA2)
        constexpr int NPR = (NQ - 1) / 2;
        R cd[4][NQ], cvv[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int r = 0; r < 4; r += 2) {
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc = __ffma2_rn(make_float2(L[i][j], L[i][j]), make_float2(vv[j][r], vv[j][r + 1]), acc);
                cvv[i][r] = acc.x;
                cvv[i][r + 1] = acc.y;
            }
#pragma unroll
            for (int pr = 0; pr < NPR; ++pr) {
                const int qq = 1 + 2 * pr;
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    acc = __ffma2_rn(make_float2(L[i][j], L[i][j]), make_float2(D[j][qq], D[j][qq + 1]), acc);
                cd[i][qq] = acc.x;
                cd[i][qq + 1] = acc.y;
            }
            if constexpr ((NQ - 1) & 1) {
                R sum = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) sum += L[i][j] * D[j][NQ - 1];
                cd[i][NQ - 1] = sum;
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) limit_scalar<P>(cd[i], cvv[i], law, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int pr = 0; pr < NPR; ++pr) {
                const int qq = 1 + 2 * pr;
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    acc = __ffma2_rn(make_float2(Rm[j][i], Rm[j][i]), make_float2(cd[i][qq], cd[i][qq + 1]), acc);
                D[j][qq] = acc.x;
                D[j][qq + 1] = acc.y;
            }
            if constexpr ((NQ - 1) & 1) {
                R sum = 0;
#pragma unroll
                for (int i = 0; i < 4; ++i) sum += Rm[j][i] * cd[i][NQ - 1];
                D[j][NQ - 1] = sum;
            }
        }
    }
    return true;
}

// s_x/dx + s_y/dy at a cell's centre point values (the 2D CFL rate; the
// half step is dt = nu / max of it).  NaN for non-physical Euler states.
template <int SYS, class R>
__device__ __forceinline__ R cfl_rate(const R* centre, const Law2D& law, R idx, R idy) {
    if constexpr (SYS == ADVECTION) {
        return fma(fabs(pick<R>(law.ax, law.ax_f)), idx, fabs(pick<R>(law.ay, law.ay_f)) * idy);
    } else if constexpr (SYS == BURGERS) {
        return fabs(centre[0]) * (idx + idy);
    } else {
        const R rho = centre[0];
        if (!positive(rho)) return cst<R>(NAN);
        const R irho = recip_t(rho), u = over(centre[1], rho, irho), v = over(centre[2], rho, irho);
        const R p = pick<R>(law.g1, law.g1_f) * fma(cst<R>(-0.5) * rho, fma(u, u, v * v), centre[3]);
        if (!positive(p)) return cst<R>(NAN);
        R ic;
        const R c = sqrt_t(over(pick<R>(law.gamma, law.gamma_f) * p, rho, irho), ic);
        return fma(fabs(u) + c, idx, (fabs(v) + c) * idy);
    }
}

// ------------------------------------------------------------- FP32-mixed

// Float-float pieces of the FP32-mixed 2D path: the cell average, the leading
// flux terms and the vertex point values carry about 48 bits, everything else
// is float (as in the 1D FP32-mixed path).
using wcc::ff;

// a * b as an unnormalised pair (hi, lo): exact product of a.hi, plus a.lo * b
__device__ __forceinline__ ff ffm_lazy(ff a, float b) {
    const ff p = wcc::two_prod(a.hi, b);
    return ff{p.hi, fmaf(a.lo, b, p.lo)};
}
// a + b + c + s + lo for O(1) floats a, b, c, a small float s and a low part
// lo: every addition of a high part is exact (two_sum), its error joins the
// low part, which is renormalised once at the end.
__device__ __forceinline__ ff ff_sum4(float a, float b, float c, float s, float lo) {
    const ff x = wcc::two_sum(a, b);
    const ff y = wcc::two_sum(x.hi, c);
    const ff z = wcc::two_sum(y.hi, s);
    return wcc::fast_two_sum(z.hi, ((lo + x.lo) + y.lo) + z.lo);
}
// a - b - c - d in float-float, in the same way
__device__ __forceinline__ ff ff_rest3(ff a, ff b, ff c, ff d) {
    const ff x = wcc::two_sum(a.hi, -b.hi);
    const ff y = wcc::two_sum(x.hi, -c.hi);
    const ff z = wcc::two_sum(y.hi, -d.hi);
    return wcc::fast_two_sum(z.hi, ((a.lo - b.lo) - (c.lo + d.lo)) + ((x.lo + y.lo) + z.lo));
}
// a + b + c + d in float-float, in the same way
__device__ __forceinline__ ff ff_sum4(ff a, ff b, ff c, ff d) {
    const ff x = wcc::two_sum(a.hi, b.hi);
    const ff y = wcc::two_sum(x.hi, c.hi);
    const ff z = wcc::two_sum(y.hi, d.hi);
    return wcc::fast_two_sum(z.hi, ((a.lo + b.lo) + (c.lo + d.lo)) + ((x.lo + y.lo) + z.lo));
}
// (a + b) - (c + d) rounded to float
__device__ __forceinline__ float ff_diff2(ff a, ff b, ff c, ff d) {
    const ff x = wcc::two_sum(a.hi, b.hi);
    const ff y = wcc::two_sum(x.hi, -c.hi);
    const ff z = wcc::two_sum(y.hi, -d.hi);
    return z.hi + (((a.lo + b.lo) - (c.lo + d.lo)) + ((x.lo + y.lo) + z.lo));
}
// a - b rounded to float where the two are close (the high parts' difference
// is then exact; otherwise its rounding is the result's)
__device__ __forceinline__ float ff_close_diff(ff a, ff b) { return (a.hi - b.hi) + (a.lo - b.lo); }
// Float-float operations without the closing renormalisation, for results
// that only feed further float-float arithmetic ((hi, lo) with lo a few ulp
// of hi is as exact a representation; every operation here reads both parts).
__device__ __forceinline__ ff ff_add_u(ff a, ff b) {
    const ff s = wcc::two_sum(a.hi, b.hi);
    return ff{s.hi, s.lo + (a.lo + b.lo)};
}
__device__ __forceinline__ ff ff_add_u(ff a, float b) {
    const ff s = wcc::two_sum(a.hi, b);
    return ff{s.hi, s.lo + a.lo};
}
__device__ __forceinline__ ff ff_mul_u(ff a, ff b) {
    const ff p = wcc::two_prod(a.hi, b.hi);
    return ff{p.hi, fmaf(a.hi, b.lo, fmaf(a.lo, b.hi, p.lo))};
}
__device__ __forceinline__ ff ff_scale(ff a, float pow2) { return ff{a.hi * pow2, a.lo * pow2}; }
// a / b for a normal b: q1 = a.hi / b.hi, then the remainder a - b q1 (its
// leading part a.hi - b.hi q1 is exact, Sterbenz) divided by b.hi; one
// reciprocal estimate serves both quotients
__device__ __forceinline__ ff ffdiv_u(ff a, ff b) {
    const float rb = __fdividef(1.f, b.hi);
    const float q1 = a.hi * rb;
    const float p = b.hi * q1;
    const float e = fmaf(b.hi, q1, -p);
    const float rem = (a.hi - p) + (a.lo - fmaf(b.lo, q1, e));
    return ff{q1, rem * rb};
}

// f(u) and g(u) at a point value u given in float-float (the (0,0,0) entries
// of the flux tables, the leading terms of Eqs. SubEq:2DFluxFU ... GL).
template <int SYS>
__device__ __forceinline__ void lead_flux_ff(const ff (&u)[nvars(SYS)], const Law2D& law, ff (&F)[nvars(SYS)],
                                             ff (&G)[nvars(SYS)]) {
    // every result feeds float-float arithmetic again (the shares take
    // hx f, hy g as exact products): no renormalisation in between; the
    // constants (a_x, a_y, gamma - 1) enter as float-float pairs
    if constexpr (SYS == ADVECTION) {
        F[0] = ff_mul_u(u[0], ff{law.ax_f, law.ax_lo_f});
        G[0] = ff_mul_u(u[0], ff{law.ay_f, law.ay_lo_f});
    } else if constexpr (SYS == BURGERS) {
        F[0] = ff_scale(ff_mul_u(u[0], u[0]), 0.5f);
        G[0] = F[0];
    } else {
        const ff vx = ffdiv_u(u[1], u[0]), vy = ffdiv_u(u[2], u[0]);
        const ff mu = ff_mul_u(u[1], vx), mv = ff_mul_u(u[1], vy), nv = ff_mul_u(u[2], vy);
        const ff p = ff_mul_u(ff_add_u(u[3], ff_scale(ff_add_u(mu, nv), -0.5f)), ff{law.g1_f, law.g1_lo_f});
        const ff Ep = ff_add_u(u[3], p);
        F[0] = u[1];
        F[1] = ff_add_u(mu, p);
        F[2] = mv;
        F[3] = ff_mul_u(Ep, vx);
        G[0] = u[2];
        G[1] = mv;
        G[2] = ff_add_u(nv, p);
        G[3] = ff_mul_u(Ep, vy);
    }
}

// The new cell's linear part in the FP32-mixed form: the cell average as the
// float-float sum of the four parents' shares, the degree-1 derivatives from
// float-float differences of the vertex point values, the rest as
// linear_cell.  rd.cf(r, v), rd.v00(r, v) (float-float) and rd.V(r, v, q)
// (float, q >= 1) read parent r.
template <int SYS, int P, class Rd>
__device__ __forceinline__ void linear_cell_mx(const Rd& rd, float (&D)[nvars(SYS)][nq(P)], ff (&ubar)[nvars(SYS)]) {
    unroll<nvars(SYS)>([&](auto vc) {
        constexpr int v = vc;
        ubar[v] = ff_sum4(rd.cf(0, v), rd.cf(1, v), rd.cf(2, v), rd.cf(3, v));
        derivatives2d<P, 1, float>(
            [&](auto qc, float& dx, float& dy) {
                if constexpr (qc == 0) {
                    dx = ff_diff2(rd.v00(1, v), rd.v00(2, v), rd.v00(0, v), rd.v00(3, v));
                    dy = ff_diff2(rd.v00(3, v), rd.v00(2, v), rd.v00(0, v), rd.v00(1, v));
                } else {
                    const float A = rd.V(2, v, qc) - rd.V(0, v, qc), B = rd.V(1, v, qc) - rd.V(3, v, qc);
                    dx = A + B;
                    dy = A - B;
                }
            },
            D[v]);
    });
}

}  // namespace wcc2d

#undef WCC2D_TIMES
