// pf_bruss.cu -- stage kernels of the epoch for the 1D Brusselator (d = 64):
// 32 interior grid points xi_i = i/33, Dirichlet u = 1, v = 3 at both ends,
//   u_i' = A + u_i^2 v_i - (B+1) u_i + D (u_{i-1} - 2 u_i + u_{i+1}),
//   v_i' = B u_i - u_i^2 v_i + D (v_{i-1} - 2 v_i + v_{i+1}),  D = alpha 33^2,
// state interleaved (u_0, v_0, u_1, v_1, ...), theta = (A, B, alpha).
//
// A particle is 16 lanes, each holding two grid points in registers, so the
// history, the increments and the error sums never leave the register file
// (one thread a particle kept 4.6 KB of them in a work area, 22 GB of DRAM
// traffic a stage-2 launch at N = 65536, and left most of the chip idle below
// that size).  The substep is the increment form of pf_fast.cuh: of the K
// Newton iterations the last takes its residual in FP64, the one before in ff,
// the earlier ones in FP32, and the linear systems are solved in FP32:
// I - gamma J is block-tridiagonal with 2x2 diagonal blocks M_i and off-diagonal
// blocks -gamma D I; each lane eliminates its second point, which leaves 16
// block rows solved by parallel cyclic reduction (4 levels of shuffles), about
// 300 FP32 instructions and 80 shuffles a warp for two particles -- the time
// of 6 FP64 instructions.  The last correction is D's low floats, known, plus
// an FP32 solution for the rest; where that rest is not small enough for FP32
// to be exact beside the state, one step of refinement in ff follows.  A
// particle the floats do not serve repeats the substep in FP64 on the same
// lanes.  Measured (GB300, S = 20, stage 1 + stage 2): N = 1000 7.3 -> 0.21 ms,
// N = 16384 8.57 -> 1.45 ms, N = 65536 23.4 -> 5.5 ms; the FP64 pipe is 60 %
// busy, three warps a sub-partition (168 registers) waiting on each other's
// results the rest (the launch bound keeps the three: at 177 registers stage 2 of N =
// 16384 took 0.97 ms, at 168 0.79); 128 registers (four warps, spills) and 64-thread blocks
// changed the epochs by less than 4 %.
#include "pf_epoch.cuh"
#include "pf_fast.cuh"
#include "pf_kernels.h"

namespace pfg {

constexpr int kBrLanes = 16;  // lanes a particle, two grid points each
constexpr int kBrThreads = 128;
constexpr int kBrPerBlock = kBrThreads / kBrLanes;

struct BrTheta {
  double A, B, D;
};

__device__ __forceinline__ BrTheta br_theta(const double* th) {
  return BrTheta{th[0], th[1], th[2] * 33.0 * 33.0};
}

// the same value s lanes lower or higher in the particle's 16 lanes (its own
// at the ends)
__device__ __forceinline__ float from_left(float v, int s) { return __shfl_up_sync(0xffffffffu, v, s, kBrLanes); }
__device__ __forceinline__ float from_right(float v, int s) { return __shfl_down_sync(0xffffffffu, v, s, kBrLanes); }
__device__ __forceinline__ double from_left(double v, int s) { return __shfl_up_sync(0xffffffffu, v, s, kBrLanes); }
__device__ __forceinline__ double from_right(double v, int s) { return __shfl_down_sync(0xffffffffu, v, s, kBrLanes); }
__device__ __forceinline__ ff from_left(ff v, int s) { return ff{from_left(v.h, s), from_left(v.l, s)}; }
__device__ __forceinline__ ff from_right(ff v, int s) { return ff{from_right(v.h, s), from_right(v.l, s)}; }

// Left and right neighbours of the lane's two points, z = (u0, v0, u1, v1);
// eu, ev are the boundary's values.
template <class T>
__device__ __forceinline__ void br_neighbours(const T (&z)[4], int g, T eu, T ev, T (&L)[4], T (&R)[4]) {
  const T lu = from_left(z[2], 1), lv = from_left(z[3], 1);
  const T ru = from_right(z[0], 1), rv = from_right(z[1], 1);
  L[0] = g == 0 ? eu : lu;
  L[1] = g == 0 ? ev : lv;
  L[2] = z[0];
  L[3] = z[1];
  R[0] = z[2];
  R[1] = z[3];
  R[2] = g == kBrLanes - 1 ? eu : ru;
  R[3] = g == kBrLanes - 1 ? ev : rv;
}

// ------------------------------------------------------- the linear systems
template <class T>
struct Mat2 {
  T a, b, c, d;
};
__device__ __forceinline__ float br_mul(float x, float y) { return __fmul_rn(x, y); }
__device__ __forceinline__ double br_mul(double x, double y) { return __dmul_rn(x, y); }
__device__ __forceinline__ float br_fma(float x, float y, float z) { return __fmaf_rn(x, y, z); }
__device__ __forceinline__ double br_fma(double x, double y, double z) { return __fma_rn(x, y, z); }
__device__ __forceinline__ float br_rcp(float x) { return f_rcp(x); }
__device__ __forceinline__ double br_rcp(double x) { return 1.0 / x; }

template <class T>
__device__ __forceinline__ Mat2<T> inverse(const Mat2<T>& m) {
  const T r = br_rcp(br_fma(m.a, m.d, -br_mul(m.b, m.c)));
  return Mat2<T>{br_mul(m.d, r), -br_mul(m.b, r), -br_mul(m.c, r), br_mul(m.a, r)};
}
template <class T>
__device__ __forceinline__ Mat2<T> product(const Mat2<T>& x, const Mat2<T>& y) {
  return Mat2<T>{br_fma(x.a, y.a, br_mul(x.b, y.c)), br_fma(x.a, y.b, br_mul(x.b, y.d)),
                 br_fma(x.c, y.a, br_mul(x.d, y.c)), br_fma(x.c, y.b, br_mul(x.d, y.d))};
}
// z - x y
template <class T>
__device__ __forceinline__ Mat2<T> minus_product(const Mat2<T>& z, const Mat2<T>& x, const Mat2<T>& y) {
  return Mat2<T>{br_fma(-x.a, y.a, br_fma(-x.b, y.c, z.a)), br_fma(-x.a, y.b, br_fma(-x.b, y.d, z.b)),
                 br_fma(-x.c, y.a, br_fma(-x.d, y.c, z.c)), br_fma(-x.c, y.b, br_fma(-x.d, y.d, z.d))};
}
template <class T>
__device__ __forceinline__ Mat2<T> scaled(const Mat2<T>& x, T s) {
  return Mat2<T>{br_mul(x.a, s), br_mul(x.b, s), br_mul(x.c, s), br_mul(x.d, s)};
}
template <class T>
__device__ __forceinline__ Mat2<T> left_of(const Mat2<T>& m, int s) {
  return Mat2<T>{from_left(m.a, s), from_left(m.b, s), from_left(m.c, s), from_left(m.d, s)};
}
template <class T>
__device__ __forceinline__ Mat2<T> right_of(const Mat2<T>& m, int s) {
  return Mat2<T>{from_right(m.a, s), from_right(m.b, s), from_right(m.c, s), from_right(m.d, s)};
}

// M_i x_i - e x_{i-1} - e x_{i+1} = b_i for the lane's points i = 2g, 2g + 1.
// The second point is eliminated, x_B = N (b_B + e (x_A + x_A+)) with N = M_B^{-1}
// and A+ the next lane's first point; the 16 rows left are brought to
//   x_A + P x_{A-s} + Q x_{A+s} = r
// and the stride s is doubled until no neighbour is left (parallel cyclic
// reduction; P is zero in the first s lanes and Q in the last, so what the
// shuffles return at the ends is multiplied by zero).
template <class T>
__device__ __forceinline__ void br_solve(const Mat2<T> (&M)[2], T e, int g, const T (&b)[4], T (&x)[4]) {
  const Mat2<T> N = inverse(M[1]);
  const T nu = br_fma(N.a, b[2], br_mul(N.b, b[3])), nv = br_fma(N.c, b[2], br_mul(N.d, b[3]));
  Mat2<T> W = left_of(N, 1);
  T wu = from_left(nu, 1), wv = from_left(nv, 1);
  if (g == 0) {
    W = Mat2<T>{0, 0, 0, 0};
    wu = wv = 0;
  }
  const T e2 = br_mul(e, e), me2 = -e2;
  Mat2<T> I = inverse(Mat2<T>{br_fma(me2, W.a + N.a, M[0].a), br_fma(me2, W.b + N.b, M[0].b),
                              br_fma(me2, W.c + N.c, M[0].c), br_fma(me2, W.d + N.d, M[0].d)});
  const T bu = br_fma(e, wu + nu, b[0]), bv = br_fma(e, wv + nv, b[1]);
  T r0 = br_fma(I.a, bu, br_mul(I.b, bv)), r1 = br_fma(I.c, bu, br_mul(I.d, bv));
  I = scaled(I, me2);
  Mat2<T> P = product(I, W), Q = product(I, N);
  if (g == kBrLanes - 1) Q = Mat2<T>{0, 0, 0, 0};
#pragma unroll
  for (int s = 1; s < kBrLanes; s *= 2) {
    const Mat2<T> Ql = left_of(Q, s), Pr = right_of(P, s);
    const T l0 = from_left(r0, s), l1 = from_left(r1, s), q0 = from_right(r0, s), q1 = from_right(r1, s);
    const Mat2<T> one{1, 0, 0, 1};
    const Mat2<T> SI = inverse(minus_product(minus_product(one, P, Ql), Q, Pr));
    const T t0 = br_fma(-P.a, l0, br_fma(-P.b, l1, br_fma(-Q.a, q0, br_fma(-Q.b, q1, r0))));
    const T t1 = br_fma(-P.c, l0, br_fma(-P.d, l1, br_fma(-Q.c, q0, br_fma(-Q.d, q1, r1))));
    r0 = br_fma(SI.a, t0, br_mul(SI.b, t1));
    r1 = br_fma(SI.c, t0, br_mul(SI.d, t1));
    if (2 * s < kBrLanes) {
      const Mat2<T> Pl = left_of(P, s), Qr = right_of(Q, s);
      const Mat2<T> mSI = scaled(SI, T(-1));
      P = product(mSI, product(P, Pl));
      Q = product(mSI, product(Q, Qr));
    }
  }
  x[0] = r0;
  x[1] = r1;
  T p0 = from_right(r0, 1), p1 = from_right(r1, 1);
  if (g == kBrLanes - 1) p0 = p1 = 0;
  const T s0 = br_mul(e, r0 + p0), s1 = br_mul(e, r1 + p1);
  x[2] = br_fma(N.a, s0, br_fma(N.b, s1, nu));
  x[3] = br_fma(N.c, s0, br_fma(N.d, s1, nv));
}

// --------------------------------------------------- right side and Jacobian
// f at y in FP64, two points a lane.
__device__ __forceinline__ void br_f(const BrTheta& T, const double (&y)[4], int g, double (&f)[4]) {
  double L[4], R[4];
  br_neighbours(y, g, 1.0, 3.0, L, R);
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const double u = y[k], v = y[k + 1], uuv = (u * u) * v;
    f[k] = fma(T.D, fma(-2.0, u, L[k] + R[k]), fma(-(T.B + 1.0), u, T.A + uuv));
    f[k + 1] = fma(T.D, fma(-2.0, v, L[k + 1] + R[k + 1]), fma(T.B, u, -uuv));
  }
}

// One substep's constants, the parameters in ff.
struct BrPar {
  ff A, B, B1, D;  // A, B, B + 1, D
};
template <class T>
struct BrDiag {
  T g, g2, gB, gD, ca, cd;  // gamma, 2 gamma, gamma B, gamma D, 1 + gamma (B+1) + 2 gamma D, 1 + 2 gamma D
};
template <class T>
__device__ __forceinline__ BrDiag<T> br_diag(T g, T B, T D) {
  const T gD = br_mul(g, D), gB = br_mul(g, B);
  const T cd = br_fma(T(2), gD, T(1));
  return BrDiag<T>{g, g + g, gB, gD, (cd + g) + gB, cd};
}
// the diagonal blocks I - gamma J at (u, v)
template <class T>
__device__ __forceinline__ Mat2<T> br_block(const BrDiag<T>& c, T u, T v) {
  const T uv = br_mul(u, v), uu = br_mul(u, u);
  return Mat2<T>{br_fma(-c.g2, uv, c.ca), -br_mul(c.g, uu), br_fma(c.g2, uv, -c.gB), br_fma(c.g, uu, c.cd)};
}

// G = D + R - gamma f(x + D) and the blocks of I - gamma J, in FP32
__device__ __forceinline__ void br_residual32(const BrPar& T, const BrDiag<float>& c, const ff (&x)[4],
                                              const ff (&Rv)[4], const ff (&Dv)[4], int g, float (&mG)[4],
                                              Mat2<float> (&M)[2]) {
  float y[4], L[4], R[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) y[k] = f_add(x[k].h, Dv[k].h);
  br_neighbours(y, g, 1.0f, 3.0f, L, R);
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const float u = y[k], v = y[k + 1], uuv = f_mul(f_mul(u, u), v);
    const float lu = f_add(f_sub(L[k], u), f_sub(R[k], u)), lv = f_add(f_sub(L[k + 1], v), f_sub(R[k + 1], v));
    const float fu = f_fma(T.D.h, lu, f_fma(-T.B1.h, u, f_add(T.A.h, uuv)));
    const float fv = f_fma(T.D.h, lv, f_fma(T.B.h, u, -uuv));
    mG[k] = f_fma(c.g, fu, -f_add(Dv[k].h, Rv[k].h));
    mG[k + 1] = f_fma(c.g, fv, -f_add(Dv[k + 1].h, Rv[k + 1].h));
    M[k / 2] = br_block(c, u, v);
  }
}

// the same with G in ff, sums not renormalised
__device__ __forceinline__ void br_residual_ff(const BrPar& T, const BrDiag<float>& c, ff gf, const ff (&x)[4],
                                               const ff (&Rv)[4], const ff (&Dv)[4], int g, float (&mG)[4],
                                               Mat2<float> (&M)[2]) {
  ff y[4], L[4], R[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) y[k] = ff_add_raw(x[k], Dv[k]);
  br_neighbours(y, g, ff{1.0f, 0.0f}, ff{3.0f, 0.0f}, L, R);
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const ff u = y[k], v = y[k + 1], uuv = ff_mul_raw(ff_mul_raw(u, u), v);
    const ff lu = ff_sub_raw(ff_add_raw(L[k], R[k]), ff_twice(u)), lv = ff_sub_raw(ff_add_raw(L[k + 1], R[k + 1]), ff_twice(v));
    const ff fu = ff_add_raw(ff_mul_raw(T.D, lu), ff_sub_raw(ff_add_raw(T.A, uuv), ff_mul_raw(T.B1, u)));
    const ff fv = ff_add_raw(ff_mul_raw(T.D, lv), ff_sub_raw(ff_mul_raw(T.B, u), uuv));
    const ff mu = ff_sub_raw(ff_mul_raw(gf, fu), ff_add_raw(Dv[k], Rv[k]));
    const ff mv = ff_sub_raw(ff_mul_raw(gf, fv), ff_add_raw(Dv[k + 1], Rv[k + 1]));
    mG[k] = f_add(mu.h, mu.l);
    mG[k + 1] = f_add(mv.h, mv.l);
    M[k / 2] = br_block(c, u.h, v.h);
  }
}

// G + (I - gamma J(y)) d in ff, for the refinement of d
__device__ __forceinline__ void br_defect(const BrPar& T, ff gf, const double (&yd)[4], const ff (&G)[4],
                                       const ff (&d)[4], int g, float (&mG)[4]) {
  ff L[4], R[4];
  br_neighbours(d, g, ff{0.0f, 0.0f}, ff{0.0f, 0.0f}, L, R);
#pragma unroll
  for (int k = 0; k < 4; k += 2) {
    const ff u = ff_from(yd[k]), v = ff_from(yd[k + 1]);
    // J d by columns: reaction 2uv du + u^2 dv, then the linear terms
    const ff rx = ff_add(ff_twice(ff_mul(ff_mul(u, v), d[k])), ff_mul(ff_mul(u, u), d[k + 1]));
    const ff lu = ff_sub(ff_add(L[k], R[k]), ff_twice(d[k]));
    const ff lv = ff_sub(ff_add(L[k + 1], R[k + 1]), ff_twice(d[k + 1]));
    const ff ju = ff_fma(T.D, lu, ff_sub(rx, ff_mul(T.B1, d[k])));
    const ff jv = ff_fma(T.D, lv, ff_sub(ff_mul(T.B, d[k]), rx));
    mG[k] = ff_sub(ff_mul(gf, ju), ff_add(G[k], d[k])).h;
    mG[k + 1] = ff_sub(ff_mul(gf, jv), ff_add(G[k + 1], d[k + 1])).h;
  }
}

// ------------------------------------------------------------- one interval
// What a lane carries: x_n with float carries, a = x_n - x_{n-1} (and its carry)
// in double and in ff, b = x_{n-1} - x_{n-2} in ff, the error sums at 2^80.
struct BrCarry {
  double x[4], a[4];
  float cx[4], ca[4];
  ff fa[4], fb[4], E[4];
};

// What substeps in FP64 add in doubles, for values beyond the floats: their part of the
// error sums and, while `b64` says so, b.  In shared memory, a column a thread:
// registers are short, and few particles use it.
struct BrWide {
  double E[4][kBrThreads], b[4][kBrThreads];
};

// One substep in FP64, on all lanes of the warp: K Newton iterations in
// increments from the same start.
template <bool ERR>
__device__ __noinline__ void br_step_fp64(const BrTheta& T, const StepCoef& c, int K, int g, BrCarry& w, BrWide* wide,
                                          bool b64, bool mine) {
  double D0[4], P[4], R[4], xn[4], h1[4];
  double f[4];
  // (a correction of 2^-13 of the state leaves a carry of 2^-38)
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    w.x[k] += (double)w.cx[k];
    w.a[k] += (double)w.ca[k];
  }
  br_f(T, w.x, g, f);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    xn[k] = w.x[k];
    h1[k] = w.x[k] - w.a[k];
    const double h2 = h1[k] - (b64 ? wide->b[k][threadIdx.x] : (double)w.fb[k].h + (double)w.fb[k].l);
    // the start and the error predictor as increments
    D0[k] = c.kind == 2 ? fma(c.pi2, h2, fma(c.pi1, h1[k], c.pi0 * xn[k])) - xn[k] : 0.0;
    P[k] = c.kind == 2 ? D0[k] : c.h * f[k];
    R[k] = xn[k] - fma(c.rho2, h1[k], c.rho1 * xn[k]);
  }
  const BrDiag<double> q = br_diag(c.gamma, T.B, T.D);
  for (int it = 0; it < K; ++it) {
    double y[4], mG[4], d[4];
    Mat2<double> M[2];
#pragma unroll
    for (int k = 0; k < 4; ++k) y[k] = xn[k] + D0[k];
    br_f(T, y, g, f);
#pragma unroll
    for (int k = 0; k < 4; ++k) mG[k] = fma(c.gamma, f[k], -(D0[k] + R[k]));
    M[0] = br_block(q, y[0], y[1]);
    M[1] = br_block(q, y[2], y[3]);
    br_solve(M, q.gD, g, mG, d);
#pragma unroll
    for (int k = 0; k < 4; ++k) D0[k] += d[k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double xk = xn[k] + D0[k];
    if (mine) {
      wide->b[k][threadIdx.x] = w.a[k];
      const double e = c.mu * (D0[k] - P[k]);
      if (ERR) wide->E[k][threadIdx.x] = fma(e, e, wide->E[k][threadIdx.x]);
    }
    w.a[k] = xk - xn[k];
    w.fb[k] = w.fa[k];
    w.fa[k] = ff_from(w.a[k]);
    w.x[k] = xk;
    w.cx[k] = w.ca[k] = 0.0f;
  }
}

// One substep in increments.  A particle whose values do not allow it (far:
// from the start) is left as it was; returns the lanes of such particles.
template <bool ERR>
__device__ __forceinline__ unsigned br_step(const BrTheta& T, const BrPar& par, const FastCoef& c, int kind, double h,
                                            int K, int g, bool far, BrCarry& w) {
  const BrDiag<float> q = br_diag(c.g.h, par.B.h, par.D.h);
  ff P[4], Dv[4], xf[4], Rf[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    xf[k] = ff_from(w.x[k]);
    xf[k].l = f_add(xf[k].l, w.cx[k]);
    ff p = ff_fma(c.pb, w.fb[k], ff_mul_raw(c.pa, w.fa[k]));
    p.l = f_fma(c.ep, xf[k].h, p.l);
    P[k] = Dv[k] = p;
    Rf[k] = ff_mul(c.fra, w.fa[k]);
  }
  for (int it = 0; it + 1 < K; ++it) {
    float mG[4], d[4];
    Mat2<float> M[2];
    if (it + 2 < K) br_residual32(par, q, xf, Rf, Dv, g, mG, M);
    else br_residual_ff(par, q, c.g, xf, Rf, Dv, g, mG, M);
    br_solve(M, q.gD, g, mG, d);
#pragma unroll
    for (int k = 0; k < 4; ++k) Dv[k] = ff_add(Dv[k], d[k]);
  }
  double y[4], f[4];
  ff G[4], dl[4];
  float lo[4], yf[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    y[k] = w.x[k] + d_from_f(Dv[k].h);
    lo[k] = Dv[k].l;
    yf[k] = f_from(y[k]);
  }
  br_f(T, y, g, f);
  Mat2<float> M[2] = {br_block(q, yf[0], yf[1]), br_block(q, yf[2], yf[3])};
  float L[4], R[4], mG[4], d[4];
  br_neighbours(lo, g, 0.0f, 0.0f, L, R);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float cor = f_fma(-c.er, xf[k].h, f_fma(c.fra.h, w.ca[k], -w.cx[k]));
    G[k] = ff_add(ff_from(fma(-c.gamma, f[k], fma(c.ra, w.a[k], d_from_f(Dv[k].h)))), cor);
    // G + (I - gamma J) lo: what the low floats leave to correct
    const Mat2<float>& m = M[k / 2];
    const float ml = (k & 1) ? f_fma(m.c, lo[k - 1], f_mul(m.d, lo[k])) : f_fma(m.a, lo[k], f_mul(m.b, lo[k + 1]));
    mG[k] = -ff_add(G[k], f_fma(-q.gD, f_add(L[k], R[k]), ml)).h;
  }
  br_solve(M, q.gD, g, mG, d);
  float md = 0.0f, my = 0.0f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    md = f_add(md, fabsf(d[k]));
    my = f_add(my, fabsf(yf[k]));
    dl[k] = two_sum(lo[k], d[k]);
  }
  // FP32 solutions are good to about 2^-20: beside y that is exact for a
  // correction of 2^-34 |y|, else the defect is solved for once more (by the warp, for
  // those of its two particles that need it: a particle's result is its own)
  const unsigned group = (threadIdx.x & 16u) ? 0xffff0000u : 0x0000ffffu;
  const unsigned refine = __ballot_sync(0xffffffffu, !(md <= 0x1.0p-34f * my));
  if (refine) {
    br_defect(par, c.g, y, G, dl, g, mG);
    br_solve(M, q.gD, g, mG, d);
    if (refine & group) {
#pragma unroll
      for (int k = 0; k < 4; ++k) dl[k] = ff_add(dl[k], d[k]);
    }
  }
  if (ERR && kind != 2) {
    // a cold start's error predictor is the explicit-Euler step
    br_f(T, w.x, g, f);
#pragma unroll
    for (int k = 0; k < 4; ++k) P[k] = ff_from(h * f[k]);
  }
  // finite, and the iterations settled (a single one: 2^-40 of it, after two FP32 solves,
  // below the last bit)
  bool ok = !far && md <= (K > 1 ? 0x1.0p-20f : 0x1.0p-13f) * my && my < 0x1.0p60f;
  if (ERR) {
    // and squares of the scaled estimates whose sum stays a float (640 of 2^116)
    float me = md;
#pragma unroll
    for (int k = 0; k < 4; ++k) me = f_add(me, f_add(fabsf(P[k].h), fabsf(Dv[k].h)));
    ok = ok && f_mul(fabsf(c.mus.h), me) < 0x1.0p58f;
  }
  const unsigned bad = __ballot_sync(0xffffffffu, !ok);
  if (bad & group) return bad;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double xn = y[k] + d_from_f(dl[k].h);
    const ff Dn = ff_add(ff_add(dl[k], Dv[k].h), -w.cx[k]);
    if (ERR) {
      const ff e = ff_mul(c.mus, ff_sub(Dn, P[k]));
      w.E[k] = ff_fma(e, e, w.E[k]);
    }
    w.fb[k] = w.fa[k];
    w.fa[k] = Dn;
    w.a[k] = xn - w.x[k];
    w.ca[k] = f_sub(dl[k].l, w.cx[k]);
    w.x[k] = xn;
    w.cx[k] = dl[k].l;
  }
  return bad;
}

// Psi over the S substeps for the warp's two particles; returns whether wide->b holds b.
template <bool ERR>
__device__ __forceinline__ bool br_propagate(const StepCoef* sc, const FastCoef* fc, int S, int K, const BrTheta& T,
                                             int g, BrCarry& w, BrWide* wide) {
  const BrPar par{ff_from(T.A), ff_from(T.B), ff_from(T.B + 1.0), ff_from(T.D)};
  const unsigned group = (threadIdx.x & 16u) ? 0xffff0000u : 0x0000ffffu;
  // the range in which the floats serve
  double big = 0.0;
#pragma unroll
  for (int k = 0; k < 4; ++k) big = fmax(big, fabs(w.x[k]));
  const double tb = fmax(fmax(fabs(T.A), fabs(T.B)), fabs(T.D));
  // (a particle with a component that is not far below the floats' 1)
  float top = f_from(big);
#pragma unroll
  for (int o = 1; o < kBrLanes; o *= 2) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
  const bool far = !(big <= kFastStateMax && tb <= kFastThetaMax && top >= (float)kFastStateMin);
  bool b64 = true;
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
    const FastCoef& c = fc[s];
    const bool step_far = far || !(c.g.h >= kFastStepMin && c.g.h <= kFastStepMax);
    const unsigned bad = br_step<ERR>(T, par, c, sc[s].kind, sc[s].h, K, g, step_far, w);
    if (bad) {
      // on a copy, so that the carry itself stays in registers
      BrCarry t = w;
      br_step_fp64<ERR>(T, sc[s], K, g, t, wide, b64, (bad & group) != 0);
      if (bad & group) w = t;
    }
    b64 = (bad & group) != 0;
  }
  return b64;
}

// The lane's four components of a particle's history from SoA rows.
__device__ __forceinline__ void br_load(const Ensemble& E, int64_t N, int64_t l, int g, BrCarry& w, BrWide* wide) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int64_t o = (int64_t)(4 * g + k) * N + l;
    const double x = E.x[o], h1 = E.h1[o], h2 = E.h2[o];
    w.x[k] = x;
    w.a[k] = x - h1;
    w.fa[k] = ff_from(w.a[k]);
    const double b = h1 - h2;
    w.fb[k] = ff_from(b);
    wide->b[k][threadIdx.x] = b;
    wide->E[k][threadIdx.x] = 0.0;
    w.cx[k] = w.ca[k] = 0.0f;
    w.E[k] = ff{0.0f, 0.0f};
  }
}

// Gaussian log-likelihood from the lanes' components, every lane adding the
// observations in their order.
__device__ __forceinline__ double br_loglik(const FilterDev& fd, const EpochParams* __restrict__ ep,
                                            const double (&x)[4]) {
  double s = 0.0;
  for (int i = 0; i < fd.m; ++i) {
    const int o = fd.obs[i], k = o & 3;
    const double mine = k == 0 ? x[0] : k == 1 ? x[1] : k == 2 ? x[2] : x[3];
    const double z = (ep->y[i] - __shfl_sync(0xffffffffu, mine, o >> 2, kBrLanes)) * ep->inv_sigma[i];
    s = fma(z, z, s);
  }
  return -0.5 * s;
}

// Step tables of a block in its dynamic shared memory; ends with a barrier.
__device__ __forceinline__ const FastCoef* br_tables(StepCoef* s_sc, const EpochParams* __restrict__ ep, int S) {
  load_steps(s_sc, ep, S);
  FastCoef* t = reinterpret_cast<FastCoef*>(s_sc + S);
  for (int i = threadIdx.x; i < S; i += blockDim.x) t[i] = fast_coef(s_sc[i]);
  __syncthreads();
  return t;
}

__device__ __forceinline__ void bstage1_body(const FilterDev& fd, const EpochParams* __restrict__ ep,
                                             int vb, int vg, const StepCoef* s_sc, const FastCoef* s_fc,
                                             BrWide* wide, double* s_red, int* s_flag) {
  const Ctrl* ctrl = fd.ctrl;
  const Ensemble src = committed(fd, ctrl->cur);
  const int64_t N = fd.N;
  const int g = threadIdx.x & (kBrLanes - 1);
  const int64_t slot = (int64_t)vb * kBrPerBlock + threadIdx.x / kBrLanes;
  const int64_t n = slot < N ? slot : N - 1;  // idle lanes repeat the last particle and write nothing
  double ph[3], th[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) ph[i] = fd.a * src.phi[i * N + n] + (1.0 - fd.a) * ctrl->phibar[i];
  to_theta<3>(fd, ph, th);
  BrCarry w;
  br_load(src, N, n, g, w, wide);
  br_propagate<false>(s_sc, s_fc, ep->S, fd.K, br_theta(th), g, w, wide);
  double x[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) x[k] = w.x[k] + (double)w.cx[k];
  const double ll = br_loglik(fd, ep, x);
  double lg = -CUDART_INF;
  if (g == 0 && slot < N) {
    fd.ll1[n] = ll;
    lg = (src.lw[n] - ctrl->logW) + ll;
    if (!finite_bits(lg)) lg = -CUDART_INF;
    fd.lg[n] = lg;
  }
  stage1_tail(fd, ep->epoch, lg, vb, vg, s_red, s_flag);
}

__device__ __forceinline__ void bstage2_body(const FilterDev& fd, const EpochParams* __restrict__ ep,
                                             int vb, int vg, const StepCoef* s_sc, const FastCoef* s_fc,
                                             BrWide* wide, double* s_red, int* s_flag) {
  const Ctrl* ctrl = fd.ctrl;
  const int cur = ctrl->cur;
  const Ensemble src = committed(fd, cur);
  const Ensemble dst = pending(fd, cur);
  const int64_t N = fd.N;
  const uint32_t epoch = ep->epoch;
  const int g = threadIdx.x & (kBrLanes - 1);
  const int64_t slot = (int64_t)vb * kBrPerBlock + threadIdx.x / kBrLanes;
  const bool live = slot < N;
  const int64_t n = live ? slot : N - 1;
  const int64_t l = fd.idx[n];
  // 4a: proliferate phi
  double z[4];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const U4 r = draw_block(fd, kRngTheta, (uint32_t)n, epoch, (uint32_t)b);
    normal_pair(r, z[2 * b], z[2 * b + 1]);
  }
  double ph[3], th[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    double lz = 0.0;
#pragma unroll
    for (int k = 0; k <= i; ++k) lz = fma(ctrl->L[i * kPMax + k], z[k], lz);
    const double shr = fd.a * src.phi[i * N + l] + (1.0 - fd.a) * ctrl->phibar[i];
    ph[i] = fma(fd.s, lz, shr);
    if (live && g == i) dst.phi[i * N + n] = ph[i];
  }
  to_theta<3>(fd, ph, th);
  BrCarry w;
  br_load(src, N, l, g, w, wide);
  // 4b, 4d: repropagate with the Milne error sums
  const bool b64 = br_propagate<true>(s_sc, s_fc, ep->S, fd.K, br_theta(th), g, w, wide);
  // 4c, 4d: innovation
  double x[4];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    const U4 r = draw_block(fd, kRngInnov, (uint32_t)n, epoch, (uint32_t)(2 * g + b));
    double z0, z1;
    normal_pair(r, z0, z1);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = 2 * b + h;
      const int64_t o = (int64_t)(4 * g + k) * N + n;
      const double E = fma((double)w.E[k].h + (double)w.E[k].l, kErrUnscale, wide->E[k][threadIdx.x]);
      const double v = pfm::sqrt_fixed(fd.kappa * E) * (h == 0 ? z0 : z1);
      const double xk = w.x[k] + (double)w.cx[k];
      const double h1 = xk - (w.a[k] + (double)w.ca[k]);
      const double h2 = h1 - (b64 ? wide->b[k][threadIdx.x] : (double)w.fb[k].h + (double)w.fb[k].l);
      x[k] = xk + v;
      if (live) {
        dst.x[o] = x[k];
        dst.h1[o] = h1 + v;
        dst.h2[o] = h2 + v;
      }
    }
  }
  // 5: new log weight
  double lwn = br_loglik(fd, ep, x) - fd.ll1[l];
  bool bad = false;
  if (!finite_bits(lwn)) {
    lwn = -CUDART_INF;
    bad = true;
  }
  if (live && g == 0) {
    dst.lw[n] = lwn;
  } else {
    lwn = -CUDART_INF;
    bad = false;
  }
  stage2_tail(fd, epoch, lwn, bad, vb, vg, s_red, s_flag);
}

template <int STAGE>
__global__ void __launch_bounds__(kBrThreads, 3) k_bstage(const __grid_constant__ FilterDev fd,
                                                     const EpochParams* __restrict__ ep) {
  extern __shared__ double s_dyn[];
  __shared__ double s_red[32];
  __shared__ BrWide s_wide;
  __shared__ int s_flag;
  if (fd.ctrl->status != PF_OK) return;
  StepCoef* s_sc = reinterpret_cast<StepCoef*>(s_dyn);
  const FastCoef* s_fc = br_tables(s_sc, ep, ep->S);
  if (STAGE == 1) bstage1_body(fd, ep, blockIdx.x, gridDim.x, s_sc, s_fc, &s_wide, s_red, &s_flag);
  else bstage2_body(fd, ep, blockIdx.x, gridDim.x, s_sc, s_fc, &s_wide, s_red, &s_flag);
}

template <int STAGE>
__global__ void __launch_bounds__(kBrThreads, 3) k_batch_bstage(const FilterDev* __restrict__ fds,
                                                           const EpochParams* const* __restrict__ eps,
                                                           const BatchTile* __restrict__ tiles) {
  extern __shared__ double s_dyn[];
  __shared__ double s_red[32];
  __shared__ BrWide s_wide;
  __shared__ int s_flag;
  const BatchTile t = tiles[blockIdx.x];
  const FilterDev& fd = *(fds + t.f);
  if (fd.ctrl->status != PF_OK) return;
  const EpochParams* ep = eps[t.f];
  StepCoef* s_sc = reinterpret_cast<StepCoef*>(s_dyn);
  const FastCoef* s_fc = br_tables(s_sc, ep, ep->S);
  const int vg = (int)((fd.N + kBrPerBlock - 1) / kBrPerBlock);
  if (STAGE == 1) bstage1_body(fd, ep, t.vb, vg, s_sc, s_fc, &s_wide, s_red, &s_flag);
  else bstage2_body(fd, ep, t.vb, vg, s_sc, s_fc, &s_wide, s_red, &s_flag);
}

int bruss_stage_blocks(int64_t N) { return (int)((N + kBrPerBlock - 1) / kBrPerBlock); }

cudaError_t launch_bruss_stage(int stage, const FilterDev& fd, const EpochParams* ep, int S,
                               cudaStream_t st) {
  const size_t smem = step_table_bytes(PF_ODE_BRUSSELATOR1D, fd.lmm, S);
  const unsigned grid = (unsigned)bruss_stage_blocks(fd.N);
  if (stage == 1) k_bstage<1><<<grid, kBrThreads, smem, st>>>(fd, ep);
  else k_bstage<2><<<grid, kBrThreads, smem, st>>>(fd, ep);
  return cudaGetLastError();
}

cudaError_t launch_batch_bruss_stage(int stage, const FilterDev* fds, const EpochParams* const* eps,
                                     const BatchTile* tiles, int ntiles, size_t smem,
                                     cudaStream_t st) {
  if (ntiles <= 0) return cudaSuccess;
  if (stage == 1) k_batch_bstage<1><<<ntiles, kBrThreads, smem, st>>>(fds, eps, tiles);
  else k_batch_bstage<2><<<ntiles, kBrThreads, smem, st>>>(fds, eps, tiles);
  return cudaGetLastError();
}

cudaError_t preload_bruss_kernels() {
  const void* ks[] = {(const void*)k_bstage<1>, (const void*)k_bstage<2>,
                      (const void*)k_batch_bstage<1>, (const void*)k_batch_bstage<2>};
  for (const void* k : ks) {
    const cudaError_t e = allow_step_table(k);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pfg
