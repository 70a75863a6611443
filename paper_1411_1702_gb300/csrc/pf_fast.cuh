// pf_fast.cuh -- the implicit substeps of the small problems with the FP64
// work cut to what FP64 is needed for.
//
// GB300 issues two FP64 lanes a clock per SM against 128 FP32 ones, and the
// propagation kernels were bound by FP64 issue (90 % of the pipe's cycles).  A
// substep is written here in increments: with y = x_n + D the LMM's equation
//   G(D) = D + R - gamma f(x_n + D) = 0
// has R = r-terms of the differences x_n - x_{n-1}, x_{n-1} - x_{n-2} (BDF) or of
// the stored derivatives (Adams-Moulton), all small beside x_n, and the
// predictor's increment P likewise.  Of the K Newton iterations
//   - the first K - 1 solve their linear system in FP32: as with the unrefined
//     reciprocals of the FP64 path, an inexact correction is repaired by the next
//     iteration's residual.  The one before the last takes its residual in ff
//     (pf_ff.cuh, sums not renormalised), those before it in FP32.  (The Adams methods
//     evaluate and solve in ff up to there: their explicit predictors are far off on
//     stiff particles, where an inexact first step would be seen in the K-th.)
//   - the last evaluates G in FP64 at the point y = x_n + (leading float of D).
//     Its correction is D's low float, known, plus a rest of about 2^-50 |y| that an
//     FP32 solution serves; what FP32 made of the point does not matter, since G
//     is evaluated at the point itself.  (A larger rest, kFastRest below, solves in ff.)
// The state stays the double of the last iteration's point plus that iteration's
// correction in ff, so a substep rounds it once, and Milne's estimate comes from
// D - P without the cancellation of y - x_p.  The result is the K-th Newton
// iterate to FP64 rounding, as before; a substep that does not satisfy this
// reasoning (a non-finite value, iterations that have not settled, an
// exponent outside the floats') is left to the FP64 path by fast_run's caller.
//
// A Robertson BDF2 substep with error sums takes 15 FP64 instructions instead
// of 89, an M1 one 16 instead of 186.  Measured (GB300, device time):
// Robertson, N = 131072, S = 50: stage 1 0.93 -> 0.237 ms, stage 2 1.08 -> 0.300 ms;
// M1 BDF2, N = 50000, S = 10: 0.16 -> 0.062 and 0.23 -> 0.076 ms (the exponentials and
// roots of pf_math.cuh and the register bounds included).  Accuracy over an interval,
// against quadruple precision on 200 particles of the prior, 2-norm of the state:
// Robertson 3e-17 (plain FP64 9e-16), M1 6e-17 (4e-16); by component at kFastRest.
#pragma once
#include "pf_ff.cuh"

namespace pfg {

// Error sums are kept in ff at 2^80 of their value, so that the squares of
// estimates from 2^-90 to 2^20 stay normal floats.
constexpr double kErrScale = 0x1.0p40, kErrUnscale = 0x1.0p-80;

// the range of states, parameters and steps for which products in the models
// below stay within the floats (anything else takes the FP64 path)
constexpr double kFastStateMin = 0x1.0p-40, kFastStateMax = 0x1.0p20;
constexpr double kFastThetaMin = 0x1.0p-40, kFastThetaMax = 0x1.0p40;
constexpr float kFastStepMin = 0x1.0p-60f, kFastStepMax = 0x1.0p40f;
// The last correction is D's low floats lo, known, and a rest.  Both limits hold for each
// component beside its own size (Robertson's y2 and y3 can be 1e-9 of y1).
//  - An FP32 solution, good to 2^-20, serves a rest of up to 2^-32; above it the rest is
//    solved for in ff (0.3 % of Robertson's substeps over its prior at S = 50, K = 2).
//  - The point is off the (K-1)-th iterate by D's rounding to a float, and that by the
//    early FP32 solves' 2^-22 of their step; the last iteration leaves both times the
//    rest.  Above 2^-15 the substep is taken with all of that in ff and FP64 (WIDE): a few
//    at the start of intervals whose parameters have just moved (stage 2: up to half a
//    dozen of 50), and every one of K = 1.  The models' kSettled is what the rest may be
//    then; a substep above it goes to FP64.  Over Robertson's prior, parameters moved by a
//    fifth, y2 and y3 are within 5e-16 (S = 50, K = 2; FP64 path 3e-15), 2e-15 (S = 10; 8e-12),
//    4e-14 (S = 5; 1e-7).  2^-17 to 2^-26 give the same at S = 50 and cost more (0.588 ms a
//    Robertson epoch at 2^-17, 0.578 here, 0.572 with no second form); with limits on the norm
//    and no second form it was 1e-13, 3e-12 and 2e-7, and up to 6e-9 for K = 1.
constexpr float kFastRest = 0x1.0p-32f, kFastSettled = 0x1.0p-15f;

// One substep's coefficients for the increment form (built in shared memory
// from the StepCoef table by fast_coef):
//   R = ra a + rb b,   P = pa a + pb b + pc c,
// BDF: a = x_n - x_{n-1}, b = x_{n-1} - x_{n-2}, c = f(t_n, x_n);
// Adams: a, b, c = f_n, f_{n-1}, f_{n-2}.
struct FastCoef {
  double gamma, ra, rb, in1;  // in1: the input at t_{n+1} (forced problems)
  ff g, fra, frb, pa, pb, pc;
  ff mus;                     // Milne's factor times 2^40 (kErrScale)
  float er, ep;               // the defects rho1 + rho2 + rho3 - 1, pi0 + pi1 + pi2 - 1 of the
                              // rounded BDF weights (0 for Adams)
};

// The entry of a StepCoef c (any struct of its fields).
template <class C>
PF_FF_FN FastCoef fast_coef(const C& c) {
  FastCoef f;
  const bool adams = c.kind > 10;
  // differences of the BDF weights are exact or nearly (they sum to one)
  f.ra = adams ? -c.rho1 : c.rho2 + c.rho3;
  f.rb = adams ? -c.rho2 : c.rho3;
  f.gamma = c.gamma;
  f.in1 = c.in1;
  f.g = ff_from(c.gamma);
  f.fra = ff_from(f.ra);
  f.frb = ff_from(f.rb);
  f.pa = ff_from(adams ? c.pi0 : -(c.pi1 + c.pi2));
  f.pb = ff_from(adams ? c.pi1 : -c.pi2);
  f.pc = ff_from(adams ? c.pi2 : c.pi3);
  f.mus = ff_from(c.mu * kErrScale);
  f.er = adams ? 0.0f : f_from(((c.rho1 - 1.0) + c.rho2) + c.rho3);
  f.ep = adams ? 0.0f : f_from(((c.pi0 - 1.0) + c.pi1) + c.pi2);
  return f;
}

#ifdef __CUDACC__
// A block's substep tables: the steps, and the increment form's coefficients where the
// kernel takes that form.  The second is formed in shared memory; the steps are copied
// there while both leave room for four blocks an SM, and read where they were uploaded
// in longer intervals (their uses are few beside the form, or the L1 cache serves them).  With
// both always in shared memory an SM held one block at 640 substeps: Robertson N = 16384
// stages 2914/3264 us.
struct StepTables {
  const StepCoef* sc;
  const FastCoef* fc;
};
constexpr int kSharedTableBytes = 54 * 1024;
__host__ __device__ constexpr int shared_steps_max(bool fast) {
  return kSharedTableBytes / (int)(sizeof(StepCoef) + (fast ? sizeof(FastCoef) : 0));
}
__host__ __device__ constexpr bool steps_shared(int S, bool fast) { return S <= shared_steps_max(fast); }

// Ends with a barrier.
__device__ __forceinline__ StepTables load_step_tables(double* s_dyn, const EpochParams* __restrict__ ep, int S,
                                                       bool fast) {
  const bool shared = steps_shared(S, fast);
  StepCoef* s_sc = reinterpret_cast<StepCoef*>(s_dyn);
  if (shared) load_steps(s_sc, ep, S);
  FastCoef* t = reinterpret_cast<FastCoef*>(shared ? s_sc + S : s_sc);
  if (fast)
    for (int i = threadIdx.x; i < S; i += blockDim.x) t[i] = fast_coef(ep->sc[i]);
  __syncthreads();
  return StepTables{shared ? s_sc : ep->sc, t};
}
#endif

// the point of the last iteration, x_n + hh, and D + R of its residual: the leading
// part in double, the rest in ff
struct FastState {
  double y[3], R64[3];
  ff cor[3];
  float lo[3];  // what D is above the point
};

// G + a, which nearly cancel
PF_FF_FN float rest_of(ff G, float a) { return f_add(f_add(G.h, a), G.l); }

// every component of d at most t of y's (false if one is not finite)
PF_FF_FN bool within(float t, float y1, float y2, float y3, float d1, float d2, float d3) {
  return fabsf(d1) <= t * fabsf(y1) && fabsf(d2) <= t * fabsf(y2) && fabsf(d3) <= t * fabsf(y3);
}

// dl = lo + d; whether d is small enough beside the state for an FP32 solution
PF_FF_FN bool rest_serves(const FastState& st, float y1, float y2, float y3, float d1, float d2, float d3,
                          ff (&dl)[3]) {
  dl[0] = two_sum(st.lo[0], d1);
  dl[1] = two_sum(st.lo[1], d2);
  dl[2] = two_sum(st.lo[2], d3);
  return within(kFastRest, y1, y2, y3, d1, d2, d3);
}

// ---------------------------------------------------------------- Robertson
struct RobertsonFast {
  static constexpr int D = 3;
  static constexpr float kSettled = 1.0f;  // f is quadratic
  struct Fk {
    ff k1, k2, k3;          // theta
  };
  struct Gk {
    ff gk1, gk2, gk3, op;   // gamma theta, 1 + gamma k1
  };
  template <class Th>
  PF_FF_FN static Fk consts(const Th& T) { return Fk{ff_from(T.k1), ff_from(T.k2), ff_from(T.k3)}; }
  template <class Th>
  PF_FF_FN static double theta_min(const Th& T) { return fmin(T.k1, fmin(T.k2, T.k3)); }
  template <class Th>
  PF_FF_FN static double theta_max(const Th& T) { return fmax(T.k1, fmax(T.k2, T.k3)); }
  PF_FF_FN static Gk scaled(const Fk& k, const FastCoef& c) {
    const ff gk1 = ff_mul(k.k1, c.g);
    return Gk{gk1, ff_mul(k.k2, c.g), ff_mul(k.k3, c.g), ff_one_plus(gk1)};
  }

  // (I - gamma J) d = -G by the elimination of Robertson::newton, in ff
  PF_FF_FN static void solve(const Gk& k, ff y2, ff y3, ff G1, ff G2, ff G3, ff (&dl)[3]) {
    const ff q = ff_mul(k.gk3, y2), p = ff_mul(k.gk3, y3), w = ff_twice(ff_mul(k.gk2, y2));
    const ff im = ff_rcp(k.op), l = ff_mul(k.gk1, im);
    const ff den = ff_fma(im, ff_fma(q, w, p), ff_one_plus(w));
    const ff num = ff_sub(ff_mul(ff_mul(q, im), G3), ff_fma(l, G1, G2));
    dl[1] = ff_div(num, den);
    dl[2] = ff_sub(ff_mul(w, dl[1]), G3);
    dl[0] = ff_mul(im, ff_fma(q, dl[2], ff_sub(ff_mul(p, dl[1]), G1)));
  }

  // the same in FP32; q, p, w as there
  PF_FF_FN static void solve32(const Gk& k, float q, float p, float w, float G1, float G2, float G3, float& d1,
                               float& d2, float& d3) {
    const float im = f_rcp(k.op.h), l = f_mul(k.gk1.h, im);
    const float den = f_fma(im, f_fma(q, w, p), f_add(1.0f, w));
    const float num = f_fma(f_mul(q, im), G3, -f_fma(l, G1, G2));
    d2 = f_mul(num, f_rcp(den));
    d3 = f_fma(w, d2, -G3);
    d1 = f_mul(im, f_fma(q, d3, f_fma(p, d2, -G1)));
  }

  // G = D + R - gamma f at y = x + D, then D -= (I - gamma J)^{-1} G, in FP32
  // (WIDE: in ff)
  template <bool WIDE>
  PF_FF_FN static void early(const Fk&, const Gk& k, const FastCoef&, const ff (&x)[3], const ff (&R)[3],
                             ff (&Dv)[3]) {
    if (WIDE) {
      const ff y1 = ff_add(x[0], Dv[0]), y2 = ff_add(x[1], Dv[1]), y3 = ff_add(x[2], Dv[2]);
      const ff ab = ff_sub(ff_mul(k.gk1, y1), ff_mul(ff_mul(k.gk3, y2), y3));
      const ff c = ff_mul(ff_mul(k.gk2, y2), y2);
      const ff g1 = ff_add(ff_add(Dv[0], R[0]), ab), g3 = ff_sub(ff_add(Dv[2], R[2]), c);
      const ff g2 = ff_add(ff_sub(ff_add(Dv[1], R[1]), ab), c);
      ff dl[3];
      solve(k, y2, y3, g1, g2, g3, dl);
      for (int i = 0; i < 3; ++i) Dv[i] = ff_add(Dv[i], dl[i]);
      return;
    }
    const ff y1 = ff_add_raw(x[0], Dv[0]), y2 = ff_add_raw(x[1], Dv[1]), y3 = ff_add_raw(x[2], Dv[2]);
    const ff q = ff_mul_raw(k.gk3, y2), t = ff_mul_raw(k.gk2, y2);
    const ff ab = ff_sub_raw(ff_mul_raw(k.gk1, y1), ff_mul_raw(q, y3));
    const ff c = ff_mul_raw(t, y2);
    const ff g1 = ff_add_raw(ff_add_raw(Dv[0], R[0]), ab), g3 = ff_sub_raw(ff_add_raw(Dv[2], R[2]), c);
    const ff g2 = ff_add_raw(ff_sub_raw(ff_add_raw(Dv[1], R[1]), ab), c);
    float d1, d2, d3;
    solve32(k, q.h, f_mul(k.gk3.h, y3.h), f_add(t.h, t.h), f_add(g1.h, g1.l), f_add(g2.h, g2.l),
            f_add(g3.h, g3.l), d1, d2, d3);
    Dv[0] = ff_add(Dv[0], d1);
    Dv[1] = ff_add(Dv[1], d2);
    Dv[2] = ff_add(Dv[2], d3);
  }

  // the same with the residual in FP32
  PF_FF_FN static void first(const Fk&, const Gk& k, const FastCoef&, const ff (&x)[3], const ff (&R)[3],
                             ff (&Dv)[3]) {
    const float y1 = f_add(x[0].h, Dv[0].h), y2 = f_add(x[1].h, Dv[1].h), y3 = f_add(x[2].h, Dv[2].h);
    const float q = f_mul(k.gk3.h, y2), t = f_mul(k.gk2.h, y2);
    const float ab = f_fma(k.gk1.h, y1, -f_mul(q, y3)), c = f_mul(t, y2);
    float d1, d2, d3;
    solve32(k, q, f_mul(k.gk3.h, y3), f_add(t, t), f_add(f_add(Dv[0].h, R[0].h), ab),
            f_add(f_sub(f_add(Dv[1].h, R[1].h), ab), c), f_sub(f_add(Dv[2].h, R[2].h), c), d1, d2, d3);
    Dv[0] = ff{f_add(Dv[0].h, d1), 0.0f};
    Dv[1] = ff{f_add(Dv[1].h, d2), 0.0f};
    Dv[2] = ff{f_add(Dv[2].h, d3), 0.0f};
  }

  // the last iteration's correction.  fy, dfy: f at the corrected point (double
  // part and ff part), if wanted.  False if the rest is above `settled` of the state.
  template <bool NEEDF, class Th>
  PF_FF_FN static bool last(const Th& T, const Fk& fk, const Gk& k, const FastCoef& c, const FastState& st,
                            float settled, ff (&dl)[3], double (&fy)[3], ff (&dfy)[3]) {
    const double y1 = st.y[0], y2 = st.y[1], y3 = st.y[2];
    const double q64 = T.k3 * y2;
    const double s64 = fma(T.k1, y1, -(q64 * y3));  // k1 y1 - k3 y2 y3 = -f1
    const double c64 = (T.k2 * y2) * y2;            // k2 y2^2 = f3
    const ff G1 = ff_add_raw(ff_from(fma(c.gamma, s64, st.R64[0])), st.cor[0]);
    const ff G2 = ff_add_raw(ff_from(fma(-c.gamma, s64, fma(c.gamma, c64, st.R64[1]))), st.cor[1]);
    const ff G3 = ff_add_raw(ff_from(fma(-c.gamma, c64, st.R64[2])), st.cor[2]);
    const float e1 = f_from(y1), e2f = f_from(y2), e3 = f_from(y3);
    // G + (I - gamma J) lo: what the low floats leave to correct
    const float q = f_mul(k.gk3.h, e2f), p = f_mul(k.gk3.h, e3), t = f_mul(k.gk2.h, e2f), w = f_add(t, t);
    const float v = f_fma(k.gk1.h, st.lo[0], -f_fma(p, st.lo[1], f_mul(q, st.lo[2])));
    const float wl = f_mul(w, st.lo[1]);
    float d1, d2, d3;
    solve32(k, q, p, w, rest_of(G1, f_add(st.lo[0], v)), rest_of(G2, f_add(f_sub(st.lo[1], v), wl)),
            rest_of(G3, f_sub(st.lo[2], wl)), d1, d2, d3);
    if (!rest_serves(st, e1, e2f, e3, d1, d2, d3, dl)) {
      if (!within(settled, e1, e2f, e3, d1, d2, d3)) return false;
      solve(k, ff_from(y2), ff_from(y3), G1, G2, G3, dl);
    }
    if (NEEDF) {
      const ff f2 = ff_from(y2), f3 = ff_from(y3);
      // f is quadratic: f(y + d) = f(y) + J d + Q(d, d), in ff beside FP64 f(y)
      const ff e2 = ff_add(f2, dl[1]);
      const ff dq = ff_add(ff_mul(f3, dl[1]), ff_mul(e2, dl[2]));      // y2 y3 changes by
      const ff ds = ff_sub(ff_mul(fk.k1, dl[0]), ff_mul(fk.k3, dq));
      const ff dc = ff_mul(fk.k2, ff_mul(dl[1], ff_add(f2, e2)));
      fy[0] = -s64;
      fy[1] = s64 - c64;
      fy[2] = c64;
      dfy[0] = ff_neg(ds);
      dfy[1] = ff_sub(ds, dc);
      dfy[2] = dc;
    }
    return true;
  }
};

// ----------------------------------------------------------------------- M1
// The fluxes j = V x/(x + k); in the last iteration j is a float jt plus dj = (V x - jt
// s)/s, s = x + k, the remainder formed by one FP64 FMA, so no FP64 reciprocal is
// needed.  (As V - u, u = V k/(x + k), it took one FP64 instruction fewer and lost what V is
// above j: x2 over an interval of AM3 1e-15 rms instead of FP64's 4e-16.)  The
// Jacobian and the early iterations take u.
struct MichaelisFast {
  static constexpr int D = 3;
  // Iterates that jump past the pole x = -k do not settle (a fifth of the prior, in the
  // first interval).
  static constexpr float kSettled = 0x1.0p-20f;
  struct Fk {
    ff fvk1, fvk2, fvd, fvc, fk1, fk2;  // V1 k1, V2 k2, V1 - V2, V2 + lambda c0, k1, k2
    float v1, v2;
  };
  struct Gk {
    ff ff0, gl;                   // input - V1, gamma lambda
  };
  static constexpr double kLambda = 0.5, kC0 = 2.0;
  template <class Th>
  PF_FF_FN static Fk consts(const Th& T) {
    return Fk{ff_from(T.v1 * T.k1), ff_from(T.v2 * T.k2), ff_from(T.v1 - T.v2), ff_from(fma(kLambda, kC0, T.v2)),
              ff_from(T.k1), ff_from(T.k2), f_from(T.v1), f_from(T.v2)};
  }
  template <class Th>
  PF_FF_FN static double theta_min(const Th& T) { return fmin(fmin(T.v1, T.v2), fmin(T.k1, T.k2)); }
  template <class Th>
  PF_FF_FN static double theta_max(const Th& T) { return fmax(fmax(T.v1, T.v2), fmax(T.k1, T.k2)); }
  template <class Th>
  PF_FF_FN static Gk scaled(const Th& T, const Fk&, const FastCoef& c) {
    return Gk{ff_from(c.in1 - T.v1), ff{0.5f * c.g.h, 0.5f * c.g.l}};
  }

  // (I - gamma J) d = -G by forward substitution, in ff; u = V k/s, r = 1/s
  PF_FF_FN static void solve(const Gk& gk, const FastCoef& c, ff u1, ff r1, ff u2, ff r2, ff G1, ff G2,
                             ff G3, ff (&dl)[3]) {
    const ff ga = ff_mul(ff_mul(c.g, u1), r1), gb = ff_mul(ff_mul(c.g, u2), r2);
    dl[0] = ff_neg(ff_div(G1, ff_one_plus(ga)));
    dl[1] = ff_div(ff_sub(ff_mul(ga, dl[0]), G2), ff_one_plus(gb));
    dl[2] = ff_div(ff_sub(ff_mul(gb, dl[1]), G3), ff_one_plus(gk.gl));
  }

  // the same in FP32; ga, gb = gamma u/s
  PF_FF_FN static void solve32(const Gk& gk, float ga, float gb, float G1, float G2, float G3, float& d1,
                               float& d2, float& d3) {
    d1 = -f_mul(G1, f_rcp(f_add(1.0f, ga)));
    d2 = f_mul(f_fma(ga, d1, -G2), f_rcp(f_add(1.0f, gb)));
    d3 = f_mul(f_fma(gb, d2, -G3), f_rcp(f_add(1.0f, gk.gl.h)));
  }

  template <bool WIDE>
  PF_FF_FN static void early(const Fk& k, const Gk& gk, const FastCoef& c, const ff (&x)[3],
                             const ff (&R)[3], ff (&Dv)[3]) {
    if (WIDE) {
      const ff s1 = ff_add(ff_add(x[0], Dv[0]), k.fk1), s2 = ff_add(ff_add(x[1], Dv[1]), k.fk2);
      const ff y3 = ff_add(x[2], Dv[2]);
      const ff u1 = ff_div(k.fvk1, s1), u2 = ff_div(k.fvk2, s2);
      const ff f1 = ff_add(gk.ff0, u1);
      const ff f2 = ff_add(ff_sub(k.fvd, u1), u2);
      const ff f3 = ff_sub(ff_sub(k.fvc, u2), ff{0.5f * y3.h, 0.5f * y3.l});
      const ff g1 = ff_sub(ff_add(Dv[0], R[0]), ff_mul(c.g, f1));
      const ff g2 = ff_sub(ff_add(Dv[1], R[1]), ff_mul(c.g, f2));
      const ff g3 = ff_sub(ff_add(Dv[2], R[2]), ff_mul(c.g, f3));
      ff dl[3];
      solve(gk, c, u1, ff_rcp(s1), u2, ff_rcp(s2), g1, g2, g3, dl);
      for (int i = 0; i < 3; ++i) Dv[i] = ff_add(Dv[i], dl[i]);
      return;
    }
    const ff s1 = ff_add(ff_add_raw(x[0], Dv[0]), k.fk1), s2 = ff_add(ff_add_raw(x[1], Dv[1]), k.fk2);
    const ff y3 = ff_add_raw(x[2], Dv[2]);
    const ff u1 = ff_div(k.fvk1, s1), u2 = ff_div(k.fvk2, s2);
    const ff f1 = ff_add_raw(gk.ff0, u1);
    const ff f2 = ff_add_raw(ff_sub_raw(k.fvd, u1), u2);
    const ff f3 = ff_sub_raw(ff_sub_raw(k.fvc, u2), ff{0.5f * y3.h, 0.5f * y3.l});
    const ff g1 = ff_sub_raw(ff_add_raw(Dv[0], R[0]), ff_mul_raw(c.g, f1));
    const ff g2 = ff_sub_raw(ff_add_raw(Dv[1], R[1]), ff_mul_raw(c.g, f2));
    const ff g3 = ff_sub_raw(ff_add_raw(Dv[2], R[2]), ff_mul_raw(c.g, f3));
    float d1, d2, d3;
    solve32(gk, f_mul(f_mul(c.g.h, u1.h), f_rcp(s1.h)), f_mul(f_mul(c.g.h, u2.h), f_rcp(s2.h)),
            f_add(g1.h, g1.l), f_add(g2.h, g2.l), f_add(g3.h, g3.l), d1, d2, d3);
    Dv[0] = ff_add(Dv[0], d1);
    Dv[1] = ff_add(Dv[1], d2);
    Dv[2] = ff_add(Dv[2], d3);
  }

  // the same with the residual in FP32
  PF_FF_FN static void first(const Fk& k, const Gk& gk, const FastCoef& c, const ff (&x)[3], const ff (&R)[3],
                             ff (&Dv)[3]) {
    const float r1 = f_rcp(f_add(f_add(x[0].h, Dv[0].h), k.fk1.h)), r2 = f_rcp(f_add(f_add(x[1].h, Dv[1].h), k.fk2.h));
    const float u1 = f_mul(k.fvk1.h, r1), u2 = f_mul(k.fvk2.h, r2), g = c.g.h;
    const float f1 = f_add(gk.ff0.h, u1), f2 = f_add(f_sub(k.fvd.h, u1), u2);
    const float f3 = f_fma(-0.5f, f_add(x[2].h, Dv[2].h), f_sub(k.fvc.h, u2));
    float d1, d2, d3;
    solve32(gk, f_mul(f_mul(g, u1), r1), f_mul(f_mul(g, u2), r2), f_fma(-g, f1, f_add(Dv[0].h, R[0].h)),
            f_fma(-g, f2, f_add(Dv[1].h, R[1].h)), f_fma(-g, f3, f_add(Dv[2].h, R[2].h)), d1, d2, d3);
    Dv[0] = ff{f_add(Dv[0].h, d1), 0.0f};
    Dv[1] = ff{f_add(Dv[1].h, d2), 0.0f};
    Dv[2] = ff{f_add(Dv[2].h, d3), 0.0f};
  }

  template <bool NEEDF, class Th>
  PF_FF_FN static bool last(const Th& T, const Fk& k, const Gk& gk, const FastCoef& c, const FastState& st,
                            float settled, ff (&dl)[3], double (&fy)[3], ff (&dfy)[3]) {
    const double s1 = st.y[0] + T.k1, s2 = st.y[1] + T.k2;
    const ff e1 = ff_from(s1), e2 = ff_from(s2);
    const ff r1 = ff_rcp(e1), r2 = ff_rcp(e2);
    const float y1 = f_from(st.y[0]), y2 = f_from(st.y[1]), y3 = f_from(st.y[2]);
    const float u1 = f_mul(k.fvk1.h, r1.h), u2 = f_mul(k.fvk2.h, r2.h);
    const double w1 = d_from_f(f_mul(f_mul(k.v1, y1), r1.h)), w2 = d_from_f(f_mul(f_mul(k.v2, y2), r2.h));
    const ff dj1 = ff_mul(ff_from(fma(-w1, s1, T.v1 * st.y[0])), r1);
    const ff dj2 = ff_mul(ff_from(fma(-w2, s2, T.v2 * st.y[1])), r2);
    fy[0] = c.in1 - w1;
    fy[1] = w1 - w2;
    fy[2] = fma(-kLambda, st.y[2] - kC0, w2);
    const ff gd1 = ff_mul_raw(c.g, dj1), gd2 = ff_mul_raw(c.g, dj2);
    const ff G1 = ff_add_raw(ff_add_raw(ff_from(fma(-c.gamma, fy[0], st.R64[0])), st.cor[0]), gd1);
    const ff G2 = ff_add_raw(ff_sub_raw(ff_add_raw(ff_from(fma(-c.gamma, fy[1], st.R64[1])), st.cor[1]), gd1), gd2);
    const ff G3 = ff_sub_raw(ff_add_raw(ff_from(fma(-c.gamma, fy[2], st.R64[2])), st.cor[2]), gd2);
    // G + (I - gamma J) lo: what the low floats leave to correct
    const float ga = f_mul(f_mul(c.g.h, u1), r1.h), gb = f_mul(f_mul(c.g.h, u2), r2.h);
    const float al = f_mul(ga, st.lo[0]), bl = f_mul(gb, st.lo[1]);
    float d1, d2, d3;
    solve32(gk, ga, gb, rest_of(G1, f_add(st.lo[0], al)), rest_of(G2, f_sub(f_add(st.lo[1], bl), al)),
            rest_of(G3, f_sub(f_fma(gk.gl.h, st.lo[2], st.lo[2]), bl)), d1, d2, d3);
    if (!rest_serves(st, y1, y2, y3, d1, d2, d3, dl)) {
      if (!within(settled, y1, y2, y3, d1, d2, d3)) return false;
      solve(gk, c, ff_mul(k.fvk1, r1), r1, ff_mul(k.fvk2, r2), r2, G1, G2, G3, dl);
    }
    if (NEEDF) {
      const ff t1 = ff_mul(k.fvk1, r1), t2 = ff_mul(k.fvk2, r2);
      // j(x + d) = j + u d/(s + d)
      const ff v1 = ff_add(dj1, ff_div(ff_mul(t1, dl[0]), ff_add(e1, dl[0])));
      const ff v2 = ff_add(dj2, ff_div(ff_mul(t2, dl[1]), ff_add(e2, dl[1])));
      dfy[0] = ff_neg(v1);
      dfy[1] = ff_sub(v1, v2);
      dfy[2] = ff_sub(v2, ff{0.5f * dl[2].h, 0.5f * dl[2].l});
    }
    return true;
  }
};

template <class Th>
PF_FF_FN RobertsonFast::Gk fast_scaled(const Th&, const RobertsonFast::Fk& k, const FastCoef& c) {
  return RobertsonFast::scaled(k, c);
}
template <class Th>
PF_FF_FN MichaelisFast::Gk fast_scaled(const Th& T, const MichaelisFast::Fk& k, const FastCoef& c) {
  return MichaelisFast::scaled(T, k, c);
}

// What a particle carries from substep to substep.
//   x + cx: x_n, the last iteration's point and its correction (Adams: h1 + c1, h2 +
//   c2: x_{n-1}, x_{n-2})
//   a + ra, b + rb: the double and ff parts of what R multiplies: BDF x_n - x_{n-1}
//   and x_{n-1} - x_{n-2} (the leading float of the increment and the rest, which
//   spares an FP64 difference), Adams f_n and f_{n-1} (all but a float)
//   fa, fb, fc: BDF x_n - x_{n-1}, x_{n-1} - x_{n-2}, f(x_n) in ff; Adams f_n, f_{n-1},
//   f_{n-2}
//   E: the error sums at 2^80 of their value
struct FastCarry {
  double x[3], h1[3], h2[3];
  ff cx[3], c1[3], c2[3];
  double a[3], b[3];
  ff ra[3], rb[3];
  ff fa[3], fb[3], fc[3], E[3];
};

// One substep.  FAM: 0 BDF2, 1 BDF3, 2 Adams-Moulton.  WIDE: every early iteration in
// ff, from a start in ff, and the last at the (K-1)-th iterate to FP64 rounding instead
// of a float's.
//  kStepSettled   done, the rest below kFastSettled
//  kStepWide      (WIDE) done, the rest above it
//  kStepUnsettled (not WIDE) w untouched, to be taken again with WIDE
//  kStepFar       w untouched, left to FP64
enum { kStepSettled, kStepWide, kStepUnsettled, kStepFar };
template <class MF, int FAM, bool ERR, bool WIDE, class Th>
PF_FF_FN int fast_iterate(const Th& T, const typename MF::Fk& fk, const FastCoef& c, int K, FastCarry& w) {
  const typename MF::Gk gk = fast_scaled(T, fk, c);
  ff P[3], Dv[3], xf[3];
  FastState st;
  for (int i = 0; i < 3; ++i) {
    xf[i] = ff_add_raw(ff_from(w.x[i]), w.cx[i]);
    if (!ERR && FAM != 2 && !WIDE) {
      // a start for the iterations only: a float does, as an early FP32 solve does
      float p = f_fma(c.pb.h, w.fb[i].h, f_fma(c.pa.h, w.fa[i].h, f_mul(c.ep, xf[i].h)));
      if (FAM == 1) p = f_fma(c.pc.h, w.fc[i].h, p);
      Dv[i] = ff{p, 0.0f};
      continue;
    }
    ff p = ff_mul_raw(c.pa, w.fa[i]);
    p = ff_fma(c.pb, w.fb[i], p);
    if (FAM != 0) p = ff_fma(c.pc, w.fc[i], p);
    if (FAM != 2) p.l = f_fma(c.ep, xf[i].h, p.l);
    P[i] = Dv[i] = p;
  }
  if (K > 1) {
    ff R[3];
    for (int i = 0; i < 3; ++i) {
      R[i] = ff_mul(c.fra, w.fa[i]);
      if (FAM != 0) R[i] = ff_fma(c.frb, w.fb[i], R[i]);
    }
    for (int it = 0; it + 1 < K; ++it) {
      if (WIDE || (FAM == 2 && (it + 2 < K || K == 2))) MF::template early<true>(fk, gk, c, xf, R, Dv);
      else if (it + 2 < K) MF::first(fk, gk, c, xf, R, Dv);
      else MF::template early<false>(fk, gk, c, xf, R, Dv);
    }
  }
  float hh[3], lw[3];  // lw: D's low float where the point has it (WIDE)
  for (int i = 0; i < 3; ++i) {
    // the point x + hh, hh the float nearest D + cx: from x_n it is hh - cx
    const ff s = ff_add(Dv[i], w.cx[i]);
    hh[i] = s.h;
    st.lo[i] = s.l;
    const double hd = d_from_f(hh[i]);
    st.y[i] = w.x[i] + hd;
    st.R64[i] = fma(c.ra, w.a[i], FAM != 0 ? fma(c.rb, w.b[i], hd) : hd);
    // the rest: R's, the carry and the weights' defect
    ff r{f_mul(c.fra.h, w.ra[i].h), 0.0f};
    if (FAM == 2) r.h = f_fma(c.frb.h, w.rb[i].h, r.h);
    else r = ff_mul_raw(c.fra, w.ra[i]);
    if (FAM == 1) r = ff_fma(c.frb, w.rb[i], r);
    if (FAM != 2) r.l = f_fma(-c.er, xf[i].h, r.l);
    st.cor[i] = ff_sub_raw(r, w.cx[i]);
    if (WIDE) {
      lw[i] = s.l;
      st.lo[i] = 0.0f;
      st.y[i] += d_from_f(s.l);
      st.cor[i] = ff_add(st.cor[i], s.l);
    }
  }
  ff dl[3], dfy[3];
  double fy[3];
  // (a single iteration has no earlier one to be off by: the ff solve of its rest is good to
  // 2^-46 of it)
  const float limit = !WIDE ? kFastSettled : K == 1 ? 1.0f : MF::kSettled;
  if (!MF::template last<FAM != 0>(T, fk, gk, c, st, limit, dl, fy, dfy)) return WIDE ? kStepFar : kStepUnsettled;
  // values still in the floats' range (and finite)
  if (!(fabsf(f_from(st.y[0])) + fabsf(f_from(st.y[1])) + fabsf(f_from(st.y[2])) < 0x1.0p24f)) return kStepFar;
  if (ERR) {
    // and squares of the scaled estimates whose sum stays a float (640 of 2^116)
    float me = 0.0f;
    for (int i = 0; i < 3; ++i) me = me + fabsf(P[i].h) + fabsf(hh[i]) + fabsf(dl[i].h);
    if (!(fabsf(c.mus.h) * me < 0x1.0p58f)) return kStepFar;
  }
  for (int i = 0; i < 3; ++i) {
    // the increment from x_n to the new state
    ff rest = ff_sub(dl[i], w.cx[i]);
    if (WIDE) rest = ff_add(rest, lw[i]);
    const ff Dn = ff_add(rest, hh[i]);
    if (ERR) {
      const ff e = ff_mul(c.mus, ff_sub(Dn, P[i]));
      w.E[i] = ff_fma(e, e, w.E[i]);
    }
    if (FAM == 2) {
      w.fc[i] = w.fb[i];
      w.fb[i] = w.fa[i];
      w.b[i] = w.a[i];
      w.rb[i] = w.ra[i];
      w.a[i] = fy[i] + d_from_f(dfy[i].h);
      w.ra[i] = ff{dfy[i].l, 0.0f};
      w.fa[i] = ff_from(w.a[i]);
      w.fa[i].l = f_add(w.fa[i].l, dfy[i].l);
    } else {
      if (FAM == 1) {
        w.b[i] = w.a[i];
        w.rb[i] = w.ra[i];
        w.fc[i] = ff_add(ff_from(fy[i]), dfy[i]);
      }
      w.fb[i] = w.fa[i];
      w.fa[i] = Dn;
      w.a[i] = d_from_f(hh[i]);
      w.ra[i] = rest;
    }
    if (FAM == 2) {
      w.h2[i] = w.h1[i];
      w.c2[i] = w.c1[i];
      w.h1[i] = w.x[i];
      w.c1[i] = w.cx[i];
    }
    w.x[i] = st.y[i];
    w.cx[i] = dl[i];
  }
  if (!WIDE) return kStepSettled;
  const float y1 = f_from(st.y[0]), y2 = f_from(st.y[1]), y3 = f_from(st.y[2]);
  return within(kFastSettled, y1, y2, y3, dl[0].h, dl[1].h, dl[2].h) ? kStepSettled : kStepWide;
}

// One substep; false, with w untouched, if it is left to FP64.  (The kernels have the two
// tries in loops of their own.)
template <class MF, int FAM, bool ERR, class Th>
PF_FF_FN bool fast_step(const Th& T, const typename MF::Fk& fk, const FastCoef& c, int K, FastCarry& w) {
  int r = fast_iterate<MF, FAM, ERR, false>(T, fk, c, K, w);
  if (r == kStepUnsettled) r = fast_iterate<MF, FAM, ERR, true>(T, fk, c, K, w);
  return r == kStepSettled || r == kStepWide;
}

PF_FF_FN double ff_value(ff a) { return (double)a.h + (double)a.l; }

// x_n, x_{n-1}, x_{n-2} of component i as doubles (the BDF past from the increments).
template <int FAM>
PF_FF_FN void fast_history(const FastCarry& w, int i, double& x, double& h1, double& h2) {
  x = w.x[i] + ff_value(w.cx[i]);
  if (FAM == 2) {
    h1 = w.h1[i] + ff_value(w.c1[i]);
    h2 = w.h2[i] + ff_value(w.c2[i]);
  } else {
    h1 = x - (w.a[i] + ff_value(w.ra[i]));
    h2 = h1 - ff_value(w.fb[i]);
  }
}

}  // namespace pfg
