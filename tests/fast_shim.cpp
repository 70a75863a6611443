// A host build of the increment form of the substeps (pf_fast.cuh), for the
// tests: one interval of one particle.  The pairs of floats round as on the
// device (the reciprocal differs in its last bit).
#include <cmath>
using std::fabs;
using std::fma;
using std::fmax;
using std::fmin;
#include "pf_fast.cuh"

using namespace pfg;

namespace {
struct Row {  // the columns of pf_substep_table's rows that the form needs, and the input
  int kind;
  double gamma, rho1, rho2, rho3, pi0, pi1, pi2, pi3, mu, in1;
};
struct ThRobertson {
  double k1, k2, k3;
};
struct ThMichaelis {
  double v1, v2, k1, k2;
};

template <class MF, int FAM, class Th>
int interval(const Th& T, const Row* rows, int S, int K, double* s, double* E) {
  const typename MF::Fk fk = MF::consts(T);
  FastCarry w{};
  for (int i = 0; i < 3; ++i) {
    w.x[i] = s[i];
    w.h1[i] = s[3 + i];
    w.h2[i] = s[6 + i];
    w.a[i] = FAM == 2 ? s[9 + i] : s[i] - s[3 + i];
    w.b[i] = FAM == 2 ? s[12 + i] : s[3 + i] - s[6 + i];
    w.fa[i] = ff_from(w.a[i]);
    w.fb[i] = ff_from(w.b[i]);
    w.fc[i] = ff_from(FAM == 2 ? s[15 + i] : FAM == 1 ? s[9 + i] : 0.0);
  }
  int n = 0;
  for (; n < S; ++n)
    if (!fast_step<MF, FAM, true>(T, fk, fast_coef(rows[n]), K, w)) break;
  for (int i = 0; i < 3; ++i) {
    fast_history<FAM>(w, i, s[i], s[3 + i], s[6 + i]);
    E[i] = ff_value(w.E[i]) * kErrUnscale;
  }
  return n;
}
}  // namespace

// model 0 Robertson, 1 M1; fam 0 BDF2, 1 BDF3, 2 Adams-Moulton; s: x_n, x_{n-1},
// x_{n-2}, then f_n (and f_{n-1}, f_{n-2}).  Returns the substeps done.
extern "C" int shim_interval(int model, int fam, const double* th, const double* rows, int S, int K,
                             double* s, double* E) {
  static thread_local Row r[640];
  for (int i = 0; i < S; ++i) {
    const double* q = rows + 11 * i;
    r[i] = Row{(int)q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], q[8], q[9], q[10]};
  }
  const ThRobertson R{th[0], th[1], th[2]};
  if (model == 0)
    return fam == 0   ? interval<RobertsonFast, 0>(R, r, S, K, s, E)
           : fam == 1 ? interval<RobertsonFast, 1>(R, r, S, K, s, E)
                      : interval<RobertsonFast, 2>(R, r, S, K, s, E);
  const ThMichaelis M{th[0], th[1], th[2], th[3]};
  return fam == 0   ? interval<MichaelisFast, 0>(M, r, S, K, s, E)
         : fam == 1 ? interval<MichaelisFast, 1>(M, r, S, K, s, E)
                    : interval<MichaelisFast, 2>(M, r, S, K, s, E);
}

// to and from pairs of floats
extern "C" void shim_pairs(const double* a, double* hl, double* back, long n) {
  for (long i = 0; i < n; ++i) {
    const ff p = ff_from(a[i]);
    hl[2 * i] = p.h;
    hl[2 * i + 1] = p.l;
    back[i] = d_from_f(p.h);
  }
}
