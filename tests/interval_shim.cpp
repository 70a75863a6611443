// A host build of the increment form's substeps (pf_fast.cuh) for the tests: one
// interval of one particle, with or without the error sums (stage 2's and stage 1's forms).
#include <cmath>
using std::fabs;
using std::fma;
using std::fmax;
using std::fmin;
#include "pf_fast.cuh"

using namespace pfg;

namespace {
struct Row {
  int kind;
  double gamma, rho1, rho2, rho3, pi0, pi1, pi2, pi3, mu, in1;
};
struct ThRobertson {
  double k1, k2, k3;
};
struct ThMichaelis {
  double v1, v2, k1, k2;
};

template <class MF, int FAM, bool ERR, class Th>
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
    if (!fast_step<MF, FAM, ERR>(T, fk, fast_coef(rows[n]), K, w)) break;
  for (int i = 0; i < 3; ++i) {
    fast_history<FAM>(w, i, s[i], s[3 + i], s[6 + i]);
    E[i] = ff_value(w.E[i]) * kErrUnscale;
  }
  return n;
}

template <class MF, class Th>
int run(int fam, int err, const Th& T, const Row* r, int S, int K, double* s, double* E) {
  if (fam == 0) return err ? interval<MF, 0, true>(T, r, S, K, s, E) : interval<MF, 0, false>(T, r, S, K, s, E);
  if (fam == 1) return err ? interval<MF, 1, true>(T, r, S, K, s, E) : interval<MF, 1, false>(T, r, S, K, s, E);
  return err ? interval<MF, 2, true>(T, r, S, K, s, E) : interval<MF, 2, false>(T, r, S, K, s, E);
}
}  // namespace

// model 0 Robertson, 1 M1; fam 0 BDF2, 1 BDF3, 2 Adams-Moulton; s: x_n, x_{n-1},
// x_{n-2}, then f_n (and f_{n-1}, f_{n-2}).  Returns the substeps done.
extern "C" int shim_run(int model, int fam, int err, const double* th, const double* rows, int S, int K, double* s,
                        double* E) {
  static thread_local Row r[640];
  for (int i = 0; i < S; ++i) {
    const double* q = rows + 11 * i;
    r[i] = Row{(int)q[0], q[1], q[2], q[3], q[4], q[5], q[6], q[7], q[8], q[9], q[10]};
  }
  if (model == 0) return run<RobertsonFast>(fam, err, ThRobertson{th[0], th[1], th[2]}, r, S, K, s, E);
  return run<MichaelisFast>(fam, err, ThMichaelis{th[0], th[1], th[2], th[3]}, r, S, K, s, E);
}
