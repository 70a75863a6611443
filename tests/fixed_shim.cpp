// A host build of the fixed-point exp and sqrt of pf_math.cuh, for the tests.
#include "pf_math.cuh"

extern "C" void shim_exp(const double* x, double* y, long n) {
  for (long i = 0; i < n; ++i) y[i] = pfm::exp_fixed(x[i]);
}

extern "C" void shim_sqrt(const double* x, double* y, long n) {
  for (long i = 0; i < n; ++i) y[i] = pfm::sqrt_fixed(x[i]);
}
