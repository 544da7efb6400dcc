// Host build of the FP64 pair exp(-y^2), erfc(y) of the half-space moments.
// Test instrumentation only.
#include "fdcgks_math.cuh"

extern "C" void probe_exp_erfc(int n, const double* y, double* e, double* ec) {
  for (int t = 0; t < n; ++t) fdk::exp_erfc(y[t], e[t], ec[t]);
}
