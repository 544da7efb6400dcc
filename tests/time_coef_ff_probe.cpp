// Host build of the mixed path's time coefficients for dt/tau <= 1 (float-float
// series) next to the FP64 form rounded to FP32.  Test instrumentation only.
#include "fdcgks_math.cuh"

using namespace fdk;

template <class T>
static void put(const TimeCoef<T>& c, double* q) {
  for (int k = 0; k < 6; ++k) { q[k] = (float)c.cn[k]; q[6 + k] = (float)c.ct[k]; }
  q[12] = (float)c.E;
  q[13] = (float)c.e1;
}

extern "C" void probe_time_coef(int n, const double* dt, const double* tau, double* series, double* fp64) {
  for (int t = 0; t < n; ++t) {
    put(time_coef_small(ff_split<float>(tau[t] / dt[t]), ff_split<float>(dt[t]), ff_split<float>(1.0 / dt[t])),
        series + 14 * t);
    put(time_coef(tau[t], dt[t], 1.0 / dt[t]), fp64 + 14 * t);
  }
}
