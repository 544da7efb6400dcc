// Host build of the FP32 series of the time coefficients (dt/tau <= 1).
// Test instrumentation only.
#include "fdcgks_math.cuh"

extern "C" void probe_time_coef_small(int n, const float* dt, const float* tau, double* out) {
  for (int t = 0; t < n; ++t) {
    const fdk::TimeCoef<float> c = fdk::time_coef_small(dt[t] / tau[t], tau[t], dt[t], 1.0f / dt[t]);
    double* q = out + 14 * t;
    for (int k = 0; k < 6; ++k) { q[k] = c.cn[k]; q[6 + k] = c.ct[k]; }
    q[12] = c.E;
    q[13] = c.e1;
  }
}
