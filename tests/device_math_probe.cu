// The conversions by shifts, the exp/erfc pair and the float-float time
// coefficients as the GPU evaluates them (nvcc) or as the host does (g++ -x
// c++).  Test instrumentation only.
#include "fdcgks_math.cuh"

using namespace fdk;

#if !defined(__CUDACC__)
#define __global__
#endif

// what: 0 est_f32 (o[0]), 1 f32_to_f64 of (float)x (o[0]), 2 exp_erfc (o[0..1]) and
// the library's pair as it was used before (o[2..3]), 3 time_coef_small of dt =
// x, tau = y (o[0..13])
FD_HD void probe_one(int what, double x, double y, double* o) {
  if (what == 0) {
    o[0] = (double)est_f32(x);
  } else if (what == 1) {
    o[0] = f32_to_f64((float)x);
  } else if (what == 2) {
    exp_erfc(x, o[0], o[1]);
    o[2] = s_exp(-x * x);
    o[3] = s_erfc_e(x, o[2]);
  } else {
    const TimeCoef<float> c =
        time_coef_small(ff_split<float>(y / x), ff_split<float>(x), ff_split<float>(1.0 / x));
    for (int k = 0; k < 6; ++k) { o[k] = c.cn[k]; o[6 + k] = c.ct[k]; }
    o[12] = c.E;
    o[13] = c.e1;
  }
}

const int STRIDE = 14;
extern "C" void probe_host(int what, int n, const double* x, const double* y, double* out) {
  for (int t = 0; t < n; ++t) probe_one(what, x[t], y[t], out + (long)STRIDE * t);
}

#if defined(__CUDACC__)
__global__ void probe_kernel(int what, int n, const double* x, const double* y, double* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) probe_one(what, x[t], y[t], out + (long)STRIDE * t);
}
extern "C" int probe_device(int what, int n, const double* x, const double* y, double* out) {
  double* d = nullptr;
  const size_t b = sizeof(double) * n;
  cudaError_t e = cudaMalloc((void**)&d, (2 + STRIDE) * b);
  if (e == cudaSuccess) e = cudaMemcpy(d, x, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(d + n, y, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(d + 2 * n, 0, STRIDE * b);
  if (e == cudaSuccess) {
    probe_kernel<<<(n + 127) / 128, 128>>>(what, n, d, d + n, d + 2 * n);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(out, d + 2 * n, STRIDE * b, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return (int)e;
}
#endif
