// Host build of the FP64 reconstructions with the FP32 saturation screen
// (double) next to the same arithmetic without it (Dual<1> has no screen).
// Test instrumentation only.
#include <cmath>

#include "fdcgks_dual.cuh"

using namespace fdk;

typedef Dual<1> D1;

extern "C" void probe_screen(int variant, double h, int n, const double* in, double* with, double* without) {
  GenoK<double> g;
  g.linear = 0;
  g.C = 20.0;
  g.tanhC = std::tanh(20.0);
  g.inv_tanhC = 1.0 / std::tanh(20.0);
  g.eps_w = 1e-6;
  g.r = variant == 1 ? 3 : 2;
  g.eps_a = variant == 1 ? 1e-15 : 1e-12;
  for (int k = 0; k < 3; ++k) {
    g.d_iface[k] = variant == 1 ? (k == 1 ? 8.0 : 1.0) : (k == 0 ? 8.0 : 1.0);
    g.d_node[k] = k == 0 ? 8.0 : 1.0;
  }
  const GenoK<D1> gd = dual_geno<1>(g);
  for (int t = 0; t < n; ++t) {
    const double* q = in + 8 * t;
    double* a = with + 7 * t;
    double* b = without + 7 * t;
    recon_interface(g, q, q + 4, h, 1.0 / h, a[0], a[1], a[2], a[3], a[4], a[5]);
    a[6] = recon_node(g, q, q + 4, h, 1.0 / h);
    D1 x[8], o[6];
    for (int k = 0; k < 8; ++k) x[k] = D1(q[k]);
    recon_interface(gd, x, x + 4, D1(h), D1(1.0 / h), o[0], o[1], o[2], o[3], o[4], o[5]);
    for (int k = 0; k < 6; ++k) b[k] = o[k].v;
    b[6] = recon_node(gd, x, x + 4, D1(h), D1(1.0 / h)).v;
  }
}
