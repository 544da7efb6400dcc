// Host build of the rule that decides whether a kernel reads a caller's device
// array itself or the copy engine stages it.  Test instrumentation only.
#include "fdcgks_internal.cuh"

extern "C" int probe_kernel_reaches(int type, int pointer_device, int device) {
  cudaPointerAttributes a = {};
  a.type = (cudaMemoryType)type;
  a.device = pointer_device;
  return fdk::kernel_reaches(a, device);
}

// bytes of staging that a run of nx x ny nodes needs, and that its point buffer has
extern "C" void probe_staging(int nx, int ny, int bounded, int mixed, long* need, long* have) {
  fdcgks_params p = {};
  p.nx = nx;
  p.ny = ny;
  for (int k = 0; k < 4; ++k) p.bc[k] = bounded;
  const fdk::Layout L = fdk::make_layout(p);
  const fdk::DenseState d = fdk::dense_areas(nullptr, L);
  *need = (long)(size_t)(d.G[1] + 8L * L.nxd * L.nyd);
  *have = (mixed ? 4L : 8L) * fdk::NPT * L.pplane;
}
