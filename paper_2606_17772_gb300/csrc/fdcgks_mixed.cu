// Mixed-precision instantiation of the FD-CGKS stage kernels: FP32
// reconstruction and flux arithmetic; the state and the S2O4 accumulation as
// float-float pairs; the time coefficients of the interface solution in FP32
// where dt/tau > 4, in FP64 (with expm1) from 1 to 4, where their terms cancel,
// and up to 1 by float-float series.
#include "fdcgks_kernels.cuh"

namespace fdk {
FDK_INSTANTIATE(float)
}  // namespace fdk
