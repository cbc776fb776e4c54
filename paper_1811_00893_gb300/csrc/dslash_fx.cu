// FP64 hopping kernels with fixed-point links (LF = 3, fx64.cuh) and no clover
// term: explicit instantiation of hop_kernels.cuh, compiled apart.
#include "hop_kernels.cuh"

namespace wl {
template struct HopKernels<kClNone, 3>;
}  // namespace wl
