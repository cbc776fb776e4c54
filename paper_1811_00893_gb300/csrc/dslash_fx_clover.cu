// FP64 hopping kernels with fixed-point links (LF = 3, fx64.cuh), both clover
// modes: explicit instantiation of hop_kernels.cuh, compiled apart.
#include "hop_kernels.cuh"

namespace wl {
template struct HopKernels<kClX2, 3>;
template struct HopKernels<kClOut, 3>;
}  // namespace wl
