// FP64 kernels of the domain-decomposed hopping term with fixed-point links
// (LF = 3, fx64.cuh), without and with the clover term: explicit instantiation
// of dd_kernels.cuh.
#include "dd_kernels.cuh"

namespace wl {
template struct DDKernels<3, kClNone>;
template struct DDKernels<3, kClX2>;
template struct DDKernels<3, kClOut>;
}  // namespace wl
