// fftfx_lg10.cu -- the fixed-point passes for transforms of 1024 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg10() { return make_fx_kernels<10>(); }
}  // namespace sg
