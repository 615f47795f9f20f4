// fftfx_lg7.cu -- the fixed-point passes for transforms of 128 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg7() { return make_fx_kernels<7>(); }
}  // namespace sg
