// fftfx_lg11.cu -- the fixed-point passes for transforms of 2048 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg11() { return make_fx_kernels<11>(); }
}  // namespace sg
