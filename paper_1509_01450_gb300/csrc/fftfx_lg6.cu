// fftfx_lg6.cu -- the fixed-point passes for transforms of 64 points.
#include "fftfx.cuh"

namespace sg {
FxKernels fx_kernels_lg6() { return make_fx_kernels<6>(); }
}  // namespace sg
