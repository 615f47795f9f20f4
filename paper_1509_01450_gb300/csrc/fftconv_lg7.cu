// fftconv_lg7.cu -- the FP32 column passes for transforms of 128 points with
// the length fixed at compile time (see FixedPassKernels in fftconv.cu).
#define SG_FFTCONV_KERNELS_ONLY
#include "fftconv.cu"

namespace sg {
FixedPassKernels fixed_pass_kernels_lg7() { return make_fixed_pass_kernels<7>(); }
}  // namespace sg
