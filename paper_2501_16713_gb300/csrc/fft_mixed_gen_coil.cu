// The mixed-radix coil-grid passes (fft_mixed_kernels.cuh) for axes of any
// oversampling factor and length: two- or three-step transforms with run-time
// radices (a translation unit of its own: one unrolled body per radix).
#include "fft_mixed_kernels.cuh"

namespace nrs {

void mixed_gen_coil_pass(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  mixed::GeneralAxis ax{x.g, x.n, x.N};
  ax.g.tw = x.tw_g;
  ax.n.tw = x.tw_n;
  mixed::run_coil_pass(a, ax, s);
}

}  // namespace nrs
