// The mixed-radix coil-grid passes (fft_mixed_kernels.cuh) at sigma 2 with
// run-time radices (a translation unit of its own: one unrolled body per radix).
#include "fft_mixed_kernels.cuh"

namespace nrs {

void mixed_rt_coil_pass(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  mixed::DoubleAxis<mixed::RtLen> ax;
  ax.l = mixed::RtLen{x.R, x.S, mix_magic(x.R), mix_magic(2 * x.R), mix_magic(x.S), x.tw_g};
  mixed::run_coil_pass(a, ax, s);
}

}  // namespace nrs
