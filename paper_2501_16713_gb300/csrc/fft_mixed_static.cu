// The mixed-radix passes (fft_mixed_kernels.cuh) with compile-time radices for
// the axis lengths of common volumes at sigma 2.
#include "fft_mixed_kernels.cuh"

namespace nrs {

namespace {
template <int R, int S>
bool pass_for(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  if (x.R != R || x.S != S) return false;
  mixed::DoubleAxis<mixed::StLen<R, S>> ax;
  ax.l.tw = x.tw_g;
  if (a.pass < 6)
    mixed::run_coil_pass(a, ax, s);
  else
    mixed::run_image_pass(a, ax, s);
  return true;
}
}  // namespace

bool mixed_static_pass(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return pass_for<4, 4>(a, x, s) ||     // 16
         pass_for<4, 8>(a, x, s) ||     // 32
         pass_for<8, 8>(a, x, s) ||     // 64
         pass_for<8, 16>(a, x, s) ||    // 128
         pass_for<12, 16>(a, x, s) ||   // 192
         pass_for<16, 16>(a, x, s);     // 256
}

}  // namespace nrs
