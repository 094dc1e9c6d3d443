// The mixed-radix passes with compile-time radices for axis lengths 224, 240 and 256 at sigma 2
// (rule and timings: fft_mixed_static.cu; a translation unit of its own to compile in
// parallel).
#include "fft_mixed_kernels.cuh"

namespace nrs {

bool mixed_static_pass_e(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return mixed::pass_for<14, 16>(a, x, s) ||  // 224
         mixed::pass_for<16, 15>(a, x, s) ||  // 240
         mixed::pass_for<16, 16>(a, x, s);  // 256
}

}  // namespace nrs
