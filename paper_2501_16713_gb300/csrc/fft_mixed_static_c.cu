// The mixed-radix passes with compile-time radices for axis lengths 144, 160 and 176 at sigma 2
// (rule and timings: fft_mixed_static.cu; a translation unit of its own to compile in
// parallel).
#include "fft_mixed_kernels.cuh"

namespace nrs {

bool mixed_static_pass_c(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return mixed::pass_for<12, 12>(a, x, s) ||  // 144
         mixed::pass_for<10, 16>(a, x, s) ||  // 160
         mixed::pass_for<16, 11>(a, x, s);  // 176
}

}  // namespace nrs
