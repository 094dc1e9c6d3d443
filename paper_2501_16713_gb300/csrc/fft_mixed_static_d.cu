// The mixed-radix passes with compile-time radices for axis lengths 192 and 208 at sigma 2
// (rule and timings: fft_mixed_static.cu; a translation unit of its own to compile in
// parallel).
#include "fft_mixed_kernels.cuh"

namespace nrs {

bool mixed_static_pass_d(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return mixed::pass_for<12, 16>(a, x, s) ||  // 192
         mixed::pass_for<16, 13>(a, x, s);  // 208
}

}  // namespace nrs
