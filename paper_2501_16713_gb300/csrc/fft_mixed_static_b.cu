// The mixed-radix passes with compile-time radices for axis lengths 96, 112 and 128 at sigma 2
// (rule and timings: fft_mixed_static.cu; a translation unit of its own to compile in
// parallel).
#include "fft_mixed_kernels.cuh"

namespace nrs {

bool mixed_static_pass_b(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return mixed::pass_for<8, 12>(a, x, s) ||  // 96
         mixed::pass_for<8, 14>(a, x, s) ||  // 112
         mixed::pass_for<8, 16>(a, x, s);  // 128
}

}  // namespace nrs
