// The mixed-radix passes (fft_mixed_kernels.cuh) with compile-time radices: every
// axis length that is a multiple of 16, up to 256, at sigma 2 (R S as factor_double,
// fft_mixed.cu, chooses them).  Other even lengths, and all rational or larger sigma,
// take run-time radices, whose one body per kernel holds radices up to 16 and spills.
// Run-time against compile-time radices, ms: four coil grids both ways 64^3 0.105 / 0.084,
// 80^3 0.217 / 0.152, 96^3 0.320 / 0.247, 144^3 0.849 / 0.676, 176^3 1.64 / 1.42, 192^3 1.89 /
// 1.59, 240^3 3.50 / 3.06; T and T^H of one image 32^3 0.040 / 0.030, 48^3 0.049 / 0.042, 96^3
// 0.133 / 0.091, 144^3 0.393 / 0.287, 208^3 1.01 / 0.79.
#include "fft_mixed_kernels.cuh"

namespace nrs {

bool mixed_static_pass_b(const MixPass& a, const MixAxis& x, cudaStream_t s);
bool mixed_static_pass_c(const MixPass& a, const MixAxis& x, cudaStream_t s);
bool mixed_static_pass_d(const MixPass& a, const MixAxis& x, cudaStream_t s);
bool mixed_static_pass_e(const MixPass& a, const MixAxis& x, cudaStream_t s);

bool mixed_static_pass(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  return mixed::pass_for<4, 4>(a, x, s) ||  // 16
         mixed::pass_for<4, 8>(a, x, s) ||  // 32
         mixed::pass_for<6, 8>(a, x, s) ||  // 48
         mixed::pass_for<8, 8>(a, x, s) ||  // 64
         mixed::pass_for<8, 10>(a, x, s) ||  // 80
         mixed_static_pass_b(a, x, s) || mixed_static_pass_c(a, x, s) ||
         mixed_static_pass_d(a, x, s) || mixed_static_pass_e(a, x, s);
}

}  // namespace nrs
