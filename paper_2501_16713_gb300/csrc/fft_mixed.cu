// Mixed-radix transforms of the coil grids and of the image-space grid: choice
// of the axis policies and the pass sequences (kernels: fft_mixed_kernels.cuh,
// instantiated in fft_mixed_static.cu, fft_mixed_rt_*.cu and fft_mixed_gen_*.cu).
#include "fft_mixed.cuh"

namespace nrs {

using namespace mixed;

namespace {

// Radices of length L: two when both can be at most 16 (fewer exchanges), else
// three with a middle one of at most 8; the most balanced choice.
bool factor(int L, MixLen* f) {
  int best = 1 << 30;
  MixLen m{};
  m.L = L;
  for (int r1 = 2; r1 <= 16; ++r1) {
    if (L % r1) continue;
    for (int r2 = 1; r2 <= 8; ++r2) {
      if ((L / r1) % r2) continue;
      const int r3 = L / r1 / r2;
      if (r3 < 2 || r3 > 16) continue;
      const int cost = (r2 > 1 ? 1000 + r2 * r2 : 0) + r1 * r1 + r3 * r3;
      if (cost < best) {
        best = cost;
        m.r1 = r1;
        m.r2 = r2;
        m.r3 = r3;
      }
    }
  }
  if (best == 1 << 30) return false;
  m.s = m.r2 * m.r3;
  m.m_s = mix_magic(m.s);
  m.m_13 = mix_magic(m.r1 * m.r3);
  m.m_12 = mix_magic(m.r1 * m.r2);
  m.m_r3 = mix_magic(m.r3);
  m.m_r1 = mix_magic(m.r1);
  *f = m;
  return true;
}

// N = R S, R even, both at most 16: the most balanced choice, R <= S on ties
// of the sum (the radix-2R steps hold two radix-R butterflies)
bool factor_double(int N, int* R, int* S) {
  int best = 1 << 30;
  for (int r = 2; r <= 16; r += 2) {
    if (N % r || N / r < 2 || N / r > 16) continue;
    const int s = N / r, cost = 2 * (r * r + s * s) + (r > s);
    if (cost < best) {
      best = cost;
      *R = r;
      *S = s;
    }
  }
  return best < (1 << 30);
}

void axis_pass(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  const bool coil = a.pass < 6;
  if (x.R > 0) {
    if (mixed_static_pass(a, x, s)) return;
    coil ? mixed_rt_coil_pass(a, x, s) : mixed_rt_image_pass(a, x, s);
  } else {
    coil ? mixed_gen_coil_pass(a, x, s) : mixed_gen_image_pass(a, x, s);
  }
}

}  // namespace

bool mix_axis(int N, int G, MixAxis* out) {
  MixAxis x{};
  x.N = N;
  x.G = G;
  if (G == 2 * N && factor_double(N, &x.R, &x.S)) {
    *out = x;
    return true;
  }
  if (!factor(G, &x.g) || !factor(N, &x.n)) return false;
  *out = x;
  return true;
}

size_t mixed_max_smem(const MixAxis* ax) {
  size_t most = 0;
  for (int a = 0; a < 3; ++a) {
    const MixAxis& x = ax[a];
    const size_t buf =
        x.R > 0 ? size_t(kLanes) * std::max(2 * x.R * (x.S | 1), x.S * (2 * x.R + 1))
                : size_t(kLanes) * std::max(x.g.r1 * (x.g.s | 1), x.n.r1 * (x.n.s | 1));
    most = std::max(most, (std::max(buf, size_t(kLanes) * x.G) + size_t(kLanes) * (x.N + 1)) *
                              sizeof(float2));
  }
  return most;
}

cudaError_t configure_mixed(const Geo& g, const MixAxis* ax) {
  const int axis[12] = {2, 1, 0, 0, 1, 2, 2, 1, 0, 0, 1, 2};
  for (int k = 0; k < 12; ++k)
    axis_pass({&g, k, 1, 1, nullptr, nullptr, nullptr, nullptr, nullptr, true}, ax[axis[k]], nullptr);
  return cudaGetLastError();
}

int launch_mixed_forward(const Geo& g, const MixAxis* ax, int C, int nph, const uint32_t* colmask,
                         const uint32_t* anymask, const float* deapod, const nrsense_c64* smaps, const nrsense_c64* m,
                         void* t1, void* t2, void* grid, cudaStream_t s) {
  axis_pass({&g, 0, C, nph, colmask, deapod, smaps, m, t1}, ax[2], s);
  axis_pass({&g, 1, C, nph, anymask, deapod, smaps, t1, t2}, ax[1], s);
  axis_pass({&g, 2, C, nph, colmask, deapod, smaps, t2, grid}, ax[0], s);
  return 3;
}

int launch_mixed_inverse(const Geo& g, const MixAxis* ax, int C, int nph, const uint32_t* colmask,
                         const uint32_t* anymask, const float* deapod, const nrsense_c64* smaps, const void* grid, void* t2,
                         void* t1, nrsense_c64* w, cudaStream_t s) {
  axis_pass({&g, 3, C, nph, colmask, deapod, smaps, grid, t2}, ax[0], s);
  axis_pass({&g, 4, C, nph, anymask, deapod, smaps, t2, t1}, ax[1], s);
  axis_pass({&g, 5, C, nph, colmask, deapod, smaps, t1, w}, ax[2], s);
  return 3;
}

int launch_mixed_image_up(const Geo& g, const MixAxis* ax, const float* deapod,
                          const nrsense_c64* x, void* t1, void* t2, nrsense_c64* u,
                          cudaStream_t s) {
  axis_pass({&g, 6, 1, 1, nullptr, deapod, nullptr, x, t1}, ax[2], s);
  axis_pass({&g, 7, 1, 1, nullptr, deapod, nullptr, t1, t2}, ax[1], s);
  axis_pass({&g, 8, 1, 1, nullptr, deapod, nullptr, t2, u}, ax[0], s);
  return 3;
}

int launch_mixed_image_down(const Geo& g, const MixAxis* ax, const float* deapod,
                            const nrsense_c64* u, void* t2, void* t1, nrsense_c64* x,
                            cudaStream_t s) {
  axis_pass({&g, 9, 1, 1, nullptr, deapod, nullptr, u, t2}, ax[0], s);
  axis_pass({&g, 10, 1, 1, nullptr, deapod, nullptr, t2, t1}, ax[1], s);
  axis_pass({&g, 11, 1, 1, nullptr, deapod, nullptr, t1, x}, ax[2], s);
  return 3;
}

}  // namespace nrs
