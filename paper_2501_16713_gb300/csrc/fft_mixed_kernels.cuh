// Passes of the mixed-radix transforms (fft_mixed.cuh) over the coil grids
// (fan-out and coil combination fused) and over the image-space grid (the N^3
// DFTs and the deapodization of T and T^H fused), as kernels templated on the
// axis policy of the transformed axis, with their launchers.
//
// Structure as in fft_pruned.cu: the forward transform of a coil grid runs
// along x over the N0 N1 data rows, along y over the N0 data planes and along z
// over every (y, x) column, loading only data; the adjoint runs z, y, x and
// stores only data.  Compact intermediates T1[slot][i0][i1][x] and
// T2[slot][i0][y][x].
//
// Image space: T's upsampling F_G^-1 (Z / C) F_N is a product of one operator
// per axis (length-N DFT, division by the axis' kernel transform,
// zero-padding, length-G inverse DFT), so each pass applies its axis' whole
// operator in shared memory and the separate N^3 transforms disappear; T^H
// likewise with the adjoint operators.
//
// Bound: HBM traffic of the compact intermediates, with the issue slots of the
// z passes close behind (at 384 points fwd_y 57 %, fwd_z 49 %, inv_z 51 % of the
// DRAM rate with 41-46 instructions per element).  16 lanes per CTA make 128-byte
// rows of every access.  Replaced cuFFT with separate fan-out, combination,
// padding and N^3 kernels: 16 coil grids of 384^3 forward 8.55 -> 3.06 ms, 16 of
// 512^3 adjoint 16.9 -> 8.2 ms, three phases of 5 grids of 168 x 120 x 264 both
// ways 1.94 -> 0.81 ms, T's 384^3 image grid 0.81 -> 0.31 ms a direction, 64^3
// images 0.078 -> 0.045 ms and 32^3 ones 0.060 -> 0.030 ms for T and T^H.
#pragma once

#include "fft_mixed.cuh"

namespace nrs {
namespace mixed {

struct Dims {
  int n0, n1, n2, g0, g1, g2;
  int C;
};

// ---- coil grids -------------------------------------------------------------

// T1[slot][i0][i1][:] = DFT_x of S_c m_j / C3 on the data rows, all coils of
// phase jj.  CTA: (block of 16 rows i1, i0, jj).
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_fwd_x_kernel(
    Dims g, AX ax, const float* __restrict__ dtab, const float2* __restrict__ smaps,
    const float2* __restrict__ m, float2* __restrict__ t1) {
  extern __shared__ float2 sy[];
  const int rb = blockIdx.x * kLanes, i0 = blockIdx.y, jj = blockIdx.z;
  const int last = g.n1 - 1 - rb;  // lanes past it repeat its row (no branch) and store nothing
  const long long nvox = (long long)g.n0 * g.n1 * g.n2;
  const int h = g.n2 / 2;
  const float d0 = __ldg(dtab + i0);
  const float* d1 = dtab + g.n0;
  const float* d2 = d1 + g.n1;
  const float2* mrow = m + jj * nvox + ((long long)i0 * g.n1 + rb) * g.n2;
#pragma unroll 1
  for (int c = 0; c < g.C; ++c) {
    const float2* srow = smaps + c * nvox + ((long long)i0 * g.n1 + rb) * g.n2;
    float2* dst = t1 + (((long long)jj * g.C + c) * g.n0 + i0) * g.n1 * g.g2 + (long long)rb * g.g2;
    auto ld = [&](int lane, int n) -> float2 {
      const int r = min(lane, last), i2 = swap_half(n, h), v = r * g.n2 + i2;
      const float2 mv = __ldg(mrow + v), sv = __ldg(srow + v);
      const float w = d0 * __ldg(d1 + rb + r) * __ldg(d2 + i2);
      return make_float2((sv.x * mv.x - sv.y * mv.y) * w, (sv.x * mv.y + sv.y * mv.x) * w);
    };
    auto st = [&](int lane, int q, auto k2, float2 v) {
      if (lane <= last) dst[lane * g.g2 + q + ax.step() * decltype(k2)::value] = v;
    };
    ax.template pad<true>(sy, ld, st);
  }
}

// Union of a CTA's two 8-point tile columns (x0 and x0 + 8): words of 32 tiles
// along the transformed axis, in shared memory (mask: [word][nt_row][nt2], row
// `row`).  Returns false when neither column has a tile.
__device__ __forceinline__ bool load_masks(const uint32_t* __restrict__ mask, int nt, int nt_row,
                                           int row, int nt2, int x0, uint32_t (*sm)[4]) {
  uint32_t v = 0;
  if (threadIdx.x < 8) {
    const int side = threadIdx.x >> 2, w = threadIdx.x & 3;
    const int tx = (x0 >> 3) + side;
    if (w < (nt + 31) / 32 && tx < nt2) v = __ldg(mask + ((long long)w * nt_row + row) * nt2 + tx);
    sm[side][w] = v;
  }
  return __syncthreads_or(v != 0u) != 0;
}

// Tile test of grid position base + step * K of a column: with a compile-time
// step the lane's mask words are in a register (at most 64 tiles: G <= 512)
// and, when the step is a multiple of 8, the bit is found by constant shifts.
template <class AX>
struct TileMask {
  const uint32_t* words;
  unsigned long long bits;
  __device__ __forceinline__ TileMask(const uint32_t* w) : words(w), bits(0) {
    if constexpr (AX::kMaskShift) bits = w[0] | (unsigned long long)w[1] << 32;
  }
  template <int K>
  __device__ __forceinline__ bool has(const AX& ax, int base, std::integral_constant<int, K>) const {
    if constexpr (AX::kMaskShift) {
      if (ax.step() % 8 == 0) return ((bits >> (base >> 3)) >> (ax.step() / 8 * K)) & 1ull;
      return (bits >> ((base + ax.step() * K) >> 3)) & 1ull;
    } else {
      const int p = base + ax.step() * K;
      return (words[p >> 8] >> ((p >> 3) & 31)) & 1u;
    }
  }
};

// Column passes: lane = 16 consecutive x; lanes past the row's end repeat its
// last column (no branch) and store nothing.  T2 columns (y, x) whose tile
// column has no tile of the union hold nothing: the y pass does not store
// (forward) or load (adjoint) them, the z pass skips them.

// T2[slot][i0][:][x] = DFT_y of T1[slot][i0][data rows][x].  CTA: (16 x, i0, slot).
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kPad) mix_fwd_y_kernel(Dims g, AX ax,
                                                                const uint32_t* __restrict__ anymask,
                                                                const float2* __restrict__ t1,
                                                                float2* __restrict__ t2) {
  extern __shared__ float2 sy[];
  __shared__ uint32_t sm[2][4];
  const int x0 = blockIdx.x * kLanes, h = g.n1 / 2, ln = threadIdx.x & (kLanes - 1);
  if (!load_masks(anymask, (g.g1 + 7) >> 3, 1, 0, (g.g2 + 7) >> 3, x0, sm)) return;
  const long long row = (long long)blockIdx.z * g.n0 + blockIdx.y;
  const bool in = x0 + ln < g.g2;
  const TileMask<AX> mask(sm[ln >> 3]);
  const float2* src = t1 + row * g.n1 * g.g2 + min(x0 + ln, g.g2 - 1);
  float2* dst = t2 + row * g.g1 * g.g2 + x0 + ln;
  auto ld = [&](int, int n) { return __ldg(src + swap_half(n, h) * g.g2); };
  auto st = [&](int, int q, auto k2, float2 v) {
    if (in && mask.has(ax, q, k2)) dst[(q + ax.step() * decltype(k2)::value) * g.g2] = v;
  };
  ax.template pad<false>(sy, ld, st);
}

// grid[slot][:][y][x] = DFT_z of T2[slot][data planes][y][x]; tiles outside the
// union over phases are not stored.  CTA: (16 x, y, slot).
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kPad) mix_fwd_z_kernel(
    Dims g, AX ax, const uint32_t* __restrict__ colmask, const float2* __restrict__ t2,
    float2* __restrict__ grid) {
  extern __shared__ float2 sy[];
  __shared__ uint32_t sm[2][4];
  const int x0 = blockIdx.x * kLanes, y = blockIdx.y, h = g.n0 / 2;
  const int ln = threadIdx.x & (kLanes - 1);
  if (!load_masks(colmask, (g.g0 + 7) >> 3, (g.g1 + 7) >> 3, y >> 3, (g.g2 + 7) >> 3, x0, sm)) return;
  const long long plane = (long long)g.g1 * g.g2, slot = blockIdx.z;
  const bool in = x0 + ln < g.g2;
  const TileMask<AX> mask(sm[ln >> 3]);
  const float2* src = t2 + slot * g.n0 * plane + (long long)y * g.g2 + min(x0 + ln, g.g2 - 1);
  float2* dst = grid + slot * g.g0 * plane + (long long)y * g.g2 + x0 + ln;
  auto ld = [&](int, int n) { return __ldg(src + swap_half(n, h) * plane); };
  auto st = [&](int, int q, auto k2, float2 v) {
    if (in && mask.has(ax, q, k2)) dst[(q + ax.step() * decltype(k2)::value) * plane] = v;
  };
  ax.template pad<false>(sy, ld, st);
}

// T2[slot][i0][y][x] = inverse DFT_z of grid[slot][:][y][x] at the data planes;
// tiles outside the union hold zeros and are not loaded.
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_inv_z_kernel(
    Dims g, AX ax, const uint32_t* __restrict__ colmask, const float2* __restrict__ grid,
    float2* __restrict__ t2) {
  extern __shared__ float2 sy[];
  __shared__ uint32_t sm[2][4];
  const int x0 = blockIdx.x * kLanes, y = blockIdx.y, h = g.n0 / 2;
  const int ln = threadIdx.x & (kLanes - 1);
  if (!load_masks(colmask, (g.g0 + 7) >> 3, (g.g1 + 7) >> 3, y >> 3, (g.g2 + 7) >> 3, x0, sm)) return;
  const long long plane = (long long)g.g1 * g.g2, slot = blockIdx.z;
  const bool in = x0 + ln < g.g2;
  const TileMask<AX> mask(sm[ln >> 3]);
  const float2* src = grid + slot * g.g0 * plane + (long long)y * g.g2 + min(x0 + ln, g.g2 - 1);
  float2* dst = t2 + slot * g.n0 * plane + (long long)y * g.g2 + x0 + ln;
  auto ld = [&](int, int j, auto n1) -> float2 {
    float2 v = make_float2(0.f, 0.f);
    if (mask.has(ax, j, n1)) v = __ldg(src + (j + ax.step() * decltype(n1)::value) * plane);
    return make_float2(v.x, -v.y);
  };
  auto st = [&](int, int n, float2 v) {
    if (in) dst[swap_half(n, h) * plane] = make_float2(v.x, -v.y);
  };
  ax.template crop<false>(sy, ld, st);
}

// T1[slot][i0][i1][x] = inverse DFT_y of T2[slot][i0][:][x] at the data rows.
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_inv_y_kernel(Dims g, AX ax,
                                                                const uint32_t* __restrict__ anymask,
                                                                const float2* __restrict__ t2,
                                                                float2* __restrict__ t1) {
  extern __shared__ float2 sy[];
  __shared__ uint32_t sm[2][4];
  const int x0 = blockIdx.x * kLanes, h = g.n1 / 2, ln = threadIdx.x & (kLanes - 1);
  load_masks(anymask, (g.g1 + 7) >> 3, 1, 0, (g.g2 + 7) >> 3, x0, sm);
  const long long row = (long long)blockIdx.z * g.n0 + blockIdx.y;
  const bool in = x0 + ln < g.g2;
  const TileMask<AX> mask(sm[ln >> 3]);
  const float2* src = t2 + row * g.g1 * g.g2 + min(x0 + ln, g.g2 - 1);
  float2* dst = t1 + row * g.n1 * g.g2 + x0 + ln;
  auto ld = [&](int, int j, auto n1) -> float2 {
    float2 v = make_float2(0.f, 0.f);
    if (mask.has(ax, j, n1)) v = __ldg(src + (j + ax.step() * decltype(n1)::value) * g.g2);
    return make_float2(v.x, -v.y);
  };
  auto st = [&](int, int n, float2 v) {
    if (in) dst[swap_half(n, h) * g.g2] = make_float2(v.x, -v.y);
  };
  ax.template crop<false>(sy, ld, st);
}

// w[jj][i0][i1][i2] = C3^-1 sum_c conj(S_c) (inverse DFT_x of T1[slot][i0][i1][:])
// at the data positions, coils summed in order (sums in shared memory: every
// output belongs to one thread).  CTA: (block of 16 rows i1, i0, jj).
template <class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_inv_x_kernel(
    Dims g, AX ax, int acc_at, const float* __restrict__ dtab, const float2* __restrict__ smaps,
    const float2* __restrict__ t1, float2* __restrict__ w) {
  extern __shared__ float2 sy[];
  float2* acc = sy + acc_at;  // [16][n2]
  const int rb = blockIdx.x * kLanes, i0 = blockIdx.y, jj = blockIdx.z;
  const int last = g.n1 - 1 - rb;  // lanes past it repeat its row (no branch) and store nothing
  const long long nvox = (long long)g.n0 * g.n1 * g.n2;
  const int h = g.n2 / 2;
#pragma unroll 1
  for (int c = 0; c < g.C; ++c) {
    const long long slot = (long long)jj * g.C + c;
    const float2* src = t1 + (slot * g.n0 + i0) * g.n1 * g.g2 + (long long)rb * g.g2;
    const float2* srow = smaps + c * nvox + ((long long)i0 * g.n1 + rb) * g.n2;
    auto ld = [&](int lane, int j, auto n1) -> float2 {
      const float2 v =
          __ldg(src + min(lane, last) * g.g2 + j + ax.step() * decltype(n1)::value);
      return make_float2(v.x, -v.y);
    };
    auto st = [&](int lane, int n, float2 v) {
      const int i2 = swap_half(n, h), o = lane * g.n2 + i2;
      const float2 s = __ldg(srow + min(lane, last) * g.n2 + i2);
      float2 a = c == 0 ? make_float2(0.f, 0.f) : acc[o];
      // conj(s) * conj(v)
      a.x = fmaf(s.x, v.x, fmaf(-s.y, v.y, a.x));
      a.y = fmaf(-s.x, v.y, fmaf(-s.y, v.x, a.y));
      acc[o] = a;
    };
    ax.template crop<true>(sy, ld, st);
  }
  const float d0 = __ldg(dtab + i0);
  float2* dst = w + jj * nvox + ((long long)i0 * g.n1 + rb) * g.n2;
  for (int o = threadIdx.x; o < min(kLanes, last + 1) * g.n2; o += blockDim.x) {
    const int lane = o / g.n2, i2 = o - lane * g.n2;
    const float dep = d0 * __ldg(dtab + g.n0 + rb + lane) * __ldg(dtab + g.n0 + g.n1 + i2);
    dst[o] = make_float2(acc[o].x * dep, acc[o].y * dep);
  }
}

// ---- image-space grid -----------------------------------------------------------

// One axis of T's upsampling (UP): out = F_G^-1 Z (scale / C) F_N in for the
// CTA's 16 lanes, or of its adjoint: out = F_N^-1 (scale / C) Z^H F_G in
// (unnormalised transforms).  sa: the transforms' buffer; sb: the spectrum
// between them, in DFT order.
template <bool UP, bool ROWS, class AX, class Ld, class St>
__device__ __forceinline__ void axis_operator(const AX& ax, float2* sa, float2* sb,
                                              const float* __restrict__ dea, float scale,
                                              const Ld& ld, const St& st) {
  const int n = ax.N(), h = n / 2;
  auto at = [&](int lane, int f) { return ROWS ? lane * (n + 1) + f : f * kLanes + lane; };
  auto keep = [&](int lane, int f, float2 v) {
    const float d = __ldg(dea + swap_half(f, h)) * scale;
    sb[at(lane, f)] = make_float2(v.x * d, -v.y * d);
  };
  auto spectrum = [&](int lane, int f) { return sb[at(lane, f)]; };
  if constexpr (UP) {
    ax.template full<ROWS>(sa, ld, keep);
    ax.template pad<ROWS>(sa, spectrum, [&](int lane, int q, auto k2, float2 v) {
      st(lane, q + ax.step() * decltype(k2)::value, make_float2(v.x, -v.y));
    });
  } else {
    ax.template crop<ROWS>(sa, [&](int lane, int j, auto n1) {
      return ld(lane, j + ax.step() * decltype(n1)::value);
    }, keep);
    ax.template full<ROWS>(sa, spectrum, [&](int lane, int k, float2 v) {
      st(lane, k, make_float2(v.x, -v.y));
    });
  }
}

// x pass, rows of N values <-> rows of G values; CTA: 16 rows of `rows`.
template <bool UP, class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_img_x_kernel(
    int rows, AX ax, int sb_at, const float* __restrict__ dea, float scale,
    const float2* __restrict__ in, float2* __restrict__ out) {
  extern __shared__ float2 sa[];
  const int r0 = blockIdx.x * kLanes, last = rows - 1 - r0;
  const int li = UP ? ax.N() : ax.G(), lo = UP ? ax.G() : ax.N();
  const float2* src = in + (long long)r0 * li;
  float2* dst = out + (long long)r0 * lo;
  axis_operator<UP, true>(
      ax, sa, sa + sb_at, dea, scale,
      [&](int lane, int p) { return __ldg(src + min(lane, last) * li + p); },
      [&](int lane, int k, float2 v) {
        if (lane <= last) dst[lane * lo + k] = v;
      });
}

// y and z passes: lanes are 16 of the `width` contiguous columns of outer
// block blockIdx.y, elements `width` apart.
template <bool UP, class AX>
__global__ void __launch_bounds__(kThreads, AX::kCrop) mix_img_col_kernel(
    long long width, AX ax, int sb_at, const float* __restrict__ dea,
    const float2* __restrict__ in, float2* __restrict__ out) {
  extern __shared__ float2 sa[];
  const long long c0 = (long long)blockIdx.x * kLanes;
  const int li = UP ? ax.N() : ax.G(), lo = UP ? ax.G() : ax.N();
  const long long col = c0 + (threadIdx.x & (kLanes - 1));
  const bool ok = col < width;
  const float2* src = in + (long long)blockIdx.y * li * width + min(col, width - 1);
  float2* dst = out + (long long)blockIdx.y * lo * width + col;
  axis_operator<UP, false>(
      ax, sa, sa + sb_at, dea, 1.0f,
      [&](int, int p) { return __ldg(src + p * width); },
      [&](int, int k, float2 v) {
        if (ok) dst[k * width] = v;
      });
}

// ---- launchers, one axis each --------------------------------------------------

// Shared-memory values of an axis' transform buffer.
template <class Len>
int buffer_elems(const DoubleAxis<Len>& a, bool rows) {
  const int r = a.l.r, s = a.l.s;
  return kLanes * (rows ? std::max(2 * r * (s | 1), s * (2 * r + 1)) : 2 * r * s);
}
inline int buffer_elems(const GeneralAxis& a, bool rows) {
  return kLanes * (rows ? std::max(a.g.r1 * (a.g.s | 1), a.n.L > 0 ? a.n.r1 * (a.n.s | 1) : 0)
                        : a.g.L);
}
// butterflies per lane of the steps of a G transform (and of an N one: image)
template <class Len>
int steps_of(const DoubleAxis<Len>& a, bool image, int* nb) {
  nb[0] = a.l.s;
  nb[1] = 2 * a.l.r;
  nb[2] = a.l.s;
  nb[3] = a.l.r;
  return image ? 4 : 2;
}
inline int steps_of(const GeneralAxis& a, bool image, int* nb) {
  int k = 0;
  for (const MixLen* f : {&a.g, &a.n}) {
    if (f == &a.n && !image) break;
    nb[k++] = f->s;
    nb[k++] = f->r1 * f->r2;
    if (f->r2 > 1) nb[k++] = f->r1 * f->r3;
  }
  return k;
}
// Threads of a CTA.  Shared memory allows only two to four CTAs per SM, so a CTA has
// to bring the warps: 256 where that leaves at most a quarter of the thread turns
// over the steps idle (384-point coil passes, 16 x (16, 24) butterflies: 3.06 ms for
// 16 grids against 3.38 with 128 threads and none idle), else the largest multiple of
// 32 that leaves at most 15 % idle, else the one that leaves the fewest.  T's
// 384-point passes: 64 threads, none idle and 6 warps per SM, 0.41 ms; 128, 0.32;
// 256, 0.31.  With 25 % allowed below 256 threads too the N = 64 passes went from
// 0.26 to 0.28 ms and run-time radices (168 x 120 x 264) from 0.81 to 0.89.
template <class AX>
int threads_for(const AX& ax, bool image) {
  int nb[6], work = 0;
  const int k = steps_of(ax, image, nb);
  for (int i = 0; i < k; ++i) work += kLanes * nb[i];
  int best = 64, best_turns = 1 << 30;
  for (int t = 64; t <= kThreads; t += 32) {
    int turns = 0;
    for (int i = 0; i < k; ++i) turns += (kLanes * nb[i] + t - 1) / t * t;
    if (100 * turns <= (t == kThreads ? 125 : 115) * work || turns < best_turns) {
      best_turns = turns;
      best = t;
    }
  }
  return best;
}

// Launch geometry of one pass: threads, dynamic shared memory, and the offset
// (in values) of the second shared buffer.
struct PassShape {
  int threads, second;
  size_t bytes;
};
template <class AX>
PassShape pass_shape(const AX& ax, bool rows, bool image, int extra) {
  PassShape p;
  p.threads = threads_for(ax, image);
  p.second = buffer_elems(ax, rows);
  p.bytes = (size_t(p.second) + size_t(kLanes) * extra) * sizeof(float2);
  return p;
}

// Launch (or, at plan time, configure) a pass' kernel.
template <class K, class... Args>
void launch_pass(const MixPass& a, K* kernel, dim3 grid, const PassShape& sh, cudaStream_t s,
                 Args... args) {
  if (a.configure)
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kMixedMaxSmem));
  else
    kernel<<<grid, sh.threads, sh.bytes, s>>>(args...);
}

inline unsigned lane_blocks(long long n) { return unsigned((n + kLanes - 1) / kLanes); }

// Coil grids: pass 0 x, 1 y, 2 z of the forward transform, 3 z, 4 y, 5 x of the inverse.
template <class AX>
void run_coil_pass(const MixPass& a, const AX& ax, cudaStream_t s) {
  const Geo& g = *a.geo;
  const Dims d{g.n0, g.n1, g.n2, g.g0, g.g1, g.g2, a.C};
  const unsigned slots = unsigned(a.C * a.nph);
  const dim3 gx(lane_blocks(g.n1), g.n0, a.nph), gy(lane_blocks(g.g2), g.n0, slots),
      gz(lane_blocks(g.g2), g.g1, slots);
  const auto* in = static_cast<const float2*>(a.in);
  auto* out = static_cast<float2*>(a.out);
  const auto* sm = reinterpret_cast<const float2*>(a.smaps);
  const PassShape sh = pass_shape(ax, a.pass == 0 || a.pass == 5, false, a.pass == 5 ? g.n2 : 0);
  switch (a.pass) {
    case 0: launch_pass(a, &mix_fwd_x_kernel<AX>, gx, sh, s, d, ax, a.deapod, sm, in, out); break;
    case 1: launch_pass(a, &mix_fwd_y_kernel<AX>, gy, sh, s, d, ax, a.colmask, in, out); break;
    case 2: launch_pass(a, &mix_fwd_z_kernel<AX>, gz, sh, s, d, ax, a.colmask, in, out); break;
    case 3: launch_pass(a, &mix_inv_z_kernel<AX>, gz, sh, s, d, ax, a.colmask, in, out); break;
    case 4: launch_pass(a, &mix_inv_y_kernel<AX>, gy, sh, s, d, ax, a.colmask, in, out); break;
    default:
      launch_pass(a, &mix_inv_x_kernel<AX>, gx, sh, s, d, ax, sh.second, a.deapod, sm, in, out);
  }
}

// Image-space grid: pass 6 x, 7 y, 8 z of T's upsampling, 9 z, 10 y, 11 x of its adjoint.
template <class AX>
void run_image_pass(const MixPass& a, const AX& ax, cudaStream_t s) {
  const Geo& g = *a.geo;
  const auto* in = static_cast<const float2*>(a.in);
  auto* out = static_cast<float2*>(a.out);
  const bool rows = a.pass == 6 || a.pass == 11;
  const PassShape sh = pass_shape(ax, rows, true, ax.N() + (rows ? 1 : 0));
  const long long plane = (long long)g.g1 * g.g2, width = g.g2;
  const int nrows = g.n0 * g.n1;
  const dim3 gx(lane_blocks(nrows)), gy(lane_blocks(width), g.n0), gz(lane_blocks(plane));
  const float scale = float(1.0 / double(g.nvox));
  const float *d1 = a.deapod + g.n0, *d2 = d1 + g.n1;
  switch (a.pass) {
    case 6:
      launch_pass(a, &mix_img_x_kernel<true, AX>, gx, sh, s, nrows, ax, sh.second, d2, scale, in, out);
      break;
    case 7:
      launch_pass(a, &mix_img_col_kernel<true, AX>, gy, sh, s, width, ax, sh.second, d1, in, out);
      break;
    case 8:
      launch_pass(a, &mix_img_col_kernel<true, AX>, gz, sh, s, plane, ax, sh.second, a.deapod, in, out);
      break;
    case 9:
      launch_pass(a, &mix_img_col_kernel<false, AX>, gz, sh, s, plane, ax, sh.second, a.deapod, in, out);
      break;
    case 10:
      launch_pass(a, &mix_img_col_kernel<false, AX>, gy, sh, s, width, ax, sh.second, d1, in, out);
      break;
    default:
      launch_pass(a, &mix_img_x_kernel<false, AX>, gx, sh, s, nrows, ax, sh.second, d2, scale, in, out);
  }
}

// The pass with compile-time radices; false: the axis has other ones.
template <int R, int S>
bool pass_for(const MixPass& a, const MixAxis& x, cudaStream_t s) {
  if (x.R != R || x.S != S) return false;
  DoubleAxis<StLen<R, S>> ax;
  ax.l.tw = x.tw_g;
  if (a.pass < 6)
    run_coil_pass(a, ax, s);
  else
    run_image_pass(a, ax, s);
  return true;
}

}  // namespace mixed
}  // namespace nrs
