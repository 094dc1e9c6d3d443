// Shared device-side definitions of the nonrigid SENSE library (sm_103a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/nrsense.h"

namespace nrs {

// Coefficients of the per-tap kernel polynomials (see kb_host.cu):
// weight of tap t for fractional offset f in [0, 1) is
//   c(f + W/2 - 1 - t) ~= sum_k c[k][t] * s^k,  s = 2f - 1.
// c: the taps of one power are neighbours, so that two taps' coefficients load and
// multiply as a pair; t: the powers of one tap, for the kernels that the compiler
// schedules better that way (kernel_weights_by_tap).
constexpr int kNumCoef = 10;
constexpr int kMaxWidth = 6;

struct alignas(8) KernelCoefs {
  float c[kNumCoef][kMaxWidth];
  float t[kMaxWidth][kNumCoef];
};

// Per-axis geometry passed by value to every kernel.
struct Geo {
  int n0, n1, n2;     // image size
  int g0, g1, g2;     // oversampled grid size
  int osf;
  long long nvox;     // n0*n1*n2
  long long ngrid;    // g0*g1*g2
};

// A point (k-space sample or displaced voxel) after plan-time preprocessing:
// fractional offsets of the first tap per axis and the first tap's grid index
// packed 10 bits per axis (axis 0 in the high bits).
__host__ __device__ inline uint32_t pack_base(int b0, int b1, int b2) {
  return (uint32_t(b0) << 20) | (uint32_t(b1) << 10) | uint32_t(b2);
}
__host__ __device__ inline void unpack_base(uint32_t p, int& b0, int& b1, int& b2) {
  b0 = int(p >> 20);
  b1 = int((p >> 10) & 1023u);
  b2 = int(p & 1023u);
}

// One block of output-stationary spreading work: the points listed in
// list[begin, end) are spread into grid tile `tile`; slot < 0 writes the tile
// to the grid directly, slot >= 0 writes a partial tile to scratch slot
// `slot` (heavy tiles are split into several items and reduced afterwards).
// The same record describes interpolation work (sorted point range of a tile).
struct SpreadItem {
  int32_t tile;
  int32_t begin;
  int32_t end;
  int32_t slot;
};

// Offsets (relative to the item's begin) of the list entries of each
// first-tap plane offset r0 in (-W, T), stored per spreading item:
// bins[b] = first entry with r0 + W - 1 >= b, b = 0 .. W + T - 1.
constexpr int kMaxBins = kMaxWidth + 16;

// Up to kMaxChunkPhases motion states are processed by one launch.  The
// per-phase point data stay in their own arrays; a launch receives this table
// by value and finds the phase of a CTA from the item prefix sums.
constexpr int kMaxChunkPhases = 16;
// Footprint classes of a point in an 8^3 tile (3 per axis: low half only, both
// halves, high half only) and the per-item offsets that delimit them.
constexpr int kCubeBins = 27 + 1;
struct SpreadItem;
struct ReduceItem;
struct PhaseTable {
  const float4* qs[kMaxChunkPhases];
  const int32_t* perm[kMaxChunkPhases];
  const int2* list[kMaxChunkPhases];
  const int32_t* bins[kMaxChunkPhases];
  const int2* clist[kMaxChunkPhases];     // class-ordered lists (8^3 tiles), or null
  const int32_t* cbins[kMaxChunkPhases];  // kCubeBins class starts per item
  const SpreadItem* items[kMaxChunkPhases];
  const ReduceItem* reduces[kMaxChunkPhases];
  long long row0[kMaxChunkPhases];    // first value/output row of the phase
  int item0[kMaxChunkPhases + 1];     // prefix sums of the launch's items per phase
  int red0[kMaxChunkPhases + 1];      // prefix sums of reduce items per phase
  int slot0[kMaxChunkPhases];         // first scratch slot of the phase
  int nphase;
  long long entries;                  // k-space spread: list entries of all items
  int longest;                        // and of the longest item
};

// Image-space points (the displaced voxels of all phases) sorted by the 8^3
// home tile of their first tap, then by cell; home tiles are grouped 2 x 2 x 2
// into 16^3 super-tiles (spread_home.cu).
struct HomeSet {
  const float4* qs;       // sorted: (f0, f1, f2, packed first tap)
  const int32_t* perm;    // sorted index -> value row
  const int32_t* tstart;  // per home tile: first sorted index (nt0 nt1 nt2 + 1 entries)
  int nt0, nt1, nt2;      // home tiles per axis (ceil(G / 8))
  int ns0, ns1, ns2;      // super-tiles per axis (ceil(G / 16))
  // per grid coordinate of each axis: (count, covers...) with every cover
  // packed as super-tile * 32 + position in its 19-point padded extent
  const int4* cover0;
  const int4* cover1;
  const int4* cover2;
};

// Image-space points (the displaced voxels of all phases) sorted by the 4^3
// block of their first tap, row-major blocks, grids of a multiple of 4 points
// per axis (spread_rows.cu).
struct RowSet {
  const float4* qs;       // sorted: (f0, f1, f2, packed first tap)
  const int32_t* perm;    // sorted index -> value row
  const int32_t* start;   // per block: first sorted index (nb0 nb1 nb2 + 1 entries)
  int nb0, nb1, nb2;      // blocks per axis (G / 4)
};

// Phase slot of work item `i` of a launch (linear search; nphase is small).
__device__ __forceinline__ int phase_of(const int* prefix, int nphase, int i) {
  int jj = 0;
  while (jj + 1 < nphase && i >= prefix[jj + 1]) ++jj;
  return jj;
}

// A split tile: partial tiles in scratch slots [first, first + count).
struct ReduceItem {
  int32_t tile;
  int32_t first;
  int32_t count;
  int32_t pad;
};

// Evaluate the W kernel weights of the three axes for fractional offsets f0, f1,
// f2, two taps per paired FMA (each part rounded as fmaf).  Home-tile spread of
// four phases at 256^3: 0.605 -> 0.590 ms; the halo-list spreads, whose
// accumulators fill the registers, are faster with one axis at a time
// (register kernel at 128^3, 8 coils: 0.540 against 0.560 ms).
template <int W>
__device__ __forceinline__ void kernel_weights3(float f0, float f1, float f2, const KernelCoefs& kc,
                                                float (&w0)[W], float (&w1)[W], float (&w2)[W]) {
  static_assert(W % 2 == 0, "tap pairs");
  const float f[3] = {f0, f1, f2};
  float2 s[3], acc[3][W / 2];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float v = fmaf(2.0f, f[a], -1.0f);
    s[a] = make_float2(v, v);
  }
#pragma unroll
  for (int k = kNumCoef - 1; k >= 0; --k)
#pragma unroll
    for (int t = 0; t < W / 2; ++t) {
      const float2 c = *reinterpret_cast<const float2*>(&kc.c[k][2 * t]);
#pragma unroll
      for (int a = 0; a < 3; ++a)
        acc[a][t] = k == kNumCoef - 1 ? c : __ffma2_rn(acc[a][t], s[a], c);
    }
#pragma unroll
  for (int t = 0; t < W / 2; ++t) {
    w0[2 * t] = acc[0][t].x;
    w0[2 * t + 1] = acc[0][t].y;
    w1[2 * t] = acc[1][t].x;
    w1[2 * t + 1] = acc[1][t].y;
    w2[2 * t] = acc[2][t].x;
    w2[2 * t + 1] = acc[2][t].y;
  }
}

// The W kernel weights of one axis.
template <int W>
__device__ __forceinline__ void kernel_weights(float f, const KernelCoefs& kc, float (&w)[W]) {
  const float s = fmaf(2.0f, f, -1.0f);
#pragma unroll
  for (int t = 0; t < W; ++t) {
    float acc = kc.c[kNumCoef - 1][t];
#pragma unroll
    for (int k = kNumCoef - 2; k >= 0; --k) acc = fmaf(acc, s, kc.c[k][t]);
    w[t] = acc;
  }
}

// The same from the tap-major coefficients (bitwise: the same operations).  Against the
// paired weights: per-voxel image interpolation at 128^3, W = 4, 0.096 / 0.101 ms, W = 6 0.434 /
// 0.464 at sigma 1.5 but 0.246 / 0.232 at sigma 2; image interpolation by super-tiles, 128^3,
// four phases at sigma 1.25, 0.250 / 0.281.  Against the power-major ones of one axis: spread of
// the compensated plans with four coils 0.124 / 0.140 ms (32^3, 40 k samples), with two 0.152 /
// 0.148.
template <int W>
__device__ __forceinline__ void kernel_weights_by_tap(float f, const KernelCoefs& kc, float (&w)[W]) {
  const float s = fmaf(2.0f, f, -1.0f);
#pragma unroll
  for (int t = 0; t < W; ++t) {
    float acc = kc.t[t][kNumCoef - 1];
#pragma unroll
    for (int k = kNumCoef - 2; k >= 0; --k) acc = fmaf(acc, s, kc.t[t][k]);
    w[t] = acc;
  }
}

// Select w[t] for a runtime t in [0, W) without dynamic register indexing.
template <int W>
__device__ __forceinline__ float select_tap(const float (&w)[W], int t) {
  float r = 0.f;
#pragma unroll
  for (int k = 0; k < W; ++k) r = (t == k) ? w[k] : r;
  return r;
}

// cp.async helpers (sm_80+): 8-byte global -> shared copy, zero-filled when
// `valid` is false.
__device__ __forceinline__ void cp_async_8(void* smem, const void* gmem, bool valid) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  const int src_size = valid ? 8 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem),
               "r"(src_size));
}
__device__ __forceinline__ void cp_async_4(void* smem, const void* gmem, bool valid) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(smem));
  const int src_size = valid ? 4 : 0;
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(s), "l"(gmem),
               "r"(src_size));
}
// asynchronous copy of one stored grid value (complex FP32: 8 bytes; complex BF16: 4)
template <typename GT>
__device__ __forceinline__ void cp_async_grid(GT* smem, const GT* gmem, bool valid) {
  if constexpr (sizeof(GT) == 8)
    cp_async_8(smem, gmem, valid);
  else
    cp_async_4(smem, gmem, valid);
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// Storage of the k-space coil grids: complex FP32 (float2) or complex BF16
// (__nv_bfloat162, round to nearest even); arithmetic is FP32 either way.
using bf162 = __nv_bfloat162;
__device__ __forceinline__ float2 grid_ld(const float2* p) { return __ldg(p); }
__device__ __forceinline__ float2 grid_ld(const bf162* p) {
  const unsigned u = __ldg(reinterpret_cast<const unsigned*>(p));
  return __bfloat1622float2(*reinterpret_cast<const bf162*>(&u));
}
__device__ __forceinline__ void grid_st(float2* p, float2 v) { *p = v; }
__device__ __forceinline__ void grid_st(bf162* p, float2 v) { *p = __float22bfloat162_rn(v); }
__device__ __forceinline__ float2 grid_ld_shared(const float2* p) { return *p; }
__device__ __forceinline__ float2 grid_ld_shared(const bf162* p) { return __bfloat1622float2(*p); }
// two consecutive stored values (coils 2q, 2q+1) from shared memory as float4
__device__ __forceinline__ float4 grid_ld2_shared(const float2* p) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 grid_ld2_shared(const bf162* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const bf162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const bf162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}

__device__ __forceinline__ int wrap_once(int i, int g) {
  // i in [0, 2g): one conditional subtract
  return i >= g ? i - g : i;
}

__device__ __forceinline__ int wrap_any(int i, int g) {
  int r = i % g;
  return r < 0 ? r + g : r;
}

}  // namespace nrs
