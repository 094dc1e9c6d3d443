// Projection Core P_j^(i) of the adjoint image-space gridding (section
// "Image-space Gridding", adjoint diagram), all phases into one grid,
//     u[g] = sum_j sum_n c3(sigma (n + d_j[n]) - g) w_j[n],
// by rows of 4^3 blocks in registers.
//
// The displaced voxels are sorted by the 4^3 block of their first tap (row-major
// blocks, first index of every block in a table).  A footprint of W taps
// reaches K blocks along an axis (K = 2 for W = 4, 3 for W = 6), so the grid
// block (z, y, x) gathers from the K^3 point blocks (z - d, y - e, x - f).  A
// warp owns a row of grid blocks along x and marches over x: one step stages
// the points of the K^2 point blocks at x (contiguous in the sorted order along
// x) and adds them to the blocks x .. x + K - 1, then block x is complete and
// is stored.  No halo lists, no shared accumulators, no partial sums to merge:
// every grid value is written exactly once and every sum has a fixed order.
//
// Staging (a lane per point) evaluates the weights, moves them to their grid
// offsets (zeros elsewhere) and stores the 16 products wz wy v of the block's
// lines and the window's x weights.  A half-warp applies one point, lane (z, y)
// its line's 4 K window values (one product, 4 K weights: 4 K paired FMAs); the
// halves' sums meet when a block is stored.  A warp's whole segment is one
// sequence of points (a lane per step holds its counts), so batches of 32 are
// full whatever the steps hold.
//
// Bound: the shared-memory data path (97 % busy before a half-warp took a whole
// point: 4 wavefronts per point and row then, 3 now) and issue (58 %).  One phase
// at 384^3, 7.1 M points: 1.085 ms by home tiles (spread_home.cu) -> 0.695 ms;
// W = 6 at 144 x 120 x 96, 1 M points: 1.25 ms by the generic halo-list kernel ->
// 0.55 ms.  A tensor-core version of the same march (lines x points times points
// x window values) measured 0.685 ms with 10 % more rounding error: not taken.
#include "plan_internal.h"

namespace nrs {

namespace {

constexpr int kRowWarps = 4;  // warps per CTA: 2 x 2 neighbouring rows (shared L1 lines)

template <int W>
struct RowStage {
  static constexpr int K = (W + 6) / 4;  // blocks a footprint reaches per axis
  float2 zyv[16];                        // [4 z + y] of the warp's block row
  float x[4 * K];                        // [4 f + x] of block f of the window
  float pad[4];                          // 176- / 192-byte records
};

// pos[r + t] = w[t], zero elsewhere (r in 0..3)
template <int W, int N>
__device__ __forceinline__ void place(const float (&w)[W], int r, float (&pos)[N]) {
  float a[W + 1];
#pragma unroll
  for (int j = 0; j <= W; ++j) {
    const float here = j < W ? w[j < W ? j : 0] : 0.f, left = j > 0 ? w[j > 0 ? j - 1 : 0] : 0.f;
    a[j] = (r & 1) ? left : here;
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const float here = j <= W ? a[j <= W ? j : 0] : 0.f;
    const float left = j >= 2 && j - 2 <= W ? a[j >= 2 && j - 2 <= W ? j - 2 : 0] : 0.f;
    pos[j] = (r & 2) ? left : here;
  }
}

// the four entries of block d of a placed row
template <int N>
__device__ __forceinline__ void pick(const float (&pos)[N], int d, float (&out)[4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    out[i] = pos[i];
#pragma unroll
    for (int k = 1; 4 * k + i < N; ++k) out[i] = d == k ? pos[4 * k + i] : out[i];
  }
}

}  // namespace

template <int W>
__global__ void __launch_bounds__(32 * kRowWarps, W == 4 ? 8 : 6)
    spread_rows_kernel(Geo g, KernelCoefs kc, RowSet rs, int seg, const float2* __restrict__ vals,
                       float2* __restrict__ grid) {
  using Stage = RowStage<W>;
  constexpr int K = Stage::K, NR = K * K;
  __shared__ __align__(16) Stage stg_all[kRowWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bz = blockIdx.z * 2 + (warp >> 1), by = blockIdx.y * 2 + (warp & 1);
  if (bz >= rs.nb0 || by >= rs.nb1) return;  // warp-uniform; no CTA barrier below
  Stage* stg = stg_all[warp];
  const int xs = blockIdx.x * seg, xe = min(xs + seg, rs.nb2);  // grid blocks of this row segment
  const int steps = xe - xs + K - 1;  // the first K - 1 only lead in; at most 32
  const int line = lane & 15, half = lane >> 4;
  // lane t: the K^2 point blocks of step t (block xs - (K - 1) + t of the rows
  // (z - d, y - e)) and the points of the steps up to t
  int beg[NR], len[NR], incl = 0;
  {
    int x = xs - (K - 1) + lane;
    if (x < 0) x += rs.nb2;
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      int pz = bz - r / K, py = by - r % K;
      if (pz < 0) pz += rs.nb0;
      if (py < 0) py += rs.nb1;
      const int32_t* st = rs.start + ((long long)pz * rs.nb1 + py) * rs.nb2 + x;
      beg[r] = lane < steps ? __ldg(st) : 0;
      len[r] = lane < steps ? __ldg(st + 1) - beg[r] : 0;
      incl += len[r];
    }
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  float2 acc[K][4];  // this half's sums of the window's blocks
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[k][i] = make_float2(0.f, 0.f);
  float4* const out = reinterpret_cast<float4*>(
      grid + ((long long)(4 * bz + (line >> 2)) * g.g1 + 4 * by + (line & 3)) * g.g2) + half;
  int step = 0, step_end = __shfl_sync(0xffffffffu, incl, 0);

  // Block xb = xs - (K - 1) + step is complete: add the halves, half h stores
  // the x pair h of every line, and the window moves on.
  auto finish_step = [&] {
    const int xb = xs - (K - 1) + step;
    float2 o[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      // the pair's value of this half, and the other half's
      const float2 mine = half ? acc[0][2 + i] : acc[0][i], give = half ? acc[0][i] : acc[0][2 + i];
      o[i] = __fadd2_rn(mine, make_float2(__shfl_xor_sync(0xffffffffu, give.x, 16),
                                          __shfl_xor_sync(0xffffffffu, give.y, 16)));
    }
    if (xb >= xs) out[2 * xb] = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        acc[k][i] = k + 1 < K ? acc[k + 1 < K ? k + 1 : k][i] : make_float2(0.f, 0.f);
    ++step;
    step_end = __shfl_sync(0xffffffffu, incl, step & 31);
  };

  for (int base = 0; base < total; base += 32) {
    const int n = min(32, total - base);
    {
      // lanes past the end repeat the last point (and are not applied)
      const int i = min(base + lane, total - 1);
      int t = 0;  // step of point i: the first with incl > i
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
        if (__shfl_sync(0xffffffffu, incl, t + d - 1) <= i) t += d;
      const int before = __shfl_sync(0xffffffffu, incl, (t - 1) & 31);
      int o = i - (t > 0 ? before : 0), r = 0, si = 0;
      bool found = false;
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        const int lk = __shfl_sync(0xffffffffu, len[k], t), bk = __shfl_sync(0xffffffffu, beg[k], t);
        if (!found && o < lk) {
          si = bk + o;
          r = k;
          found = true;
        }
        o -= lk;
      }
      const float4 p = __ldg(rs.qs + si);
      const float2 v = __ldg(vals + __ldg(rs.perm + si));
      const uint32_t pk = __float_as_uint(p.w);
      const int dz = r / K, dy = r - dz * K;
      float wz[W], wy[W], wx[W], pos[4 * K], z4[4], y4[4];
      kernel_weights3<W>(p.x, p.y, p.z, kc, wz, wy, wx);
      Stage& d = stg[lane];
      place<W>(wx, int(pk) & 3, pos);
#pragma unroll
      for (int f = 0; f < K; ++f)
        reinterpret_cast<float4*>(d.x)[f] =
            make_float4(pos[4 * f], pos[4 * f + 1], pos[4 * f + 2], pos[4 * f + 3]);
      place<W>(wz, int(pk >> 20) & 3, pos);
      pick(pos, dz, z4);
      place<W>(wy, int(pk >> 10) & 3, pos);
      pick(pos, dy, y4);
#pragma unroll
      for (int z = 0; z < 4; ++z)
#pragma unroll
        for (int y = 0; y < 4; y += 2) {
          const float wa = z4[z] * y4[y], wb = z4[z] * y4[y + 1];
          const float2 a = __fmul2_rn(make_float2(wa, wa), v), b = __fmul2_rn(make_float2(wb, wb), v);
          reinterpret_cast<float4*>(d.zyv)[2 * z + y / 2] = make_float4(a.x, a.y, b.x, b.y);
        }
    }
    __syncwarp();
    int p = 0;
    for (;;) {
      // points of this batch that belong to the current step
      const int pe = min(n, step_end - base);
      // this half's point p + half, its line's product and the window's weights
      auto apply = [&](int k, bool live) {
        const Stage& rec = stg[live ? k + half : k];
        float2 c = rec.zyv[line];
        if (!live) c = make_float2(0.f, 0.f);
#pragma unroll
        for (int f = 0; f < K; ++f) {
          const float4 x4 = *reinterpret_cast<const float4*>(rec.x + 4 * f);
          acc[f][0] = __ffma2_rn(make_float2(x4.x, x4.x), c, acc[f][0]);
          acc[f][1] = __ffma2_rn(make_float2(x4.y, x4.y), c, acc[f][1]);
          acc[f][2] = __ffma2_rn(make_float2(x4.z, x4.z), c, acc[f][2]);
          acc[f][3] = __ffma2_rn(make_float2(x4.w, x4.w), c, acc[f][3]);
        }
      };
#pragma unroll 1
      for (; p + 4 <= pe; p += 4) {
        apply(p, true);
        apply(p + 2, true);
      }
      if (p + 2 <= pe) {
        apply(p, true);
        p += 2;
      }
      if (p < pe) {
        // an odd last point: half 1 adds zeros
        apply(p, half == 0);
        p += 1;
      }
      if (step_end > base + n || step >= steps) break;  // the step goes on in the next batch
      finish_step();
      if (step >= steps) break;
    }
    __syncwarp();
  }
  while (step < steps) finish_step();
}

// Blocks of a row per warp: long segments repeat fewer lead-in steps, short ones
// fill the chip; at least four warps per resident slot where the grid has them.
int row_segment(const RowSet& rs) {
  const long long rows = (long long)rs.nb0 * rs.nb1;
  const long long want = 4LL * 152 * 28;
  long long seg = rows * rs.nb2 / want;
  seg = std::max<long long>(4, std::min<long long>(seg, 30));  // steps: at most 32
  return int(std::min<long long>(seg, rs.nb2));
}

// Points that a warp of launch_spread_rows visits, the largest over its warps.
__global__ void row_load_kernel(RowSet rs, int K, int seg, int segs, int32_t* __restrict__ most) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)rs.nb0 * rs.nb1 * segs) return;
  const int xs = int(i % segs) * seg, xe = min(xs + seg, rs.nb2), lead = xs - (K - 1);
  const int by = int(i / segs % rs.nb1), bz = int(i / segs / rs.nb1);
  int load = 0;
  for (int d = 0; d < K; ++d)
    for (int e = 0; e < K; ++e) {
      const int pz = bz >= d ? bz - d : bz - d + rs.nb0, py = by >= e ? by - e : by - e + rs.nb1;
      const int32_t* st = rs.start + ((long long)pz * rs.nb1 + py) * rs.nb2;
      load += st[xe] - st[max(lead, 0)];
      if (lead < 0) load += st[rs.nb2] - st[rs.nb2 + lead];
    }
  atomicMax(most, load);
}

int launch_row_load(int W, const RowSet& rs, int32_t* most, cudaStream_t s) {
  const int seg = row_segment(rs), segs = (rs.nb2 + seg - 1) / seg;
  const long long n = (long long)rs.nb0 * rs.nb1 * segs;
  row_load_kernel<<<unsigned((n + 255) / 256), 256, 0, s>>>(rs, W == 4 ? 2 : 3, seg, segs, most);
  return 1;
}

int launch_spread_rows(const Geo& g, int W, const KernelCoefs& kc, const RowSet& rs,
                       const nrsense_c64* vals, nrsense_c64* grid, cudaStream_t s) {
  const int seg = row_segment(rs);
  const dim3 gd((rs.nb2 + seg - 1) / seg, (rs.nb1 + 1) / 2, (rs.nb0 + 1) / 2);
  const auto* v = reinterpret_cast<const float2*>(vals);
  auto* u = reinterpret_cast<float2*>(grid);
  if (W == 4)
    spread_rows_kernel<4><<<gd, 32 * kRowWarps, 0, s>>>(g, kc, rs, seg, v, u);
  else
    spread_rows_kernel<6><<<gd, 32 * kRowWarps, 0, s>>>(g, kc, rs, seg, v, u);
  return 1;
}

}  // namespace nrs
