// Plan-time sort of the displaced voxels on the device: positions
// q = sigma (n + d_j[n]) in FP64, first tap and fraction, stable order by the
// 4^3 block (row spread) or by the 8^3 home tile and cell (home-tile spread) of
// the first tap.
//
// Three passes over the points: decompose and count per group; scatter to the
// group's range in any order; rank every point among its group by (cell, index)
// and write its record there.  The rank makes the order independent of the
// scatter's.  A group's points are read by all its members, at 8 to a few hundred
// points per group from L1; a displacement that gathers more than kMaxGroup
// points in a group is left to the host's sort.  64^3, two phases (524 k points):
// 62 ms on the host -> 0.55 ms.
#include "plan_internal.h"

namespace nrs {

namespace {

constexpr int kMaxGroup = 8192;
constexpr int kScanItems = 2048;  // counts per CTA of the scan (256 threads x 8)

__device__ __forceinline__ void decompose_dev(double q, int G, int W, int* base, float* frac) {
  const double fl = floor(q);
  long long b = (long long)fl - (W / 2 - 1);
  b %= G;
  if (b < 0) b += G;
  *base = int(b);
  *frac = float(q - fl);
}

// info[0]: 1 if a displacement is not finite or beyond 1e6 voxels
__global__ void image_points_kernel(Geo g, int W, double sigma, long long n,
                                    const float* __restrict__ disp, int shift, int nb1, int nb2,
                                    float4* __restrict__ q, int32_t* __restrict__ key,
                                    int32_t* __restrict__ count, int32_t* __restrict__ info) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const long long j = i / g.nvox, v = i - j * g.nvox;
  const int i2 = int(v % g.n2), i1 = int((v / g.n2) % g.n1), i0 = int(v / ((long long)g.n1 * g.n2));
  const int ii[3] = {i0, i1, i2}, gs[3] = {g.g0, g.g1, g.g2};
  int b[3];
  float f[3];
  bool bad = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    float d = __ldg(disp + (3 * j + a) * g.nvox + v);
    if (!isfinite(d) || fabsf(d) > 1e6f) {
      bad = true;
      d = 0.f;
    }
    decompose_dev(__dadd_rn(__dmul_rn(sigma, double(ii[a])), __dmul_rn(sigma, double(d))), gs[a], W,
                  &b[a], &f[a]);
  }
  if (bad) atomicOr(info, 1);
  q[i] = make_float4(f[0], f[1], f[2], __uint_as_float(pack_base(b[0], b[1], b[2])));
  const int k = ((b[0] >> shift) * nb1 + (b[1] >> shift)) * nb2 + (b[2] >> shift);
  key[i] = k;
  atomicAdd(count + k, 1);
}

// start[i] = counts before i within the CTA's 2048, total of the CTA, largest count
__global__ void __launch_bounds__(256) scan_local_kernel(const int32_t* __restrict__ count,
                                                         long long n, int32_t* __restrict__ start,
                                                         int32_t* __restrict__ totals,
                                                         int32_t* __restrict__ info) {
  __shared__ int warp_sum[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long base = blockIdx.x * (long long)kScanItems + threadIdx.x * 8;
  int c[8], sum = 0, most = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    c[k] = base + k < n ? count[base + k] : 0;
    most = max(most, c[k]);
    sum += c[k];
  }
  int incl = sum;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += t;
    most = max(most, __shfl_xor_sync(0xffffffffu, most, d));
  }
  if (lane == 31) warp_sum[warp] = incl;
  if (lane == 0 && most > 0) atomicMax(info + 1, most);
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    before += w < warp ? warp_sum[w] : 0;
    total += warp_sum[w];
  }
  int at = before + incl - sum;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (base + k < n) start[base + k] = at;
    at += c[k];
  }
  if (threadIdx.x == 0) totals[blockIdx.x] = total;
}

// totals -> sums before, one CTA
__global__ void __launch_bounds__(1024) scan_totals_kernel(int32_t* __restrict__ totals, int n) {
  __shared__ int warp_sum[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int carry = 0;
  for (int base = 0; base < n; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = i < n ? totals[i] : 0;
    int incl = v;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += t;
    }
    if (lane == 31) warp_sum[warp] = incl;
    __syncthreads();
    int before = carry, all = carry;
    for (int w = 0; w < 32; ++w) {
      before += w < warp ? warp_sum[w] : 0;
      all += warp_sum[w];
    }
    if (i < n) totals[i] = before + incl - v;
    carry = all;
    __syncthreads();
  }
}

// start += the CTA's offset; fill = 0 (the counts' array); start[n] = points
__global__ void scan_add_kernel(long long n, const int32_t* __restrict__ totals, int32_t points,
                                int32_t* __restrict__ start, int32_t* __restrict__ fill) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) {
    start[i] += totals[i / kScanItems];
    fill[i] = 0;
  } else if (i == n) {
    start[n] = points;
  }
}

__global__ void group_scatter_kernel(long long n, int cells, const float4* __restrict__ q,
                                     const int32_t* __restrict__ key,
                                     const int32_t* __restrict__ start, int32_t* __restrict__ fill,
                                     unsigned long long* __restrict__ order) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int k = key[i];
  unsigned long long cell = 0;
  if (cells) {
    const uint32_t pk = __float_as_uint(q[i].w);
    cell = (((pk >> 20) & 7u) * 8 + ((pk >> 10) & 7u)) * 8 + (pk & 7u);
  }
  order[start[k] + atomicAdd(fill + k, 1)] = cell << 32 | (unsigned long long)i;
}

__global__ void group_rank_kernel(long long n, const float4* __restrict__ q,
                                  const int32_t* __restrict__ key,
                                  const int32_t* __restrict__ start,
                                  const unsigned long long* __restrict__ order,
                                  float4* __restrict__ qs, int32_t* __restrict__ perm) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= n) return;
  const unsigned long long u = order[p];
  const uint32_t i = uint32_t(u);
  const int k = key[i], s = start[k], e = start[k + 1];
  int r = 0;
  for (int t = s; t < e; ++t) r += order[t] < u ? 1 : 0;
  qs[s + r] = q[i];
  perm[s + r] = int32_t(i);
}

}  // namespace

// Sort n = P N^3 displaced voxels (disp: device) into groups of edge 1 << shift
// (cells: also by cell within the group) into qs, perm (n entries) and start
// (groups + 1 entries), all device arrays of the caller.  *bad: a displacement is
// not finite or too large.  *done = false (and nothing usable): a group is too
// crowded for the rank.  Synchronises.
nrsense_status sort_image_points(const Geo& g, int W, double sigma, long long n, const float* disp,
                                 int shift, bool cells, float4* qs, int32_t* perm, int32_t* start,
                                 bool* bad, bool* done, cudaStream_t s) {
  const int e = 1 << shift;
  const int nb1 = (g.g1 + e - 1) / e, nb2 = (g.g2 + e - 1) / e;
  const long long groups = (long long)((g.g0 + e - 1) / e) * nb1 * nb2;
  const int tiles = int((groups + kScanItems - 1) / kScanItems);
  // one temporary allocation: records, order, keys, counts, totals, info
  const size_t bytes = size_t(n) * (16 + 8 + 4) + size_t(groups) * 4 + size_t(tiles) * 4 + 8;
  unsigned char* tmp = nullptr;
  if (cudaMalloc(&tmp, bytes) != cudaSuccess) {
    cudaGetLastError();
    return NRSENSE_ERR_OOM;
  }
  auto* q = reinterpret_cast<float4*>(tmp);
  auto* order = reinterpret_cast<unsigned long long*>(q + n);
  auto* info = reinterpret_cast<int32_t*>(order + n);
  auto* key = info + 2;
  auto* count = key + n;
  auto* totals = count + groups;
  int32_t h[2] = {0, 0};
  const unsigned nb = unsigned((n + 255) / 256);
  bool ok = cudaMemsetAsync(info, 0, 8, s) == cudaSuccess &&
            cudaMemsetAsync(count, 0, size_t(groups) * 4, s) == cudaSuccess;
  if (ok) {
    image_points_kernel<<<nb, 256, 0, s>>>(g, W, sigma, n, disp, shift, nb1, nb2, q, key, count, info);
    scan_local_kernel<<<tiles, 256, 0, s>>>(count, groups, start, totals, info);
    ok = cudaMemcpyAsync(h, info, 8, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
         cudaStreamSynchronize(s) == cudaSuccess;
  }
  *bad = h[0] != 0;
  *done = ok && h[0] == 0 && h[1] <= kMaxGroup;
  if (*done) {
    scan_totals_kernel<<<1, 1024, 0, s>>>(totals, tiles);
    scan_add_kernel<<<unsigned((groups + 256) / 256), 256, 0, s>>>(groups, totals, int32_t(n), start,
                                                                   count);
    group_scatter_kernel<<<nb, 256, 0, s>>>(n, cells ? 1 : 0, q, key, start, count, order);
    group_rank_kernel<<<nb, 256, 0, s>>>(n, q, key, start, order, qs, perm);
    ok = cudaGetLastError() == cudaSuccess && cudaStreamSynchronize(s) == cudaSuccess;
  }
  cudaFree(tmp);
  return ok ? NRSENSE_OK : NRSENSE_ERR_CUDA;
}

}  // namespace nrs
