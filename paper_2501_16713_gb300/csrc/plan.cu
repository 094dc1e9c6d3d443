// Plan construction for the nonrigid SENSE operator (host, plan time).
//
// nrsense_plan_create validates the problem statement (stacked SENSE
// equation: P motion states sharing one image, C coils, M_j samples per
// state), evaluates the kernel polynomials and deapodization tables in FP64,
// decomposes every k-space sample position q = omega G / (2 pi) and every
// displaced voxel position q = sigma (n + d_j[n]) into first tap and fraction,
// sorts the points into 8^3 grid tiles, builds the per-tile halo lists and
// work items of the output-stationary spreading kernels, and creates the cuFFT
// plans and work buffers.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <new>
#include <thread>
#include <vector>

#include "kb_host.h"
#include <cufftXt.h>

#include "plan_internal.h"

using namespace nrs;

namespace {

// Host-side fault injection for the error paths (NRSENSE_FAULT=alloc|cufft|upload;
// alloc:N: allocations of a plan that holds N already).
bool fault_requested(const char* what, const nrsense_plan_s* p = nullptr) {
  const char* f = std::getenv("NRSENSE_FAULT");
  if (f == nullptr) return false;
  const size_t n = std::strlen(what);
  if (std::strncmp(f, what, n) != 0) return false;
  return f[n] == '\0' || (f[n] == ':' && p != nullptr &&
                          p->allocations.size() >= size_t(std::atoll(f + n + 1)));
}

nrsense_status dev_alloc(nrsense_plan_s* p, void** ptr, size_t bytes) {
  *ptr = nullptr;
  if (bytes == 0) return NRSENSE_OK;
  if (fault_requested("alloc", p)) return NRSENSE_ERR_OOM;
  if (cudaMalloc(ptr, bytes) != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return NRSENSE_ERR_OOM;
  }
  p->allocations.push_back(*ptr);
  p->allocation_bytes.push_back(bytes);
  p->device_bytes += (long long)bytes;
  return NRSENSE_OK;
}

// free one tracked allocation (null: no-op)
void dev_free(nrsense_plan_s* p, void* ptr) {
  if (ptr == nullptr) return;
  for (size_t i = 0; i < p->allocations.size(); ++i)
    if (p->allocations[i] == ptr) {
      cudaFree(ptr);
      p->device_bytes -= (long long)p->allocation_bytes[i];
      p->allocations.erase(p->allocations.begin() + long(i));
      p->allocation_bytes.erase(p->allocation_bytes.begin() + long(i));
      return;
    }
}

// Frees what the plan allocated since its construction unless kept: the arrays of
// a point order are the plan's only once all of them are there.
struct Rollback {
  nrsense_plan_s* p;
  size_t mark;
  bool keep = false;
  explicit Rollback(nrsense_plan_s* plan) : p(plan), mark(plan->allocations.size()) {}
  Rollback(const Rollback&) = delete;
  Rollback& operator=(const Rollback&) = delete;
  ~Rollback() {
    while (!keep && p->allocations.size() > mark) dev_free(p, p->allocations.back());
  }
};

void free_pointset(nrsense_plan_s* p, PointSet* ps) {
  void* arrs[] = {ps->qs, ps->perm, ps->list, ps->items, ps->bins, ps->reduces, ps->iitems,
                  ps->clist, ps->cbins};
  for (void* a : arrs) dev_free(p, a);
  *ps = PointSet{};
}

template <typename T>
nrsense_status dev_alloc_n(nrsense_plan_s* p, T** ptr, long long n) {
  return dev_alloc(p, reinterpret_cast<void**>(ptr), size_t(n) * sizeof(T));
}

template <typename T>
nrsense_status upload(T* dst, const std::vector<T>& src, cudaStream_t s) {
  if (src.empty()) return NRSENSE_OK;
  if (fault_requested("upload")) return NRSENSE_ERR_CUDA;
  if (cudaMemcpyAsync(dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s) !=
      cudaSuccess)
    return NRSENSE_ERR_CUDA;
  // host vectors are freed by the caller after return: wait here
  if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  return NRSENSE_OK;
}

#define NRS_TRY(expr)                          \
  do {                                         \
    nrsense_status _st = (expr);               \
    if (_st != NRSENSE_OK) return _st;         \
  } while (0)

struct HostPoint {
  float f[3];
  int b[3];
  int32_t row;
};

// Decompose a position on the periodic grid: first tap index (mod G) and the
// fractional offset f = q - floor(q) of the kernel's centre cell.
inline void decompose(double q, int G, int W, int* base, float* frac) {
  const double fl = std::floor(q);
  long long b = (long long)fl - (W / 2 - 1);
  if (b < 0 || b >= G) {
    b %= G;
    if (b < 0) b += G;
  }
  *base = int(b);
  *frac = float(q - fl);
}

// Morton (Z-order) code of a tile, 10 bits per axis: work items in this
// order keep neighbouring tiles (which share halo data) close in time.
uint64_t morton3(const TilePlan& tp, long long tile) {
  const long long tz = tile / ((long long)tp.nt1 * tp.nt2);
  const long long rem = tile - tz * tp.nt1 * tp.nt2;
  const long long ty = rem / tp.nt2, tx = rem - ty * tp.nt2;
  uint64_t m = 0;
  for (int b = 0; b < 10; ++b) {
    m |= uint64_t((tx >> b) & 1) << (3 * b);
    m |= uint64_t((ty >> b) & 1) << (3 * b + 1);
    m |= uint64_t((tz >> b) & 1) << (3 * b + 2);
  }
  return m;
}

TilePlan make_tileplan(const Geo& g, int T) {
  TilePlan tp;
  tp.t0 = tp.t1 = tp.t2 = T;
  tp.nt0 = (g.g0 + T - 1) / T;
  tp.nt1 = (g.g1 + T - 1) / T;
  tp.nt2 = (g.g2 + T - 1) / T;
  tp.ntiles = (long long)tp.nt0 * tp.nt1 * tp.nt2;
  return tp;
}

// Tiles (edge 1 << sh) along one axis of G points that the W taps from b touch: 1 or
// 2, or up to 3 where they wrap past a ragged last tile.
inline int touched_tiles(int b, int W, int G, int sh, int* out) {
  if (b + W <= G) {  // no wrap: a footprint is no longer than a tile
    out[0] = b >> sh;
    out[1] = (b + W - 1) >> sh;
    return out[1] == out[0] ? 1 : 2;
  }
  int n = 0;
  for (int t = 0; t < W; ++t) {
    int gi = b + t;
    if (gi >= G) gi -= G;
    const int ti = gi >> sh;
    bool seen = false;
    for (int k = 0; k < n; ++k) seen |= (out[k] == ti);
    if (!seen) out[n++] = ti;
  }
  return n;
}

// Mark every tile touched by a footprint of the given points.
void mark_touched_tiles(const nrsense_plan_s* p, const TilePlan& tp,
                        const std::vector<HostPoint>& pts, std::vector<char>& mask) {
  const Geo& g = p->geo;
  const int sh = tp.t0 == 16 ? 4 : 3;
  for (const HostPoint& h : pts) {
    int t0[8], t1[8], t2[8];
    const int n0 = touched_tiles(h.b[0], p->W, g.g0, sh, t0);
    const int n1 = touched_tiles(h.b[1], p->W, g.g1, sh, t1);
    const int n2 = touched_tiles(h.b[2], p->W, g.g2, sh, t2);
    for (int a = 0; a < n0; ++a)
      for (int b = 0; b < n1; ++b)
        for (int c = 0; c < n2; ++c) mask[((long long)t0[a] * tp.nt1 + t1[b]) * tp.nt2 + t2[c]] = 1;
  }
}

// The host side of a point set: what upload_pointset copies to the device.
struct HostSet {
  TilePlan tp{};
  long long npts = 0, list_len = 0;
  int occupied = 0, slots = 0, longest_item = 0;
  bool cube = false;
  std::vector<float4> qs;
  std::vector<int32_t> perm, bins, cbins;
  std::vector<int2> list, clist;
  std::vector<SpreadItem> items, iitems;
  std::vector<ReduceItem> reds;
};

// Sort points into tiles, build halo lists and work items (host only: the phases
// of a plan run in threads of their own).
// tp: tiles of this set; write_mask: tiles that must be written even without
// points (NULL = every tile); interp: also build interpolation work items.
nrsense_status compute_pointset(const Geo& g, int W, const std::vector<HostPoint>& pts,
                                const TilePlan& tp, const std::vector<char>* write_mask,
                                bool interp, int max_item, HostSet* hs) {
  hs->tp = tp;
  const long long npts = (long long)pts.size();
  hs->npts = npts;
  if (npts >= (1ll << 31)) return NRSENSE_ERR_ARG;
  const int gsz[3] = {g.g0, g.g1, g.g2};
  const int sh = tp.t0 == 16 ? 4 : 3, tmask = (1 << sh) - 1;  // tiles of 8 or 16 points per axis

  // order: tile of the first tap, cell inside the tile, input order (counting
  // sort by tile, then each tile's (cell, index) keys)
  std::vector<int64_t> first(tp.ntiles + 1, 0);
  auto tile_id = [&](const HostPoint& h) {
    return ((long long)(h.b[0] >> sh) * tp.nt1 + (h.b[1] >> sh)) * tp.nt2 + (h.b[2] >> sh);
  };
  for (const HostPoint& h : pts) first[tile_id(h) + 1]++;
  for (long long t = 0; t < tp.ntiles; ++t) first[t + 1] += first[t];
  std::vector<uint64_t> ko((size_t)npts);
  {
    std::vector<int64_t> at(first.begin(), first.end() - 1);
    for (long long i = 0; i < npts; ++i) {
      const HostPoint& h = pts[(size_t)i];
      const uint64_t cell =
          ((uint64_t(h.b[0] & tmask) << sh | uint64_t(h.b[1] & tmask)) << sh) | uint64_t(h.b[2] & tmask);
      ko[(size_t)at[tile_id(h)]++] = cell << 32 | uint64_t(i);
    }
  }
  for (long long t = 0; t < tp.ntiles; ++t)
    if (first[t + 1] - first[t] > 1) std::sort(ko.begin() + first[t], ko.begin() + first[t + 1]);
  // interpolation items: sorted ranges of points sharing a first-tap tile
  std::vector<SpreadItem>& iitems = hs->iitems;
  if (interp) {
    for (long long t = 0; t < tp.ntiles; ++t)
      for (long long cb = first[t]; cb < first[t + 1]; cb += kInterpMaxItem)
        iitems.push_back({int32_t(t), int32_t(cb),
                          int32_t(std::min<long long>(first[t + 1], cb + kInterpMaxItem)), -1});
    std::stable_sort(iitems.begin(), iitems.end(), [&](const SpreadItem& a, const SpreadItem& b) {
      return morton3(tp, a.tile) < morton3(tp, b.tile);
    });
  }

  std::vector<float4>& qs = hs->qs;
  std::vector<int32_t>& perm = hs->perm;
  qs.resize((size_t)npts);
  perm.resize((size_t)npts);
  std::vector<uint32_t> base((size_t)npts);  // packed first taps in sorted order
  for (long long s_i = 0; s_i < npts; ++s_i) {
    const HostPoint& h = pts[(size_t)(ko[(size_t)s_i] & 0xffffffffu)];
    const uint32_t packed = pack_base(h.b[0], h.b[1], h.b[2]);
    float w;
    std::memcpy(&w, &packed, sizeof(w));
    qs[(size_t)s_i] = make_float4(h.f[0], h.f[1], h.f[2], w);
    perm[(size_t)s_i] = h.row;
    base[(size_t)s_i] = packed;
  }
  std::vector<uint64_t>().swap(ko);
  auto axis0 = [&](int32_t si) { return int(base[(size_t)si] >> 20); };

  // halo lists: every tile touched by a point's W^3 footprint
  auto each_tile = [&](uint32_t packed, auto&& f) {
    int b0, b1, b2, t0[8], t1[8], t2[8];
    unpack_base(packed, b0, b1, b2);
    const int n0 = touched_tiles(b0, W, gsz[0], sh, t0), n1 = touched_tiles(b1, W, gsz[1], sh, t1),
              n2 = touched_tiles(b2, W, gsz[2], sh, t2);
    for (int a = 0; a < n0; ++a)
      for (int b = 0; b < n1; ++b)
        for (int c = 0; c < n2; ++c) f(((long long)t0[a] * tp.nt1 + t1[b]) * tp.nt2 + t2[c]);
  };
  std::vector<int64_t> counts(tp.ntiles + 1, 0);
  for (long long s_i = 0; s_i < npts; ++s_i)
    each_tile(base[(size_t)s_i], [&](long long t) { counts[t + 1]++; });
  for (long long t = 0; t < tp.ntiles; ++t) counts[t + 1] += counts[t];
  const long long list_len = counts[tp.ntiles];
  if (list_len >= (1ll << 31)) return NRSENSE_ERR_ARG;
  std::vector<int32_t> list(list_len);  // sorted indices; paired with rows below
  {
    std::vector<int64_t> fill(counts.begin(), counts.end() - 1);
    for (long long s_i = 0; s_i < npts; ++s_i)
      each_tile(base[(size_t)s_i], [&](long long t) { list[fill[t]++] = int32_t(s_i); });
  }
  hs->list_len = list_len;
  // within each tile, order the points by the plane offset of their first tap
  // (axis 0) relative to the tile origin, so the spreading warp that owns a
  // plane finds its points in one contiguous range (stable: ties keep order)
  {
    const int nb = W + tp.t0;  // offsets in (-W, T)
    std::vector<int32_t> tmp;
    std::vector<int64_t> bcount(nb + 1);
    for (long long t = 0; t < tp.ntiles; ++t) {
      const long long b = counts[t], e = counts[t + 1];
      if (e - b < 2) continue;
      const int o0 = int(t / ((long long)tp.nt1 * tp.nt2)) * tp.t0;
      auto key = [&](int32_t si) {
        int r = axis0(si) - o0;
        if (r < 0) r += g.g0;
        if (r >= tp.t0) r -= g.g0;
        return r + W - 1;
      };
      std::fill(bcount.begin(), bcount.end(), 0);
      for (long long i = b; i < e; ++i) bcount[key(list[i]) + 1]++;
      for (int k = 0; k < nb; ++k) bcount[k + 1] += bcount[k];
      tmp.assign(list.begin() + b, list.begin() + e);
      for (int32_t si : tmp) list[b + bcount[key(si)]++] = si;
    }
  }

  // work items: occupied tiles, plus empty tiles in write_mask (they write
  // zeros); heavy tiles split
  std::vector<SpreadItem>& items = hs->items;
  std::vector<ReduceItem>& reds = hs->reds;
  int slots = 0, occupied = 0;
  for (long long t = 0; t < tp.ntiles; ++t) {
    const long long b = counts[t], e = counts[t + 1];
    const long long L = e - b;
    if (L > 0) occupied++;
    if (L == 0 && write_mask != nullptr && !(*write_mask)[t]) continue;
    if (L <= max_item) {
      items.push_back({int32_t(t), int32_t(b), int32_t(e), -1});
    } else {
      // deal the (r0-sorted) entries round-robin into chunks, so every chunk
      // spans all planes of the tile and keeps the r0 order
      const int nchunk = int((L + max_item - 1) / max_item);
      std::vector<int32_t> seg(list.begin() + b, list.begin() + e);
      long long w = b;
      ReduceItem r{int32_t(t), slots, nchunk, 0};
      for (int k = 0; k < nchunk; ++k) {
        const long long cb = w;
        for (long long i = k; i < L; i += nchunk) list[w++] = seg[i];
        items.push_back({int32_t(t), int32_t(cb), int32_t(w), slots + k});
      }
      slots += nchunk;
      reds.push_back(r);
    }
  }
  // Morton order of tiles (chunks of a tile stay adjacent)
  std::stable_sort(items.begin(), items.end(), [&](const SpreadItem& a, const SpreadItem& b) {
    return morton3(tp, a.tile) < morton3(tp, b.tile);
  });
  hs->slots = slots;
  hs->occupied = occupied;
  for (const SpreadItem& it : items) hs->longest_item = std::max(hs->longest_item, it.end - it.begin);
  // per item: first entry of each first-tap plane offset bin (list sorted by
  // r0 within every tile, so within every item)
  const int nb = W + tp.t0 + 1;
  std::vector<int32_t>& bins = hs->bins;
  bins.resize(items.size() * nb);
  for (size_t k = 0; k < items.size(); ++k) {
    const SpreadItem& itm = items[k];
    const int o0 = int(itm.tile / ((long long)tp.nt1 * tp.nt2)) * tp.t0;
    int32_t* bk = bins.data() + k * nb;
    int e = itm.begin;
    for (int bb = 0; bb < nb - 1; ++bb) {
      // advance past entries with r0 + W - 1 < bb
      while (e < itm.end) {
        int r = axis0(list[e]) - o0;
        if (r < 0) r += g.g0;
        if (r >= tp.t0) r -= g.g0;
        if (r + W - 1 >= bb) break;
        ++e;
      }
      bk[bb] = e - itm.begin;
    }
    bk[nb - 1] = itm.end - itm.begin;
  }
  // class-ordered copy for the tensor-core spread over 4^3 sub-blocks (8^3
  // tiles): along each axis the first-tap offset r in [1 - W, 7] puts a
  // footprint in the low half of the tile only (r <= 4 - W), in both halves
  // (r <= 3) or in the high half only (r >= 4); the entries of every item
  // are ordered by class 9 c0 + 3 c1 + c2 (stable), with 28 offsets per item
  const bool cube = interp && tp.t0 == 8 && tp.t1 == 8 && tp.t2 == 8;
  std::vector<int2>& clist2 = hs->clist;
  std::vector<int32_t>& cbins = hs->cbins;
  hs->cube = cube;
  if (cube) {
    clist2.resize(list_len);
    cbins.assign(items.size() * kCubeBins, 0);
    std::vector<int32_t> cls;
    for (size_t k = 0; k < items.size(); ++k) {
      const SpreadItem& itm = items[k];
      const long long t = itm.tile;
      const int o[3] = {int(t / ((long long)tp.nt1 * tp.nt2)) * 8, int((t / tp.nt2) % tp.nt1) * 8,
                        int(t % tp.nt2) * 8};
      const int n = itm.end - itm.begin;
      cls.resize(n);
      int32_t* cb = cbins.data() + k * kCubeBins;
      for (int i = 0; i < n; ++i) {
        int hb[3], c = 0;
        unpack_base(base[(size_t)list[itm.begin + i]], hb[0], hb[1], hb[2]);
        for (int a = 0; a < 3; ++a) {
          int r = hb[a] - o[a];
          if (r < 0) r += gsz[a];
          if (r >= 8) r -= gsz[a];
          c = 3 * c + (r <= 4 - W ? 0 : r < 4 ? 1 : 2);
        }
        cls[i] = c;
        cb[c + 1]++;
      }
      for (int c = 0; c < kCubeBins - 1; ++c) cb[c + 1] += cb[c];
      std::vector<int32_t> at(cb, cb + kCubeBins - 1);
      for (int i = 0; i < n; ++i) {
        const int32_t si = list[itm.begin + i];
        clist2[itm.begin + at[cls[i]]++] = make_int2(si, perm[si]);
      }
    }
  }
  hs->list.resize(list_len);
  for (long long i = 0; i < list_len; ++i) hs->list[i] = make_int2(list[i], perm[list[i]]);
  return NRSENSE_OK;
}

nrsense_status upload_pointset(nrsense_plan_s* p, const HostSet& hs, PointSet* ps, cudaStream_t s) {
  ps->tp = hs.tp;
  ps->npts = hs.npts;
  ps->list_len = hs.list_len;
  ps->n_items = int(hs.items.size());
  ps->n_reduces = int(hs.reds.size());
  ps->n_slots = hs.slots;
  ps->n_occupied = hs.occupied;
  ps->longest_item = hs.longest_item;
  ps->n_iitems = int(hs.iitems.size());
  auto put = [&](auto** dst, const auto& src) -> nrsense_status {
    NRS_TRY(dev_alloc_n(p, dst, std::max<long long>((long long)src.size(), 1)));
    return upload(*dst, src, s);
  };
  NRS_TRY(put(&ps->qs, hs.qs));
  NRS_TRY(put(&ps->perm, hs.perm));
  NRS_TRY(put(&ps->list, hs.list));
  NRS_TRY(put(&ps->items, hs.items));
  NRS_TRY(put(&ps->bins, hs.bins));
  NRS_TRY(put(&ps->reduces, hs.reds));
  NRS_TRY(put(&ps->iitems, hs.iitems));
  if (hs.cube) {
    NRS_TRY(put(&ps->clist, hs.clist));
    NRS_TRY(put(&ps->cbins, hs.cbins));
  }
  return NRSENSE_OK;
}

nrsense_status build_pointset(nrsense_plan_s* p, const std::vector<HostPoint>& pts, PointSet* ps,
                              const TilePlan& tp, const std::vector<char>* write_mask, bool interp,
                              int max_item, cudaStream_t s) {
  HostSet hs;
  NRS_TRY(compute_pointset(p->geo, p->W, pts, tp, write_mask, interp, max_item, &hs));
  return upload_pointset(p, hs, ps, s);
}

// samples whose host lists a plan's creation holds at once (several phases)
constexpr long long kHostListPoints = 8 << 20;

// f(j) for j < n in threads (at most one per core); the first failure's status.
template <class F>
nrsense_status for_phases(int n, F&& f) {
  const int nt = std::min<int>(n, std::max(1u, std::thread::hardware_concurrency()));
  std::vector<nrsense_status> st((size_t)n, NRSENSE_OK);
  auto work = [&](int k) {
    for (int j = k; j < n; j += nt) {
      try {
        st[(size_t)j] = f(j);
      } catch (const std::exception&) {
        st[(size_t)j] = NRSENSE_ERR_OOM;
      }
    }
  };
  std::vector<std::thread> pool;
  int started = 1;
  try {
    pool.reserve((size_t)nt);
    for (; started < nt; ++started) pool.emplace_back(work, started);
  } catch (const std::exception&) {
    // no more threads, or no memory for their state: this one takes the rest
  }
  work(0);
  for (std::thread& t : pool) t.join();
  for (int k = started; k < nt; ++k) work(k);
  for (nrsense_status v : st)
    if (v != NRSENSE_OK) return v;
  return NRSENSE_OK;
}

// Displaced voxel positions from the plan's displacements, on the host.
nrsense_status host_image_points(nrsense_plan_s* p, std::vector<HostPoint>& pts, cudaStream_t s) {
  const Geo& g = p->geo;
  const long long nd = (long long)p->P * 3 * g.nvox;
  const double sigma = double(g.g0) / double(g.n0);
  std::vector<float> hd((size_t)nd);
  if (cudaMemcpyAsync(hd.data(), p->disp, size_t(nd) * sizeof(float), cudaMemcpyDeviceToHost, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return NRSENSE_ERR_CUDA;
  for (long long i = 0; i < nd; ++i)
    if (!std::isfinite(hd[i]) || std::fabs(hd[i]) > 1e6f) return NRSENSE_ERR_ARG;
  pts.resize((size_t)(p->P * g.nvox));
  const int gs[3] = {g.g0, g.g1, g.g2};
  for (int j = 0; j < p->P; ++j) {
    const float* dj = hd.data() + (long long)j * 3 * g.nvox;
    for (long long v = 0; v < g.nvox; ++v) {
      const int i2 = int(v % g.n2);
      const int i1 = int((v / g.n2) % g.n1);
      const int i0 = int(v / ((long long)g.n1 * g.n2));
      const int ii[3] = {i0, i1, i2};
      HostPoint& h = pts[(size_t)(j * g.nvox + v)];
      for (int a = 0; a < 3; ++a) {
        // q = sigma * (n + d) = sigma*n + sigma*d in FP64 (sigma*n exact)
        const double q = sigma * double(ii[a]) + sigma * double(dj[a * g.nvox + v]);
        decompose(q, gs[a], p->W, &h.b[a], &h.f[a]);
      }
      h.row = int32_t(j * g.nvox + v);
    }
  }
  return NRSENSE_OK;
}

// The displaced voxels grouped by the block of edge 1 << shift of their first tap
// (cells: by cell within it), stable: on the device (plan_image.cu), or on the
// host where a group is too crowded for that.
nrsense_status sorted_image_points(nrsense_plan_s* p, int shift, bool cells, const float4** qs,
                                   const int32_t** perm, const int32_t** start, cudaStream_t s) {
  const Geo& g = p->geo;
  const int e = 1 << shift, m = e - 1;
  const int nb1 = (g.g1 + m) / e, nb2 = (g.g2 + m) / e;
  const size_t groups = (size_t)((g.g0 + m) / e) * nb1 * nb2;
  const long long n = (long long)p->P * g.nvox;
  float4* dq = nullptr;
  int32_t *dp = nullptr, *ds = nullptr;
  NRS_TRY(dev_alloc_n(p, &dq, n));
  NRS_TRY(dev_alloc_n(p, &dp, n));
  NRS_TRY(dev_alloc_n(p, &ds, (long long)groups + 1));
  *qs = dq;
  *perm = dp;
  *start = ds;
  if (fault_requested("upload")) return NRSENSE_ERR_CUDA;
  bool bad = false, done = false;
  NRS_TRY(sort_image_points(g, p->W, double(g.g0) / double(g.n0), n, p->disp, shift, cells, dq, dp, ds,
                            &bad, &done, s));
  if (bad) return NRSENSE_ERR_ARG;
  if (done) return NRSENSE_OK;
  std::vector<HostPoint> pts;
  NRS_TRY(host_image_points(p, pts, s));
  std::vector<std::pair<uint64_t, int32_t>> ko((size_t)n);  // (group, cell), index
  std::vector<int32_t> st(groups + 1, 0);
  for (long long i = 0; i < n; ++i) {
    const HostPoint& h = pts[(size_t)i];
    const uint64_t k = ((uint64_t)(h.b[0] >> shift) * nb1 + (h.b[1] >> shift)) * nb2 + (h.b[2] >> shift);
    const uint64_t cell = cells ? (((h.b[0] & m) * e) + (h.b[1] & m)) * e + (h.b[2] & m) : 0;
    ko[(size_t)i] = {k << 32 | cell, int32_t(i)};
    st[(size_t)k + 1]++;
  }
  std::sort(ko.begin(), ko.end());
  for (size_t k = 0; k < groups; ++k) st[k + 1] += st[k];
  std::vector<float4> hq((size_t)n);
  std::vector<int32_t> hp((size_t)n);
  for (long long k = 0; k < n; ++k) {
    const HostPoint& h = pts[(size_t)ko[(size_t)k].second];
    const uint32_t packed = pack_base(h.b[0], h.b[1], h.b[2]);
    float w;
    std::memcpy(&w, &packed, sizeof(w));
    hq[(size_t)k] = make_float4(h.f[0], h.f[1], h.f[2], w);
    hp[(size_t)k] = h.row;
  }
  NRS_TRY(upload(dq, hq, s));
  NRS_TRY(upload(dp, hp, s));
  return upload(ds, st, s);
}

// Image-space points sorted by the 8^3 home tile of their first tap, then by
// cell (the order of the home-tile spread, spread_home.cu), with the first
// sorted index of every home tile, and the super-tile scratch.
nrsense_status build_home_set(nrsense_plan_s* p, cudaStream_t s) {
  const Geo& g = p->geo;
  if (p->home_scratch != nullptr) return NRSENSE_OK;  // built
  Rollback undo(p);
  HomeSet hs{};
  hs.nt0 = (g.g0 + 7) / 8;
  hs.nt1 = (g.g1 + 7) / 8;
  hs.nt2 = (g.g2 + 7) / 8;
  hs.ns0 = (g.g0 + 15) / 16;
  hs.ns1 = (g.g1 + 15) / 16;
  hs.ns2 = (g.g2 + 15) / 16;
  NRS_TRY(sorted_image_points(p, 3, true, &hs.qs, &hs.perm, &hs.tstart, s));
  // per axis and coordinate: the super-tiles whose 3-point-padded extents
  // cover it (directly or wrapped around the periodic grid), increasing
  const int gsz[3] = {g.g0, g.g1, g.g2}, nsz[3] = {hs.ns0, hs.ns1, hs.ns2};
  const int4** cov[3] = {&hs.cover0, &hs.cover1, &hs.cover2};
  for (int a = 0; a < 3; ++a) {
    std::vector<int4> tab(gsz[a]);
    for (int x = 0; x < gsz[a]; ++x) {
      int e[3] = {0, 0, 0}, n = 0;
      for (int c = 0; c < nsz[a]; ++c) {
        const int o = 16 * c, ext = std::min(16, gsz[a] - o);
        for (int u : {x, x + gsz[a]})
          if (u >= o && u < o + ext + 3) {
            if (n == 3) return NRSENSE_ERR_ARG;  // cannot happen for grids >= 11 points
            e[n++] = c * 32 + (u - o);
          }
      }
      tab[x] = make_int4(n, e[0], e[1], e[2]);
    }
    int4* dtab = nullptr;
    NRS_TRY(dev_alloc_n(p, &dtab, (long long)tab.size()));
    NRS_TRY(upload(dtab, tab, s));
    if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
    *cov[a] = dtab;
  }
  if (configure_home_kernels() != cudaSuccess) return NRSENSE_ERR_CUDA;
  nrsense_c64* scratch = nullptr;
  NRS_TRY(dev_alloc_n(p, &scratch, home_scratch_elems(hs)));
  undo.keep = true;
  p->ihome = hs;
  p->home_scratch = scratch;
  return NRSENSE_OK;
}

// Image-space points sorted by the 4^3 block of their first tap (stable), with
// the first sorted index of every block (spread_rows.cu); not kept (rows_ok stays
// false) where the displacement gathers the points in so few rows that the warp with
// the most of them decides the time: a row is one warp's, about 30 (W = 4) or 48 ns a
// point, while the home tiles (W = 4) and the split halo lists (W = 6) deal a crowd to
// more warps.  T^H of images contracted about their centre, points of the fullest warp,
// rows against home tiles: 64^3 540 0.053 / 0.053 ms, 1280 0.092 / 0.082; 128^3 1656
// 0.262 / 0.304, 4096 0.361 / 0.296, 15876 0.825 / 0.447.  W = 6 against halo lists: 64^3
// 3456 0.35 / 0.70, 16000 0.94 / 1.00, 78400 3.7 / 1.05; 128^3 9792 1.21 / 2.64, 34400
// 3.15 / 2.81, 172800 9.5 / 2.93.  Motion of some voxels stays far below: 160 to 1250 at
// 16^3 to 192^3.
nrsense_status build_row_set(nrsense_plan_s* p, cudaStream_t s) {
  const Geo& g = p->geo;
  Rollback undo(p);
  RowSet rs{};
  rs.nb0 = g.g0 / 4;
  rs.nb1 = g.g1 / 4;
  rs.nb2 = g.g2 / 4;
  NRS_TRY(sorted_image_points(p, 2, false, &rs.qs, &rs.perm, &rs.start, s));
  int32_t* most = nullptr;
  int32_t load = 0;
  NRS_TRY(dev_alloc_n(p, &most, 1));
  if (cudaMemsetAsync(most, 0, sizeof(load), s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  launch_row_load(p->W, rs, most, s);
  if (cudaMemcpyAsync(&load, most, sizeof(load), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return NRSENSE_ERR_CUDA;
  dev_free(p, most);
  const long long n = (long long)p->P * g.nvox;
  if (load > (p->W == 4 ? 400 + n / 1000 : 16000 + n / 128)) return NRSENSE_OK;
  undo.keep = true;
  p->irows = rs;
  p->rows_ok = true;
  return NRSENSE_OK;
}

// scratch for split tiles of the k-space spread: slots x coil chunks x tile x
// chunk coils (grown, never shrunk)
nrsense_status ensure_scratch(nrsense_plan_s* p) {
  long long need = 0;
  auto tile_pts = [](const PointSet& ps) {
    return (long long)ps.tp.t0 * ps.tp.t1 * ps.tp.t2;
  };
  if (p->C > 0) {
    const int cc = spread_coil_chunk(p->C);
    const int chunks = (p->C + cc - 1) / cc;
    for (int j0 = 0; j0 < p->P; j0 += p->phase_chunk) {
      long long slots = 0;
      for (int j = j0; j < std::min(p->P, j0 + p->phase_chunk); ++j) slots += p->kpts[j].n_slots;
      need = std::max(need, slots * chunks * tile_pts(p->kpts[j0]) * cc);
    }
  }
  if (need <= p->scratch_elems) return NRSENSE_OK;
  nrsense_c64* larger = nullptr;
  NRS_TRY(dev_alloc_n(p, &larger, need));
  dev_free(p, p->b_scratch);
  p->b_scratch = larger;
  p->scratch_elems = need;
  p->epoch += 1;  // captured graphs hold the old address
  return NRSENSE_OK;
}

// halo lists of the displaced voxels (the spread over per-tile lists)
nrsense_status build_image_lists(nrsense_plan_s* p, cudaStream_t s) {
  if (p->ipts.qs != nullptr) return NRSENSE_OK;  // built
  Rollback undo(p);
  std::vector<HostPoint> pts;
  NRS_TRY(host_image_points(p, pts, s));
  PointSet lists;
  NRS_TRY(build_pointset(p, pts, &lists, p->itiles, nullptr, /*interp=*/false, kSpreadMaxItemImage, s));
  // partial tiles of their own: the k-space spread's scratch stays where it is
  nrsense_c64* scratch = nullptr;
  NRS_TRY(dev_alloc_n(p, &scratch, (long long)lists.n_slots * lists.tp.t0 * lists.tp.t1 * lists.tp.t2));
  undo.keep = true;
  p->ipts = lists;
  p->image_scratch = scratch;
  return NRSENSE_OK;
}

nrsense_status cufft_check(cufftResult r) {
  return r == CUFFT_SUCCESS ? NRSENSE_OK : NRSENSE_ERR_CUFFT;
}

// Radices and twiddle tables of the mixed-radix passes, where every axis has
// them.  Compensated and BF16-storage plans keep the cuFFT path: the one asks
// for its accuracy, the other rounds its coil grids to 8 bits, where any change
// of the last FP32 bit before it moves results by a BF16 step.
nrsense_status create_mixed(nrsense_plan_s* p, cudaStream_t s) {
  const Geo& g = p->geo;
  const int gs[3] = {g.g0, g.g1, g.g2}, ns[3] = {g.n0, g.n1, g.n2};
  if (p->comp_spread || p->grid_bf16) return NRSENSE_OK;
  MixAxis ax[3];
  for (int a = 0; a < 3; ++a)
    if (!mix_axis(ns[a], gs[a], &ax[a])) return NRSENSE_OK;
  if (mixed_max_smem(ax) > kMixedMaxSmem) return NRSENSE_OK;
  std::vector<float2> tw;
  for (int k = 0; k < 6; ++k) {
    const int L = k < 3 ? gs[k] : ns[k - 3];
    for (int j = 0; j < L; ++j)
      tw.push_back(make_float2(float(std::cos(2.0 * M_PI * j / L)), float(-std::sin(2.0 * M_PI * j / L))));
  }
  float2* d = nullptr;
  NRS_TRY(dev_alloc_n(p, &d, (long long)tw.size()));
  NRS_TRY(upload(d, tw, s));
  const float2* dn = d + gs[0] + gs[1] + gs[2];
  for (int a = 0; a < 3; ++a) {
    ax[a].tw_g = d;
    ax[a].tw_n = dn;
    d += gs[a];
    dn += ns[a];
    p->mix[a] = ax[a];
  }
  if (configure_mixed(g, p->mix) != cudaSuccess) return NRSENSE_ERR_CUDA;
  p->image_mixed = !p->identity_warp;
  return NRSENSE_OK;
}

nrsense_status create_impl(nrsense_plan_s* p, const nrsense_desc* desc, const int64_t* n_samples,
                           const float* coords, const float* disp, const nrsense_c64* smaps,
                           cudaStream_t s) {
  const nrsense_desc& d = *desc;
  for (int a = 0; a < 3; ++a)
    if (d.n[a] < 4 || (d.n[a] & 1)) return NRSENSE_ERR_ARG;
  // oversampled grid: osf * n, or given per axis (a rational sigma = G / n)
  const bool explicit_grid = d.grid[0] > 0 && d.grid[1] > 0 && d.grid[2] > 0;
  if (!explicit_grid && (d.grid[0] != 0 || d.grid[1] != 0 || d.grid[2] != 0)) return NRSENSE_ERR_ARG;
  int gsize[3];
  if (explicit_grid) {
    for (int a = 0; a < 3; ++a) {
      gsize[a] = d.grid[a];
      if (4 * gsize[a] < 5 * d.n[a] || gsize[a] > 4 * d.n[a]) return NRSENSE_ERR_ARG;
      if ((long long)gsize[a] * d.n[0] != (long long)gsize[0] * d.n[a]) return NRSENSE_ERR_ARG;
    }
  } else {
    if (d.osf < 2 || d.osf > 4) return NRSENSE_ERR_ARG;
    for (int a = 0; a < 3; ++a) gsize[a] = d.osf * d.n[a];
  }
  if (d.kb_width != 4 && d.kb_width != 6) return NRSENSE_ERR_ARG;
  if (d.n_phases < 1 || d.n_coils < 0) return NRSENSE_ERR_ARG;
  if (d.precision != NRSENSE_FP32 && d.precision != NRSENSE_BF16_STORE &&
      d.precision != NRSENSE_FP32_COMPENSATED)
    return NRSENSE_ERR_ARG;
  if (d.precision == NRSENSE_FP32_COMPENSATED && d.kb_width != 4) return NRSENSE_ERR_ARG;
  if (d.precision == NRSENSE_BF16_STORE)  // cuFFT's BF16 transforms: power-of-two sizes
    for (int a = 0; a < 3; ++a) {
      const int ga = gsize[a];
      if (ga & (ga - 1)) return NRSENSE_ERR_ARG;
    }
  if (!(d.kb_beta >= 0.0) || !std::isfinite(d.kb_beta)) return NRSENSE_ERR_ARG;
  p->desc = d;
  p->identity_warp = (d.flags & NRSENSE_IDENTITY_WARP) != 0;
  p->grid_bf16 = d.precision == NRSENSE_BF16_STORE;
  p->comp_spread = d.precision == NRSENSE_FP32_COMPENSATED;
  p->P = d.n_phases;
  p->C = d.n_coils;
  p->W = d.kb_width;
  Geo& g = p->geo;
  g.n0 = d.n[0]; g.n1 = d.n[1]; g.n2 = d.n[2];
  g.g0 = gsize[0]; g.g1 = gsize[1]; g.g2 = gsize[2];
  // integer sigma (0 when sigma = G / n is not an integer)
  g.osf = (g.g0 % g.n0 == 0) ? g.g0 / g.n0 : 0;
  const double sigma = double(g.g0) / double(g.n0);
  if (g.g0 > 1024 || g.g1 > 1024 || g.g2 > 1024) return NRSENSE_ERR_ARG;  // 10-bit packed taps
  // a tile and a kernel footprint must not wrap onto each other
  const int gmin = kSpreadTile + d.kb_width - 1;
  if (g.g0 < gmin || g.g1 < gmin || g.g2 < gmin) return NRSENSE_ERR_ARG;
  g.nvox = (long long)g.n0 * g.n1 * g.n2;
  g.ngrid = (long long)g.g0 * g.g1 * g.g2;
  if ((long long)p->P * g.nvox >= (1ll << 31)) return NRSENSE_ERR_ARG;
  if (!p->identity_warp && disp == nullptr) return NRSENSE_ERR_ARG;
  if (p->C > 0 && (coords == nullptr || smaps == nullptr || n_samples == nullptr))
    return NRSENSE_ERR_ARG;
  p->beta = d.kb_beta > 0 ? d.kb_beta : beatty_beta(p->W, sigma);
  if (!(p->beta > 0)) return NRSENSE_ERR_ARG;
  p->poly_err = fit_kernel_polys(p->W, p->beta, &p->kc);

  if (configure_kernels() != cudaSuccess) return NRSENSE_ERR_CUDA;
  const TilePlan ktiles = make_tileplan(g, kSpreadTile);
  const TilePlan itiles =
      make_tileplan(g, spread_tile_edge(p->W, 1, std::min(g.g0, std::min(g.g1, g.g2))));
  p->ktiles = ktiles;
  p->itiles = itiles;

  // deapodization: 1/C(m/G) for m in [-N/2, N/2), per axis
  {
    std::vector<float> tab;
    const int ns[3] = {g.n0, g.n1, g.n2}, gs[3] = {g.g0, g.g1, g.g2};
    for (int a = 0; a < 3; ++a)
      for (int m = -ns[a] / 2; m < ns[a] / 2; ++m)
        tab.push_back(float(1.0 / kb_kernel_ft(double(m) / gs[a], p->W, p->beta)));
    NRS_TRY(dev_alloc_n(p, &p->deapod, (long long)tab.size()));
    NRS_TRY(upload(p->deapod, tab, s));
  }
  NRS_TRY(dev_alloc_n(p, &p->d_status, 1));
  if (cudaMemsetAsync(p->d_status, 0, sizeof(int32_t), s) != cudaSuccess) return NRSENSE_ERR_CUDA;

  // displacements: copy, validate, and build the image-space point set
  if (!p->identity_warp) {
    const long long nd = (long long)p->P * 3 * g.nvox;
    NRS_TRY(dev_alloc_n(p, &p->disp, nd));
    if (cudaMemcpyAsync(p->disp, disp, size_t(nd) * sizeof(float), cudaMemcpyDeviceToDevice, s) !=
        cudaSuccess)
      return NRSENSE_ERR_CUDA;
    if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
    p->ipts.tp = itiles;
    // the point order of the spread that the plan starts with (the others are
    // built when a tuning choice needs them).  Rows against home tiles, points per
    // grid value: 1/8 (one phase at sigma 2) 0.695 against 1.08 ms at 384^3, 1/4
    // (two phases) 0.40 against 0.40 ms at 256^3, 1/2 0.76 against 0.59: the home
    // tiles' fixed cost per tile (accumulators, merge, rims) against the rows' four
    // visits per point
    const bool rows = !p->comp_spread && !p->grid_bf16 && g.g0 % 4 == 0 && g.g1 % 4 == 0 &&
                      g.g2 % 4 == 0;
    p->home_ok = p->W == 4 && !p->comp_spread;
    if (p->home_ok) p->spread_image_variant = kSpreadHome;
    if (rows && (p->W != 4 || 6 * p->P * g.nvox <= g.ngrid)) NRS_TRY(build_row_set(p, s));
    p->rows_sparse = p->rows_ok && p->W == 4;
    if (!p->rows_ok) NRS_TRY(p->home_ok ? build_home_set(p, s) : build_image_lists(p, s));
    // Interpolation until the plan is tuned (the same values, but for the last bit where a
    // negative displacement below 1e-7 rounds up to the grid point in FP64): a thread per
    // voxel, or from super-tiles staged in shared memory.  Per voxel at sigma 2: 0.324
    // against 0.429 ms at 192^3 with one phase, 0.302 against 0.311 at 128^3 with four;
    // but 0.571 against 0.480 with eight (0.248 against 0.202 at 96^3, equal at 64^3; without
    // the rigid shifts that part the phases' taps 0.542 against 0.563).
    // A rational sigma decomposes every position in FP64, which the super-tiles' sorted
    // points hold ready: 0.387 against 0.101 ms at 128^3, sigma 1.5; with no more CTAs
    // than SMs that hides (0.014 against 0.020 ms at 32^3; 0.030 against 0.019 at 48^3).
    const bool many = 4 * p->P * g.nvox >= 3 * g.ngrid && g.nvox > 64 * 64 * 64;
    p->interp_home = p->home_ok && (g.osf == 0 ? g.nvox > 152 * 256 : many);
    if (p->interp_home) NRS_TRY(build_home_set(p, s));
  }

  // coils and k-space
  if (p->C > 0) {
    p->M.assign(n_samples, n_samples + p->P);
    p->off.resize(p->P);
    long long tot = 0;
    for (int j = 0; j < p->P; ++j) {
      if (p->M[j] < 0 || p->M[j] >= (1ll << 31)) return NRSENSE_ERR_ARG;
      p->off[j] = tot;
      tot += p->M[j];
    }
    p->Mtot = tot;
    const long long nm = g.nvox * p->C;
    NRS_TRY(dev_alloc_n(p, &p->smaps, nm));
    if (cudaMemcpyAsync(p->smaps, smaps, size_t(nm) * sizeof(nrsense_c64), cudaMemcpyDeviceToDevice,
                        s) != cudaSuccess)
      return NRSENSE_ERR_CUDA;

    std::vector<float> hc(size_t(3 * tot));
    if (tot > 0) {
      if (cudaMemcpyAsync(hc.data(), coords, size_t(3 * tot) * sizeof(float),
                          cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess)
        return NRSENSE_ERR_CUDA;
    }
    p->kpts.resize(p->P);
    const int gs[3] = {g.g0, g.g1, g.g2};
    std::vector<std::vector<HostPoint>> all((size_t)p->P);
    std::vector<std::vector<char>> touch((size_t)p->P);
    NRS_TRY(for_phases(p->P, [&](int j) -> nrsense_status {
      std::vector<HostPoint>& pts = all[(size_t)j];
      pts.resize((size_t)p->M[j]);
      for (long long i = 0; i < p->M[j]; ++i) {
        HostPoint& h = pts[(size_t)i];
        for (int a = 0; a < 3; ++a) {
          const float om = hc[size_t(3 * (p->off[j] + i) + a)];
          if (!std::isfinite(om)) return NRSENSE_ERR_ARG;
          // q = omega G / (2 pi) in FP64; periodic, so any finite omega wraps
          const double q = double(om) * double(gs[a]) / (2.0 * M_PI);
          decompose(q, gs[a], p->W, &h.b[a], &h.f[a]);
        }
        h.row = int32_t(i);
      }
      touch[(size_t)j].assign((size_t)ktiles.ntiles, 0);
      mark_touched_tiles(p, ktiles, pts, touch[(size_t)j]);
      return NRSENSE_OK;
    }));
    // all phases share one spread target: each phase writes every tile that
    // any phase occupies (zeros where it has no points), the rest stay zero
    std::vector<char> uni((size_t)ktiles.ntiles, 0);
    for (const std::vector<char>& t : touch)
      for (size_t k = 0; k < uni.size(); ++k) uni[k] |= t[k];
    long long nuni = 0;
    for (char u : uni) nuni += u != 0;
    p->kuni_fraction = double(nuni) / double(uni.size());
    // per (y, x) tile column, a bit per z tile of the union: the pruned
    // transforms store (forward) and load (adjoint) only those tiles
    {
      const size_t cols = (size_t)ktiles.nt1 * ktiles.nt2;
      std::vector<uint32_t> cm(cols * ((ktiles.nt0 + 31) / 32), 0u);
      std::vector<char> any(cols, 0);
      for (long long t = 0; t < ktiles.ntiles; ++t)
        if (uni[(size_t)t]) {
          const size_t col = size_t(t) % cols, z = size_t(t) / cols;
          cm[(z >> 5) * cols + col] |= 1u << (z & 31);
          any[col] = 1;
        }
      long long ncol = 0;
      for (char v : any) ncol += v;
      p->kcol_fraction = ktiles.nt0 <= 32 ? double(ncol) / double(cols) : 1.0;
      NRS_TRY(dev_alloc_n(p, &p->kcolmask, (long long)cm.size()));
      NRS_TRY(upload(p->kcolmask, cm, s));
      std::vector<uint32_t> am((size_t)ktiles.nt2 * ((ktiles.nt1 + 31) / 32), 0u);
      for (size_t c = 0; c < cols; ++c)
        if (any[c]) {
          const size_t y = c / ktiles.nt2;
          am[(y >> 5) * ktiles.nt2 + c % ktiles.nt2] |= 1u << (y & 31);
        }
      NRS_TRY(dev_alloc_n(p, &p->kanymask, (long long)am.size()));
      NRS_TRY(upload(p->kanymask, am, s));
    }
    // The phases' lists in turn, as many at once as hold kHostListPoints samples
    // together: about 120 bytes of host memory a sample, 1 GB, beside the samples' own
    // records (one phase alone takes what it needs).
    for (int j0 = 0; j0 < p->P;) {
      int j1 = j0;
      for (long long n = 0; j1 < p->P && (j1 == j0 || n + p->M[j1] <= kHostListPoints); ++j1) n += p->M[j1];
      std::vector<HostSet> sets((size_t)(j1 - j0));
      NRS_TRY(for_phases(j1 - j0, [&](int k) -> nrsense_status {
        std::vector<HostPoint>& pts = all[(size_t)(j0 + k)];
        const nrsense_status st = compute_pointset(g, p->W, pts, ktiles, &uni, /*interp=*/true,
                                                   p->spread_max_item, &sets[(size_t)k]);
        std::vector<HostPoint>().swap(pts);
        return st;
      }));
      for (; j0 < j1; ++j0) {
        HostSet& hs = sets[sets.size() - size_t(j1 - j0)];
        NRS_TRY(upload_pointset(p, hs, &p->kpts[(size_t)j0], s));
        hs = HostSet{};
      }
    }
    p->kunion.swap(uni);
  }

  // cuFFT plans
  if (fault_requested("cufft")) return NRSENSE_ERR_CUFFT;
  if (!p->identity_warp) {
    NRS_TRY(cufft_check(cufftPlan3d(&p->fft_n, g.n0, g.n1, g.n2, CUFFT_C2C)));
    p->have_fft_n = true;
    NRS_TRY(cufft_check(cufftPlan3d(&p->fft_g, g.g0, g.g1, g.g2, CUFFT_C2C)));
    p->have_fft_g = true;
  }
  if (p->C > 0) {
    // phases per launch: as many as half of the free memory allows (four
    // coil-grid buffers per phase plus about one for cuFFT's work area)
    const long long elem = p->grid_bf16 ? 4 : 8;  // bytes per stored complex value
    const long long per_phase = 5LL * p->C * g.ngrid * elem;
    int pc = d.phase_chunk;
    if (pc <= 0) {
      size_t free_b = 0, total_b = 0;
      if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) return NRSENSE_ERR_CUDA;
      pc = int(std::max<long long>(1, (long long)(free_b / 2) / per_phase));
    }
    pc = std::max(1, std::min(pc, std::min(p->P, kMaxChunkPhases)));
    p->phase_chunk = pc;
    // pruned coil-grid transforms (FP32 C2C or BF16 through cufftXt)
    const long long plane = (long long)g.g1 * g.g2;
    long long n2[2] = {g.g1, g.g2};
    long long nz[1] = {g.g0};
    auto make = [&](cufftHandle* h, int rank, long long* n, long long* emb, long long stride,
                    long long dist, long long batch) -> nrsense_status {
      if (cufftCreate(h) != CUFFT_SUCCESS) return NRSENSE_ERR_CUFFT;
      size_t work = 0;
      const cufftResult r =
          p->grid_bf16
              ? cufftXtMakePlanMany(*h, rank, n, emb, stride, dist, CUDA_C_16BF, emb, stride, dist,
                                    CUDA_C_16BF, batch, &work, CUDA_C_16BF)
              : cufftMakePlanMany64(*h, rank, n, emb, stride, dist, emb, stride, dist, CUFFT_C2C,
                                    batch, &work);
      if (r != CUFFT_SUCCESS) {
        cufftDestroy(*h);
        return NRSENSE_ERR_CUFFT;
      }
      return NRSENSE_OK;
    };
    NRS_TRY(make(&p->fft_p2, 2, n2, n2, 1, plane, g.n0));
    nrsense_status st2 = make(&p->fft_p2h, 2, n2, n2, 1, plane, g.n0 / 2);
    if (st2 != NRSENSE_OK) {
      cufftDestroy(p->fft_p2);
      return st2;
    }
    st2 = make(&p->fft_z, 1, nz, nz, plane, 1, plane);
    if (st2 != NRSENSE_OK) {
      cufftDestroy(p->fft_p2);
      cufftDestroy(p->fft_p2h);
      return st2;
    }
    p->have_gc = true;
  }

  // work buffers
  NRS_TRY(dev_alloc_n(p, &p->b_m, (long long)p->P * g.nvox));
  NRS_TRY(dev_alloc_n(p, &p->b_tmp, g.nvox));
  if (!p->identity_warp) {
    NRS_TRY(dev_alloc_n(p, &p->b_xhat, g.nvox));
    NRS_TRY(dev_alloc_n(p, &p->b_upad, g.ngrid));
    NRS_TRY(dev_alloc_n(p, &p->b_ugrid, g.ngrid));
    if (cudaMemsetAsync(p->b_upad, 0, size_t(g.ngrid) * sizeof(nrsense_c64), s) != cudaSuccess)
      return NRSENSE_ERR_CUDA;
    // the pruned image-space passes: their T1 and T2 (6 N^3 values) fit in b_upad (8 N^3)
    p->image_fft_ok = pruned_image_fft_supported(g) && !p->comp_spread;
    p->image_fft_pruned = p->image_fft_ok;
  }
  NRS_TRY(create_mixed(p, s));
  if (p->C > 0) {
    const size_t cgb = size_t(g.ngrid) * p->C * p->phase_chunk * (p->grid_bf16 ? 4 : 8);
    NRS_TRY(dev_alloc(p, &p->b_xpad, cgb));
    NRS_TRY(dev_alloc(p, &p->b_xwork, cgb));
    NRS_TRY(dev_alloc(p, &p->b_xspread, cgb));
    NRS_TRY(dev_alloc(p, &p->b_xmid, cgb));
    if (cudaMemsetAsync(p->b_xmid, 0, cgb, s) != cudaSuccess) return NRSENSE_ERR_CUDA;
    // own pruned transforms where supported (chosen by default; the autotuner
    // times both paths)
    p->fft_pruned_ok = pruned_fft_supported(g, p->C, p->grid_bf16) && init_pruned_fft() == cudaSuccess;
    p->fft_pruned = p->fft_pruned_ok;
    // Power-of-two grids up to 256 have both kinds of passes; the mixed-radix ones are the
    // faster along 128 points, the power-of-two ones along 256 and, barely, along 32 and
    // 64.  Mixed against power-of-two, ms forward and adjoint, 8 coils, one / four phases: 128^3
    // grid 0.147 / 0.474 against 0.154 / 0.530, z y x = 128 128 64 0.083 / 0.251 against 0.084 /
    // 0.275, 128 128 256 0.253 / 0.863 against 0.275 / 0.957; but 64 128 128 0.099 / 0.260 against
    // 0.087 / 0.266, 128 64 32 0.051 against 0.046, 256^3 0.86 / 3.39 against 0.79 / 3.11.  So by
    // the two axes whose passes run over the padded columns.
    // Grids of 1024 points along z and about as many along another axis stay with
    // cuFFT: at 1024 points, its best length, the in-place passes hold 131 KB of shared
    // memory, a CTA per SM, and transform the zero half too.  Two coils forward and
    // adjoint, own passes against cuFFT: 1024^3 40.9 / 31.8 ms (24.6 / 22.5 at sigma 4),
    // 1024 x 192 x 960 13.3 / 11.9, 1024 x 1024 x 64 (four coils) 4.6 / 3.9; but 1024 x 864 x
    // 864 25.1 / 31.1, 512 x 1024 x 1024 14.8 / 18.9, 960^3 34.4 / 47.1.
    const bool cufft_1024 = g.g0 == 1024 && (g.g1 == 1024 || g.g2 >= 896);
    p->coil_mixed = p->mix[0].N > 0 && !cufft_1024 &&
                    (!p->fft_pruned_ok || (g.g0 == 128 && g.g1 == 128));
    // tensor maps of the interpolation input (TMA-staged halos, W = 4)
    const long long slots = (long long)p->C * p->phase_chunk;
    // a test-only limit on the halo wait (0 makes every TMA-staged CTA time out)
    if (const char* lim = std::getenv("NRSENSE_TMA_POLL_LIMIT")) p->tma_poll_limit = std::atoll(lim);
    p->tma_ok = p->W == 4 &&
                make_grid_tensor_map(&p->tmap_xwork4, p->b_xwork, g, slots, p->grid_bf16, 4) &&
                make_grid_tensor_map(&p->tmap_xwork8, p->b_xwork, g, slots, p->grid_bf16, 8) &&
                make_grid_tensor_map(&p->tmap_xwork2, p->b_xwork, g, slots, p->grid_bf16, 2);
    // launch choices until the plan is tuned.  Interpolation from TMA-staged halos
    // of 4 coils (bitwise the per-value staging's results; 1.60 against 2.97 ms
    // at 128^3, 8 coils, 4 phases; the tuned choice there).  FP32 spread by
    // sub-blocks: on the tensor cores with sums of the register kernel's accuracy
    // (CubeSum::kHalves; 5 to 8 coils and chunks of 8; 256^3, 16 coils, 3 M samples: below
    // 4.5 ms against 6.50 of the register kernel), or by FMAs (1 and 2 coils, where that is the faster one:
    // few_pays, kernels_spread.cu; with 3 and 4 coils the register kernel is the faster
    // one on dense samples, 0.495 against 0.634 ms at 128^3, and the tuner times both).
    // BF16 grids keep the register kernel and its exact summation order.
    if (p->tma_ok) {
      p->interp_tma = true;
      p->interp_coils = p->C <= 2 ? 2 : 4;
    }
    if (p->W == 4 && !p->grid_bf16 && !p->comp_spread && (p->C <= 2 || p->C > 4))
      p->spread_variant = kSpreadCubeExact;
    // empty tiles of the spread target are never written: zero them once
    if (cudaMemsetAsync(p->b_xspread, 0, cgb, s) != cudaSuccess) return NRSENSE_ERR_CUDA;
    NRS_TRY(dev_alloc_n(p, &p->b_y, std::max<long long>(p->Mtot * p->C, 1)));
    if (cudaMemsetAsync(p->b_xpad, 0, cgb, s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  }
  NRS_TRY(ensure_scratch(p));
  if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  return NRSENSE_OK;
}

void release(nrsense_plan_s* p) {
  cg_release(p);
  fista_release(p);
  motion_release(p);
  for (cudaEvent_t e : p->prof_events) cudaEventDestroy(e);
  p->prof_events.clear();
  if (p->have_fft_n) cufftDestroy(p->fft_n);
  if (p->have_fft_g) cufftDestroy(p->fft_g);
  if (p->have_gc) {
    cufftDestroy(p->fft_p2);
    cufftDestroy(p->fft_p2h);
    cufftDestroy(p->fft_z);
    p->have_gc = false;
  }
  for (void* a : p->allocations) cudaFree(a);
  p->allocations.clear();
  p->allocation_bytes.clear();
}

}  // namespace

namespace nrs {

nrsense_status ensure_image_sets(nrsense_plan_s* p, bool lists, bool home, cudaStream_t s) {
  if (p->identity_warp) return NRSENSE_OK;
  try {
    if (lists) NRS_TRY(build_image_lists(p, s));
    if (home) NRS_TRY(build_home_set(p, s));
  } catch (const std::bad_alloc&) {
    return NRSENSE_ERR_OOM;
  }
  return NRSENSE_OK;
}

static nrsense_status retile_impl(nrsense_plan_s* p, int max_item, cudaStream_t s) {
  p->epoch += 1;  // point-set buffers are rebuilt
  if (max_item < 64 || max_item > (1 << 16)) return NRSENSE_ERR_ARG;
  if (p->C == 0 || max_item == p->spread_max_item) {
    p->spread_max_item = p->C == 0 ? p->spread_max_item : max_item;
    return NRSENSE_OK;
  }
  if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  for (int j = 0; j < p->P; ++j) {
    PointSet& ps = p->kpts[j];
    // the sorted points, back to host records (their order is kept by the
    // stable sort of build_pointset)
    std::vector<float4> qs((size_t)ps.npts);
    std::vector<int32_t> perm((size_t)ps.npts);
    if (ps.npts > 0 &&
        (cudaMemcpyAsync(qs.data(), ps.qs, qs.size() * sizeof(float4), cudaMemcpyDeviceToHost,
                         s) != cudaSuccess ||
         cudaMemcpyAsync(perm.data(), ps.perm, perm.size() * sizeof(int32_t),
                         cudaMemcpyDeviceToHost, s) != cudaSuccess ||
         cudaStreamSynchronize(s) != cudaSuccess))
      return NRSENSE_ERR_CUDA;
    std::vector<HostPoint> pts((size_t)ps.npts);
    for (size_t i = 0; i < pts.size(); ++i) {
      uint32_t packed;
      std::memcpy(&packed, &qs[i].w, sizeof(packed));
      unpack_base(packed, pts[i].b[0], pts[i].b[1], pts[i].b[2]);
      pts[i].f[0] = qs[i].x;
      pts[i].f[1] = qs[i].y;
      pts[i].f[2] = qs[i].z;
      pts[i].row = perm[i];
    }
    // the phase's new items replace the old ones once they and the scratch that they
    // need are there: a refused allocation leaves every phase with items that fit
    PointSet fresh;
    {
      Rollback undo(p);
      NRS_TRY(build_pointset(p, pts, &fresh, ps.tp, &p->kunion, /*interp=*/true, max_item, s));
      undo.keep = true;
    }
    std::swap(ps, fresh);
    const nrsense_status st = ensure_scratch(p);
    if (st != NRSENSE_OK) std::swap(ps, fresh);
    free_pointset(p, &fresh);
    if (st != NRSENSE_OK) return st;
  }
  p->spread_max_item = max_item;
  return cudaStreamSynchronize(s) == cudaSuccess ? NRSENSE_OK : NRSENSE_ERR_CUDA;
}

nrsense_status retile_kspace(nrsense_plan_s* p, int max_item, cudaStream_t s) {
  try {
    return retile_impl(p, max_item, s);
  } catch (const std::bad_alloc&) {
    return NRSENSE_ERR_OOM;
  }
}

}  // namespace nrs

extern "C" {

nrsense_status nrsense_plan_create(const nrsense_desc* desc, const int64_t* n_samples_host,
                                   const float* coords_dev, const float* disp_dev,
                                   const nrsense_c64* smaps_dev, void* stream,
                                   nrsense_plan_t* out) {
  if (desc == nullptr || out == nullptr) return NRSENSE_ERR_ARG;
  *out = nullptr;
  auto* p = new (std::nothrow) nrsense_plan_s();
  if (p == nullptr) return NRSENSE_ERR_OOM;
  nrsense_status st;
  try {
    st = create_impl(p, desc, n_samples_host, coords_dev, disp_dev, smaps_dev,
                     static_cast<cudaStream_t>(stream));
  } catch (const std::bad_alloc&) {
    st = NRSENSE_ERR_OOM;
  }
  if (st != NRSENSE_OK) {
    cudaStreamSynchronize(static_cast<cudaStream_t>(stream));
    release(p);
    delete p;
    return st;
  }
  *out = p;
  return NRSENSE_OK;
}

nrsense_status nrsense_plan_destroy(nrsense_plan_t plan) {
  if (plan == nullptr) return NRSENSE_OK;
  cudaDeviceSynchronize();
  release(plan);
  delete plan;
  return NRSENSE_OK;
}

nrsense_status nrsense_plan_info(nrsense_plan_t p, nrsense_info* out) {
  if (p == nullptr || out == nullptr) return NRSENSE_ERR_ARG;
  std::memset(out, 0, sizeof(*out));
  out->grid[0] = p->geo.g0;
  out->grid[1] = p->geo.g1;
  out->grid[2] = p->geo.g2;
  out->kb_beta = p->beta;
  out->kernel_poly_err = p->poly_err;
  out->total_samples = p->Mtot;
  const TilePlan& ktp = p->kpts.empty() ? p->ipts.tp : p->kpts[0].tp;
  out->tile[0] = ktp.t0;
  out->tile[1] = ktp.t1;
  out->tile[2] = ktp.t2;
  out->n_tiles = ktp.ntiles;
  long long occ = 0, items = 0, split = 0;
  for (const auto& k : p->kpts) {
    occ += k.n_occupied;
    items += k.n_items;
    split += k.n_reduces;
  }
  out->occupied_fraction =
      p->kpts.empty() ? 0.0 : double(occ) / (double(ktp.ntiles) * double(p->kpts.size()));
  out->spread_items = items;
  out->split_tiles = split;
  out->device_bytes = p->device_bytes;
  out->phase_chunk = p->phase_chunk;
  out->union_fraction = p->kuni_fraction;
  out->union_columns = p->kcol_fraction;
  return NRSENSE_OK;
}

nrsense_status nrsense_profile_start(nrsense_plan_t p, int32_t max_launches) {
  if (p == nullptr || max_launches < 0 || max_launches > (1 << 20)) return NRSENSE_ERR_ARG;
  while (p->prof_events.size() < size_t(2 * max_launches)) {
    cudaEvent_t e;
    if (cudaEventCreate(&e) != cudaSuccess) return NRSENSE_ERR_CUDA;
    p->prof_events.push_back(e);
  }
  p->prof_stage.clear();
  p->prof_on = true;
  p->launches_at_start = p->launches;
  return NRSENSE_OK;
}

nrsense_status nrsense_profile_stop(nrsense_plan_t p, double* ms, int64_t* count,
                                    int64_t* own_kernels) {
  if (p == nullptr) return NRSENSE_ERR_ARG;
  p->prof_on = false;
  if (cudaDeviceSynchronize() != cudaSuccess) return NRSENSE_ERR_CUDA;
  if (ms) for (int i = 0; i < NRSENSE_NUM_STAGES; ++i) ms[i] = 0.0;
  if (count) for (int i = 0; i < NRSENSE_NUM_STAGES; ++i) count[i] = 0;
  for (size_t k = 0; k < p->prof_stage.size(); ++k) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, p->prof_events[2 * k], p->prof_events[2 * k + 1]) != cudaSuccess)
      return NRSENSE_ERR_CUDA;
    const int st = p->prof_stage[k];
    if (ms) ms[st] += double(t);
    if (count) count[st] += 1;
  }
  if (own_kernels) *own_kernels = p->launches - p->launches_at_start;
  p->prof_stage.clear();
  return NRSENSE_OK;
}

const char* nrsense_stage_name(int32_t st) {
  static const char* names[NRSENSE_NUM_STAGES] = {
      "fft_n", "fft_g", "fft_gc", "deapod_pad", "interp_image", "spread_image", "crop_deapod",
      "coil_fanout_pad", "interp_kspace", "spread_kspace", "crop_coilsum", "vector", "solver",
      "cnn", "fista", "fft_pruned"};
  return (st >= 0 && st < NRSENSE_NUM_STAGES) ? names[st] : "unknown";
}

const char* nrsense_status_string(nrsense_status s) {
  switch (s) {
    case NRSENSE_OK: return "ok";
    case NRSENSE_ERR_ARG: return "invalid argument";
    case NRSENSE_ERR_OOM: return "out of memory";
    case NRSENSE_ERR_CUFFT: return "cuFFT failure";
    case NRSENSE_ERR_CUDA: return "CUDA runtime failure";
    case NRSENSE_ERR_BREAKDOWN: return "CG breakdown";
    case NRSENSE_ERR_NOT_CONVERGED: return "CG not converged";
    case NRSENSE_ERR_TIMEOUT: return "device wait timed out";
    case NRSENSE_ERR_STATE: return "call not valid for this plan";
    default: return "unknown status";
  }
}

nrsense_status nrsense_device_status(nrsense_plan_t p, int32_t clear, int32_t* out_host,
                                     void* stream) {
  if (p == nullptr || out_host == nullptr) return NRSENSE_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(out_host, p->d_status, sizeof(int32_t), cudaMemcpyDeviceToHost, s) !=
      cudaSuccess)
    return NRSENSE_ERR_CUDA;
  if (clear && cudaMemsetAsync(p->d_status, 0, sizeof(int32_t), s) != cudaSuccess)
    return NRSENSE_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return NRSENSE_ERR_CUDA;
  return NRSENSE_OK;
}

}  // extern "C"
