// DFTs of 16 rows or columns per CTA for the axis lengths that the power-of-two
// passes of fft_pruned.cu do not cover (device code of the fft_mixed*.cu
// files).  An axis holds N data values centred on a periodic grid of G points
// (data at [0, N/2) and [G - N/2, G)); "wrapped order" numbers them by grid
// position modulo N, which for a spectrum is DFT order.  An axis policy has
//   pad(ld, st)   length-G DFT of the zero-padded data: ld(lane, n'),
//   crop(ld, st)  length-G DFT of a full input, only the data outputs: st(lane, n', v),
//   full(ld, st)  length-N DFT,
// always exp(-2 pi i n k / L) (an inverse transform conjugates in its functors).
//
// DoubleAxis (G = 2N, N = R S with R even, R and S at most 16): a length-G
// transform in two steps, radix 2R and radix S, whose zero half is never
// computed: a radix-2R butterfly with R nonzero inputs is two radix-R ones
// (even outputs of v, odd outputs of v W_2R^n), with R wanted outputs two
// radix-R ones of the even and the odd inputs.  One exchange through shared
// memory per transform.  The radices are template values for N a multiple of 16 up
// to 256 (strides, masks and twiddle indices become constants) and run-time values, with one unrolled body per radix behind a CTA-uniform
// switch, for the rest.
// GeneralAxis (N and G each r1 r2 r3 with r1 and r3 in 2..16 and r2 in 1..8: of the
// lengths of 16 to 1024 without a prime above 13 all but 625, 729, 875, 891, 972 and
// 1000): in place, decimation in frequency, two or three steps.
#pragma once

#include <type_traits>

#include "plan_internal.h"

namespace nrs {
namespace mixed {

constexpr int kLanes = 16;     // rows or columns per CTA
constexpr int kThreads = 256;  // most threads per CTA

// cos and sin of 2 pi j / r at compile time (Taylor series about 0 after
// reduction to [-pi, pi])
constexpr double ct_angle(int j, int r) {
  j %= r;
  if (2 * j > r) j -= r;
  return 6.283185307179586476925286766559 * double(j) / double(r);
}
constexpr double ct_cos(int j, int r) {
  const double x = ct_angle(j, r), x2 = x * x;
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 20; ++k) {
    term *= -x2 / double((2 * k - 1) * (2 * k));
    sum += term;
  }
  return sum;
}
constexpr double ct_sin(int j, int r) {
  const double x = ct_angle(j, r), x2 = x * x;
  double term = x, sum = x;
  for (int k = 1; k < 20; ++k) {
    term *= -x2 / double((2 * k) * (2 * k + 1));
    sum += term;
  }
  return sum;
}

template <int B, int E, class F>
__device__ __forceinline__ void unroll(F&& f) {
  if constexpr (B < E) {
    f(std::integral_constant<int, B>{});
    unroll<B + 1, E>(f);
  }
}

__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

// a * exp(-2 pi i J / R)
template <int J, int R>
__device__ __forceinline__ float2 rotate(float2 a) {
  constexpr int j = J % R;
  if constexpr (j == 0) {
    return a;
  } else if constexpr (4 * j == R) {
    return make_float2(a.y, -a.x);
  } else if constexpr (2 * j == R) {
    return make_float2(-a.x, -a.y);
  } else if constexpr (4 * j == 3 * R) {
    return make_float2(-a.y, a.x);
  } else {
    constexpr float c = float(ct_cos(j, R)), s = float(ct_sin(j, R));
    return make_float2(a.x * c + a.y * s, a.y * c - a.x * s);
  }
}

constexpr int small_factor(int r) {  // composite radices split off 4, else the smallest prime
  if (r % 4 == 0 && r > 4) return 4;
  for (int p = 2; p * p <= r; ++p)
    if (r % p == 0) return p;
  return r;
}

// a[k] = sum_n a[n] exp(-2 pi i n k / R), natural order, in registers
template <int R>
__device__ __forceinline__ void dft(float2 (&a)[R]) {
  if constexpr (R == 1) {
  } else if constexpr (R == 2) {
    const float2 u = a[0], v = a[1];
    a[0] = make_float2(u.x + v.x, u.y + v.y);
    a[1] = make_float2(u.x - v.x, u.y - v.y);
  } else if constexpr (R == 4) {
    const float2 s0 = make_float2(a[0].x + a[2].x, a[0].y + a[2].y);
    const float2 d0 = make_float2(a[0].x - a[2].x, a[0].y - a[2].y);
    const float2 s1 = make_float2(a[1].x + a[3].x, a[1].y + a[3].y);
    const float2 d1 = make_float2(a[1].x - a[3].x, a[1].y - a[3].y);
    a[0] = make_float2(s0.x + s1.x, s0.y + s1.y);
    a[2] = make_float2(s0.x - s1.x, s0.y - s1.y);
    a[1] = make_float2(d0.x + d1.y, d0.y - d1.x);
    a[3] = make_float2(d0.x - d1.y, d0.y + d1.x);
  } else if constexpr (small_factor(R) == R) {
    // odd prime: X[k], X[R - k] = a0 + sum_j cos_jk s_j -+ i sum_j sin_jk d_j
    constexpr int H = (R - 1) / 2;
    float2 s[H], d[H];
    unroll<0, H>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      s[j] = make_float2(a[j + 1].x + a[R - 1 - j].x, a[j + 1].y + a[R - 1 - j].y);
      d[j] = make_float2(a[j + 1].x - a[R - 1 - j].x, a[j + 1].y - a[R - 1 - j].y);
    });
    const float2 a0 = a[0];
    float2 sum = a0;
    unroll<0, H>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      sum.x += s[j].x;
      sum.y += s[j].y;
    });
    a[0] = sum;
    unroll<1, H + 1>([&](auto kc) {
      constexpr int k = decltype(kc)::value;
      float2 e = a0, o = make_float2(0.f, 0.f);
      unroll<0, H>([&](auto jc) {
        constexpr int j = decltype(jc)::value;
        constexpr float c = float(ct_cos((j + 1) * k, R)), sn = float(ct_sin((j + 1) * k, R));
        e.x = fmaf(c, s[j].x, e.x);
        e.y = fmaf(c, s[j].y, e.y);
        o.x = fmaf(sn, d[j].x, o.x);
        o.y = fmaf(sn, d[j].y, o.y);
      });
      a[k] = make_float2(e.x + o.y, e.y - o.x);
      a[R - k] = make_float2(e.x - o.y, e.y + o.x);
    });
  } else {
    // R = P Q, n = Q n1 + n2, k = k1 + P k2
    constexpr int P = small_factor(R), Q = R / P;
    float2 b[P][Q];
    unroll<0, Q>([&](auto nc) {
      constexpr int n2 = decltype(nc)::value;
      float2 t[P];
      unroll<0, P>([&](auto pc) {
        constexpr int n1 = decltype(pc)::value;
        t[n1] = a[Q * n1 + n2];
      });
      dft<P>(t);
      unroll<0, P>([&](auto pc) {
        constexpr int k1 = decltype(pc)::value;
        b[k1][n2] = rotate<k1 * n2, R>(t[k1]);
      });
    });
    unroll<0, P>([&](auto pc) {
      constexpr int k1 = decltype(pc)::value;
      dft<Q>(b[k1]);
      unroll<0, Q>([&](auto qc) {
        constexpr int k2 = decltype(qc)::value;
        a[k1 + P * k2] = b[k1][k2];
      });
    });
  }
}

// f(integral_constant<R>) for the radix r (CTA-uniform) out of 2..16; EVEN: even ones
template <bool EVEN = false, class F>
__device__ __forceinline__ void with_radix(int r, F&& f) {
  unroll<1, 9>([&](auto hc) {
    constexpr int R = 2 * decltype(hc)::value;
    if (r == R) f(std::integral_constant<int, R>{});
    if constexpr (!EVEN && R > 2)
      if (r == R - 1) f(std::integral_constant<int, R - 1>{});
  });
}
// the middle radix of a three-step length is at most 8
template <class F>
__device__ __forceinline__ void with_middle(int r, F&& f) {
  unroll<2, 9>([&](auto rc) {
    if (r == decltype(rc)::value) f(rc);
  });
}

// q = x / d for x < 2^16, d >= 2 (m = ceil(2^32 / d), exact in this range)
__device__ __forceinline__ int fast_div(int x, unsigned m) { return int(__umulhi(unsigned(x), m)); }

// Shared-memory index of element (group k1, offset o) of a lane, groups of s
// elements, g groups.  Columns keep the lane fastest (a half-warp covers the
// 16 lanes' 128 bytes); rows keep the element fastest and pad every group to
// an odd pitch, so a step whose lanes walk over the groups meets distinct banks.
template <bool ROWS>
__device__ __forceinline__ int sidx(int s, int g, int lane, int k1, int o) {
  return ROWS ? (lane * g + k1) * (s | 1) + o : (k1 * s + o) * kLanes + lane;
}

// Run f(lane, j) for every butterfly j < nb of every lane of the CTA.
template <bool ROWS, class Div, class F>
__device__ __forceinline__ void for_butterflies(int nb, const Div& div, F&& f) {
  if constexpr (ROWS) {
    for (int b = threadIdx.x; b < kLanes * nb; b += blockDim.x) {
      const int lane = div(b);
      f(lane, b - lane * nb);
    }
  } else {
    const int lane = threadIdx.x & (kLanes - 1);
    for (int j = threadIdx.x / kLanes; j < nb; j += blockDim.x / kLanes) f(lane, j);
  }
}

// Radices and twiddles of a DoubleAxis: template values, or (RtLen) run-time ones.
template <int R_, int S_>
struct StLen {
  static constexpr bool kStatic = true;
  // CTAs per SM of the pad and the crop kernels (their butterflies hold 2R and
  // max(2R, S) values in registers)
  static constexpr int kPad = R_ <= 8 ? 4 : 3, kCrop = R_ <= 8 ? 3 : 2;
  static constexpr int r = R_, s = S_;
  const float2* tw;    // exp(-2 pi i j / 2N), j < 2N
  template <class F>
  __device__ __forceinline__ void with_r(F&& f) const { f(std::integral_constant<int, R_>{}); }
  template <class F>
  __device__ __forceinline__ void with_s(F&& f) const { f(std::integral_constant<int, S_>{}); }
  __device__ __forceinline__ int div_r(int x) const { return x / R_; }
  __device__ __forceinline__ int div_2r(int x) const { return x / (2 * R_); }
  __device__ __forceinline__ int div_s(int x) const { return x / S_; }
};
struct RtLen {
  static constexpr bool kStatic = false;
  static constexpr int kPad = 3, kCrop = 2;
  int r, s;
  unsigned m_r, m_2r, m_s;
  const float2* tw;
  template <class F>
  __device__ __forceinline__ void with_r(F&& f) const { with_radix<true>(r, f); }
  template <class F>
  __device__ __forceinline__ void with_s(F&& f) const { with_radix(s, f); }
  __device__ __forceinline__ int div_r(int x) const { return fast_div(x, m_r); }
  __device__ __forceinline__ int div_2r(int x) const { return fast_div(x, m_2r); }
  __device__ __forceinline__ int div_s(int x) const { return fast_div(x, m_s); }
};

// Grid positions: pad's st gets (lane, q, k2, v) for position q + step k2 and
// crop's ld (lane, j, n1) for position j + step n1, with k2 and n1 compile-time
// values, so that a functor can test a tile mask with constant shifts.
template <class Len>
struct DoubleAxis {
  static constexpr bool kMaskShift = Len::kStatic;  // step is a compile-time value
  static constexpr int kPad = Len::kPad, kCrop = Len::kCrop;
  Len l;
  __host__ __device__ __forceinline__ int N() const { return l.r * l.s; }
  __host__ __device__ __forceinline__ int G() const { return 2 * l.r * l.s; }
  __host__ __device__ __forceinline__ int step() const { return 2 * l.r; }

  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void pad(float2* sy, const Ld& ld, const St& st) const {
    l.with_r([&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for_butterflies<ROWS>(l.s, [&](int x) { return l.div_s(x); }, [&](int lane, int j) {
        float2 v[R], e[R];
        unroll<0, R>([&](auto ic) {
          constexpr int n1 = decltype(ic)::value;
          v[n1] = ld(lane, l.s * n1 + j);
        });
        unroll<0, R>([&](auto ic) { e[decltype(ic)::value] = v[decltype(ic)::value]; });
        dft<R>(e);
        unroll<0, R>([&](auto ic) {
          constexpr int k1 = decltype(ic)::value;
          sy[sidx<ROWS>(l.s, 2 * l.r, lane, 2 * k1, j)] =
              k1 == 0 ? e[0] : cmul(e[k1], __ldg(l.tw + j * 2 * k1));
        });
        // grid index of input n1: n1, or n1 + R in the upper half of the data
        unroll<0, R>([&](auto ic) {
          constexpr int n1 = decltype(ic)::value;
          v[n1] = rotate<n1 + (n1 >= R / 2 ? R : 0), 2 * R>(v[n1]);
        });
        dft<R>(v);
        unroll<0, R>([&](auto ic) {
          constexpr int k1 = decltype(ic)::value;
          sy[sidx<ROWS>(l.s, 2 * l.r, lane, 2 * k1 + 1, j)] =
              cmul(v[k1], __ldg(l.tw + j * (2 * k1 + 1)));
        });
      });
    });
    __syncthreads();
    l.with_s([&](auto sc) {
      constexpr int S = decltype(sc)::value;
      for_butterflies<ROWS>(2 * l.r, [&](int x) { return l.div_2r(x); }, [&](int lane, int q) {
        float2 b[S];
        unroll<0, S>([&](auto ic) {
          constexpr int o = decltype(ic)::value;
          b[o] = sy[sidx<ROWS>(S, 2 * l.r, lane, q, o)];
        });
        dft<S>(b);
        unroll<0, S>([&](auto ic) { st(lane, q, ic, b[decltype(ic)::value]); });
      });
    });
    __syncthreads();
  }

  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void crop(float2* sy, const Ld& ld, const St& st) const {
    l.with_s([&](auto sc) {
      constexpr int S = decltype(sc)::value;
      for_butterflies<ROWS>(2 * l.r, [&](int x) { return l.div_2r(x); }, [&](int lane, int j) {
        float2 a[S];
        unroll<0, S>([&](auto ic) { a[decltype(ic)::value] = ld(lane, j, ic); });
        dft<S>(a);
        unroll<0, S>([&](auto ic) {
          constexpr int k1 = decltype(ic)::value;
          sy[sidx<ROWS>(2 * l.r, S, lane, k1, j)] =
              k1 == 0 ? a[0] : cmul(a[k1], __ldg(l.tw + j * k1));
        });
      });
    });
    __syncthreads();
    l.with_r([&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for_butterflies<ROWS>(l.s, [&](int x) { return l.div_s(x); }, [&](int lane, int k1) {
        float2 e[R], o[R];
        unroll<0, R>([&](auto ic) {
          constexpr int m = decltype(ic)::value;
          e[m] = sy[sidx<ROWS>(2 * R, l.s, lane, k1, 2 * m)];
        });
        dft<R>(e);
        unroll<0, R>([&](auto ic) {
          constexpr int m = decltype(ic)::value;
          o[m] = sy[sidx<ROWS>(2 * R, l.s, lane, k1, 2 * m + 1)];
        });
        dft<R>(o);
        unroll<0, R>([&](auto ic) {
          constexpr int m = decltype(ic)::value;
          // wanted outputs k2 = m, or m + R in the upper half of the data
          const float2 w = rotate<m + (m >= R / 2 ? R : 0), 2 * R>(o[m]);
          st(lane, k1 + l.s * m, make_float2(e[m].x + w.x, e[m].y + w.y));
        });
      });
    });
    __syncthreads();
  }

  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void full(float2* sy, const Ld& ld, const St& st) const {
    l.with_r([&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for_butterflies<ROWS>(l.s, [&](int x) { return l.div_s(x); }, [&](int lane, int j) {
        float2 v[R];
        unroll<0, R>([&](auto ic) {
          constexpr int n1 = decltype(ic)::value;
          v[n1] = ld(lane, l.s * n1 + j);
        });
        dft<R>(v);
        unroll<0, R>([&](auto ic) {
          constexpr int k1 = decltype(ic)::value;
          sy[sidx<ROWS>(l.s, l.r, lane, k1, j)] =
              k1 == 0 ? v[0] : cmul(v[k1], __ldg(l.tw + 2 * j * k1));
        });
      });
    });
    __syncthreads();
    l.with_s([&](auto sc) {
      constexpr int S = decltype(sc)::value;
      for_butterflies<ROWS>(l.r, [&](int x) { return l.div_r(x); }, [&](int lane, int k1) {
        float2 b[S];
        unroll<0, S>([&](auto ic) {
          constexpr int o = decltype(ic)::value;
          b[o] = sy[sidx<ROWS>(S, l.r, lane, k1, o)];
        });
        dft<S>(b);
        unroll<0, S>([&](auto ic) {
          constexpr int k2 = decltype(ic)::value;
          st(lane, k1 + l.r * k2, b[k2]);
        });
      });
    });
    __syncthreads();
  }
};

// In-place DFT of any supported length: with n = r2 r3 n1 + r3 n2 + n3 and
// k = k1 + r1 k2 + r1 r2 k3,
//   X[k] = sum_n3 W_L^(n3 (k1 + r1 k2)) W_r3^(n3 k3)
//          sum_n2 W_(r1 r2)^(n2 k1) W_r2^(n2 k2)  sum_n1 W_r1^(n1 k1) x[n]
// (r2 = 1: two steps).
template <bool ROWS, class Ld, class St>
__device__ __forceinline__ void fft_lanes(const MixLen& f, float2* sy, const Ld& ld, const St& st) {
  with_radix(f.r1, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for_butterflies<ROWS>(f.s, [&](int x) { return fast_div(x, f.m_s); }, [&](int lane, int j) {
      float2 v[R];
      unroll<0, R>([&](auto ic) {
        constexpr int n1 = decltype(ic)::value;
        v[n1] = ld(lane, f.s * n1 + j);
      });
      dft<R>(v);
      // W_(r1 r2)^(n2 k1) with three steps, W_L^(n3 k1) with two
      const int t = f.r2 > 1 ? f.r3 * fast_div(j, f.m_r3) : j;
      unroll<0, R>([&](auto ic) {
        constexpr int k1 = decltype(ic)::value;
        sy[sidx<ROWS>(f.s, f.r1, lane, k1, j)] =
            k1 == 0 ? v[0] : cmul(v[k1], __ldg(f.tw + t * k1));
      });
    });
  });
  __syncthreads();
  if (f.r2 > 1) {
    with_middle(f.r2, [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      for_butterflies<ROWS>(f.r1 * f.r3, [&](int x) { return fast_div(x, f.m_13); },
                            [&](int lane, int j) {
        const int k1 = fast_div(j, f.m_r3), n3 = j - k1 * f.r3;
        float2 v[R];
        unroll<0, R>([&](auto ic) {
          constexpr int n2 = decltype(ic)::value;
          v[n2] = sy[sidx<ROWS>(f.s, f.r1, lane, k1, n2 * f.r3 + n3)];
        });
        dft<R>(v);
        unroll<0, R>([&](auto ic) {
          constexpr int k2 = decltype(ic)::value;
          sy[sidx<ROWS>(f.s, f.r1, lane, k1, k2 * f.r3 + n3)] =
              cmul(v[k2], __ldg(f.tw + n3 * (k1 + f.r1 * k2)));
        });
      });
    });
    __syncthreads();
  }
  with_radix(f.r3, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    for_butterflies<ROWS>(f.r1 * f.r2, [&](int x) { return fast_div(x, f.m_12); },
                          [&](int lane, int j) {
      const int k2 = f.r2 > 1 ? fast_div(j, f.m_r1) : 0, k1 = j - k2 * f.r1;
      float2 v[R];
      unroll<0, R>([&](auto ic) {
        constexpr int n3 = decltype(ic)::value;
        v[n3] = sy[sidx<ROWS>(f.s, f.r1, lane, k1, k2 * f.r3 + n3)];
      });
      dft<R>(v);
      unroll<0, R>([&](auto ic) {
        constexpr int k3 = decltype(ic)::value;
        st(lane, j + f.r1 * f.r2 * k3, v[k3]);
      });
    });
  });
  __syncthreads();
}

struct GeneralAxis {
  static constexpr bool kMaskShift = false;
  static constexpr int kPad = 3, kCrop = 3;
  MixLen g, n;
  int nn;  // N
  __host__ __device__ __forceinline__ int N() const { return nn; }
  __host__ __device__ __forceinline__ int G() const { return g.L; }
  __host__ __device__ __forceinline__ int step() const { return 0; }
  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void pad(float2* sy, const Ld& ld, const St& st) const {
    const int h = nn / 2;
    fft_lanes<ROWS>(g, sy,
                    [&](int lane, int p) -> float2 {
                      if (p >= h && p < g.L - h) return make_float2(0.f, 0.f);
                      return ld(lane, p < h ? p : p - (g.L - nn));
                    },
                    [&](int lane, int k, float2 v) {
                      st(lane, k, std::integral_constant<int, 0>{}, v);
                    });
  }
  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void crop(float2* sy, const Ld& ld, const St& st) const {
    const int h = nn / 2;
    fft_lanes<ROWS>(g, sy,
                    [&](int lane, int p) { return ld(lane, p, std::integral_constant<int, 0>{}); },
                    [&](int lane, int k, float2 v) {
                      if (k < h || k >= g.L - h) st(lane, k < h ? k : k - (g.L - nn), v);
                    });
  }
  template <bool ROWS, class Ld, class St>
  __device__ __forceinline__ void full(float2* sy, const Ld& ld, const St& st) const {
    fft_lanes<ROWS>(n, sy, ld, st);
  }
};

// centred index of wrapped index n' (and back: the map is its own inverse)
__device__ __forceinline__ int swap_half(int i, int h) { return i < h ? i + h : i - h; }

}  // namespace mixed
}  // namespace nrs
