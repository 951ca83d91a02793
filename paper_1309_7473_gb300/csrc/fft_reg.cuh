// Register-resident Stockham FFT used by the fast-path time-ordered-data kernels.
//
// A thread owns E elements of one length-L sequence (L = product of the stage
// radices, every radix divides E): on entry x[e] holds the element at position
// i + e (L/E), 0 <= i < L/E, and on exit x[e] holds the transform at that same
// position.  Every stage's butterflies read their inputs from those natural
// positions (butterfly ib = i + (L/E) u, input m at ib + m L/R is register
// u + m E/R), so only the outputs of non-final stages go through shared memory:
// a sequence of S stages costs S - 1 exchanges, each one store and one load per
// element, instead of a load and a store per stage.  Twiddles w_{PR}^{mk} come
// from a table of w_L^e, e < L (forward sign, conjugated for SIGN > 0): the powers
// of two are loaded and the other exponents formed as products.
#pragma once

#include "common.cuh"
#include "fft.cuh"

// Stage twiddles w^m, m < R: 1 (default) by recurrence from one loaded w (two live
// registers, relative error growing to ~R ulp); 0 from the loaded w, w^2, w^4, w^8
// and products (at most three roundings, more live registers).
#ifndef CMM_TW_MODE
#define CMM_TW_MODE 1
#endif

namespace cmm {

constexpr int clog2(int v) { return v <= 1 ? 0 : 1 + clog2(v / 2); }

template <int... Rs> struct RadProd;
template <> struct RadProd<> { static constexpr int value = 1; };
template <int R, int... Rs> struct RadProd<R, Rs...> { static constexpr int value = R * RadProd<Rs...>::value; };

// the real type of a complex pair
template <typename V> struct RealOf;
template <> struct RealOf<float2> { using t = float; };
template <> struct RealOf<double2> { using t = double; };

// FP64 takes every stage twiddle from the table: loads cost nothing beside its pipe.
template <int SIGN, int E, int L, int P, typename V, typename Addr, int R, int... REST>
__device__ __forceinline__ void rfft_stages(V (&x)[E], const int i, const V* __restrict__ tw, const Addr& ad) {
  using T = typename RealOf<V>::t;
  static_assert(E % R == 0, "every radix must divide the elements per thread");
  constexpr int NB = E / R;
  constexpr bool LAST = sizeof...(REST) == 0;
  if constexpr (!LAST) __syncthreads();
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int ib = i + (L / E) * u;
    const int k = ib & (P - 1);
    V z[R];
#pragma unroll
    for (int m = 0; m < R; ++m) z[m] = x[u + m * NB];
    if constexpr (P > 1 && sizeof(T) == 8) {
      const int b = k * (L / (P * R));
#pragma unroll
      for (int m = 1; m < R; ++m) {
        const V w = __ldg(tw + m * b);
        z[m] = SIGN > 0 ? cmulc(z[m], w) : cmul(z[m], w);
      }
    } else if constexpr (P > 1) {
      // one or four L1 loads per butterfly instead of R - 1, the rest on the FP32 pipe
      const int b = k * (L / (P * R));
#if CMM_TW_MODE == 1
      // w^m by recurrence from w (two live twiddles)
      float2 w1 = __ldg(tw + b);
      if (SIGN > 0) w1.y = -w1.y;
      float2 wm = w1;
#pragma unroll
      for (int m = 1; m < R; ++m) {
        z[m] = cmul(z[m], wm);
        if (m + 1 < R) wm = cmul(wm, w1);
      }
#else
      float2 wp[R];
#pragma unroll
      for (int m = 1; m < R; m *= 2) {
        wp[m] = __ldg(tw + m * b);
        if (SIGN > 0) wp[m].y = -wp[m].y;
      }
#pragma unroll
      for (int m = 3; m < R; ++m)
        if (m & (m - 1)) wp[m] = cmul(wp[m & (m - 1)], wp[m & -m]);
#pragma unroll
      for (int m = 1; m < R; ++m) z[m] = cmul(z[m], wp[m]);
#endif
    }
    dft_reg<T, clog2(R), SIGN>(z);
    if constexpr (LAST) {
#pragma unroll
      for (int q = 0; q < R; ++q) x[u + q * NB] = z[q];
    } else {
      // outputs at (ib - k) R + k + q P: one base index, constant offsets
      const int b = ad.base((ib - k) * R + k);
#pragma unroll
      for (int q = 0; q < R; ++q) ad.st_at(b, q * P, z[q]);
    }
  }
  if constexpr (!LAST) {
    __syncthreads();
    const int b = ad.base(i);
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = ad.ld_at(b, e * (L / E));
    rfft_stages<SIGN, E, L, P * R, V, Addr, REST...>(x, i, tw, ad);
  }
}

template <int SIGN, int E, int... RS, typename V, typename Addr>
__device__ __forceinline__ void rfft(V (&x)[E], const int i, const V* __restrict__ tw, const Addr& ad) {
  rfft_stages<SIGN, E, RadProd<RS...>::value, 1, V, Addr, RS...>(x, i, tw, ad);
}

// One contiguous row (pass F), padded by one element every 2^PS positions.
// st_at / ld_at address position pos + o from base(pos) with a constant offset o;
// exact whenever the low PS bits of pos and o do not carry into each other, which
// holds for every access of the register FFT (either pos is a multiple of 2^PS
// and o < 2^PS, or o is a multiple of 2^PS, or o is a multiple of a power of two
// p < 2^PS and pos < p).
template <int PS>
struct RowAddr {
  float2* buf;
  __device__ __forceinline__ int idx(int pos) const { return pos + (pos >> PS); }
  __device__ __forceinline__ void st(int pos, float2 v) const { buf[idx(pos)] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return buf[idx(pos)]; }
  __device__ __forceinline__ int base(int pos) const { return idx(pos); }
  __device__ __forceinline__ void st_at(int b, int o, float2 v) const { buf[b + o + (o >> PS)] = v; }
  __device__ __forceinline__ float2 ld_at(int b, int o) const { return buf[b + o + (o >> PS)]; }
};

// ------------------------------------------------------------------ two sequences a thread
// Two complex numbers side by side: lane x of re and im is the first, lane y the
// second.  Sums and constant rotations of both are one packed FP32 instruction per
// part, a product by i is a renaming, and a stage twiddle serves both (one
// recurrence for two sequences).
template <typename T>
struct __align__(16) Cx2 {
  V2<T> re, im;
};

__device__ __forceinline__ float2 pfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 pfma(double2 a, double2 b, double2 c) {
  return double2{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}

template <typename T>
__device__ __forceinline__ Cx2<T> cx_add(const Cx2<T>& a, const Cx2<T>& b) {
  return Cx2<T>{padd(a.re, b.re), padd(a.im, b.im)};
}
template <typename T>
__device__ __forceinline__ Cx2<T> cx_sub(const Cx2<T>& a, const Cx2<T>& b) {
  return Cx2<T>{psub(a.re, b.re), psub(a.im, b.im)};
}
// a (c + i s), the same (c, s) for both numbers
template <typename T>
__device__ __forceinline__ Cx2<T> cx_mul(const Cx2<T>& a, T c, T s) {
  const V2<T> cc{c, c}, ss{s, s}, ns{-s, -s};
  return Cx2<T>{pfma(a.im, ns, pmul(a.re, cc)), pfma(a.re, ss, pmul(a.im, cc))};
}

// v exp(SIGN 2 pi i m / 32), m known at compile time after unrolling
template <typename T, int SIGN>
__device__ __forceinline__ Cx2<T> cx_rot32(const Cx2<T>& v, int m) {
  m &= 31;
  if (m == 0) return v;
  const Cx2<T> pos{V2<T>{-v.im.x, -v.im.y}, v.re}, neg{v.im, V2<T>{-v.re.x, -v.re.y}};   // i v, -i v
  if (m == 8) return SIGN < 0 ? neg : pos;
  if (m == 24) return SIGN < 0 ? pos : neg;
  if (m == 16) return Cx2<T>{V2<T>{-v.re.x, -v.re.y}, V2<T>{-v.im.x, -v.im.y}};
  return cx_mul<T>(v, (T)cos32(m), (T)(SIGN * sin32(m)));
}

// a + SIGN i b and a - SIGN i b: parts swapped by name, no instruction of their own
template <typename T, int SIGN>
__device__ __forceinline__ void cx_addsub_i(const Cx2<T>& a, const Cx2<T>& b, Cx2<T>& plus, Cx2<T>& minus) {
  const Cx2<T> p{psub(a.re, b.im), padd(a.im, b.re)}, m{padd(a.re, b.im), psub(a.im, b.re)};
  plus = SIGN > 0 ? p : m;
  minus = SIGN > 0 ? m : p;
}

template <typename T, int SIGN>
__device__ __forceinline__ void cx_dft4(Cx2<T>& x0, Cx2<T>& x1, Cx2<T>& x2, Cx2<T>& x3) {
  const Cx2<T> a0 = cx_add(x0, x2), a1 = cx_sub(x0, x2), a2 = cx_add(x1, x3), d = cx_sub(x1, x3);
  x0 = cx_add(a0, a2);
  x2 = cx_sub(a0, a2);
  cx_addsub_i<T, SIGN>(a1, d, x1, x3);
}

// x_q <- sum_j x_j w_R^{j q}, R = 2^LR <= 16 (4 x 4 for 16, 4 x 2 for 8, else radix-2 stages)
template <typename T, int LR, int SIGN>
__device__ __forceinline__ void cx_dft(Cx2<T>* x) {
  if constexpr (LR == 2) {
    cx_dft4<T, SIGN>(x[0], x[1], x[2], x[3]);
  } else if constexpr (LR == 3) {
    Cx2<T> e[4] = {x[0], x[2], x[4], x[6]}, o[4] = {x[1], x[3], x[5], x[7]};
    cx_dft4<T, SIGN>(e[0], e[1], e[2], e[3]);
    cx_dft4<T, SIGN>(o[0], o[1], o[2], o[3]);
    o[1] = cx_rot32<T, SIGN>(o[1], 4);
    o[3] = cx_rot32<T, SIGN>(o[3], 12);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k == 2) {
        cx_addsub_i<T, SIGN>(e[2], o[2], x[2], x[6]);
      } else {
        x[k] = cx_add(e[k], o[k]);
        x[k + 4] = cx_sub(e[k], o[k]);
      }
    }
  } else if constexpr (LR == 4) {
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) cx_dft4<T, SIGN>(x[n1], x[n1 + 4], x[n1 + 8], x[n1 + 12]);
#pragma unroll
    for (int n1 = 1; n1 < 4; ++n1)
#pragma unroll
      for (int k2 = 1; k2 < 4; ++k2) x[n1 + 4 * k2] = cx_rot32<T, SIGN>(x[n1 + 4 * k2], 2 * n1 * k2);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) cx_dft4<T, SIGN>(x[4 * k2], x[4 * k2 + 1], x[4 * k2 + 2], x[4 * k2 + 3]);
    Cx2<T> t[16];
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2)
#pragma unroll
      for (int k1 = 0; k1 < 4; ++k1) t[k2 + 4 * k1] = x[4 * k2 + k1];
#pragma unroll
    for (int e = 0; e < 16; ++e) x[e] = t[e];
  } else {
    constexpr int R = 1 << LR;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int j = bitrev(i, LR);
      if (i < j) {
        const Cx2<T> t = x[i];
        x[i] = x[j];
        x[j] = t;
      }
    }
#pragma unroll
    for (int half = 1; half < R; half *= 2)
#pragma unroll
      for (int start = 0; start < R; start += 2 * half)
#pragma unroll
        for (int j = 0; j < half; ++j) {
          const Cx2<T> t = cx_rot32<T, SIGN>(x[start + j + half], j * (32 / (2 * half)));
          const Cx2<T> u = x[start + j];
          x[start + j] = cx_add(u, t);
          x[start + j + half] = cx_sub(u, t);
        }
  }
}

// Stages of rfft on two sequences of the same length at once.  FRESH: no thread still
// reads the buffer, so the first exchange needs no barrier before its stores.
template <typename T, int SIGN, bool FRESH, int E, int L, int P, typename Addr, int R, int... REST>
__device__ __forceinline__ void rfft2_stages(Cx2<T> (&x)[E], const int i, const V2<T>* __restrict__ tw,
                                             const Addr& ad) {
  static_assert(E % R == 0, "every radix must divide the elements per thread");
  constexpr int NB = E / R;
  constexpr bool LAST = sizeof...(REST) == 0;
  if constexpr (!LAST && !FRESH) __syncthreads();
#pragma unroll
  for (int u = 0; u < NB; ++u) {
    const int ib = i + (L / E) * u;
    const int k = ib & (P - 1);
    Cx2<T> z[R];
#pragma unroll
    for (int m = 0; m < R; ++m) z[m] = x[u + m * NB];
    if constexpr (P > 1 && sizeof(T) == 8) {
      const int b = k * (L / (P * R));
#pragma unroll
      for (int m = 1; m < R; ++m) {
        const V2<T> w = __ldg(tw + m * b);
        z[m] = cx_mul<T>(z[m], w.x, SIGN > 0 ? -w.y : w.y);
      }
    } else if constexpr (P > 1) {
      const int b = k * (L / (P * R));
      V2<T> w1 = __ldg(tw + b);
      if (SIGN > 0) w1.y = -w1.y;
      // four chains of step w^4 instead of one of step w: the same products, depth 5
      // instead of 14, and a rounding error that grows with the depth (operator error
      // at 32 detectors x 2^16 samples 2.6e-7 -> 2.2e-7; the same time)
      V2<T> wq[4];
      wq[0] = w1;
      wq[1] = cmul(w1, w1);
      wq[2] = cmul(wq[1], w1);
      wq[3] = cmul(wq[1], wq[1]);
      const V2<T> w4 = wq[3];
#pragma unroll
      for (int m = 1; m < R; ++m) {
        z[m] = cx_mul<T>(z[m], wq[(m - 1) & 3].x, wq[(m - 1) & 3].y);
        if (m + 4 < R) wq[(m - 1) & 3] = cmul(wq[(m - 1) & 3], w4);
      }
    }
    cx_dft<T, clog2(R), SIGN>(z);
    if constexpr (LAST) {
#pragma unroll
      for (int q = 0; q < R; ++q) x[u + q * NB] = z[q];
    } else {
      const int b = ad.base((ib - k) * R + k);
#pragma unroll
      for (int q = 0; q < R; ++q) ad.st_at(b, q * P, z[q]);
    }
  }
  if constexpr (!LAST) {
    __syncthreads();
    const int b = ad.base(i);
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = ad.ld_at(b, e * (L / E));
    rfft2_stages<T, SIGN, false, E, L, P * R, Addr, REST...>(x, i, tw, ad);
  }
}

template <typename T, int SIGN, bool FRESH, int E, int... RS, typename Addr>
__device__ __forceinline__ void rfft2(Cx2<T> (&x)[E], const int i, const V2<T>* __restrict__ tw, const Addr& ad) {
  rfft2_stages<T, SIGN, FRESH, E, RadProd<RS...>::value, 1, Addr, RS...>(x, i, tw, ad);
}

// One contiguous row of Cx2 elements, padded by one element every 2^PS positions (as
// RowAddr): eight lanes of a 16-byte access phase fall on distinct bank groups.
template <typename T, int PS>
struct RowAddr2 {
  Cx2<T>* buf;
  __device__ __forceinline__ int base(int pos) const { return pos + (pos >> PS); }
  __device__ __forceinline__ void st_at(int b, int o, const Cx2<T>& v) const {
    if constexpr (sizeof(T) == 4)
      *reinterpret_cast<float4*>(buf + b + o + (o >> PS)) = make_float4(v.re.x, v.re.y, v.im.x, v.im.y);
    else
      buf[b + o + (o >> PS)] = v;
  }
  __device__ __forceinline__ Cx2<T> ld_at(int b, int o) const {
    if constexpr (sizeof(T) == 4) {
      const float4 v = *reinterpret_cast<const float4*>(buf + b + o + (o >> PS));
      return Cx2<T>{V2<T>{v.x, v.y}, V2<T>{v.z, v.w}};
    } else {
      return buf[b + o + (o >> PS)];
    }
  }
};

}  // namespace cmm
