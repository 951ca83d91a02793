// Kernels of the pair-packed path of A = P^T N^-1 P (Eq. 2; pointing of Eq. 1 with the response
// of Sec. Test setup; N^-1 the per-detector Fourier-diagonal noise filter of the
// Introduction and Sec. Test setup): FP32 compute (FP32 or BF16 spectrum storage, with or
// without noise correlated between detectors, tod_pair.cu) and FP64 (tod_pair64.cu).
//
// Two detectors in one sequence share its rounding: about 1e-7 of the larger one's values
// (2^-9 in BF16) reaches the smaller.  Weights and stored data therefore travel in powers
// of two per detector that make both of order one: w = u w', z = f s, and the filtered
// data are h y' with h = u / f (kept with the inverse transform's 1 / n_t).  Powers of two
// change no bit of detectors that are alike.
//
// Two detectors d1, d2 share one complex sequence of n_t points, z(t) = s1(t) +
// i s2(t): each complex element is one time sample of both detectors, so the
// boresight and rotation tables are read once per element for the two of them, by
// lanes on consecutive samples (coalesced).  With Z = FFT(z), the real spectra are
// S1(k) = (Z(k) + conj Z(n_t - k)) / 2 and i S2(k) = (Z(k) - conj Z(n_t - k)) / 2, so
// the filtered sequence y = y1 + i y2 has
//     Y(k) = a Z(k) + b conj Z(n_t - k),  a = (w1 + w2) / 2,  b = (w1 - w2) / 2,
// w_j = w_dj at the frequency index min(k, n_t - k) of the n_t-point DFT: each bin
// pair (k, n_t - k) is filtered with four real products and no split twiddle.
// n_t = R C as a four-step FFT over t = c + C kr (c < C contiguous, kr < R):
//
//   k_pair_fwd:     P m for both detectors at (c, kr), the R-point column FFTs over
//                   kr (register-resident, one shared-memory exchange), times
//                   w_{n_t}^{c k1}.
//   k_pair_filter:  row pairs (k1, R - k1): C-point row FFTs, the pair filter in
//                   registers, the inverse row FFTs and the conjugate twiddle.
//
// Storage rule of the spectrum between the passes.  With v[kr] the column transform,
// row k1 < R / 2 holds v[k1] w_{n_t}^{c k1} and row R - k1 (k1 = 1 .. R / 2) holds
// conj(v[R - k1]) w_{n_t}^{c k1}.  The same C-point FFT over c of the two rows then
// gives Z(k) and conj Z(n_t - k) at the same position, k = k1 + R pos:
// sum_c conj(v[R - k1]) w_{n_t}^{c k1} w_C^{c pos} = conj sum_c v[R - k1] w_{n_t}^{-c k}.
// So one thread holds both members of every bin pair: no exchange with a partner, one
// weight evaluation and one stage twiddle for the two, and the sums of both rows are
// packed instructions.  With (A, B) = (Z(k), conj Z(n_t - k)) the filter is
// (A, B) <- (a A + b B, a B + b A), and the inverse row FFT and twiddle are again the
// same for both; the last pass conjugates the rows from R / 2 up.  Rows 0 and R / 2
// pair with themselves: B = conj A, and A = conj(B) w_C^c.
//
//   k_pair_inv_bin: inverse column FFTs into a padded tile; each lane then takes 8
//                   consecutive samples of a row and bins them for each detector
//                   with a run accumulator (one vector FP32 reduction per run into
//                   the L2-resident partial map of its group of kFlushDets = 256
//                   detectors).
//   k_fast_flush_maps (tod_fast.cu) sums a launch's partial maps in FP64 into the
//   FP64 map, so no FP32 sum covers more than 256 detectors.  The FP64 form reduces its
//   runs straight into the FP64 map.
//
// A chunk with an odd number of detectors pairs its last detector with nothing
// (the imaginary part stays zero and is not binned).
#pragma once

#include <math.h>

#include <algorithm>
#include <vector>

#include "common.cuh"
#include "fft_reg.cuh"
#include "tod_common.cuh"
#include "tod_fast.cuh"

namespace cmm {

// A binning run in the frame of the scan rotation: for samples of one detector on
// one pixel, sums of u, u cos 2phi_t and u sin 2phi_t; the detector angle psi_d
// enters once, when the run is reduced: sum u cos 2(psi + phi) = cos 2psi * sum u
// cos 2phi - sin 2psi * sum u sin 2phi (and the sine likewise), with the inverse
// FFT's 1/N and the detector's u / f in st = h and (sx, sy) = (cos, sin 2psi) st.
template <typename T>
struct PairRun {
  int cur = -1;
  T t = 0, c = 0, s = 0;
};

template <int NC>
__device__ __forceinline__ void pair_run_close(float* acc32, const PairRun<float>& r, int skip, float st, float sx,
                                               float sy) {
  if (r.cur >= 0 && r.cur != skip) {
    if (NC == 1) red_add(acc32 + r.cur, st * r.t);
    else red_add4(acc32 + 4 * r.cur, st * r.t, fmaf(sx, r.c, -sy * r.s), fmaf(sy, r.c, sx * r.s));
  }
}
// FP64: straight into the FP64 map
template <int NC>
__device__ __forceinline__ void pair_run_close(double* acc, const PairRun<double>& r, int skip, double st, double sx,
                                               double sy) {
  if (r.cur >= 0 && r.cur != skip) {
    if (NC == 1) {
      atomicAdd(acc + r.cur, st * r.t);
    } else {
      double* dst = acc + 4 * (long long)r.cur;
      atomicAdd(dst, st * r.t);
      atomicAdd(dst + 1, fma(sx, r.c, -sy * r.s));
      atomicAdd(dst + 2, fma(sy, r.c, sx * r.s));
    }
  }
}

// Launch shapes: 16 columns a block, so that half a warp reads 16 consecutive samples (32
// columns at R <= 128 left too few blocks to balance: A at 128 x 2^17 149 against 143 us),
// for 32 resident warps per SM forward and 24 in the binning.  FP64: 8 columns, small
// blocks of a pipe that few warps fill (A at 32 x 2^16: 395 us, 405 with 32 columns).
template <typename T, int R> struct PairShape {
  static constexpr int J = 16;
  static constexpr int THREADS = J * R / kE;
  static constexpr int MINB = 1024 / THREADS, MINB_INV = 768 / THREADS;
};
template <int R> struct PairShape<double, R> {
  static constexpr int J = 8;
  static constexpr int THREADS = J * R / kE;
  static constexpr int MINB = 1, MINB_INV = 1;
};

// (cos 2phi, sin 2phi) of the fixed-point pair (c, s) of a boresight record, in FP32:
// (c^2 - s^2, 2 c s) / (c^2 + s^2), the integers converted exactly on the FP32 pipe
__device__ __forceinline__ float2 rot2_of_bore(const int4 b) {
  const float cf = small_int_to_float(b.z + 32768) - 32768.0f;
  const float sf = small_int_to_float(b.w + 32768) - 32768.0f;
  const float inv = __fdividef(1.0f, fmaf(cf, cf, sf * sf));
  return make_float2((cf - sf) * (cf + sf) * inv, 2.0f * cf * sf * inv);
}

// w_d / u at frequency index kf (0 <= kf <= n_t / 2) from the detector's table (cf.x = 1 / u)
template <typename T>
__device__ __forceinline__ T pair_table(const TodArgs& a, int d, const V4<T>& cf, int kf) {
  return cf.x * __ldg(reinterpret_cast<const T*>(a.wtab) + (size_t)d * (a.n_t / 2 + 1) + kf);
}

// w of one detector from log2 of its frequency index
__device__ __forceinline__ float law_weight(const float4 cf, float lk) {
  return cf.w != 0.0f ? cf.x : __fdividef(cf.x, 1.0f + exp2f(fmaf(-cf.y, lk, cf.z)));
}

// w_d1 and w_d2 at frequency index kf: from the tables, else the law with log2(kf) shared
__device__ __forceinline__ void pair_weights(const TodArgs& a, int d1, int d2, const float4 cf1, const float4 cf2,
                                             bool two, int kf, float& w1, float& w2) {
  if (a.wtab) {
    w1 = pair_table<float>(a, d1, cf1, kf);
    w2 = two ? pair_table<float>(a, d2, cf2, kf) : 0.f;
  } else {
    const float lk = __log2f(small_int_to_float(kf == 0 ? 1 : kf));
    w1 = law_weight(cf1, lk);
    w2 = two ? law_weight(cf2, lk) : 0.f;
  }
}

// The pair filter's a, b = (w_d1 +- w_d2) / 2
__device__ __forceinline__ void pair_ab(const TodArgs& a, int d1, int d2, const float4 cf1, const float4 cf2, bool two,
                                        int kf, float& ha, float& hb) {
  float w1, w2;
  pair_weights(a, d1, d2, cf1, cf2, two, kf, w1, w2);
  ha = 0.5f * (w1 + w2);
  hb = 0.5f * (w1 - w2);
}

// 2^y, |y| < kExp2Max, by table and Taylor series: y = n / 64 + r with |r| <= 1 / 128,
// 2^y = 2^(n div 64) 2^((n mod 64) / 64) e^(r ln 2), the series to r^5 (the next term is
// below 4e-17).  Nine FP64 instructions; relative error below 2.5e-16.
constexpr double kExp2Max = 500.0;
constexpr int kExp2Tab = 64;
__device__ __forceinline__ double exp2_tab(double y, const double* __restrict__ tab) {
  constexpr double kRound = 6755399441055744.0;   // 1.5 2^52: the low word of y 64 + it is n
  constexpr double l1 = 0.69314718055994530942, l2 = l1 * l1 / 2, l3 = l2 * l1 / 3, l4 = l3 * l1 / 4, l5 = l4 * l1 / 5;
  const double t = fma(y, (double)kExp2Tab, kRound);
  const int n = __double2loint(t);
  const double r = fma(t - kRound, -1.0 / kExp2Tab, y);
  const double p = r * fma(r, fma(r, fma(r, fma(r, l5, l4), l3), l2), l1);
  const double s = __ldg(tab + (n & (kExp2Tab - 1)));
  const double v = fma(s, p, s);
  return __hiloint2double(__double2hiint(v) + ((n >> 6) << 20), __double2loint(v));
}

// FP64: its pipe takes 16 cycles an instruction, so log2(kf) comes from the operator's
// table, the powers of two from exp2_tab and both weights from one reciprocal,
// w_j = x_j / d_j = x_j d_i / (d_1 d_2).  Laws too steep for that take the plain form.
__device__ __forceinline__ void pair_ab(const TodArgs& a, int d1, int d2, const double4_32a& cf1, const double4_32a& cf2,
                                        bool two, int kf, double& ha, double& hb) {
  if (a.wtab) {
    const double w1 = pair_table<double>(a, d1, cf1, kf);
    const double w2 = two ? pair_table<double>(a, d2, cf2, kf) : 0.0;
    ha = 0.5 * (w1 + w2);
    hb = 0.5 * (w1 - w2);
    return;
  }
  const double lk = __ldg(a.lg2 + kf);
  const double y1 = fma(-cf1.y, lk, cf1.z), y2 = fma(-cf2.y, lk, cf2.z);
  const int top = __double2hiint(kExp2Max);   // |y| < kExp2Max by the high words (false for NaN)
  double e1, e2, x2 = two ? cf2.x : 0.0;
  if ((__double2hiint(y1) & 0x7fffffff) < top && (__double2hiint(y2) & 0x7fffffff) < top) {
    const double* tab = a.lg2 + a.n_t / 2 + 1;
    e1 = cf1.w != 0.0 ? 0.0 : exp2_tab(y1, tab);   // white noise: d = 1
    e2 = cf2.w != 0.0 ? 0.0 : exp2_tab(y2, tab);
    e1 += 1.0;
    e2 += 1.0;
    const double h = 0.5 * __drcp_rn(e1 * e2);
    const double u = cf1.x * e2, v = x2 * e1;
    ha = (u + v) * h;
    hb = (u - v) * h;
  } else {
    e1 = cf1.w != 0.0 ? 0.0 : exp2(y1);
    e2 = cf2.w != 0.0 ? 0.0 : exp2(y2);
    const double w1 = cf1.x / (1.0 + e1), w2 = x2 / (1.0 + e2);
    ha = 0.5 * (w1 + w2);
    hb = 0.5 * (w1 - w2);
  }
}

// (P m)(t) of one detector from its pixel, the rotation (cos, sin 2phi) and the gather copy
template <typename T, int NC>
__device__ __forceinline__ T pair_project(const TodArgs& a, int p, const V2<T> pol, const V2<T> r2) {
  if (NC == 1) return __ldg((const T*)a.gather + p);
  V4<T> g;
  if constexpr (sizeof(T) == 4) g = __ldg((const float4*)a.gather + p);
  else g = reinterpret_cast<const V4<T>*>(a.gather)[p];
  const T c = pol.x * r2.x - pol.y * r2.y;
  const T s = pol.y * r2.x + pol.x * r2.y;
  return fma(s, g.z, fma(c, g.y, g.x));
}

// ------------------------------------------------------------------ pass T (forward)
// Second half of the forward pass: the column FFT of x[e] at rows i + e TPC of column c,
// and the twiddled spectrum rows of pair q.
template <typename T, typename S, int R, typename Addr>
__device__ __forceinline__ void pair_fwd_store(const TodArgs& a, V2<T> (&x)[kE], int q, int c, int i, const Addr& ad) {
  using V = V2<T>;
  constexpr int TPC = R / kE;
  const V* tw = reinterpret_cast<const V*>(a.tw);
  ColPlan<R>::template run<-1>(x, i, tw + a.twl.R_off, ad);
  // four-step twiddle w_N^(c k1), k1 = kr for kr = i + e TPC < R / 2 and k1 = R - kr, the
  // value conjugated, above (see the storage rule at the top): by recurrence in FP32; in
  // FP64, whose products cost the same either way, each from the tables
  S* Y = reinterpret_cast<S*>(a.spec) + (size_t)q * a.N + c + i * a.C;
  if constexpr (sizeof(T) == 8) {
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int k1 = e < kE / 2 ? i + e * TPC : R - i - e * TPC;
      const V w = tw_N(a, tw, c * k1);
      Store<T, S>::st(Y + e * (TPC * a.C), e < kE / 2 ? cmul(x[e], w) : cmulc(w, x[e]));
    }
  } else {
    const V step = tw_N(a, tw, c * TPC);
    V w = tw_N(a, tw, c * i);
#pragma unroll
    for (int e = 0; e < kE / 2; ++e) {
      Store<T, S>::st(Y + e * (TPC * a.C), cmul(x[e], w));
      w = cmul(w, step);
    }
    w = tw_N(a, tw, c * (TPC - i));
#pragma unroll
    for (int e = kE - 1; e >= kE / 2; --e) {
      Store<T, S>::st(Y + e * (TPC * a.C), cmulc(w, x[e]));
      w = cmul(w, step);
    }
  }
}

template <typename T, int NC, typename S, int R, bool PERIODIC, bool CACHED>
__global__ void __launch_bounds__(PairShape<T, R>::THREADS, PairShape<T, R>::MINB) k_pair_fwd(const TodArgs a, int nd) {
  using V = V2<T>;
  constexpr int TPC = R / kE;
  constexpr int J = PairShape<T, R>::J;
  if (a.done && *a.done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* smf = reinterpret_cast<V*>(smraw);
  const int cl = threadIdx.x % J;
  const int i = threadIdx.x / J;
  const int c = blockIdx.x * J + cl;
  const ColJ<J, V> ad{smf, cl};
  const int q = blockIdx.y;   // pair within the chunk
  const bool two = 2 * q + 1 < nd;
  const int d1 = a.d0 + 2 * q, d2 = two ? d1 + 1 : d1;
  const int2 off1 = a.det_off[d1], off2 = a.det_off[d2];
  const V* pol = reinterpret_cast<const V*>(a.pol);
  const V pol1 = pol[d1], pol2 = pol[d2];
  const int npix = (int)a.npix;
  V x[kE];
#pragma unroll
  for (int e = 0; e < kE; ++e) {
    const int t = c + (i + e * TPC) * a.C;
    int p1, p2;
    V r2{(T)0, (T)0};
    if constexpr (CACHED) {   // FP32 and BF16 operators
      p1 = __ldcs(a.pix + (size_t)d1 * a.n_t + t);
      p2 = __ldcs(a.pix + (size_t)d2 * a.n_t + t);
      if (NC == 3) r2 = __ldg(a.rot2 + t);
    } else {
      const int4 b = __ldg(a.bore + t);
      p1 = pixel_fast<PERIODIC>(b, off1, a.ny, a.nx, npix);
      p2 = pixel_fast<PERIODIC>(b, off2, a.ny, a.nx, npix);
      if constexpr (NC == 3 && sizeof(T) == 4) r2 = rot2_of_bore(b);
      else if constexpr (NC == 3) r2 = __ldg(a.rot64 + t);
    }
    const T v1 = pair_project<T, NC>(a, p1, pol1, r2);
    const T v2 = pair_project<T, NC>(a, p2, pol2, r2);
    x[e] = V{v1, two ? v2 : (T)0};
  }
  pair_fwd_store<T, S, R>(a, x, q, c, i, ad);
}

// The sum of squares of a thread's values in FP64, by itself, where those of type T leave
// its range; NaN where a value is not finite.
template <typename T>
__device__ __noinline__ void add_squares_far(double* out, const T (&v)[kE]) {
  T m = 0;
  bool finite = true;
  for (int e = 0; e < kE; ++e) {
    finite = finite && isfinite(v[e]);
    m = max(m, abs(v[e]));
  }
  if (!finite) {
    atomicAdd(out, (double)NAN);
  } else if (m > (T)0) {
    double d = 0.0;
    for (int e = 0; e < kE; ++e) {
      const double q = (double)v[e] / (double)m;
      d += q * q;
    }
    const double mm = min(max((double)m, 1e-150), 1e150);   // its square within FP64
    atomicAdd(out, d * mm * mm);
  }
}

// The warp's sums of squares of both numbers of x, in lane 0.
template <typename T>
__device__ __forceinline__ V2<T> warp_squares(const V2<T> (&x)[kE], bool on1, bool on2, double* out) {
  constexpr T lo = sizeof(T) == 4 ? (T)1e-24 : (T)1e-200, hi = sizeof(T) == 4 ? (T)1e30 : (T)1e200;
  V2<T> s{(T)0, (T)0};
#pragma unroll
  for (int e = 0; e < kE; ++e) s = pfma(x[e], x[e], s);
  const bool far1 = on1 && !(s.x > lo && s.x < hi), far2 = on2 && !(s.y > lo && s.y < hi);   // zero and NaN too
  if (far1 || far2) {
    T v[kE];
    for (int j = 0; j < 2; ++j) {
      if (!(j ? far2 : far1)) continue;
#pragma unroll
      for (int e = 0; e < kE; ++e) v[e] = j ? x[e].y : x[e].x;
      add_squares_far<T>(out + j, v);
      (j ? s.y : s.x) = (T)0;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s.x += __shfl_xor_sync(0xffffffffu, s.x, o);
    s.y += __shfl_xor_sync(0xffffffffu, s.y, o);
  }
  return s;
}

// The same from stored time-ordered data D [n_det][n_t] (the right-hand side): a half-warp
// reads 16 consecutive samples of either detector, times its factor f; a detector of factor
// 0 (no weight, or not finite) counts as zero.
//
// Data may be as loud as they like (a glitch, a drift, a cut detector), so the noise model's
// guess of f is checked against the data: the first pass sums their squares on the way,
// k_tod_gains lists the pairs whose detectors differ, and the LIST form transforms those
// again with measured factors.  Reading the data for their level before the transform would
// cost every call a pass over them (537 MB at 256 x 2^19: 80 us).  One FP64 atomic per
// block and detector, and no load waits for a factor: with one atomic per warp, whose
// blocks meet on the addresses of a few pairs, and with such waits 935 us a right-hand
// side of 256 x 2^19, now 840; 825 without the factors, of which 8 us are the two small
// kernels when no pair is listed, and 1350 in the one-detector packing, whose forward pass
// from stored data is the generic kernel.
template <typename T, typename S, int R, typename D, bool LIST>
__global__ void __launch_bounds__(PairShape<T, R>::THREADS, PairShape<T, R>::MINB) k_pair_fwd_tod(const TodArgs a, int nd) {
  using V = V2<T>;
  constexpr int TPC = R / kE;
  constexpr int J = PairShape<T, R>::J;
  if (a.done && *a.done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ V sums[PairShape<T, R>::THREADS / 32];
  const int cl = threadIdx.x % J;
  const int i = threadIdx.x / J;
  const int c = blockIdx.x * J + cl;
  const ColJ<J, V> ad{reinterpret_cast<V*>(smraw), cl};
  const int nq = LIST ? a.tod_list[0] : (int)gridDim.y;
  for (int j = blockIdx.y; j < nq; j += gridDim.y) {   // LIST: over the listed pairs, else once
    const int q = LIST ? a.tod_list[1 + j] : j;
    const bool two = 2 * q + 1 < nd;
    const int d1 = a.d0 + 2 * q, d2 = two ? d1 + 1 : d1;
    const T f1 = (T)a.tod_f[d1], f2 = two ? (T)a.tod_f[d2] : (T)0;
    const D* t1 = reinterpret_cast<const D*>(a.tod) + (size_t)d1 * a.n_t + c;
    const D* t2 = reinterpret_cast<const D*>(a.tod) + (size_t)d2 * a.n_t + c;
    const bool on1 = f1 != (T)0, on2 = f2 != (T)0;   // uniform over the block
    V x[kE];
#pragma unroll
    for (int e = 0; e < kE; ++e) {
      const int o = (i + e * TPC) * a.C;
      x[e] = pmul(V{f1, f2}, V{(T)__ldcs(t1 + o), (T)__ldcs(t2 + o)});
    }
    if (!on1 || !on2) {   // whatever is stored there, NaN too
#pragma unroll
      for (int e = 0; e < kE; ++e) x[e] = V{on1 ? x[e].x : (T)0, on2 ? x[e].y : (T)0};
    }
    if constexpr (!LIST) {
      const V s = warp_squares<T>(x, on1, on2, a.tod_norm + d1);
      if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = s;
    }
    pair_fwd_store<T, S, R>(a, x, q, c, i, ad);   // with barriers between its stages
    if constexpr (LIST) {
      __syncthreads();   // the next pair reuses the exchange buffer
    } else if (threadIdx.x < (two ? 2 : 1)) {
      double s = 0.0;
      for (int w = 0; w < PairShape<T, R>::THREADS / 32; ++w) s += widen(threadIdx.x ? sums[w].y : sums[w].x);
      if (s > 0.0) atomicAdd(a.tod_norm + d1 + threadIdx.x, s);
    }
  }
}

// ------------------------------------------------------------------ pass F (filter)
// Both rows of a pair in one thread (2 x 16 complex values): 118 registers, 16 resident
// warps per SM, 95M warp instructions on 64 detectors x 2^20 samples where one row a
// thread (32 warps, the partner's values through shared memory) took 151M; 2.85 -> 2.44
// ms at 1024 x 2^20.  It is now bound by latency (issue 48 %, FP32 pipe 55 % active,
// DRAM 37 %): 24 warps at 80 registers spill (2.99 ms).  Rows shorter than 128 threads
// share a CTA of 128 (64: the same times; 256: 85 against 74 us at 128 x 2^18).
// FP64: 8 points of both rows a thread and one block per SM.
template <typename T, int C, int E> struct PairFilterShape {
  static constexpr int TPR = C / E;   // threads per row pair
  static constexpr int LEAST = sizeof(T) == 8 ? 32 : 128;
  static constexpr int THREADS = TPR > LEAST ? TPR : LEAST;
  static constexpr int PAIRS = THREADS / TPR;   // row pairs per CTA
  static constexpr int MINB = sizeof(T) == 8 ? 1 : 512 / THREADS;
};

// The spectrum slots of the cross-detector step: slot k1 C + pos holds bin k = k1 + R pos,
// k1 = 0 .. R / 2 (rows 0 and R / 2 hold every bin twice, conjugated).
__host__ __device__ __forceinline__ int pair_corr_slots(int R, int C) { return (R / 2 + 1) * C; }

// Modes.  kPairFull: the whole pass.  With noise correlated between detectors the pass is
// cut around k_pair_corr: kPairSplit stores the forward transforms, Z(k) in row k1 and
// conj Z(n - k) in row R - k1 (rows 0 and R / 2: Z(k) alone, whose partner is in the same
// row); kPairMerge starts from those, y_j = w_j (S_j - sum_m V_jm s_m) with the spectra
// S_1 = (A + B) / 2 and S_2 = (A - B) / 2i of the two detectors, and inverts
// (A, B) = (y_1 + i y_2, y_1 - i y_2).
constexpr int kPairFull = 0, kPairSplit = 1, kPairMerge = 2;

template <typename T, typename S, int MODE, int E, int... RC>
__global__ void __launch_bounds__(PairFilterShape<T, RadProd<RC...>::value, E>::THREADS,
                                  PairFilterShape<T, RadProd<RC...>::value, E>::MINB)
    k_pair_filter(const TodArgs a, int nd) {
  using V = V2<T>;
  constexpr int C = RadProd<RC...>::value;
  constexpr int TPR = C / E;
  constexpr int PAIRS = PairFilterShape<T, C, E>::PAIRS;
  constexpr int PS = clog2(E);
  constexpr int ROWLEN = C + (C >> PS);
  if (a.done && *a.done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int rs = threadIdx.x / TPR;
  const int i = threadIdx.x % TPR;
  const int k1 = blockIdx.x * PAIRS + rs;
  const bool ok = k1 <= (a.R >> 1);
  const bool lo = k1 == 0, mid = k1 == (a.R >> 1);   // rows paired with themselves
  const int q = blockIdx.y;
  const bool two = 2 * q + 1 < nd;
  const int d1 = a.d0 + 2 * q, d2 = two ? d1 + 1 : d1;
  const V* tw = reinterpret_cast<const V*>(a.tw);
  S* Ya = reinterpret_cast<S*>(a.spec) + (size_t)q * a.N + k1 * C + i;
  S* Yb = lo ? Ya : Ya + (a.R - 2 * k1) * C;   // row R - k1
  const RowAddr2<T, PS> ad{reinterpret_cast<Cx2<T>*>(smraw) + rs * ROWLEN};
  Cx2<T> x[E];
  if constexpr (MODE == kPairMerge) {
    if (lo || mid) {   // the partner position of the same row, conjugated
      const S* row = Ya - i;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int pos = i + e * TPR;
        const V A = Store<T, S>::ld(row + pos), B = Store<T, S>::ld(row + (lo ? (C - pos) & (C - 1) : C - 1 - pos));
        x[e] = Cx2<T>{V{A.x, B.x}, V{A.y, -B.y}};
      }
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const V A = ok ? Store<T, S>::ld(Ya + e * TPR) : V{(T)0, (T)0};
        const V B = ok ? Store<T, S>::ld(Yb + e * TPR) : V{(T)0, (T)0};
        x[e] = Cx2<T>{V{A.x, B.x}, V{A.y, B.y}};
      }
    }
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const V A = ok ? Store<T, S>::ld(Ya + e * TPR) : V{(T)0, (T)0};
      const V B = ok ? Store<T, S>::ld(Yb + e * TPR) : V{(T)0, (T)0};
      x[e] = Cx2<T>{V{A.x, B.x}, V{A.y, B.y}};
    }
    if (lo) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[e].im.y = -x[e].im.x;   // B = conj A
    } else if (mid) {
      // row R / 2 is stored as B = conj(y) w_N^(c R / 2): A = conj(B) w_C^c
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const V A = cmul(V{x[e].re.y, -x[e].im.y}, __ldg(tw + a.twl.C_off + i + e * TPR));
        x[e].re.x = A.x;
        x[e].im.x = A.y;
      }
    }
    rfft2<T, -1, true, E, RC...>(x, i, tw + a.twl.C_off, ad);
  }
  if constexpr (MODE == kPairSplit) {
    if (ok) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        Store<T, S>::st(Ya + e * TPR, V{x[e].re.x, x[e].im.x});
        if (!lo && !mid) Store<T, S>::st(Yb + e * TPR, V{x[e].re.y, x[e].im.y});
      }
    }
    return;
  }
  {
    const V4<T> cf1 = reinterpret_cast<const V4<T>*>(a.coef)[d1];
    const V4<T> cf2 = reinterpret_cast<const V4<T>*>(a.coef)[d2];
    const int n = (int)a.N;
    float tv1[kMaxCorrModes], tv2[kMaxCorrModes];   // the detectors' templates, as their data times f
    const int slots = pair_corr_slots(a.R, C);
    if constexpr (MODE == kPairMerge) {
      const float f1 = a.tod_f ? a.tod_f[d1] : 1.f, f2 = a.tod_f ? a.tod_f[d2] : 1.f;
#pragma unroll
      for (int j = 0; j < kMaxCorrModes; ++j) {
        tv1[j] = j < a.corr_r ? f1 * a.corrV[d1 * a.corr_r + j] : 0.f;
        tv2[j] = j < a.corr_r ? f2 * a.corrV[d2 * a.corr_r + j] : 0.f;
      }
    }
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int k = k1 + a.R * (i + e * TPR);
      const int kf = ok ? min(k, n - k) : 0;
      if constexpr (MODE == kPairMerge) {
        T w1, w2;
        pair_weights(a, d1, d2, cf1, cf2, two, kf, w1, w2);
        V p1{(T)0, (T)0}, p2{(T)0, (T)0};
        const float2* sol = a.corr_s + (ok ? k1 * C + i + e * TPR : 0);
#pragma unroll
        for (int j = 0; j < kMaxCorrModes; ++j)
          if (j < a.corr_r) {
            const float2 sj = __ldg(sol + j * slots);
            p1 = V{fmaf(tv1[j], sj.x, p1.x), fmaf(tv1[j], sj.y, p1.y)};
            p2 = V{fmaf(tv2[j], sj.x, p2.x), fmaf(tv2[j], sj.y, p2.y)};
          }
        const Cx2<T> v = x[e];
        const T h = (T)0.5;
        const V y1{w1 * (h * (v.re.x + v.re.y) - p1.x), w1 * (h * (v.im.x + v.im.y) - p1.y)};
        const V y2{w2 * (h * (v.im.x - v.im.y) - p2.x), w2 * (h * (v.re.y - v.re.x) - p2.y)};
        x[e] = Cx2<T>{V{y1.x - y2.y, y1.x + y2.y}, V{y1.y + y2.x, y1.y - y2.x}};
      } else {
        T ha, hb;
        pair_ab(a, d1, d2, cf1, cf2, two, kf, ha, hb);
        const V h{ha, ha}, g{hb, hb};
        x[e].re = pfma(h, x[e].re, pmul(g, V{x[e].re.y, x[e].re.x}));
        x[e].im = pfma(h, x[e].im, pmul(g, V{x[e].im.y, x[e].im.x}));
      }
    }
  }
  rfft2<T, 1, MODE == kPairMerge, E, RC...>(x, i, tw + a.twl.C_off, ad);
  if (ok) {
    // conj(w_N^(k1 c)), c = i + e TPR, for both rows: by recurrence, or from the tables
    V w = tw_N(a, tw, k1 * i);
    const V stp = tw_N(a, tw, k1 * TPR);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const Cx2<T> y = cx_mul<T>(x[e], w.x, -w.y);
      if (!mid) Store<T, S>::st(Ya + e * TPR, V{y.re.x, y.im.x});
      if (!lo) Store<T, S>::st(Yb + e * TPR, V{y.re.y, y.im.y});
      if constexpr (sizeof(T) == 4) w = cmul(w, stp);
      else if (e + 1 < E) w = tw_N(a, tw, k1 * (i + (e + 1) * TPR));
    }
  }
}

// ------------------------------------------------------------------ correlated noise
// Cross-detector step, one thread per slot: t_j = sum_d V_dj w_d(k) S_d(k) over all
// detectors, s = M(k)^-1 t (see k_corr_minv).  Bound by its one read of the spectra
// (4 bytes a sample in FP32) beside the weights; log2(k) is shared by all detectors, whose
// coefficients and templates are staged in shared memory.  1024 x 2^20, three modes: 0.93
// ms (4.6 TB/s) beside 1.31 ms for kPairSplit and 2.73 for kPairMerge, which reads every
// bin's solution from L2 once per pair of detectors (8 points a thread: 2.84 ms; pairs
// varying fastest over the blocks: 2.89).  A with three modes 13.9 -> 9.95 ms against the
// one-detector packing, 192 x 2^19 1.39 -> 0.99.
constexpr int kCorrThreads = 256, kCorrStage = 64;   // pairs staged at a time

template <typename S, int RM>
__global__ void __launch_bounds__(kCorrThreads) k_pair_corr(const TodArgs a, int n_det) {
  __shared__ float4 coef[2 * kCorrStage];
  __shared__ float V[2 * kCorrStage][RM];
  if (a.done && *a.done) return;
  const int slots = pair_corr_slots(a.R, a.C);
  const int slot = min((int)(blockIdx.x * kCorrThreads + threadIdx.x), slots - 1);
  const int k1 = slot >> a.logC, pos = slot & (a.C - 1);
  const int k = k1 + a.R * pos, n = (int)a.N, kf = min(k, n - k);
  const bool self = k1 == 0 || 2 * k1 == a.R;   // the partner bin in the same row
  const int other = k1 == 0 ? ((a.C - pos) & (a.C - 1)) : self ? k1 * a.C + a.C - 1 - pos : (a.R - k1) * a.C + pos;
  const S* Ya = reinterpret_cast<const S*>(a.spec) + slot;
  const S* Yb = reinterpret_cast<const S*>(a.spec) + other;
  const float lk = __log2f(small_int_to_float(kf == 0 ? 1 : kf));
  const int pairs = (n_det + 1) / 2;
  float2 t[RM];
#pragma unroll
  for (int j = 0; j < RM; ++j) t[j] = make_float2(0.f, 0.f);
  for (int q0 = 0; q0 < pairs; q0 += kCorrStage) {
    const int nq = min(kCorrStage, pairs - q0);
    __syncthreads();
    for (int d = threadIdx.x; d < 2 * nq; d += kCorrThreads) {
      const int dd = a.d0 + min(2 * q0 + d, n_det - 1);
      const bool real = 2 * q0 + d < n_det;   // the missing partner of an odd last detector
      coef[d] = reinterpret_cast<const float4*>(a.coef)[dd];
      const float h = (float)a.n_t * a.tod_h[dd];   // w V S = (w / u) (u / f V) (f S)
#pragma unroll
      for (int j = 0; j < RM; ++j) V[d][j] = real ? h * a.corrV[dd * RM + j] : 0.f;
    }
    __syncthreads();
#pragma unroll 4
    for (int q = 0; q < nq; ++q) {
      const size_t o = (size_t)(q0 + q) * a.N;
      const float2 A = Store<float, S>::ld(Ya + o);
      float2 B = Store<float, S>::ld(Yb + o);
      if (self) B.y = -B.y;
      float w1, w2;
      if (a.wtab) {
        const int d1 = a.d0 + 2 * (q0 + q);
        w1 = pair_table<float>(a, d1, coef[2 * q], kf);
        w2 = pair_table<float>(a, min(d1 + 1, a.d0 + n_det - 1), coef[2 * q + 1], kf);
      } else {
        w1 = law_weight(coef[2 * q], lk);
        w2 = law_weight(coef[2 * q + 1], lk);
      }
      w1 *= 0.5f;
      w2 *= 0.5f;
      const float2 s1 = make_float2(w1 * (A.x + B.x), w1 * (A.y + B.y));
      const float2 s2 = make_float2(w2 * (A.y - B.y), w2 * (B.x - A.x));
#pragma unroll
      for (int j = 0; j < RM; ++j) {
        const float v1 = V[2 * q][j], v2 = V[2 * q + 1][j];
        t[j].x = fmaf(v1, s1.x, fmaf(v2, s2.x, t[j].x));
        t[j].y = fmaf(v1, s1.y, fmaf(v2, s2.y, t[j].y));
      }
    }
  }
  if ((int)(blockIdx.x * kCorrThreads + threadIdx.x) >= slots) return;
  const float* m = a.corr_minv + (size_t)slot * RM * RM;
#pragma unroll
  for (int j = 0; j < RM; ++j) {
    float sx = 0.f, sy = 0.f;
#pragma unroll
    for (int l = 0; l < RM; ++l) {
      sx = fmaf(m[j * RM + l], t[l].x, sx);
      sy = fmaf(m[j * RM + l], t[l].y, sy);
    }
    a.corr_s[j * slots + slot] = make_float2(sx, sy);
  }
}

// ------------------------------------------------------------------ pass T' (inverse + P^T)
template <typename T, int NC, typename S, int R, bool PERIODIC, bool CACHED>
__global__ void __launch_bounds__(PairShape<T, R>::THREADS, PairShape<T, R>::MINB_INV)
    k_pair_inv_bin(const TodArgs a, int nd) {
  using V = V2<T>;
  constexpr int TPC = R / kE;
  constexpr int J = PairShape<T, R>::J;
  constexpr int NT = PairShape<T, R>::THREADS;
  constexpr int BS = J + 2;    // row stride of the binning tile (the pad spreads rows over the banks)
  constexpr int SPL = 8;              // consecutive samples per lane
  constexpr int LPR = J / SPL;        // lanes per row
  constexpr int RPP = NT / LPR;       // rows per binning pass
  // Pixel staging: rows of PS ints; a lane's 8 pixels are two 16-byte chunks interleaved
  // with its row neighbour's and permuted by an XOR with the row, so that the staging
  // stores and the eight lanes of a quarter-warp load spread over the 4-bank groups.
  constexpr int PS = 16;
  static_assert(LPR >= 1 && RPP <= R && R % RPP == 0 && (RPP * J) % NT == 0, "binning layout");
  if (a.done && *a.done) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  V* smf = reinterpret_cast<V*>(smraw);
  const int cl = threadIdx.x % J;
  const int i = threadIdx.x / J;
  const int c = blockIdx.x * J + cl;
  const int c0 = blockIdx.x * J;
  const V* tw = reinterpret_cast<const V*>(a.tw);
  const ColJ<J, V> ad{smf, cl};
  const int q = blockIdx.y;
  const bool two = 2 * q + 1 < nd;
  const int d1 = a.d0 + 2 * q, d2 = two ? d1 + 1 : d1;
  // FP32: the partial map of this pair's group of detectors (whole pairs per group)
  T* acc;
  if constexpr (sizeof(T) == 4) acc = a.acc32 + (long long)((2 * q) / a.flush_dets) * a.acc32_map;
  else acc = a.acc;
  const int npix = (int)a.npix;
  const S* Y = reinterpret_cast<const S*>(a.spec) + (size_t)q * a.N + c + i * a.C;
  V x[kE];
#pragma unroll
  for (int e = 0; e < kE; ++e) {
    x[e] = Store<T, S>::ld(Y + e * (TPC * a.C));
    if (e >= kE / 2) x[e].y = -x[e].y;   // rows R / 2 and above are stored conjugated
  }
  ColPlan<R>::template run<1>(x, i, tw + a.twl.R_off, ad);
  __syncthreads();
  // y(t) for t = c + C kr into a tile of rows kr
#pragma unroll
  for (int e = 0; e < kE; ++e) smf[(i + e * TPC) * BS + cl] = x[e];
  __syncthreads();
  const int bq = threadIdx.x % LPR;
  const int br = threadIdx.x / LPR;
  const V* pol = reinterpret_cast<const V*>(a.pol);
  const V pol1 = pol[d1], pol2 = pol[d2];
  const int2 off1 = a.det_off[d1], off2 = a.det_off[d2];
  int* pst = reinterpret_cast<int*>(smf + R * BS);   // pixels of one pass: [detector][RPP][PS]
  for (int kr0 = 0; kr0 < R; kr0 += RPP) {
    const int kr = kr0 + br;
    const int tq = c0 + SPL * bq + kr * a.C;   // the lane's first sample
    // the lane's 8 rotations (64 bytes, 64-byte aligned: tq is a multiple of 8),
    // issued before the staging so that they are in flight across its barrier
    V r2[8];
    if constexpr (NC == 3) {
      if constexpr (sizeof(T) == 8) {
#pragma unroll
        for (int k = 0; k < 8; ++k) r2[k] = __ldg(a.rot64 + tq + k);
      } else if constexpr (CMM_V8) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float v[8];
          ld_nc_v8(a.rot2 + tq + 4 * h, v);
#pragma unroll
          for (int k = 0; k < 4; ++k) r2[4 * h + k] = make_float2(v[2 * k], v[2 * k + 1]);
        }
      } else {
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(a.rot2 + tq + k));
          r2[k] = make_float2(v.x, v.y);
          r2[k + 1] = make_float2(v.z, v.w);
        }
      }
    }
    if constexpr (!CACHED) {
      // pixels of both detectors for the pass's RPP x J samples, lanes on
      // consecutive samples (coalesced boresight reads)
#pragma unroll
      for (int k = 0; k < RPP * J / NT; ++k) {
        const int sidx = threadIdx.x + k * NT;
        const int rr = sidx / J, col = sidx % J;
        const int4 b = __ldg(a.bore + c0 + col + (kr0 + rr) * a.C);
        // column col = 8 bq + 4 h + w of the row goes to chunk (2 h + bq) ^ (row & 3)
        const int sw = (((((col >> 1) & 2) | ((col >> 3) & 1)) ^ (rr & 3)) << 2) | (col & 3);
        pst[rr * PS + sw] = pixel_fast<PERIODIC>(b, off1, a.ny, a.nx, npix);
        pst[(RPP + rr) * PS + sw] = pixel_fast<PERIODIC>(b, off2, a.ny, a.nx, npix);
      }
      __syncthreads();
    }
    // the lane's 8 filtered samples of both detectors (real part: d1, imaginary: d2)
    V yv[8];
    if constexpr (sizeof(T) == 4) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 v = reinterpret_cast<const float4*>(smf)[(kr * BS + 8 * bq) / 2 + j];
        yv[2 * j] = V{v.x, v.y};
        yv[2 * j + 1] = V{v.z, v.w};
      }
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) yv[k] = smf[kr * BS + 8 * bq + k];
    }
#pragma unroll
    for (int dd = 0; dd < 2; ++dd) {
      if (dd == 1 && !two) break;
      int p[8];
      int4 P0, P1;
      if constexpr (CACHED && CMM_V8) {
        // 32 bytes, 32-byte aligned (tq and n_t are multiples of 8)
        ld_cs_v8(a.pix + (size_t)(dd ? d2 : d1) * a.n_t + tq, p);
        P0 = make_int4(p[0], p[1], p[2], p[3]);
        P1 = make_int4(p[4], p[5], p[6], p[7]);
      } else if constexpr (CACHED) {
        const int* pixd = a.pix + (size_t)(dd ? d2 : d1) * a.n_t + tq;
        P0 = __ldcs(reinterpret_cast<const int4*>(pixd));
        P1 = __ldcs(reinterpret_cast<const int4*>(pixd + 4));
      } else {
        const int* prow = pst + (dd * RPP + br) * PS;
        P0 = *reinterpret_cast<const int4*>(prow + ((bq ^ (br & 3)) << 2));
        P1 = *reinterpret_cast<const int4*>(prow + (((2 | bq) ^ (br & 3)) << 2));
      }
      p[0] = P0.x; p[1] = P0.y; p[2] = P0.z; p[3] = P0.w;
      p[4] = P1.x; p[5] = P1.y; p[6] = P1.z; p[7] = P1.w;
      const V pl = dd ? pol2 : pol1;
      // loaded here: held in registers through the pass they cost it 1.3 % (301 x 2^19)
      const T st = (T)__ldg(a.tod_h + (dd ? d2 : d1)), sx = st * pl.x, sy = st * pl.y;
      PairRun<T> run;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const T u = dd ? yv[k].y : yv[k].x;
        if (p[k] != run.cur) {
          pair_run_close<NC>(acc, run, npix, st, sx, sy);
          run.cur = p[k];
          run.t = run.c = run.s = 0;
        }
        run.t += u;
        if (NC == 3) {
          run.c = fma(r2[k].x, u, run.c);
          run.s = fma(r2[k].y, u, run.s);
        }
      }
      pair_run_close<NC>(acc, run, npix, st, sx, sy);
    }
    if constexpr (!CACHED) __syncthreads();   // the staging is rewritten by the next pass
  }
}

// ------------------------------------------------------------------ dispatch

template <typename T, int NC, typename S, int R, bool PERIODIC, bool CACHED>
inline int run_pair_T_c(const TodArgs& a, int nd, int pass, cudaStream_t st, bool attr_only) {
  constexpr int J = PairShape<T, R>::J;
  constexpr int NT = PairShape<T, R>::THREADS;
  // forward: FFT tile R x J complex.  inverse: binning tile R x (J + 2) complex and the
  // pixel staging of one pass (2 detectors x RPP rows x PS ints)
  constexpr int RPP = NT / (J / 8);   // rows per binning pass
  const int smem_f = (int)(sizeof(V2<T>) * R * J);
  constexpr int PS = 16;
  // (the pixel-cache instances stage no pixels: less shared memory leaves more L1)
  const int smem_i = (int)(sizeof(V2<T>) * R * (J + 2) + (CACHED ? 0 : sizeof(int) * 2 * RPP * PS));
  if (attr_only) {
    CMM_CUDA(cudaFuncSetAttribute(k_pair_fwd<T, NC, S, R, PERIODIC, CACHED>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  smem_f));
    CMM_CUDA(cudaFuncSetAttribute(k_pair_inv_bin<T, NC, S, R, PERIODIC, CACHED>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, smem_i));
    return CMM_OK;
  }
  const dim3 g(a.C / J, (nd + 1) / 2);
  if (pass == 0) k_pair_fwd<T, NC, S, R, PERIODIC, CACHED><<<g, NT, smem_f, st>>>(a, nd);
  else k_pair_inv_bin<T, NC, S, R, PERIODIC, CACHED><<<g, NT, smem_i, st>>>(a, nd);
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}

// The cached-pixel kernels exist only for the non-periodic map.
template <typename T, int NC, typename S, int R, bool PERIODIC>
inline int run_pair_T(const TodArgs& a, int nd, int pass, cudaStream_t st, bool attr_only) {
  if constexpr (!PERIODIC && sizeof(T) == 4) {
    if (attr_only) CMM_TRY((run_pair_T_c<T, NC, S, R, false, true>(a, nd, pass, st, true)));
    else if (a.pix) return run_pair_T_c<T, NC, S, R, false, true>(a, nd, pass, st, false);
  }
  return run_pair_T_c<T, NC, S, R, PERIODIC, false>(a, nd, pass, st, attr_only);
}

template <typename T, int NC, typename S, bool PERIODIC>
inline int dispatch_pair_T_p(const TodArgs& a, int nd, int pass, cudaStream_t st, bool attr_only) {
  if (a.logR == 6) return run_pair_T<T, NC, S, 64, PERIODIC>(a, nd, pass, st, attr_only);
  if (a.logR == 7) return run_pair_T<T, NC, S, 128, PERIODIC>(a, nd, pass, st, attr_only);
  return run_pair_T<T, NC, S, 256, PERIODIC>(a, nd, pass, st, attr_only);
}

template <typename T, int NC, typename S>
inline int dispatch_pair_T(const TodArgs& a, int nd, int pass, cudaStream_t st, bool attr_only) {
  return a.periodic ? dispatch_pair_T_p<T, NC, S, true>(a, nd, pass, st, attr_only)
                    : dispatch_pair_T_p<T, NC, S, false>(a, nd, pass, st, attr_only);
}

// Forward pass from stored data (a.tod).
// LIST: the pairs of a.tod_list, whose number the device knows; few blocks, since the list
// is empty for data like their noise model (8 to a column: 3 us at 256 x 2^19).
template <typename T, typename S, int R, bool LIST>
inline int run_pair_D(const TodArgs& a, int nd, bool f64, cudaStream_t st, bool attr_only) {
  constexpr int J = PairShape<T, R>::J;
  const int smem = (int)(sizeof(V2<T>) * R * J);
  const auto k = f64 ? k_pair_fwd_tod<T, S, R, double, LIST> : k_pair_fwd_tod<T, S, R, float, LIST>;
  if (attr_only) {
    CMM_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    return CMM_OK;
  }
  const int pairs = (nd + 1) / 2;
  k<<<dim3(a.C / J, LIST ? std::min(pairs, 8) : pairs), PairShape<T, R>::THREADS, smem, st>>>(a, nd);
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}

template <typename T, typename S, bool LIST>
inline int dispatch_pair_D(const TodArgs& a, int nd, bool f64, cudaStream_t st, bool attr_only) {
  if (a.logR == 6) return run_pair_D<T, S, 64, LIST>(a, nd, f64, st, attr_only);
  if (a.logR == 7) return run_pair_D<T, S, 128, LIST>(a, nd, f64, st, attr_only);
  return run_pair_D<T, S, 256, LIST>(a, nd, f64, st, attr_only);
}

int launch_tod_gains(const cmm_op* op, const TodArgs& a, int nd, cudaStream_t st);

// The whole forward pass from stored data; leaves the factors in a for the passes after it.
template <typename T, typename S>
inline int pair_fwd_stored(const cmm_op* op, TodArgs& a, int nd, const void* tod, bool f64, cudaStream_t st) {
  a.tod = tod;
  a.tod_f = op->nz->tod_guess;
  CMM_TRY((dispatch_pair_D<T, S, false>(a, nd, f64, st, false)));
  CMM_TRY(launch_tod_gains(op, a, nd, st));
  a.tod_f = op->tod_f;
  return dispatch_pair_D<T, S, true>(a, nd, f64, st, false);
}

// The path's coefficients: those of A, then those of stored data.
inline const char* pair_coef(const cmm_op* op) {
  return op->prec == CMM_PREC_F64 ? reinterpret_cast<const char*>(op->nz->pair64)
                                  : reinterpret_cast<const char*>(op->nz->pair32);
}

// The factors of stored data in the passes after the forward one.
inline void stored_gains(const cmm_op* op, TodArgs& a) {
  a.coef = pair_coef(op) + op->pt->n_det * (op->prec == CMM_PREC_F64 ? sizeof(double4_32a) : sizeof(float4));
  a.tod_f = op->tod_f;
  a.tod_h = op->tod_h;
}

template <typename T, typename S, int MODE, int E, int... RC>
inline int run_pair_F(const TodArgs& a, int nd, cudaStream_t st, bool attr_only) {
  constexpr int C = RadProd<RC...>::value;
  constexpr int PAIRS = PairFilterShape<T, C, E>::PAIRS;
  constexpr int PS = clog2(E);
  const size_t smem = sizeof(Cx2<T>) * PAIRS * (C + (C >> PS));
  if (attr_only) {
    CMM_CUDA(cudaFuncSetAttribute(k_pair_filter<T, S, MODE, E, RC...>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    return CMM_OK;
  }
  const int nrp = a.R / 2 + 1;
  const dim3 g((nrp + PAIRS - 1) / PAIRS, (nd + 1) / 2);
  k_pair_filter<T, S, MODE, E, RC...><<<g, PairFilterShape<T, C, E>::THREADS, smem, st>>>(a, nd);
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}

template <typename T, typename S, int MODE = kPairFull>
inline int dispatch_pair_F(const TodArgs& a, int nd, cudaStream_t st, bool attr_only) {
  if constexpr (sizeof(T) == 4) {
    switch (a.logC) {
      // short rows: 8 points a thread, twice the threads (row transforms of 32 x 2^16 take
      // 10.3 against 12.4 us); from 1024 points on the third exchange costs more (75
      // against 74 us at 1024, 2.82 against 2.45 ms at 4096)
      case 7: return run_pair_F<T, S, MODE, 8, 8, 8, 2>(a, nd, st, attr_only);
      case 8: return run_pair_F<T, S, MODE, 8, 8, 8, 4>(a, nd, st, attr_only);
      case 9: return run_pair_F<T, S, MODE, 8, 8, 8, 8>(a, nd, st, attr_only);
      case 10: return run_pair_F<T, S, MODE, 16, 16, 16, 4>(a, nd, st, attr_only);
      case 11: return run_pair_F<T, S, MODE, 16, 16, 16, 8>(a, nd, st, attr_only);
      case 12: return run_pair_F<T, S, MODE, 16, 16, 16, 16>(a, nd, st, attr_only);
    }
  } else {
    switch (a.logC) {
      case 7: return run_pair_F<T, S, MODE, 8, 8, 8, 2>(a, nd, st, attr_only);
      case 8: return run_pair_F<T, S, MODE, 8, 8, 8, 4>(a, nd, st, attr_only);
      case 9: return run_pair_F<T, S, MODE, 8, 8, 8, 8>(a, nd, st, attr_only);
      case 10: return run_pair_F<T, S, MODE, 8, 8, 8, 8, 2>(a, nd, st, attr_only);
      case 11: return run_pair_F<T, S, MODE, 8, 8, 8, 8, 4>(a, nd, st, attr_only);
      case 12: return run_pair_F<T, S, MODE, 8, 8, 8, 8, 8>(a, nd, st, attr_only);
    }
  }
  return fail(CMM_ERR_UNSUPPORTED, "pair path: row length out of range");
}

inline TodArgs pair_args(const cmm_op* op, int d0) {
  TodArgs a = make_args(op, d0);
  a.N = op->pt->n_t;
  a.R = op->pR;
  a.C = op->pC;
  a.logR = op->plogR;
  a.logC = op->plogC;
  a.tw = op->tw_pair;
  a.twl = tw_layout(op->pR, op->pC);
  a.coef = pair_coef(op);
  return a;
}

// Twiddle tables of the pair split: w_R, w_C, and the low part of w_{n_t}
template <typename T>
inline int pair_twiddles(cmm_op* op) {
  const TwLayout l = tw_layout(op->pR, op->pC);
  std::vector<V2<T>> h(l.total);
  auto fill = [&](int64_t off, int count, double L) {
    for (int e = 0; e < count; ++e) {
      const double ang = -2.0 * M_PI * (double)e / L;
      h[off + e] = V2<T>{(T)std::cos(ang), (T)std::sin(ang)};
    }
  };
  fill(l.R_off, op->pR, op->pR);
  fill(l.C_off, op->pC, op->pC);
  fill(l.Nlo_off, op->pC, (double)op->pt->n_t);
  void* d = nullptr;
  if (cudaMalloc(&d, sizeof(V2<T>) * l.total) != cudaSuccess) {
    cudaGetLastError();
    return fail(CMM_ERR_OOM, "twiddle table allocation failed");
  }
  op->tw_pair = d;
  CMM_CUDA(cudaMemcpy(op->tw_pair, h.data(), sizeof(V2<T>) * l.total, cudaMemcpyHostToDevice));
  return CMM_OK;
}

template <typename T, typename S>
inline int prepare_pair_s(cmm_op* op) {
  TodArgs a = pair_args(op, 0);
  for (const bool f64 : {false, true}) {
    CMM_TRY((dispatch_pair_D<T, S, false>(a, 0, f64, nullptr, true)));
    CMM_TRY((dispatch_pair_D<T, S, true>(a, 0, f64, nullptr, true)));
  }
  if (op->pt->ncomp == 1) CMM_TRY((dispatch_pair_T<T, 1, S>(a, 0, 0, nullptr, true)));
  else CMM_TRY((dispatch_pair_T<T, 3, S>(a, 0, 0, nullptr, true)));
  if constexpr (sizeof(T) == 4) {
    CMM_TRY((dispatch_pair_F<T, S, kPairSplit>(a, 0, nullptr, true)));
    CMM_TRY((dispatch_pair_F<T, S, kPairMerge>(a, 0, nullptr, true)));
  }
  return dispatch_pair_F<T, S>(a, 0, nullptr, true);
}

}  // namespace cmm
