// The circulant preconditioner's apply z = Sigma^-1 F^-1 H^-1 F Sigma^-1 r (Eq. 12) of
// TQU maps in three kernels:
//
//   k_circ_rows_fwd:  Sigma^-1 r and the row transforms,
//   k_circ_cols:      the column transforms, the per-mode products, and the inverse
//                     column transforms, a column and its mirror (the modes f and -f)
//                     in one block,
//   k_circ_rows_inv:  the inverse row transforms, Sigma^-1 and the partial sums of r^T z.
//
// The three real planes travel as two complex ones, T + i Q and U, interleaved per pixel
// as one Cx2 (two complex numbers that every transform treats alike): one 16-byte (FP32)
// access, one twiddle and packed sums for the two.  A real plane's spectrum is Hermitian,
// so X_T and X_Q at f are unpacked from T + i Q at f and -f, and H_{-f} = conj H_f: the
// blocks of half of the modes are stored, in the order in which k_circ_cols reads them.
//
// The transforms are mixed-radix Stockham passes in place: every thread takes one
// butterfly of up to 12 points into registers, so most sides up to a thousand take three
// passes (900 = 9 10 10, 1200 = 12 10 10), the first reading global memory and the last
// writing it.  Against one kernel per step (seven, with double-buffered passes of radix 2
// to 5, five for 900 and 1200) the planes cross L2
// four times instead of ten.  One apply after another on one stream, FP32: 1200 x 900 155 ->
// 69 us (rows 19, columns 26, rows 22; 117 MB of maps and blocks: 17 us of HBM), 600 x 450
// 77 -> 34, 256 x 256 51 -> 25, 64 x 64 35 -> 23 (FP64 58 -> 42); three maps at 1200 x 900 on
// three streams 130 -> 50 us an apply.  What bounds it now is latency at 24 warps per SM,
// and in the last kernel the FP64 pipe (z and its product with r).
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "circ.cuh"
#include "fft_reg.cuh"
#include "map_kernels.cuh"

namespace cmm {

namespace {

// ------------------------------------------------------------------ roots of unity
// cos and sin by their Taylor series, |x| <= pi / 4 (14 terms: below 1e-17)
constexpr double series_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k <= 14; ++k) {
    t *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    s += t;
  }
  return s;
}
constexpr double series_sin(double x) {
  double t = x, s = x;
  for (int k = 1; k <= 14; ++k) {
    t *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    s += t;
  }
  return s;
}
// cos(2 pi j / n), the angle brought to at most pi / 4 in whole numbers
constexpr double root_cos(int j, int n) {
  j = ((j % n) + n) % n;
  if (2 * j > n) j = n - j;
  double sg = 1.0;
  if (4 * j > n) {   // cos x = -cos(pi - x)
    sg = -1.0;
    j = n - 2 * j;
    n *= 2;
  }
  if (8 * j > n) return sg * series_sin(6.28318530717958647693 * (n - 4 * j) / (4.0 * n));
  return sg * series_cos(6.28318530717958647693 * j / n);
}
constexpr double root_sin(int j, int n) { return root_cos(4 * j - n, 4 * n); }

template <int I, int N, typename F>
__device__ __forceinline__ void static_for(const F& f) {
  if constexpr (I < N) {
    f(std::integral_constant<int, I>{});
    static_for<I + 1, N>(f);
  }
}

// ------------------------------------------------------------------ short transforms
template <typename T>
__device__ __forceinline__ Cx2<T> cx_axpy(T c, const Cx2<T>& a, const Cx2<T>& b) {   // c a + b
  const V2<T> cc{c, c};
  return Cx2<T>{pfma(cc, a.re, b.re), pfma(cc, a.im, b.im)};
}
template <typename T>
__device__ __forceinline__ Cx2<T> cx_scale(T c, const Cx2<T>& a) {
  const V2<T> cc{c, c};
  return Cx2<T>{pmul(cc, a.re), pmul(cc, a.im)};
}
// a (c + i s).  In FP32 with what the rounded constants lack, added before the products
// are rounded: every butterfly uses the same constants, so their errors do not average out
// over a line as those of the stage twiddles do.
template <typename T>
__device__ __forceinline__ Cx2<T> cx_mul_const(const Cx2<T>& a, double c, double s) {
  if constexpr (sizeof(T) == 8) {
    return cx_mul<T>(a, c, s);
  } else {
    const T ch = (T)c, sh = (T)s, cl = (T)(c - (double)ch), sl = (T)(s - (double)sh);
    const V2<T> cc{ch, ch}, ss{sh, sh}, ns{-sh, -sh}, dc{cl, cl}, ds{sl, sl}, dn{-sl, -sl};
    return Cx2<T>{pfma(a.im, ns, pfma(a.re, cc, pfma(a.im, dn, pmul(a.re, dc)))),
                  pfma(a.re, ss, pfma(a.im, cc, pfma(a.re, ds, pmul(a.im, dc))))};
  }
}
// x_q <- sum_j x_j exp(SIGN 2 pi i j q / N): direct forms for 2 to 5, N = A B else
// (A-point transforms, the constants w_N^(b c), B-point transforms)
template <typename T, int N, int SIGN>
__device__ __forceinline__ void cx_dft_n(Cx2<T>* x) {
  if constexpr (N == 2) {
    const Cx2<T> a = x[0];
    x[0] = cx_add(a, x[1]);
    x[1] = cx_sub(a, x[1]);
  } else if constexpr (N == 3) {
    const Cx2<T> t = cx_add(x[1], x[2]), u = cx_scale<T>((T)root_sin(1, 3), cx_sub(x[1], x[2]));
    const Cx2<T> m = cx_axpy<T>((T)-0.5, t, x[0]);
    x[0] = cx_add(x[0], t);
    cx_addsub_i<T, SIGN>(m, u, x[1], x[2]);
  } else if constexpr (N == 4) {
    cx_dft4<T, SIGN>(x[0], x[1], x[2], x[3]);
  } else if constexpr (N == 5) {
    constexpr double c1 = root_cos(1, 5), c2 = root_cos(2, 5), s1 = root_sin(1, 5), s2 = root_sin(2, 5);
    const Cx2<T> a1 = cx_add(x[1], x[4]), a2 = cx_add(x[2], x[3]), b1 = cx_sub(x[1], x[4]), b2 = cx_sub(x[2], x[3]);
    const Cx2<T> m1 = cx_axpy<T>((T)c1, a1, cx_axpy<T>((T)c2, a2, x[0]));
    const Cx2<T> m2 = cx_axpy<T>((T)c2, a1, cx_axpy<T>((T)c1, a2, x[0]));
    const Cx2<T> u1 = cx_axpy<T>((T)s1, b1, cx_scale<T>((T)s2, b2));
    const Cx2<T> u2 = cx_axpy<T>((T)s2, b1, cx_scale<T>((T)-s1, b2));
    x[0] = cx_add(x[0], cx_add(a1, a2));
    cx_addsub_i<T, SIGN>(m1, u1, x[1], x[4]);
    cx_addsub_i<T, SIGN>(m2, u2, x[2], x[3]);
  } else {
    constexpr int A = N == 16 ? 4 : N == 12 ? 4 : N == 8 ? 4 : N % 5 == 0 ? 5 : 3;
    constexpr int B = N / A;
    static_assert(A * B == N, "radix");
    Cx2<T> y[B][A];
    static_for<0, B>([&](auto bi) {
      constexpr int b = decltype(bi)::value;
      static_for<0, A>([&](auto ai) { y[b][decltype(ai)::value] = x[B * decltype(ai)::value + b]; });
      cx_dft_n<T, A, SIGN>(y[b]);
      static_for<0, A>([&](auto ci) {
        constexpr int c = decltype(ci)::value;
        constexpr double wr = root_cos(b * c, N), wi = SIGN * root_sin(b * c, N);
        if constexpr (b * c == 0) {
        } else if constexpr (4 * b * c == N) {   // SIGN i
          const Cx2<T> v = y[b][c];
          y[b][c] = SIGN > 0 ? Cx2<T>{V2<T>{-v.im.x, -v.im.y}, v.re} : Cx2<T>{v.im, V2<T>{-v.re.x, -v.re.y}};
        } else {
          y[b][c] = cx_mul_const<T>(y[b][c], wr, wi);
        }
      });
    });
    static_for<0, A>([&](auto ci) {
      constexpr int c = decltype(ci)::value;
      Cx2<T> z[B];
      static_for<0, B>([&](auto bi) { z[decltype(bi)::value] = y[decltype(bi)::value][c]; });
      cx_dft_n<T, B, SIGN>(z);
      static_for<0, B>([&](auto di) { x[c + A * decltype(di)::value] = z[decltype(di)::value]; });
    });
  }
}

// Launch shapes.  FP32: at most 12 points a thread (48 registers of data), two columns
// beside each other to make whole 32-byte sectors, and registers for three row blocks and
// two column blocks per SM (two and one: 1.35 times the time of an apply at 1200 x 900, four
// row blocks 1.03 times, both with twiddles formed in registers).  FP64: at most 6 points,
// since its pipe takes as long for a warp with few lanes as for a full one, so small maps
// want many threads a line (64 x 64: 45 us an apply in radix 4, 76 in radix 8).
template <typename T> struct CircKernel {
  static constexpr int kMaxRad = sizeof(T) == 4 ? 12 : 6;
  static constexpr int kRowThreads = sizeof(T) == 4 ? 256 : 512, kRowBlocks = sizeof(T) == 4 ? 3 : 1;
  static constexpr int kColThreads = sizeof(T) == 4 ? 448 : 512, kColBlocks = sizeof(T) == 4 ? 2 : 1;
  static constexpr int kCols = sizeof(T) == 4 ? 2 : 1;
};

// Inputs i + m nbf of one butterfly, from load(pos) or from buf (positions through
// at(pos)), its stage twiddles (for a pass after the first) and its transform.
template <typename T, int SIGN, int R, typename At, typename Load>
__device__ __forceinline__ void butterfly_in(Cx2<T> (&x)[CircKernel<T>::kMaxRad], int i, int nbf, bool rd, bool twiddle,
                                             const V2<T>* tw, int step, const Cx2<T>* buf, const At& at,
                                             const Load& load) {
  if (rd) {
#pragma unroll
    for (int m = 0; m < R; ++m) x[m] = buf[at(i + m * nbf)];
  } else {
#pragma unroll
    for (int m = 0; m < R; ++m) x[m] = load(i + m * nbf);
  }
  if (twiddle) {
    // w^m from the table: powers formed in registers lose digits (an apply at 1200 x 900 is 6 %
    // faster with them, but 3e-7 from the line FFTs instead of 1.5e-7)
#pragma unroll
    for (int m = 1; m < R; ++m) {
      const V2<T> w = __ldg(tw + m * step);
      x[m] = cx_mul<T>(x[m], w.x, SIGN > 0 ? -w.y : w.y);
    }
  }
  cx_dft_n<T, R, SIGN>(x);
}

template <typename T, int R, typename At, typename Store>
__device__ __forceinline__ void butterfly_out(const Cx2<T> (&x)[CircKernel<T>::kMaxRad], int i, int k, int p, bool wr, Cx2<T>* buf,
                                              const At& at, const Store& store) {
  if (wr) {
    const int base = (i - k) * R + k;
#pragma unroll
    for (int q = 0; q < R; ++q) buf[at(base + q * p)] = x[q];
  } else {
#pragma unroll
    for (int q = 0; q < R; ++q) store(i + q * p, x[q]);
  }
}

// The code of one radix f(std::integral_constant<int, R>): exact loops for every radix
// (loops over kMaxRad points under predicates took 1.4 times as long).
template <typename T, typename F>
__device__ __forceinline__ void for_radix(int R, const F& f) {
  switch (R) {
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    default:
      if constexpr (CircKernel<T>::kMaxRad == 12) {
        if (R == 6) f(std::integral_constant<int, 6>{});
        else if (R == 8) f(std::integral_constant<int, 8>{});
        else if (R == 9) f(std::integral_constant<int, 9>{});
        else if (R == 10) f(std::integral_constant<int, 10>{});
        else f(std::integral_constant<int, 12>{});
      } else {
        f(std::integral_constant<int, 6>{});
      }
  }
}

// The passes of one line, in place in buf.  Inputs come from load() and outputs go to
// store() unless IN_BUF / OUT_BUF: then they are in buf (OUT_BUF: visible to the block on
// return).  Thread i of the line takes butterfly i of every pass that has that many.
// Every thread of the block calls this (barriers); `on`: the thread's line exists.  The
// points of every radix share one array: one per case would be live across the barrier.
template <typename T, int SIGN, bool IN_BUF, bool OUT_BUF, typename At, typename Load, typename Store>
__device__ __forceinline__ void line_fft(const CircLine& ln, const V2<T>* __restrict__ tw, int i, bool on,
                                         Cx2<T>* buf, const At& at, const Load& load, const Store& store) {
  int p = 1;
  for (int st = 0; st < ln.nrad; ++st) {
    const int R = ln.rad[st], nbf = ln.nbf[st];
    const bool act = on && i < nbf;
    const bool rd = IN_BUF || st > 0, wr = OUT_BUF || st < ln.nrad - 1;
    const int k = i - fast_div(i, ln.mp[st]) * p;
    Cx2<T> x[CircKernel<T>::kMaxRad];
    if (act)
      for_radix<T>(R, [&](auto r) {
        butterfly_in<T, SIGN, decltype(r)::value>(x, i, nbf, rd, st > 0, tw, k * ln.step[st], buf, at, load);
      });
    if (rd && wr) __syncthreads();   // every input of this pass has been read
    if (act)
      for_radix<T>(R, [&](auto r) { butterfly_out<T, decltype(r)::value>(x, i, k, p, wr, buf, at, store); });
    if (wr) __syncthreads();
    p *= R;
  }
}

// line position -> buffer index of a row: one element of padding every 16 keeps the
// strided stores of the first pass off one bank group
__host__ __device__ constexpr int row_len(int L) { return L + (L >> 4) + 1; }

// ------------------------------------------------------------------ kernels
// Rows rows * blockIdx.x .. + rows - 1, ln.width threads a row.
template <typename T>
__global__ void __launch_bounds__(CircKernel<T>::kRowThreads, CircKernel<T>::kRowBlocks)
    k_circ_rows_fwd(const double* __restrict__ r, const T* __restrict__ blk, Cx2<T>* __restrict__ planes, const CircLine ln,
                    int ny, int rows, const V2<T>* __restrict__ tw, const int* done) {
  if (done && *done) return;
  extern __shared__ __align__(32) unsigned char smem[];
  const int s = threadIdx.x / ln.width, i = threadIdx.x - s * ln.width;
  const int y = blockIdx.x * rows + s;
  const long long npix = (long long)ny * ln.L, p0 = (long long)y * ln.L;
  const double* rr = r + p0;
  const T* br = blk + 6 * p0;
  Cx2<T>* pr = planes + p0;
  Cx2<T>* buf = reinterpret_cast<Cx2<T>*>(smem) + s * row_len(ln.L);
  line_fft<T, -1, false, false>(
      ln, tw, i, s < rows && y < ny, buf, [](int pos) { return pos + (pos >> 4); },
      [&](int pos) {
        const V2<T>* b = reinterpret_cast<const V2<T>*>(br) + 3 * pos;
        const V2<T> b0 = b[0], b1 = b[1], b2 = b[2];
        const T x0 = (T)rr[pos], x1 = (T)rr[npix + pos], x2 = (T)rr[2 * npix + pos];
        return Cx2<T>{V2<T>{b0.x * x0 + b0.y * x1 + b1.x * x2, b1.x * x0 + b2.x * x1 + b2.y * x2},
                      V2<T>{b0.y * x0 + b1.y * x1 + b2.x * x2, (T)0}};
      },
      [&](int pos, const Cx2<T>& v) { pr[pos] = v; });
}

// Columns kx = J blockIdx.x .. + J - 1 (kx <= nx / 2) and their mirrors nx - kx; NS = 2 J
// lines, interleaved in the buffer, and NS ln.width threads.
template <typename T, int J>
__global__ void __launch_bounds__(CircKernel<T>::kColThreads, CircKernel<T>::kColBlocks)
    k_circ_cols(Cx2<T>* __restrict__ planes, const T* __restrict__ hinv, const CircLine ln, int nx,
                const V2<T>* __restrict__ tw, const int* done) {
  if (done && *done) return;
  constexpr int NS = 2 * J;
  extern __shared__ __align__(32) unsigned char smem[];
  Cx2<T>* buf = reinterpret_cast<Cx2<T>*>(smem);
  const int ny = ln.L;
  const int s = threadIdx.x % NS, i = threadIdx.x / NS;
  const int kx = blockIdx.x * J + s % J;
  const bool mirror = s >= J;
  const bool self = kx == 0 || 2 * kx == nx;   // its own mirror: the second copy is not written
  Cx2<T>* g = planes + (mirror && kx ? nx - kx : kx);
  const auto at = [&](int pos) { return pos * NS + s; };
  line_fft<T, -1, false, true>(
      ln, tw, i, kx <= nx / 2, buf, at,
      [&](int pos) { return g[(long long)pos * nx]; }, [](int, const Cx2<T>&) {});
  // Y = H^-1 X at f = (ky, kx) and -f; X_T, X_Q from T + i Q at both, X_U their mean
  const T* H = hinv + (size_t)blockIdx.x * J * ny * 9;
  const T h = (T)0.5;
  for (int t = threadIdx.x; t < J * ny; t += blockDim.x) {
    const int c = t % J, ky = t / J;
    if ((int)blockIdx.x * J + c > nx / 2) continue;
    Cx2<T>& F = buf[ky * NS + c];
    Cx2<T>& G = buf[(ky ? ny - ky : 0) * NS + J + c];
    const T xr[3] = {h * (F.re.x + G.re.x), h * (F.im.x + G.im.x), h * (F.re.y + G.re.y)};
    const T xi[3] = {h * (F.im.x - G.im.x), h * (G.re.x - F.re.x), h * (F.im.y - G.im.y)};
    T o[9];
#pragma unroll
    for (int j = 0; j < 9; ++j) o[j] = H[9 * (size_t)t + j];
    T yr[3], yi[3];
    mode_mul3<T>(o, xr, xi, yr, yi);
    F = Cx2<T>{V2<T>{yr[0] - yi[1], yr[2]}, V2<T>{yi[0] + yr[1], yi[2]}};
    G = Cx2<T>{V2<T>{yr[0] + yi[1], yr[2]}, V2<T>{yr[1] - yi[0], -yi[2]}};
  }
  __syncthreads();
  line_fft<T, 1, true, false>(
      ln, tw, i, kx <= nx / 2, buf, at, [](int) { return Cx2<T>{}; },
      [&](int pos, const Cx2<T>& v) {
        if (!(mirror && self)) g[(long long)pos * nx] = v;
      });
}

// Row groups blockIdx.x, + gridDim.x, ...: z = Sigma^-1 of the scaled real parts, and the
// block's partial sum of r^T z (fixed order; block 0 clears the partials of no block).
template <typename T>
__global__ void __launch_bounds__(CircKernel<T>::kRowThreads, CircKernel<T>::kRowBlocks)
    k_circ_rows_inv(const Cx2<T>* __restrict__ planes, const T* __restrict__ blk, double* __restrict__ z, const CircLine ln,
                    int ny, int rows, const V2<T>* __restrict__ tw, const double* __restrict__ r,
                    double* __restrict__ partial, const int* done) {
  if (done && *done) return;
  extern __shared__ __align__(32) unsigned char smem[];
  const int s = threadIdx.x / ln.width, i = threadIdx.x - s * ln.width;
  const long long npix = (long long)ny * ln.L;
  const T sc = (T)(1.0 / (double)npix);
  Cx2<T>* buf = reinterpret_cast<Cx2<T>*>(smem) + s * row_len(ln.L);
  const int groups = (ny + rows - 1) / rows;
  double acc = 0.0;
  for (int gi = blockIdx.x; gi < groups; gi += gridDim.x) {
    const int y = gi * rows + s;
    const long long p0 = (long long)y * ln.L;
    const double* rr = r + p0;
    double* zr = z + p0;
    const T* br = blk + 6 * p0;
    const Cx2<T>* pr = planes + p0;
    line_fft<T, 1, false, false>(
        ln, tw, i, s < rows && y < ny, buf, [](int pos) { return pos + (pos >> 4); },
        [&](int pos) { return pr[pos]; },
        [&](int pos, const Cx2<T>& v) {
          const V2<T>* b = reinterpret_cast<const V2<T>*>(br) + 3 * pos;
          const V2<T> b0 = b[0], b1 = b[1], b2 = b[2];
          const T x0 = v.re.x * sc, x1 = v.im.x * sc, x2 = v.re.y * sc;
          const double y0 = widen(b0.x * x0 + b0.y * x1 + b1.x * x2);
          const double y1 = widen(b0.y * x0 + b1.y * x1 + b2.x * x2);
          const double y2 = widen(b1.x * x0 + b2.x * x1 + b2.y * x2);
          zr[pos] = y0;
          zr[npix + pos] = y1;
          zr[2 * npix + pos] = y2;
          if (partial) acc += rr[pos] * y0 + rr[npix + pos] * y1 + rr[2 * npix + pos] * y2;
        });
    __syncthreads();   // the next group rewrites the buffer
  }
  if (!partial) return;
  __shared__ double sum[32];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sum[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double v = 0.0;
    for (int w = 0; w < (int)blockDim.x / 32; ++w) v += sum[w];
    partial[blockIdx.x] = v;
  }
  if (blockIdx.x == 0)
    for (int b = gridDim.x + threadIdx.x; b < kRedBlocks; b += blockDim.x) partial[b] = 0.0;
}

// ------------------------------------------------------------------ plans
// Fewest passes, then the largest smallest radix (the fewest threads a line); odd radices
// first, whose strided first stores meet no bank twice.
bool best_radices(int L, int left, const int* allowed, int nallowed, int* rad, int n, int* best, int* best_min) {
  if (left == 0) {
    if (L != 1) return false;
    int mn = 99;
    for (int j = 0; j < n; ++j) mn = std::min(mn, rad[j]);
    if (mn > *best_min) {
      *best_min = mn;
      std::copy(rad, rad + n, best);
    }
    return true;
  }
  bool any = false;
  for (int a = 0; a < nallowed; ++a)
    if (L % allowed[a] == 0 && (n == 0 || allowed[a] <= rad[n - 1])) {
      rad[n] = allowed[a];
      any |= best_radices(L / allowed[a], left - 1, allowed, nallowed, rad, n + 1, best, best_min);
    }
  return any;
}

template <typename T>
bool plan_line(int L, CircLine& ln) {
  static const int radices[] = {12, 10, 9, 8, 6, 5, 4, 3, 2};
  constexpr int skip = CircKernel<T>::kMaxRad == 12 ? 0 : 4;
  ln.L = L;
  int rad[kCircPasses], best[kCircPasses], mn = 0;
  for (int n = 1; n <= kCircPasses; ++n)
    if (best_radices(L, n, radices + skip, 9 - skip, rad, 0, best, &mn)) {
      std::stable_sort(best, best + n, [](int a, int b) { return (a & 1) > (b & 1); });
      int p = 1;
      ln.nrad = n;
      for (int st = 0; st < n; ++st) {
        ln.rad[st] = best[st];
        ln.nbf[st] = L / best[st];
        ln.step[st] = L / (p * best[st]);
        ln.mp[st] = fast_div_magic((unsigned)p);
        p *= best[st];
      }
      ln.width = L / mn;
      return true;
    }
  return false;
}

template <typename T> size_t smem_rows(const CircPlan& p) { return sizeof(Cx2<T>) * p.rows * row_len(p.x.L); }
template <typename T> size_t smem_cols(const CircPlan& p) { return sizeof(Cx2<T>) * 2 * p.J * p.y.L; }
int round32(int v) { return (v + 31) / 32 * 32; }

}  // namespace

template <typename T>
CircPlan circ_plan(int ny, int nx) {
  CircPlan p;
  p.ny = ny;
  p.nx = nx;
  p.J = CircKernel<T>::kCols;
  if (ny >= 65536 || nx >= 65536 || !plan_line<T>(nx, p.x) || !plan_line<T>(ny, p.y)) return p;
  // whole warps, and more than one row a block only while two blocks per SM are left
  const int fill = std::max((32 + p.x.width - 1) / p.x.width, (ny + 2 * kSMs - 1) / (2 * kSMs));
  p.rows = std::max(1, std::min(fill, 256 / p.x.width));
  // one column a block where two (375 = 5 5 5 3: 125 threads a line) do not fit
  const auto cols_fit = [&] {
    return 2 * p.J * p.y.width <= CircKernel<T>::kColThreads && smem_cols<T>(p) <= 200 * 1024;
  };
  if (!cols_fit()) p.J = 1;
  p.ok = p.x.width <= CircKernel<T>::kRowThreads && smem_rows<T>(p) <= 200 * 1024 && cols_fit();
  return p;
}
template CircPlan circ_plan<float>(int, int);
template CircPlan circ_plan<double>(int, int);

template <typename T>
int circ_prepare(const CircPlan& p) {
  constexpr int J = CircKernel<T>::kCols;
  CMM_CUDA(cudaFuncSetAttribute(p.J == 1 ? k_circ_cols<T, 1> : k_circ_cols<T, J>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  CMM_CUDA(cudaFuncSetAttribute(k_circ_rows_fwd<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  CMM_CUDA(cudaFuncSetAttribute(k_circ_rows_inv<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
  return CMM_OK;
}
template int circ_prepare<float>(const CircPlan&);
template int circ_prepare<double>(const CircPlan&);

template <typename T>
int launch_circ_apply(const CircPlan& p, const V2<T>* tw, const T* blk, const T* hinv, const double* r, double* z,
                      void* planes_, double* partial, const int* done, cudaStream_t s) {
  constexpr int J = CircKernel<T>::kCols;
  Cx2<T>* planes = static_cast<Cx2<T>*>(planes_);
  const int groups = (p.ny + p.rows - 1) / p.rows, nt = round32(p.rows * p.x.width);
  k_circ_rows_fwd<T><<<groups, nt, smem_rows<T>(p), s>>>(r, blk, planes, p.x, p.ny, p.rows, tw, done);
  CMM_LAUNCH_CHECK();
  const auto cols = p.J == 1 ? k_circ_cols<T, 1> : k_circ_cols<T, J>;
  cols<<<(p.nx / 2 + p.J) / p.J, round32(2 * p.J * p.y.width), smem_cols<T>(p), s>>>(planes, hinv, p.y, p.nx, tw + p.nx,
                                                                                     done);
  CMM_LAUNCH_CHECK();
  k_circ_rows_inv<T><<<std::min(groups, kRedBlocks), nt, smem_rows<T>(p), s>>>(planes, blk, z, p.x, p.ny, p.rows, tw, r,
                                                                               partial, done);
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}
template int launch_circ_apply<float>(const CircPlan&, const float2*, const float*, const float*, const double*, double*,
                                      void*, double*, const int*, cudaStream_t);
template int launch_circ_apply<double>(const CircPlan&, const double2*, const double*, const double*, const double*,
                                       double*, void*, double*, const int*, cudaStream_t);

}  // namespace cmm
