// Two-detector path of the FP32 and BF16 operators: sizes, tables and launches of the
// kernels of tod_pair.cuh.
#include "map_kernels.cuh"
#include "tod_pair.cuh"

namespace cmm {

// Split of the pair sequence, n_t = 2^log_nt points: R = 64 below 2^16, 128 for 2^16
// and 2^17, 256 from 2^18 (rows C = n_t / R of 128 to 4096 points).
bool pair_path_sizes(int log_nt, int* logR, int* logC) {
  if (log_nt < 13 || log_nt > 20) return false;
  *logR = log_nt < 16 ? 6 : (log_nt < 18 ? 7 : 8);
  *logC = log_nt - *logR;
  return true;
}

// Whether the path can serve the operator's applications (the hit limit is that of the
// FP32 partial maps; correlated noise is for FP32 and BF16), and whether it does.
bool pair_path_fits(const cmm_op* op) {
  return op->pR > 0 && op->tw_pair &&
         (op->prec == CMM_PREC_F64 ? op->nz->corr_r == 0 : op->pt->max_hits <= kF32HitLimit);
}

int pair_corr_slots_of(const cmm_op* op) { return pair_corr_slots(op->pR, op->pC); }

bool pair_path_ok(const cmm_op* op) { return op->pair && pair_path_fits(op); }

int launch_flush_to_map(const TodArgs& a, int nc, int maps, bool add_acc, const uint8_t* mask, const ApplyOut& out,
                        cudaStream_t st);
int launch_flush_maps(const TodArgs& a, int nc, int maps, cudaStream_t st);

// ------------------------------------------------------------------ factors of stored data
// One block after the first forward pass: from every detector's sum of squares (cleared for
// the next call) its factors f and h = u / (n_t f), and the list of pairs to transform again.
// unit: u / n_t.
//
// level = mean square of f s.  A pair whose rms differ by less than kTodBalance keeps the
// guesses: its quieter detector then carries at most about kTodBalance times its own
// rounding (FP32 2.5e-7, alone 3e-7).  Else both take the power of two nearest 1 / rms.
// Without weight: f = h = 0, and for an all-zero detector h = 0, as their filtered data are
// exactly zero.  Not finite: NaN for that detector alone, f = 0 keeps it out of its
// partner's sequence.  With correlated noise a detector's filtered data also hold the common
// modes, whose size is that of all detectors' data: no level is then taken below their
// weighted mean square.
constexpr double kTodBalance = 4.0;
constexpr int kGainThreads = 1024;

__global__ void __launch_bounds__(kGainThreads) k_tod_gains(double* norm, const float* __restrict__ guess,
                                                            const float* __restrict__ unit, float* __restrict__ f,
                                                            float* __restrict__ h, int* __restrict__ list, int d0, int nd,
                                                            double per, bool corr, const int* done) {
  if (done && *done) return;
  __shared__ int count;
  __shared__ double common;
  if (threadIdx.x == 0) count = 0;
  if (corr) {
    double su = 0.0, sr = 0.0;
    for (int d = d0 + threadIdx.x; d < d0 + nd; d += kGainThreads) {
      const double f0 = (double)guess[d], ms = norm[d] * per;
      if (f0 > 0.0 && isfinite(ms)) {
        su += (double)unit[d];
        sr += (double)unit[d] * (ms / (f0 * f0));
      }
    }
    su = block_sum_warps(su);
    __syncthreads();
    sr = block_sum_warps(sr);
    if (threadIdx.x == 0) common = su > 0.0 ? sr / su : 0.0;
  }
  __syncthreads();
  for (int q = threadIdx.x; 2 * q < nd; q += kGainThreads) {
    double level[2] = {0.0, 0.0};
    bool again = false;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int d = d0 + 2 * q + j;
      if (2 * q + j >= nd) break;
      const double ms = norm[d] * per;
      const float f0 = guess[d];
      norm[d] = 0.0;
      f[d] = f0;
      if (f0 == 0.0f) {
        h[d] = 0.0f;
      } else if (!isfinite(ms)) {
        f[d] = 0.0f;
        h[d] = NAN;
        again = true;
      } else {
        level[j] = corr ? fmax(ms, common * ((double)f0 * f0)) : ms;
        h[d] = level[j] > 0.0 ? unit[d] / f0 : 0.0f;
      }
    }
    if (level[0] > 0.0 && level[1] > 0.0 &&
        fmax(level[0], level[1]) > kTodBalance * kTodBalance * fmin(level[0], level[1])) {
      again = true;
      for (int j = 0; j < 2; ++j) {
        const int d = d0 + 2 * q + j;
        // the guess over sqrt(level), within 2^+-100, and h within FP32
        const int eu = ilogbf(unit[d]);
        const int ef = (int)fmin(100.0, fmax(-100.0, ilogbf(guess[d]) - rint(0.5 * log2(level[j]))));
        f[d] = scalbnf(1.0f, min(max(ef, eu - 126), eu + 126));
        h[d] = unit[d] / f[d];
      }
    }
    if (again) list[1 + atomicAdd(&count, 1)] = q;
  }
  __syncthreads();
  if (threadIdx.x == 0) list[0] = count;
}

int launch_tod_gains(const cmm_op* op, const TodArgs& a, int nd, cudaStream_t st) {
  k_tod_gains<<<1, kGainThreads, 0, st>>>(op->tod_norm, op->nz->tod_guess, op->nz->unit + op->pt->n_det, op->tod_f,
                                          op->tod_h, op->tod_list, a.d0, nd, 1.0 / (double)op->pt->n_t, a.corr_r > 0,
                                          a.done);
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}

template <typename S>
static int run_corr(const TodArgs& a, int nd, cudaStream_t st) {
  const int g = (pair_corr_slots(a.R, a.C) + kCorrThreads - 1) / kCorrThreads;
  switch (a.corr_r) {
    case 1: k_pair_corr<S, 1><<<g, kCorrThreads, 0, st>>>(a, nd); break;
    case 2: k_pair_corr<S, 2><<<g, kCorrThreads, 0, st>>>(a, nd); break;
    case 3: k_pair_corr<S, 3><<<g, kCorrThreads, 0, st>>>(a, nd); break;
    default: k_pair_corr<S, 4><<<g, kCorrThreads, 0, st>>>(a, nd); break;
  }
  CMM_LAUNCH_CHECK();
  return CMM_OK;
}
static_assert(kMaxCorrModes == 4, "k_pair_corr instances");

template <typename S>
static int apply_pair_s(cmm_op* op, int d0, int nd, const void* tod, int tod_is_f64, const ApplyOut& out, int pass) {
  TodArgs a = pair_args(op, d0);
  if (tod) stored_gains(op, a);
  cudaStream_t st = op->ctx->stream;
  const int nc = op->pt->ncomp;
  if (pass < 0 || pass == 0) {
    TraceRange tr("A: P m + column FFTs (two detectors per sequence)");
    if (tod) CMM_TRY((pair_fwd_stored<float, S>(op, a, nd, tod, tod_is_f64 != 0, st)));
    else if (nc == 1) CMM_TRY((dispatch_pair_T<float, 1, S>(a, nd, 0, st, false)));
    else CMM_TRY((dispatch_pair_T<float, 3, S>(a, nd, 0, st, false)));
  }
  if (pass < 0 || pass == 1) {
    TraceRange tr("A: row FFTs + N^-1");
    if (a.corr_r > 0) {
      // correlated noise: forward rows, the cross-detector solve over the whole chunk, back
      CMM_TRY((dispatch_pair_F<float, S, kPairSplit>(a, nd, st, false)));
      CMM_TRY(run_corr<S>(a, nd, st));
      CMM_TRY((dispatch_pair_F<float, S, kPairMerge>(a, nd, st, false)));
    } else {
      CMM_TRY((dispatch_pair_F<float, S>(a, nd, st, false)));
    }
  }
  if (pass < 0 || pass == 2) {
    TraceRange tr("A: inverse column FFTs + P^T");
    // one launch bins up to acc32_maps groups of kFlushDets detectors, each group into its
    // own FP32 partial map; one flush then adds them all in FP64 into the accumulator, the
    // application's last one into the result
    const bool acc = apply_uses_acc(op);
    const int per_launch = op->acc32_maps * kFlushDets;   // even: whole pairs per group
    for (int g0 = 0; g0 < nd; g0 += per_launch) {
      TodArgs b = a;
      const int gn = std::min(per_launch, nd - g0);
      b.d0 = a.d0 + g0;
      b.spec = reinterpret_cast<S*>(a.spec) + (long long)(g0 / 2) * a.N;
      b.flush_dets = kFlushDets;
      b.acc32_map = (long long)op->acc_stride * (a.npix + 1);
      if (nc == 1) CMM_TRY((dispatch_pair_T<float, 1, S>(b, gn, 2, st, false)));
      else CMM_TRY((dispatch_pair_T<float, 3, S>(b, gn, 2, st, false)));
      const int maps = (gn + kFlushDets - 1) / kFlushDets;
      if (d0 + g0 + gn == op->pt->n_det) CMM_TRY(launch_flush_to_map(b, nc, maps, acc, op->pt->mask, out, st));
      else CMM_TRY(launch_flush_maps(b, nc, maps, st));
    }
  }
  return CMM_OK;
}

// tod: stored data [n_det][n_t] in place of P m, or nullptr.
int launch_apply_chunk_pair(cmm_op* op, int d0, int nd, const void* tod, int tod_is_f64, const ApplyOut& out, int pass) {
  if (op->prec == CMM_PREC_F64) return launch_apply_chunk_pair64(op, d0, nd, tod, tod_is_f64, pass);
  if (op->prec == CMM_PREC_BF16) return apply_pair_s<__nv_bfloat162>(op, d0, nd, tod, tod_is_f64, out, pass);
  return apply_pair_s<float2>(op, d0, nd, tod, tod_is_f64, out, pass);
}

// The split, which n_samp fixes, its tables and the kernels' shared-memory attributes.
int prepare_pair(cmm_op* op) {
  int lr = 0, lc = 0;
  if (!pair_path_sizes(ilog2_ll(op->pt->n_t), &lr, &lc)) return CMM_OK;
  op->plogR = lr;
  op->plogC = lc;
  op->pR = 1 << lr;
  op->pC = 1 << lc;
  if (!op->tod_norm) {
    const size_t n = (size_t)op->pt->n_det;
    if (cudaMalloc(&op->tod_norm, (sizeof(double) + 2 * sizeof(float)) * n + sizeof(int) * (1 + (n + 1) / 2)) !=
        cudaSuccess) {
      op->tod_norm = nullptr;
      cudaGetLastError();
      return fail(CMM_ERR_OOM, "factors of stored data");
    }
    op->tod_f = reinterpret_cast<float*>(op->tod_norm + n);
    op->tod_h = op->tod_f + n;
    op->tod_list = reinterpret_cast<int*>(op->tod_h + n);
    CMM_CUDA(cudaMemsetAsync(op->tod_norm, 0, sizeof(double) * n, op->ctx->stream));
  }
  if (op->prec == CMM_PREC_F64) return prepare_pair64(op);
  if (!op->tw_pair) CMM_TRY(pair_twiddles<float>(op));
  return op->prec == CMM_PREC_BF16 ? prepare_pair_s<float, __nv_bfloat162>(op) : prepare_pair_s<float, float2>(op);
}

}  // namespace cmm
