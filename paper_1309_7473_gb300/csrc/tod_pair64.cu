// Two-detector path of the FP64 operators (kernels of tod_pair.cuh).
//
// GB300 issues one FP64 warp instruction in 16 cycles per SM, so the FP64 application is
// bound by the count of FP64 instructions and by nothing else.  Against the generic
// kernels (one detector a sequence, tod.cu) the pair form needs no split twiddle, the
// rotation comes from a table instead of two divisions a sample and pass, a weight takes
// 18 FP64 instructions instead of a logarithm, a power and a division, runs of samples on
// a pixel are summed before they are reduced, and no thread idles in the row transforms.
// A at 32 detectors x 2^16 samples: 834 -> 401 us (forward 138 -> 98, filter 550 -> 200,
// inverse 133 -> 90), at 128 x 2^18 10.19 -> 5.57 ms, at 64 x 2^20 21.1 -> 12.2 ms.
#include "tod_pair.cuh"

namespace cmm {

__global__ void k_rot64(const int4* __restrict__ bore, long long n, double2* __restrict__ out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    double2 r;
    sample_response<double>(bore[t], double2{1.0, 0.0}, r.x, r.y);
    out[t] = r;
  }
}

// log2 of the frequency indices, then exp2_tab's powers 2^(j / 64)
__global__ void k_lg2(long long n, double* __restrict__ out) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n + kExp2Tab;
       k += (long long)gridDim.x * blockDim.x)
    out[k] = k < n ? log2((double)(k == 0 ? 1 : k)) : exp2((double)(k - n) / kExp2Tab);
}

int launch_apply_chunk_pair64(cmm_op* op, int d0, int nd, const void* tod, int tod_is_f64, int pass) {
  TodArgs a = pair_args(op, d0);
  if (tod) stored_gains(op, a);
  cudaStream_t st = op->ctx->stream;
  const bool t_only = op->pt->ncomp == 1;
  if (pass < 0 || pass == 0) {
    TraceRange tr("A: P m + column FFTs (two detectors per sequence, FP64)");
    if (tod) CMM_TRY((pair_fwd_stored<double, double2>(op, a, nd, tod, tod_is_f64 != 0, st)));
    else if (t_only) CMM_TRY((dispatch_pair_T<double, 1, double2>(a, nd, 0, st, false)));
    else CMM_TRY((dispatch_pair_T<double, 3, double2>(a, nd, 0, st, false)));
  }
  if (pass < 0 || pass == 1) {
    TraceRange tr("A: row FFTs + N^-1 (FP64)");
    CMM_TRY((dispatch_pair_F<double, double2>(a, nd, st, false)));
  }
  if (pass < 0 || pass == 2) {
    TraceRange tr("A: inverse column FFTs + P^T (FP64)");
    if (t_only) CMM_TRY((dispatch_pair_T<double, 1, double2>(a, nd, 2, st, false)));
    else CMM_TRY((dispatch_pair_T<double, 3, double2>(a, nd, 2, st, false)));
  }
  return CMM_OK;
}

// The FP64 tables: twiddles, (cos 2phi, sin 2phi) per sample and log2 per frequency
// index (20 bytes a sample of one detector, kept by the operator).
int prepare_pair64(cmm_op* op) {
  const long long n_t = op->pt->n_t;
  cudaStream_t st = op->ctx->stream;
  if (!op->tw_pair) CMM_TRY(pair_twiddles<double>(op));
  if (!op->rot64) {
    if (cudaMalloc(&op->rot64, sizeof(double2) * n_t) != cudaSuccess ||
        cudaMalloc(&op->lg2, sizeof(double) * (n_t / 2 + 1 + kExp2Tab)) != cudaSuccess) {
      cudaGetLastError();
      return fail(CMM_ERR_OOM, "FP64 rotation and frequency tables");
    }
    k_rot64<<<(int)std::min<long long>((n_t + 255) / 256, 4096), 256, 0, st>>>(op->pt->bore, n_t, op->rot64);
    CMM_LAUNCH_CHECK();
    k_lg2<<<(int)std::min<long long>((n_t / 2 + 256) / 256, 4096), 256, 0, st>>>(n_t / 2 + 1, op->lg2);
    CMM_LAUNCH_CHECK();
  }
  return prepare_pair_s<double, double2>(op);
}

}  // namespace cmm
