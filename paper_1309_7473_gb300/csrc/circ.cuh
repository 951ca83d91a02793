// Plan and launches of the fused circulant apply (circ.cu).
#pragma once

#include "common.cuh"
#include "fft.cuh"

namespace cmm {

constexpr int kCircPasses = 8;

// In-place passes of one line: radices, butterflies and table step per pass
struct CircLine {
  int L = 0, nrad = 0, width = 0;   // width: threads per line, the most butterflies of a pass
  int rad[kCircPasses], nbf[kCircPasses], step[kCircPasses];
  unsigned mp[kCircPasses];         // magic of the division by the product of the earlier radices
};

struct CircPlan {
  bool ok = false;
  int ny = 0, nx = 0;
  CircLine x, y;
  int rows = 1;   // rows per block of the row kernels
  int J = 1;      // columns (and mirrors) per block of the column kernel
  int64_t modes() const { return (int64_t)((nx / 2 + J) / J) * J * ny; }   // stored mode blocks
};

// ok = false where a block cannot hold the lines: a line takes L / (its smallest radix)
// threads, of which a row may have 256 (FP64 512) and a column and its mirror together 448
// (FP64 512), or more than 200 KB of shared memory.  In FP32 (radices to 12) every side of
// 2, 3 and 5 below 675 and most up to 1200 fit; columns of 675 = 9 5 5 3 and 1024 = 8 8 4 4
// do not.  In FP64 (radices to 6) one small radix costs more: columns of 640, 800, 810, 960,
// 972, 1000, 1125, 1152 and 1200 do not fit.  The line FFTs of map.cu serve those sides.
template <typename T> CircPlan circ_plan(int ny, int nx);
// Opts the kernels into the plan's shared memory (before any stream capture).
template <typename T> int circ_prepare(const CircPlan& p);
// z = M_C r of a TQU map and, with `partial`, the kRedBlocks partial sums of r^T z.
// blk: Sigma^-1 [npix][6]; hinv: the mode blocks in the plan's order; planes: npix Cx2;
// tw: w_nx^e, e < nx, then w_ny^e, e < ny.
template <typename T>
int launch_circ_apply(const CircPlan& p, const V2<T>* tw, const T* blk, const T* hinv, const double* r, double* z,
                      void* planes, double* partial, const int* done, cudaStream_t s);

}  // namespace cmm
