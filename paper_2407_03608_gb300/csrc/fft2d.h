// Shared by the row transforms of the pruned 2-D path (fft2d.cu, rows2d.cu).
#pragma once

#include "fft_core.h"
#include "kernels.h"

namespace gpn {

using fft::cpx;

// entries of one high-part twiddle table (W^{64 q}, q <= N2 / 64)
__host__ __device__ constexpr int tw_hi(int n2) { return n2 / 64 + 1; }
// a launch of the row kernels
template <typename T>
struct RowsArgs {
  const T* gin;            // spreading grids (forward input), (R*C) x nf x nf
  T* gout;                 // interp grids (inverse output)
  cpx<T>* X;               // forward row output / inverse row input: [cr][M+1][nf]
  const cpx<T>* tw;        // two-level tables: W_{N2} (hi, lo), then W_nf (hi, lo)
  long long nf;
  long long G;             // nf^2
  int M;
  int row0;                // first row of item 0 (a multiple of RB)
  int row_hi;
  long long npairs;        // RB-row groups per grid
  long long nitems;        // npairs * C * R
  int col_lo, col_hi;
};

// FP32 inverse row transforms of length nf = 2^(L+1) of `grids` grids (rows2d.cu); the row groups
// of `a` are the kernel's own
void rows_pairs_inv(int L, const RowsArgs<float>& a, int row_lo, int grids, cudaStream_t st);

}  // namespace gpn
