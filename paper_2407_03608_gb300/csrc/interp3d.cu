// Steps (4b) + (5) of Sec. 4.2 in three dimensions, on the box grids of fft3d.cu:
//   out_i = sum_zyx psi(z) psi(y) psi(x) sum_k w_k(x_i) g_k[z][y][x]  (+ shift * alpha_i).
//
// One warp a point, straight from the grid through L1: the channels are innermost, so one row
// (z, y) of the support is width * Cp adjacent values, which the lanes read in S coalesced
// loads.  A lane's position in that row fixes its cell x and channel k for the whole point, so
// psi(x) w_k is formed once per lane and slot, and a row costs S loads and S + 1 multiply-adds.
// Points come in bin order and a block takes consecutive ones, so the rows of neighbouring
// points are served by L1.  Sums: a row's slots, then the rows of a plane weighted by psi(y),
// then the planes weighted by psi(z); the 32 partial sums are added in float-float (FP32
// plans) or float64.
//
// Bound: latency of the L1/L2 loads and issue (about 9 instructions a row).  On 2e6 points, ms:
// the staged kernel of interp.cu 15.1 (8 channels, width 9, nf 512) and 26.7 (10, 9, nf 864); here
// with 48 warps an SM 4.35 and 6.00, with 64 4.17 and 5.35.  Loads of two channels with packed
// sums need 48 registers: 4.95; sorting the points finer than by bins changes nothing.
#include <algorithm>

#include "kernels.h"

namespace gpn {

namespace {

// the rows are short chains of loads, so what counts is warps in flight: up to three loads a row
// 64 an SM (32 registers, a few spilled outside the loop), above that what the registers allow
template <int S>
constexpr int kWarps = S <= 3 ? 16 : 8;
constexpr int kPointsPerBlock = 64;

template <typename T>
struct Interp3Args {
  const int* l0[3];
  const T* xi[3];
  const T* wk;
  long long n;
  const T* grid;
  GridView v;
  int width, C, Cp;
  T beta, inv_halfw;
  const double* alpha;   // sorted order (may be null)
  double shift;
  const double* dcorr;   // per-point addition to the shift (may be null)
  double* out;           // sorted order, n x R
};

__device__ __forceinline__ double warp_total(float v) {
  dd s{v, 0.0f};
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += shfl_xor_val(s, o);
  return (double)s;
}
__device__ __forceinline__ double warp_total(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// S: loads a row, ceil(width Cp / 32)
template <typename T, int S>
__global__ void __launch_bounds__(32 * kWarps<S>, S <= 3 ? 4 : 1) k_interp3d(Interp3Args<T> a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = a.width, r = blockIdx.y;
  const long long s0 = a.v.stride[0], s1 = a.v.stride[1];
  const T* grid = a.grid + r * a.v.rstride + lane;
  const double* alpha = a.alpha ? a.alpha + (size_t)r * a.n : nullptr;
  const int last = W * a.Cp - 32 * (S - 1);   // lanes of the last slot inside the row
  int xs[S], ks[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    xs[s] = (s * 32 + lane) / a.Cp;
    ks[s] = (s * 32 + lane) - xs[s] * a.Cp;
  }
  const long long p1 = min(a.n, (long long)(blockIdx.x + 1) * kPointsPerBlock);
  for (long long p = (long long)blockIdx.x * kPointsPerBlock + warp; p < p1; p += kWarps<S>) {
    const int lz = a.l0[0][p] - a.v.lo[0], ly = a.l0[1][p] - a.v.lo[1], lx = a.l0[2][p] - a.v.lo[2];
    T pz = T(0), py = T(0), px = T(0);
    if (lane < W) {
      pz = psi_at<T>(lane, a.xi[0][p], a.beta, a.inv_halfw);
      py = psi_at<T>(lane, a.xi[1][p], a.beta, a.inv_halfw);
      px = psi_at<T>(lane, a.xi[2][p], a.beta, a.inv_halfw);
    }
    T v[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const T q = shfl_val(px, xs[s] & 31);
      const bool in = (s + 1 < S || lane < last) && ks[s] < a.C;
      v[s] = in ? q * a.wk[p * a.C + ks[s]] : T(0);
    }
    const T* g = grid + lz * s0 + ly * s1 + lx * a.v.stride[2];
    T acc = T(0);
    for (int z = 0; z < W; ++z) {
      const T* gz = g + z * s0;
      T plane = T(0);
#pragma unroll 3
      for (int y = 0; y < W; ++y) {
        const T* gy = gz + y * s1;
        T row = T(0);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const T u = (s + 1 < S || lane < last) ? __ldg(gy + 32 * s) : T(0);
          row += v[s] * u;
        }
        plane += shfl_val(py, y) * row;
      }
      acc += shfl_val(pz, z) * plane;
    }
    double res = warp_total(acc);
    if (lane == 0) {
      if (alpha) res += (a.dcorr ? a.shift + a.dcorr[p] : a.shift) * alpha[p];
      a.out[(size_t)r * a.n + p] = res;
    }
  }
}

template <typename T, int S>
void dispatch(const Interp3Args<T>& a, dim3 grid, cudaStream_t st) {
  if (a.width * a.Cp <= 32 * S)
    k_interp3d<T, S><<<grid, 32 * kWarps<S>, 0, st>>>(a);
  else if constexpr (S < kMaxWidth * kMaxChannels / 32)
    dispatch<T, S + 1>(a, grid, st);
}

template <typename T>
void impl(Plan& plan, const PointSet& ps, const double* alpha_sorted, double shift, double* out_sorted, int R,
          cudaStream_t st) {
  const GridGeom& g = plan.geom;
  Interp3Args<T> a{};
  for (int q = 0; q < 3; ++q) {
    a.l0[q] = ps.cell0[q];
    a.xi[q] = (const T*)ps.xi[q];
  }
  a.wk = (const T*)ps.wk;
  a.n = ps.n;
  a.grid = (const T*)plan.grid_out;
  a.v = plan.view;
  a.width = g.width;
  a.C = g.C;
  a.Cp = plan.box3.Cp;
  a.beta = es_beta_arg<T>(g.beta);
  a.inv_halfw = (T)(2.0 / g.width);
  a.alpha = alpha_sorted;
  a.shift = shift;
  a.dcorr = (&ps == &plan.pts) ? plan.dcorr : nullptr;
  a.out = out_sorted;
  dispatch<T, 1>(a, dim3((unsigned)((ps.n + kPointsPerBlock - 1) / kPointsPerBlock), (unsigned)R), st);
  GPN_CUDA(cudaGetLastError());
}

}  // namespace

void launch_interp3d(Plan& plan, const PointSet& ps, const double* alpha_sorted, double shift, double* out_sorted,
                     int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    impl<float>(plan, ps, alpha_sorted, shift, out_sorted, R, st);
  else
    impl<double>(plan, ps, alpha_sorted, shift, out_sorted, R, st);
}

}  // namespace gpn
