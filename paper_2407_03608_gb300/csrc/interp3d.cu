// Steps (4b) + (5) of Sec. 4.2 in three dimensions, on the box grids of fft3d.cu:
//   out_i = sum_zyx psi(z) psi(y) psi(x) sum_k w_k(x_i) g_k[z][y][x]  (+ shift * alpha_i).
//
// One warp a point, straight from the grid through L1: the channels are innermost, so one row
// (z, y) of the support is width * Cp adjacent values, which the lanes read in S coalesced
// loads; a row costs S loads and S multiply-adds.  A lane's position in the row fixes its cell x
// and channel k for the whole point.  Points come in bin order and a block takes consecutive ones,
// so the rows of neighbouring points are served by L1.  Sums: a slot's rows weighted by psi(y), the
// planes weighted by psi(z); then the slots pass through shared memory, lane k sums channel k over
// x, and the products w_k beta_k, whose signs alternate, are formed and added in float64.
//
// Bound: latency of the L1/L2 loads and issue (about 9 instructions a row).  On 2e6 points, ms:
// the staged kernel of interp.cu 15.1 (8 channels, width 9, nf 512) and 26.7 (10, 9, nf 864); here
// 4.27 and 5.61, 7 channels in float64 (2e5 points) 2.83.  What the loop's registers allow decides:
// indexed rows instead of running pointers 4.98 and 6.25, unrolled by 3 as well 5.19 and 7.63, 48
// warps an SM instead of 64 in that form 5.27 and 6.97.  Mixing the channels of a lane in one FP32 sum 4.17 and
// 5.44.  Sorting the points finer than by bins changes nothing.
#include <algorithm>

#include "kernels.h"

namespace gpn {

namespace {

// the rows are short chains of loads, so what counts is warps in flight: up to three loads a row
// 64 an SM (32 registers, a few spilled outside the loop), above that what the registers allow
template <int S>
constexpr int kWarps = S <= 3 ? 16 : 8;
// points a block takes, at most and where they still give two blocks an SM: 1000 points of 4 channels
// at width 7 48 us with 64 a block, 18 with as many as warps (the staged kernel 18)
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
  int fold;              // half the power of two that holds C lanes
  int per;               // points a block
  T beta, inv_halfw;
  const double* alpha;   // sorted order (may be null)
  double shift;
  const double* dcorr;   // per-point addition to the shift (may be null)
  double* out;           // sorted order, n x R
};

// S: loads a row, ceil(width Cp / 32)
template <typename T, int S>
__global__ void __launch_bounds__(32 * kWarps<S>, S <= 3 ? 4 : 1) k_interp3d(Interp3Args<T> a) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = a.width, r = blockIdx.y;
  const long long s0 = a.v.stride[0], s1 = a.v.stride[1];
  const T* grid = a.grid + r * a.v.rstride + lane;
  const double* alpha = a.alpha ? a.alpha + (size_t)r * a.n : nullptr;
  const int last = W * a.Cp - 32 * (S - 1);   // lanes of the last slot inside the row
  __shared__ T s_sum[kWarps<S>][32 * S];   // a point's sums over z and y, in the order of a row
  T* sums = s_sum[warp];
  const long long p1 = min(a.n, (long long)(blockIdx.x + 1) * a.per);
  for (long long p = (long long)blockIdx.x * a.per + warp; p < p1; p += kWarps<S>) {
    const int lz = a.l0[0][p] - a.v.lo[0], ly = a.l0[1][p] - a.v.lo[1], lx = a.l0[2][p] - a.v.lo[2];
    T pz = T(0), py = T(0), px = T(0);
    if (lane < W) {
      pz = psi_at<T>(lane, a.xi[0][p], a.beta, a.inv_halfw);
      py = psi_at<T>(lane, a.xi[1][p], a.beta, a.inv_halfw);
      px = psi_at<T>(lane, a.xi[2][p], a.beta, a.inv_halfw);
    }
    const T* g = grid + lz * s0 + ly * s1 + lx * a.v.stride[2];
    T acc[S];
#pragma unroll
    for (int s = 0; s < S; ++s) acc[s] = T(0);
    for (int z = 0; z < W; ++z, g += s0) {
      const T* gy = g;
      T plane[S];
#pragma unroll
      for (int s = 0; s < S; ++s) plane[s] = T(0);
#pragma unroll 4
      for (int y = 0; y < W; ++y, gy += s1) {
        const T wy = shfl_val(py, y);
#pragma unroll
        for (int s = 0; s < S; ++s) plane[s] += wy * ((s + 1 < S || lane < last) ? __ldg(gy + 32 * s) : T(0));
      }
      const T wz = shfl_val(pz, z);
#pragma unroll
      for (int s = 0; s < S; ++s) acc[s] += wz * plane[s];
    }
    // lane k: the sum of channel k over x, times w_k in float64
#pragma unroll
    for (int s = 0; s < S; ++s) sums[32 * s + lane] = acc[s];
    __syncwarp();
    T beta = T(0);
    const T* sk = sums + min(lane, a.C - 1);
    for (int x = 0; x < W; ++x) beta += shfl_val(px, x) * sk[x * a.Cp];
    double res = lane < a.C ? (double)a.wk[p * a.C + lane] * (double)beta : 0.0;
    for (int o = a.fold; o > 0; o >>= 1) res += __shfl_xor_sync(0xffffffffu, res, o);
    __syncwarp();   // the next point's sums take the place of these
    if (lane == 0) {
      if (alpha) res += (a.dcorr ? a.shift + a.dcorr[p] : a.shift) * alpha[p];
      a.out[(size_t)r * a.n + p] = res;
    }
  }
}

template <typename T, int S>
void dispatch(Interp3Args<T> a, int R, cudaStream_t st) {
  if (a.width * a.Cp <= 32 * S) {
    const long long rounds = a.n / (304 * kWarps<S>);
    a.per = (int)std::max<long long>(1, std::min<long long>(kPointsPerBlock / kWarps<S>, rounds)) * kWarps<S>;
    k_interp3d<T, S><<<dim3((unsigned)((a.n + a.per - 1) / a.per), (unsigned)R), 32 * kWarps<S>, 0, st>>>(a);
  } else if constexpr (S < kMaxWidth * kMaxChannels / 32) {
    dispatch<T, S + 1>(a, R, st);
  }
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
  for (int w = 1; w < g.C; w *= 2) a.fold = w;
  a.beta = es_beta_arg<T>(g.beta);
  a.inv_halfw = (T)(2.0 / g.width);
  a.alpha = alpha_sorted;
  a.shift = shift;
  a.dcorr = (&ps == &plan.pts) ? plan.dcorr : nullptr;
  a.out = out_sorted;
  dispatch<T, 1>(a, R, st);
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
