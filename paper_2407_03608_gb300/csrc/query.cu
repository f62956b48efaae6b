// Query points of the posterior mean (Eq. postmean) without binning: their cells, offsets and
// Chebyshev weights in the caller's order, and the 2-D interpolation straight from the grid.
//
// Binning a query set costs a sort, a dozen allocations and two host round trips; a query needs
// width^2 cells of every channel, which one warp reads in coalesced half-warp rows.
// Bound: L2 and DRAM latency of the unsorted supports (2-D, 1e5 queries, 8 channels, width 8:
// 0.27 ms).  A posterior mean at 1e5 queries on that plan: 1.93 -> 1.33 ms.
#include <algorithm>
#include <type_traits>

#include "kernels.h"

namespace gpn {

namespace {

template <typename T>
struct QueryPointArgs {
  const double* x;       // n x d row-major
  const double* w;       // paper-native fields
  const double* sig;
  long long n;
  int d, width;
  long long nf;
  double centre[kMaxDim];
  double inv_h, half_nf, half_w;
  int* l0[kMaxDim];
  T* xi[kMaxDim];
  T* wk;                 // [n][C]
  ChebArgs cb;
};

// the same arithmetic as the binned points: g = (x - centre)/h + nf/2, l0 = ceil(g - width/2)
// (every query lies in the plan's box, so its support lies in the grid; the clamp only guards
// the reads)
template <typename T>
__global__ void __launch_bounds__(128) k_query_points(QueryPointArgs<T> a) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= a.n) return;
  for (int q = 0; q < a.d; ++q) {
    const double g = (a.x[i * a.d + q] - a.centre[q]) * a.inv_h + a.half_nf;
    const double l0 = fmin(fmax(ceil(g - a.half_w), 0.0), (double)(a.nf - a.width));
    a.l0[q][i] = (int)l0;
    a.xi[q][i] = (T)(g - l0);
  }
  double v[kMaxChannels];
  cheb_weights(a.w[i], a.sig[i], a.cb, v);
  for (int k = 0; k < a.cb.C; ++k) a.wk[i * a.cb.C + k] = (T)v[k];
}

template <typename T>
struct QueryInterpArgs {
  const int* l0y;
  const int* l0x;
  const T* xiy;
  const T* xix;
  const T* wk;
  long long n;
  const T* grid;         // [k][y][x]
  long long nf, G;
  int width, C;
  T beta, inv_halfw;
  double* mu;
};

// w_k s_k and its sum: exact products in float-float for FP32, float-float for float-float,
// float64 for float64
template <typename T>
using Sum = typename std::conditional<std::is_same<T, double>::value, double, dd>::type;
__device__ __forceinline__ dd widen_product(float a, float b) {
  const float p = ffops::mul(a, b);
  return {p, ffops::fma(a, b, -p)};
}
__device__ __forceinline__ dd widen_product(dd a, dd b) { return a * b; }
__device__ __forceinline__ double widen_product(double a, double b) { return a * b; }
__device__ __forceinline__ dd scale_sum(float a, dd b) { return dd(a, 0.0f) * b; }
__device__ __forceinline__ dd scale_sum(dd a, dd b) { return a * b; }
__device__ __forceinline__ double scale_sum(double a, double b) { return a * b; }

// One warp a query: half-warp h takes the support's rows h, h + 2, ..., lane j of it column j.
template <typename T>
__global__ void __launch_bounds__(256) k_query_interp2(QueryInterpArgs<T> a) {
  const int lane = threadIdx.x & 31, j = lane & 15, h = lane >> 4, W = a.width;
  const long long q = blockIdx.x * (long long)(blockDim.x / 32) + threadIdx.x / 32;
  if (q >= a.n) return;
  const bool in = j < W;
  const T py = in ? psi_at<T>(j, a.xiy[q], a.beta, a.inv_halfw) : T(0);
  const T px = in ? psi_at<T>(j, a.xix[q], a.beta, a.inv_halfw) : T(0);
  T pr[kMaxWidth / 2];   // psi of this half-warp's rows
#pragma unroll
  for (int i = 0; i < kMaxWidth / 2; ++i) pr[i] = shfl_val(py, 2 * i + h);
  const T* g = a.grid + (a.l0y[q] + h) * a.nf + a.l0x[q] + j;
  Sum<T> res(0.0);
#pragma unroll 2
  for (int k = 0; k < a.C; ++k, g += a.G) {
    T s = T(0);
#pragma unroll
    for (int i = 0; i < kMaxWidth / 2; ++i)
      if (in && 2 * i + h < W) madd(s, pr[i], ldg_val(g + 2 * i * a.nf));
    res += widen_product(a.wk[q * a.C + k], s);
  }
  res = scale_sum(px, res);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) res += shfl_xor_val(res, o);
  if (lane == 0) a.mu[q] = (double)res;
}

template <typename T>
void points_impl(const Plan& plan, PointSet& qs, const double* x, const double* w, const double* sig, void* work,
                 cudaStream_t st) {
  const Hyper& h = plan.h;
  QueryPointArgs<T> a{};
  a.x = x;
  a.w = w;
  a.sig = sig;
  a.n = qs.n;
  a.d = h.d;
  a.width = h.width;
  a.nf = h.nf;
  const double P = 1.0 / h.dw;   // the same operations as the training points' binning
  a.inv_h = h.nf / P;
  a.half_nf = 0.5 * h.nf;
  a.half_w = 0.5 * h.width;
  T* t = (T*)work;
  a.wk = t;
  t += (size_t)qs.n * plan.geom.C;
  for (int q = 0; q < h.d; ++q, t += qs.n) {
    a.centre[q] = 0.5 * (h.box_lo[q] + h.box_hi[q]);
    a.xi[q] = t;
    qs.xi[q] = t;
  }
  for (int q = 0; q < h.d; ++q) qs.cell0[q] = a.l0[q] = (int*)t + (size_t)q * qs.n;
  qs.wk = a.wk;
  a.cb.C = plan.geom.C;
  a.cb.d = h.d;
  for (int k = 0; k < a.cb.C; ++k) {
    a.cb.nodes[k] = plan.tb.nodes[k];
    a.cb.bary[k] = plan.tb.bary[k];
  }
  k_query_points<T><<<blocks_for(qs.n, 128), 128, 0, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

template <typename T>
void interp_impl(const Plan& plan, const PointSet& qs, double* mu, cudaStream_t st) {
  const GridGeom& g = plan.geom;
  QueryInterpArgs<T> a{qs.cell0[0],
                       qs.cell0[1],
                       (const T*)qs.xi[0],
                       (const T*)qs.xi[1],
                       (const T*)qs.wk,
                       qs.n,
                       (const T*)plan.grid_out,
                       g.nf,
                       plan.grid_elems,
                       g.width,
                       g.C,
                       es_beta_arg<T>(g.beta),
                       (T)(2.0 / g.width),
                       mu};
  k_query_interp2<T><<<blocks_for(qs.n, 8), 256, 0, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

}  // namespace

// Query sets evaluated without binning: the 1-D, 2-D and 3-D box plans', up to the sizes where
// the unsorted reads of the supports cost more than the sort.  A posterior mean without / with
// binning, ms (training points, grid, channels in brackets):
//   1-D FP32         [1e5, nf 32768, 8]       1e5 queries .19 / .65   1e6 .83 / 1.48   4e6 2.4 / 2.9
//   1-D float64      [1e5, nf 32768, 8]       1e5 .43 / .84           1e6 1.4 / 2.4    4e6 4.4 / 5.8
//   2-D FP32         [1e6, nf 8192, 8]        1e4 4.41 / 4.92         1e5 4.73 / 5.63  2.6e5 5.31 / 5.96
//                    [1e4, nf 512, 5]         1e4 .14 / .29           1e5 .25 / .74    2.6e5 .43 / 1.09
//                    [1e5, nf 4096, 8]        1e5 1.36 / 1.79         2.5e5 1.82 / 2.18   1e6 4.25 / 2.73
//   2-D float-float  [1e6, nf 4096, 7]        1e5 4.41 / 4.95         2.6e5 5.20 / 5.25
//                    [1e5, nf 4096]           1e5 4.28 / 4.66         2.5e5 5.16 / 5.14   1e6 9.73 / 6.19
//   2-D float64      [1e5, nf 2048, 6]        1e4 3.10 / 3.27         1.3e5 3.97 / 4.08
//                    [1e5, nf 4096]           1e5 4.70 / 4.74         2.5e5 5.89 / 5.41   1e6 11.9 / 7.28
//   3-D FP32         [2e6, nf 540, 7]         1e4 9.43 / 9.99         1e5 9.77 / 10.7     2.6e5 10.4 / 11.4
//                    [2e6, nf 800, 8]         1e4 27.3 / 28.2         1e5 27.8 / 29.4     2.6e5 28.7 / 30.2
//                    [2e4, nf 140, 5]         1e4 .37 / .55           1e5 .54 / 1.18      2.6e5 .87 / 1.72
//   3-D float64      [2e4, nf 256, 6]         1e4 9.28 / 9.47         1e5 11.0 / 11.8     2.6e5 14.2 / 15.2
// So the grids' size against the L2 moves the line little, and in 3-D nothing lost up to the count
// that was measured, where the line is drawn.  (2-D float64: the kernel values of an unbinned query
// are not tabulated, and their float64 arithmetic sets the line.  The 3-D interpolation has gained since.)
bool query_unbinned(const Plan& plan, long long n) {
  if (plan.geom.d == 1) return n < (1ll << 31);   // (more are refused by the binning, as ever)
  if (plan.geom.d == 3) return plan.box3.on && n <= (1 << 18);
  return n <= (plan.precision == GP_FP64 ? 1 << 17 : 1 << 18);
}

size_t query_work_bytes(const Plan& plan, long long n) {
  return (size_t)n * ((size_t)(plan.geom.C + plan.geom.d) * plan.real_size + plan.geom.d * sizeof(int));
}

void build_query_points(const Plan& plan, PointSet& qs, const double* x, const double* w, const double* sig,
                        long long n, void* work, cudaStream_t st) {
  qs.n = n;
  if (plan.precision == GP_FP32)
    points_impl<float>(plan, qs, x, w, sig, work, st);
  else if (plan.precision == GP_DF64)
    points_impl<dd>(plan, qs, x, w, sig, work, st);
  else
    points_impl<double>(plan, qs, x, w, sig, work, st);
}

// mu in the order of the queries, from plan.grid_out
void launch_query_mean(Plan& plan, const PointSet& qs, double* mu, cudaStream_t st) {
  if (plan.geom.d != 2) return launch_interp(plan, qs, nullptr, 0.0, mu, 1, st);
  if (plan.precision == GP_FP32)
    interp_impl<float>(plan, qs, mu, st);
  else if (plan.precision == GP_DF64)
    interp_impl<dd>(plan, qs, mu, st);
  else
    interp_impl<double>(plan, qs, mu, st);
}

}  // namespace gpn
