// One-dimensional plans: spreading, interpolation, and the transforms with step (3) of
// Sec. 4.2 between them (nf = 2^a).
//
// A 1-D workload is small (N = 2000 points, C = 15 channels of 8192 cells at the paper's
// accuracy), so what counts is how many SMs share a step and how many launches there are.
//
// Transforms.  A channel's real row of nf values is an h = nf/2 point complex sequence
// z[j] = x[2j] + i x[2j+1].  S blocks share one transform without exchanging data: block q
// computes the outputs Z[q + S k] from the h/S sums
//   u[n] = W_h^{n q} sum_{s<S} z[n + s h/S] W_S^{s q},   Z[q + S k] = FFT_{h/S}(u)[k],
// at the price of forming its own S-term sums (18 additions and products for S = 8 against
// the sub-transform's 30 to 40 an element).  With S = 8 the 15 channels of the N = 2000
// workload occupy 120 SMs instead of 15; the FP64 pipe (2 multiply-adds a clock and SM) is
// what bounds them.  The inverse has the same form.
// Step 3 then works on the complex sequences themselves: one thread takes the pair of
// entries (k, h - k) of a channel, splits them into the real row's modes X[k] and X[h - k],
// multiplies by A' across the channels (through shared memory) and merges the products back
// into the pair, in place.
//
// Points are sorted by their first support cell (not only by bin), so the points that reach
// a group of cells are one contiguous run.
//
// Bound: latency (five launches of 7 to 15 us), the FP64 pipe in the float64 transforms.  A matvec,
// against the tiled or atomic spread, row or cuFFT transforms and a lane-a-point interpolation:
// N = 2000 float64 (15 channels, nf 8192) 235 -> 57 us, N = 1e5 FP32 with 4 right-hand sides (10
// channels, nf 65536) 217 -> 127 us.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fft_core.h"
#include "kernels.h"

namespace gpn {

namespace {

using fft::cpx;

template <typename T>
struct alignas(2 * sizeof(T)) RawC {
  T x, y;
};
template <typename T>
__device__ __forceinline__ cpx<T> load_c(const cpx<T>* p) {
  const RawC<T> v = *reinterpret_cast<const RawC<T>*>(p);
  return {v.x, v.y};
}
template <typename T>
__device__ __forceinline__ void store_c(cpx<T>* p, cpx<T> v) {
  *reinterpret_cast<RawC<T>*>(p) = RawC<T>{v.x, v.y};
}

// The sum of exact products of FP32 values, in three words (about 72 bits): float64's precision on
// the FP32 pipe (float64 sums run at a sixtieth of its rate, conversions at a sixteenth).  Largest
// error over 2e5 sums of up to 32 terms, relative to the largest term: 3.1e-16, float64 1.7e-15, two words
// 4.6e-14.
struct Sum3 {
  float a = 0.0f, b = 0.0f, c = 0.0f;

  // + x + y, |y| below |x|'s last place or so
  __device__ __forceinline__ void add(float x, float y) {
    const dd s = two_sum(a, x), t = two_sum(b, s.lo), u = two_sum(t.hi, y);
    a = s.hi;
    b = u.hi;
    c = ffops::add(c, ffops::add(t.lo, u.lo));
  }
  __device__ __forceinline__ explicit operator double() const { return (double)a + ((double)b + (double)c); }
};
__device__ __forceinline__ void set_product(double& sum, double w, double b) { sum = w * b; }
__device__ __forceinline__ void set_product(Sum3& sum, float w, float b) {
  sum.a = ffops::mul(w, b);
  sum.b = ffops::fma(w, b, -sum.a);
  sum.c = 0.0f;
}
__device__ __forceinline__ void add_product(double& sum, double w, double b) { sum += w * b; }
__device__ __forceinline__ void add_product(Sum3& sum, float w, float b) {
  const float p = ffops::mul(w, b);
  sum.add(p, ffops::fma(w, b, -p));
}
__device__ __forceinline__ void add_value(double& sum, double x) { sum += x; }
__device__ __forceinline__ void add_value(Sum3& sum, float x) { sum.add(x, 0.0f); }
template <typename T>
using SumOf = typename std::conditional<sizeof(T) == 4, Sum3, double>::type;

// + the same of lane ^ o
__device__ __forceinline__ void add_lane(double& sum, int o) { sum += shfl_xor_val(sum, o); }
__device__ __forceinline__ void add_lane(Sum3& sum, int o) {
  const float x = shfl_xor_val(sum.a, o), y = shfl_xor_val(sum.b, o), z = shfl_xor_val(sum.c, o);
  sum.add(x, y);
  sum.c = ffops::add(sum.c, z);
}

// ---- spreading --------------------------------------------------------------------------

constexpr int kSpreadThreads = 256;
constexpr int kChunk = 128;     // points staged at a time

template <typename T>
struct Spread1Args {
  const int* l0;
  const int* perm;       // sorted position -> caller index, when alpha is in the caller's order
  const T* xi;
  const T* psi;          // tabulated kernel values [n][width] (null: evaluate)
  const T* wk;           // [n][C]
  const int* start;      // start[c]: first sorted point with l0 >= c, c <= nf (null: searched for)
  int cell0, cell1;      // cells the points reach
  int cells;             // cells a block
  const double* alpha;   // n x R column-major
  long long n;
  T* grid;               // [r][k][nf]
  long long nf;
  T* scratch;            // the parts' sums [part][r][k][cell1 - cell0], with more than one part
  int width, C, R;
  T beta, inv_halfw;
};

// first of the n sorted cells l0 that is >= c
__device__ __forceinline__ int first_at(const int* __restrict__ l0, int n, int c) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (l0[mid] < c)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// One thread takes one (cell, channel) pair, one block a run of `cells` cells.  The points that
// reach the run are one contiguous run of the cell-sorted points; the block stages their kernel
// values, weights and the alpha of RB right-hand sides in shared memory, kChunk points at a
// time, and every thread walks the points that reach its own cell (again contiguous), so that every multiply-add is a needed
// one.  The order of the sums is the points' order (results do not depend on scheduling), and
// every cell the points reach is written, so the grid needs no clearing.
// SEARCH: without the table of the cells' first points (a template parameter: with both in one
// kernel the compiler gives up the walk's unrolled form, 1.5 times the time with RB = 4).
template <typename T, int RB, bool SEARCH>
__global__ void __launch_bounds__(kSpreadThreads) k_spread1d(Spread1Args<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int W = a.width, C = a.C, r0 = blockIdx.y * RB, tid = threadIdx.x;
  T* s_wk = reinterpret_cast<T*>(smem_raw);   // [kChunk][C]
  T* s_psi = s_wk + kChunk * C;               // [kChunk][W]
  T* s_amp = s_psi + kChunk * W;              // [kChunk][RB]: alpha, converted once a point
  int* s_l0 = reinterpret_cast<int*>(s_amp + kChunk * RB);
  const int c0 = a.cell0 + blockIdx.x * a.cells, c1 = min(c0 + a.cells, a.cell1);
  const auto start = [&](int c) {
    if constexpr (SEARCH) return first_at(a.l0, (int)a.n, c);
    return a.start[c];
  };
  const int p0 = start(max(0, c0 - W + 1)), p1 = start(c1);
  const int ci = tid / C, k = tid - ci * C, cell = c0 + ci;
  const int pi = tid / W, j = tid - pi * W, pstep = kSpreadThreads / W;
  const bool on = ci < a.cells && cell < c1;
  const int q0 = on ? start(max(0, cell - W + 1)) : 0, q1 = on ? start(cell + 1) : 0;
  const double* alpha = a.alpha + (size_t)r0 * a.n;
  // this block's part of the run's chunks
  const int chunks = (p1 - p0 + kChunk - 1) / kChunk, parts = gridDim.z;
  const int b0 = p0 + (int)((long long)chunks * blockIdx.z / parts) * kChunk;
  const int b1 = min(p1, p0 + (int)((long long)chunks * (blockIdx.z + 1) / parts) * kChunk);
  T acc[RB];
#pragma unroll
  for (int r = 0; r < RB; ++r) acc[r] = T(0);
  for (int base = b0; base < b1; base += kChunk) {
    const int m = min(kChunk, b1 - base);
    for (int i = tid; i < m; i += kSpreadThreads) {
      s_l0[i] = a.l0[base + i];
      const int q = a.perm ? a.perm[base + i] : base + i;
#pragma unroll
      for (int r = 0; r < RB; ++r) s_amp[i * RB + r] = r0 + r < a.R ? (T)alpha[(size_t)r * a.n + q] : T(0);
    }
    if (pi < pstep)
      for (int q = pi; q < m; q += pstep)
        s_psi[q * W + j] = a.psi ? a.psi[(size_t)(base + q) * W + j]
                                 : psi_at<T>(j, a.xi[base + q], a.beta, a.inv_halfw);
    for (int i = tid; i < m * C; i += kSpreadThreads) s_wk[i] = a.wk[(size_t)base * C + i];
    __syncthreads();
    const int e = min(q1 - base, m);
    T part[RB];   // a chunk's sum on its own: dense cells add their points in two levels
#pragma unroll
    for (int r = 0; r < RB; ++r) part[r] = T(0);
#pragma unroll 4
    for (int q = max(q0 - base, 0); q < e; ++q) {
      const T v = s_psi[q * W + (cell - s_l0[q])] * s_wk[q * C + k];
#pragma unroll
      for (int r = 0; r < RB; ++r) part[r] += v * s_amp[q * RB + r];
    }
#pragma unroll
    for (int r = 0; r < RB; ++r) acc[r] += part[r];
    __syncthreads();
  }
  // the run's sums leave through shared memory, cells fastest
  T* s_out = reinterpret_cast<T*>(smem_raw);
  const int nc = c1 - c0, span = a.cell1 - a.cell0;
  T* out = parts > 1 ? a.scratch + (size_t)blockIdx.z * a.R * C * span + (c0 - a.cell0) : a.grid + c0;
  const long long pitch = parts > 1 ? span : a.nf;
#pragma unroll
  for (int r = 0; r < RB; ++r) {
    if (r0 + r >= a.R) break;
    if (on) s_out[k * a.cells + ci] = acc[r];
    __syncthreads();
    for (int i = tid; i < nc * C; i += kSpreadThreads) {
      const int kk = i / nc, c = i - kk * nc;
      out[((size_t)(r0 + r) * C + kk) * pitch + c] = s_out[kk * a.cells + c];
    }
    __syncthreads();
  }
}

// the parts' sums, in their order: one thread a (right-hand side, channel, cell)
template <typename T>
__global__ void __launch_bounds__(256) k_spread1d_sum(Spread1Args<T> a, int parts) {
  const int span = a.cell1 - a.cell0, total = a.R * a.C * span, i = blockIdx.x * 256 + threadIdx.x;
  if (i >= total) return;
  SumOf<T> s{};
  for (int p = 0; p < parts; ++p) add_value(s, a.scratch[(size_t)p * total + i]);
  a.grid[(size_t)(i / span) * a.nf + a.cell0 + i % span] = (T)(double)s;
}

// right-hand sides a block takes, and cells of a block's run
constexpr int spread_rhs(int R) { return R <= 2 ? R : 4; }
int spread_cells(int C) { return std::max(1, kSpreadThreads / C); }

// Parts the points of a run are divided into.  A short grid has few runs (64 cells of 4 channels:
// one), and a thread walks all points of its cell: parts of a chunk or more, up to two blocks an SM.
// nf = 64, 4 channels, ms a product without / with parts (and with the atomic or tiled spread of
// before): float64 n = 1e4 1.01 / .056 (.76), 1e5 with 5 right-hand sides 21.1 / .24 (7.6), FP32 1e5
// 3.71 / .084 (2.9); nf = 1024, 6 channels, n = 1e6: float64 8.80 / .59 (67), FP32 3.04 / .18 (32).  The
// spread alone at n = 1e6, us, FP32 / float64: 94 runs 439 / 1630 whole and 138 / 600 in parts, 154 runs
// 365 / 1330 and 215 / 956, 187 runs 240 / 914 and 138 / 579; 307 runs (whole by the rule) 206 / 977.
int spread_parts(const Plan& plan, int R) {
  const int span = plan.line_cell1 - plan.line_cell0, cells = spread_cells(plan.geom.C);
  const long long blocks = (long long)((span + cells - 1) / cells) * ((R + spread_rhs(R) - 1) / spread_rhs(R));
  if (!plan.spare || blocks >= 304) return 1;
  const double points = (double)plan.pts.n * std::min(1.0, (double)(cells + plan.geom.width - 1) / span);   // a run's
  return (int)std::max(1.0, std::min((double)((304 + blocks - 1) / blocks), points / kChunk));
}

template <typename T, int RB>
void spread_launch(const Spread1Args<T>& a, int R, int parts, cudaStream_t st) {
  const size_t smem = kChunk * ((a.C + a.width + RB) * sizeof(T) + sizeof(int));
  void (*k)(Spread1Args<T>) = a.start ? k_spread1d<T, RB, false> : k_spread1d<T, RB, true>;
  GPN_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int blocks = (a.cell1 - a.cell0 + a.cells - 1) / a.cells;
  k<<<dim3((unsigned)blocks, (unsigned)((R + RB - 1) / RB), (unsigned)parts), kSpreadThreads, smem, st>>>(a);
  if (parts > 1) k_spread1d_sum<T><<<blocks_for((long long)R * a.C * (a.cell1 - a.cell0), 256), 256, 0, st>>>(a, parts);
}

template <typename T>
void spread_impl(Plan& plan, const double* alpha, const int* perm, int R, cudaStream_t st) {
  const GridGeom& g = plan.geom;
  const PointSet& ps = plan.pts;
  Spread1Args<T> a{};
  a.l0 = ps.cell0[0];
  a.perm = perm;
  a.xi = (const T*)ps.xi[0];
  a.psi = (const T*)ps.psi[0];
  a.wk = (const T*)ps.wk;
  a.start = plan.line_start;
  a.cell0 = plan.line_cell0;
  a.cell1 = plan.line_cell1;
  a.cells = spread_cells(g.C);
  a.alpha = alpha;
  a.n = ps.n;
  a.grid = (T*)plan.grid;
  a.nf = g.nf;
  a.width = g.width;
  a.C = g.C;
  a.beta = es_beta_arg<T>(g.beta);
  a.inv_halfw = (T)(2.0 / g.width);
  a.R = R;
  a.scratch = (T*)plan.line_scratch;
  const int parts = spread_parts(plan, R);
  // several right-hand sides a block share the staged points
  switch (spread_rhs(R)) {
    case 1: spread_launch<T, 1>(a, R, parts, st); break;
    case 2: spread_launch<T, 2>(a, R, parts, st); break;
    default: spread_launch<T, 4>(a, R, parts, st);
  }
  GPN_CUDA(cudaGetLastError());
}

// start[c], c = 0 .. nf
__global__ void k_line_start(const int* __restrict__ l0, int n, int cells, int* __restrict__ start) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c <= cells) start[c] = first_at(l0, n, c);
}

// ---- interpolation ------------------------------------------------------------------------

template <typename T>
struct Interp1Args {
  const int* l0;
  const int* perm;       // sorted position -> caller index, when alpha and out are in the caller's order
  const T* xi;
  const T* psi;
  const T* wk;
  long long n;
  const T* grid;         // [r][k][nf]
  long long nf;
  int width, C;
  T beta, inv_halfw;
  const double* alpha;   // sorted order (may be null)
  double shift;
  const double* dcorr;   // per-point addition to the shift (may be null)
  double* out;           // sorted order, n x R
};

template <typename T>
__device__ __forceinline__ void finish_point(const Interp1Args<T>& a, long long p, int r, double res) {
  const long long i = (size_t)r * a.n + (a.perm ? a.perm[p] : p);
  if (a.alpha) res += (a.dcorr ? a.shift + a.dcorr[p] : a.shift) * a.alpha[i];
  a.out[i] = res;
}

// Sixteen lanes a point: lane j holds psi(j), lane k sums channel k (k + 16, ...) over the W
// cells; the products w_k beta_k are added exactly (see add_product).  For point sets too small to fill the
// chip with a thread a point (and for float64, whose kernel values it spreads over the lanes).
template <typename T>
__global__ void __launch_bounds__(128) k_interp1d_lanes(Interp1Args<T> a) {
  const int gl = threadIdx.x & 15, r = blockIdx.y, W = a.width;
  const long long p = blockIdx.x * (long long)(blockDim.x / 16) + threadIdx.x / 16;
  const bool on = p < a.n;
  const long long q = on ? p : a.n - 1;
  const T* g = a.grid + (size_t)r * a.C * a.nf + a.l0[q];
  T pj = T(0);
  if (gl < W) pj = a.psi ? a.psi[q * W + gl] : psi_at<T>(gl, a.xi[q], a.beta, a.inv_halfw);
  SumOf<T> part{};
  for (int k0 = 0; k0 < a.C; k0 += 16) {
    const bool in = k0 + gl < a.C;
    const int k = in ? k0 + gl : a.C - 1;
    const T* gk = g + (size_t)k * a.nf;
    const T w = in ? a.wk[q * a.C + k] : T(0);
    T v[kMaxWidth], s = T(0);   // every cell is loaded before the first sum
#pragma unroll
    for (int j = 0; j < kMaxWidth; ++j) v[j] = j < W ? __ldg(gk + j) : T(0);
#pragma unroll
    for (int j = 0; j < kMaxWidth; ++j)
      if (j < W) s += __shfl_sync(0xffffffffu, pj, j, 16) * v[j];
    if (k0 == 0)
      set_product(part, w, s);
    else
      add_product(part, w, s);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) add_lane(part, o);
  if (on && gl == 0) finish_point(a, p, r, (double)part);
}

// A thread a point, NC = C channels in registers (32 with the extra ones unused): neighbouring
// points read neighbouring cells; the points' weights (rows of C values) come through shared
// memory, a row a lane would touch a line each.
constexpr int kInterpThreads = 128;
template <typename T, int NC>
__global__ void __launch_bounds__(kInterpThreads) k_interp1d(Interp1Args<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* s_wk = reinterpret_cast<T*>(smem_raw);   // [kInterpThreads][C | 1]
  const long long p0 = blockIdx.x * (long long)kInterpThreads, p = p0 + threadIdx.x;
  const int r = blockIdx.y, W = a.width, C = NC <= 16 ? NC : a.C;
  const int m = (int)min((long long)kInterpThreads, a.n - p0) * C;
  for (int i = threadIdx.x; i < m; i += kInterpThreads) {
    const int q = i / C;
    s_wk[q * (C | 1) + (i - q * C)] = a.wk[p0 * C + i];
  }
  const bool on = p < a.n;
  const T* g = a.grid + (size_t)r * C * a.nf + (on ? a.l0[p] : 0);
  const T x = on ? a.xi[p] : T(0);
  T acc[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) acc[k] = T(0);
  if (on) {
    for (int j = 0; j < W; ++j) {
      const T ps = a.psi ? a.psi[p * W + j] : psi_at<T>(j, x, a.beta, a.inv_halfw);
#pragma unroll
      for (int k = 0; k < NC; ++k)
        if (NC <= 16 || k < C) acc[k] += ps * __ldg(g + (size_t)k * a.nf + j);
    }
  }
  __syncthreads();
  if (!on) return;
  const T* w = s_wk + threadIdx.x * (C | 1);
  SumOf<T> res{};
#pragma unroll
  for (int k = 0; k < NC; ++k)
    if (NC <= 16 || k < C) add_product(res, w[k], acc[k]);
  finish_point(a, p, r, (double)res);
}

template <typename T, int NC>
void interp_dispatch(const Interp1Args<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 16) {
    k_interp1d<T, 32><<<grid, kInterpThreads, sizeof(T) * kInterpThreads * (a.C | 1), st>>>(a);
  } else {
    if (a.C == NC)
      k_interp1d<T, NC><<<grid, kInterpThreads, sizeof(T) * kInterpThreads * (a.C | 1), st>>>(a);
    else
      interp_dispatch<T, NC + 1>(a, grid, st);
  }
}

template <typename T>
void interp_impl(Plan& plan, const PointSet& ps, const double* alpha, double shift, double* out, const int* perm, int R,
                 cudaStream_t st) {
  const GridGeom& g = plan.geom;
  Interp1Args<T> a{ps.cell0[0],
                   perm,
                   (const T*)ps.xi[0],
                   (const T*)ps.psi[0],
                   (const T*)ps.wk,
                   ps.n,
                   (const T*)plan.grid_out,
                   g.nf,
                   g.width,
                   g.C,
                   es_beta_arg<T>(g.beta),
                   (T)(2.0 / g.width),
                   alpha,
                   shift,
                   (&ps == &plan.pts) ? plan.dcorr : nullptr,
                   out};
  // a thread a point once the points fill half of the chip's threads (152 SMs x 1024)
  if (ps.n * R >= 152ll * 1024)
    interp_dispatch<T, 1>(a, dim3((unsigned)((ps.n + kInterpThreads - 1) / kInterpThreads), (unsigned)R), st);
  else
    k_interp1d_lanes<T><<<dim3((unsigned)((ps.n + 7) / 8), (unsigned)R), 128, 0, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

// ---- transforms -----------------------------------------------------------------------------

constexpr int kMaxSplit = 8;
// blocks wanted in a launch: three quarters of the SMs (a second wave for a few blocks more would
// cost a whole sub-transform; the 15 channels of the N = 2000 workload take 120 blocks at S = 8)
constexpr int kLineBlocks = 114;

// The passes of the N-point sub-transform: one of radix r0 (2 or 4, or 1: none), then np of
// radix R; a thread holds NB butterflies of radix R.  The passes run as one loop over the same
// code: a block runs each pass once, so unrolled passes would be bound by instruction fetches
// (measured: 31 us for 512-point float64 sub-transforms with unrolled radix-8 passes, an
// estimated 7 us of which is arithmetic).
struct LinePlan {
  int N = 0, R = 0, NB = 0, r0 = 1, np = 0;
};

template <typename T>
struct LineArgs {
  const cpx<T>* in;      // forward: grid rows as pairs [cr][h]; inverse: spectra [cr][h]
  cpx<T>* out;
  const cpx<T>* tw;      // exp(-2 pi i k / nf), k < nf
  const cpx<T>* ptw;     // pass twiddles of the h / S point transform
  int N, r0, np;
  int h;
  int lo, hi;            // pairs of the row that hold data or are read by the interpolation
};

// a * exp(-+ 2 pi i q / 4)
template <bool INV, typename T>
__device__ __forceinline__ cpx<T> quarter_turns(cpx<T> a, int q) {
  if (q & 1) a = fft::rot90<INV>(a);
  return q & 2 ? cpx<T>{-a.x, -a.y} : a;
}

// padded shared-memory index: the first passes store at strides of 4 and 8 elements, which would
// fall in a few banks
template <typename T>
__device__ __forceinline__ int spos(int n) { return n + (n >> (sizeof(T) == 4 ? 4 : 3)); }

// one Stockham pass in place, NB butterflies a thread (J threads)
template <int R, int NB, bool INV, typename T>
__device__ __forceinline__ void line_pass(cpx<T>* s, int N, int J, int Ns, int t, const cpx<T>* tw) {
  const int nbf = N / R;
  cpx<T> v[NB][R], w[NB][R];
  // the twiddles (global memory) are on their way before the barrier
  if (Ns > 1) {
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int r = 1; r < R; ++r) w[b][r] = load_c(tw + (r - 1) * Ns + ((t + b * J) & (Ns - 1)));
  }
#pragma unroll
  for (int b = 0; b < NB; ++b)
#pragma unroll
    for (int r = 0; r < R; ++r) v[b][r] = load_c(s + spos<T>(t + b * J + r * nbf));
  __syncthreads();
#pragma unroll
  for (int b = 0; b < NB; ++b) {
    const int j = t + b * J, k = j & (Ns - 1);
    if (Ns > 1) {
#pragma unroll
      for (int r = 1; r < R; ++r) {
        if (INV) w[b][r].y = -w[b][r].y;
        v[b][r] = fft::cmul(v[b][r], w[b][r]);
      }
    }
    fft::dft<INV, R>(v[b]);
#pragma unroll
    for (int r = 0; r < R; ++r) store_c(s + spos<T>((j - k) * R + k + r * Ns), v[b][r]);
  }
  __syncthreads();
}

// blockIdx = (output residue q, channel and right-hand side); N / (R NB) threads
template <typename T, bool INV, int S, int R, int NB>
__global__ void __launch_bounds__(512) k_line(LineArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.N, J = blockDim.x, t = threadIdx.x, q = blockIdx.x;
  const cpx<T>* src = a.in + (size_t)blockIdx.y * a.h;
  cpx<T>* dst = a.out + (size_t)blockIdx.y * a.h;
  auto twid = [&](int i) {
    cpx<T> w = load_c(a.tw + i);
    if (INV) w.y = -w.y;
    return w;
  };
  const cpx<T> w8 = S == 8 ? twid(q * (a.h / 4)) : cpx<T>{T(1), T(0)};   // W_8^q
#pragma unroll 4
  for (int n = t; n < N; n += J) {
    cpx<T> z[S];
#pragma unroll
    for (int i = 0; i < S; ++i) {
      const int j = n + i * N;
      z[i] = INV || (j >= a.lo && j < a.hi) ? load_c(src + j) : cpx<T>{T(0), T(0)};
    }
    // W_S^{i q}: the halves pair up with the sign (-1)^q, the quarters with quarter turns
    if constexpr (S > 1) {
      const cpx<T> w = twid(2 * n * q);
#pragma unroll
      for (int i = 0; i < S / 2; ++i) z[i] = q & 1 ? z[i] - z[i + S / 2] : z[i] + z[i + S / 2];
      if constexpr (S == 4) z[0] = z[0] + quarter_turns<INV>(z[1], q & 3);
      if constexpr (S == 8) {
        const cpx<T> u0 = z[0] + quarter_turns<INV>(z[2], q & 3), u1 = z[1] + quarter_turns<INV>(z[3], q & 3);
        z[0] = u0 + (q & 1 ? fft::cmul(u1, w8) : quarter_turns<INV>(u1, q / 2));
      }
      z[0] = fft::cmul(z[0], w);
    }
    store_c(s + spos<T>(n), z[0]);
  }
  __syncthreads();
  const cpx<T>* tw = a.ptw;
  int ns = a.r0;
  if (a.r0 == 2) line_pass<2, R * NB / 2, INV, T>(s, N, J, 1, t, tw);
  if (a.r0 == 4) line_pass<4, (R * NB > 4 ? R * NB / 4 : 1), INV, T>(s, N, J, 1, t, tw);
#pragma unroll 1
  for (int p = 0; p < a.np; ++p) {
    line_pass<R, NB, INV, T>(s, N, J, ns, t, tw);
    if (ns > 1) tw += (R - 1) * ns;
    ns *= R;
  }
  for (int n = t; n < N; n += J) {
    const int j = q + S * n;
    if (!INV || (j >= a.lo && j < a.hi)) store_c(dst + j, load_c(s + spos<T>(n)));
  }
}

// ---- step 3 on the pairs (k, h - k) -----------------------------------------------------------

constexpr int kDiagK = 16;   // pairs a block

template <typename T>
struct LineDiagArgs {
  cpx<T>* Z;             // [r][C][h], in place
  const cpx<T>* tw;      // exp(-2 pi i k / nf)
  const T* A;            // packed upper triangle [p][f], f = 0..M
  long long n_freq;
  int h, M, C;
};

// blockIdx = (pair group, right-hand side), blockDim = (kDiagK pairs, C channels)
template <typename T>
__global__ void __launch_bounds__(1024) k_line_diag(LineDiagArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s_lo = reinterpret_cast<cpx<T>*>(smem_raw);   // [C][kDiagK]: X[k]
  const int C = a.C, tx = threadIdx.x, c = threadIdx.y, h = a.h;
  cpx<T>* s_hi = s_lo + C * kDiagK;                     // X[h - k]
  const int k = blockIdx.x * kDiagK + tx, kn = h - k;
  const bool on = k <= h / 2, lo = on && k <= a.M, hi = on && kn <= a.M;
  const cpx<T> w = on ? load_c(a.tw + k) : cpx<T>{T(1), T(0)};
  const int rowp = c * C - c * (c - 1) / 2;
  cpx<T>* Z = a.Z + ((size_t)blockIdx.y * C + c) * h;
  cpx<T> zk{T(0), T(0)}, zn{T(0), T(0)};
  if (lo) {
    zk = load_c(Z + k);
    zn = load_c(Z + (kn & (h - 1)));
  }
  // with c = conj Z[h-k], e = Z[k] + c, o = Z[k] - c, p = W^k o: X[k] = (e - i p) / 2 and
  // X[h-k] = conj(e + i p) / 2
  {
    const cpx<T> e{zk.x + zn.x, zk.y - zn.y}, o{zk.x - zn.x, zk.y + zn.y}, p = fft::cmul(w, o);
    store_c(s_lo + c * kDiagK + tx, {T(0.5) * (e.x + p.y), T(0.5) * (e.y - p.x)});
    if (hi) store_c(s_hi + c * kDiagK + tx, {T(0.5) * (e.x - p.y), -T(0.5) * (e.y + p.x)});
  }
  __syncthreads();
  cpx<T> a0{T(0), T(0)}, a1{T(0), T(0)};
  if (lo) {
#pragma unroll 5
    for (int l = 0; l < C; ++l) {
      const int p = l >= c ? rowp + (l - c) : l * C - l * (l - 1) / 2 + (c - l);
      const T* Ap = a.A + (size_t)p * a.n_freq;
      const T v = __ldg(Ap + k);
      const cpx<T> b = load_c(s_lo + l * kDiagK + tx);
      a0.x += v * b.x;
      a0.y += v * b.y;
      if (hi) {
        const T vn = __ldg(Ap + kn);
        const cpx<T> bn = load_c(s_hi + l * kDiagK + tx);
        a1.x += vn * bn.x;
        a1.y += vn * bn.y;
      }
    }
  }
  if (on) {
    // with c = conj a1, e = a0 + c, o = a0 - c, p = conj(W^k) o: Z[k] = e + i p, Z[h-k] = conj(e - i p)
    const cpx<T> e{a0.x + a1.x, a0.y - a1.y}, o{a0.x - a1.x, a0.y + a1.y}, p = fft::cmul(fft::conj(w), o);
    store_c(Z + k, {e.x - p.y, e.y + p.x});
    if (k != 0 && kn != k) store_c(Z + kn, {e.x + p.y, p.x - e.y});
  }
}

// Radix 4 up to 1024 points (256 threads), radix 8 above in FP32 and four butterflies of radix
// 4 a thread in float64 (whose radix-8 butterflies would not fit the registers)
LinePlan line_passes(int n, int precision) {
  LinePlan m;
  m.N = n;
  m.R = precision == GP_FP32 && n > 1024 ? 8 : 4;
  m.NB = n <= 1024 ? 1 : (m.R == 8 ? (n <= 4096 ? 1 : 2) : 4);
  int rest = n;
  while (rest % m.R == 0) {
    rest /= m.R;
    ++m.np;
  }
  m.r0 = rest;
  const size_t bytes = (precision == GP_FP32 ? 8 : 16) * (size_t)n;
  if (n < 4 || n / (m.R * m.NB) > 512 || bytes > (size_t(128) << 10)) m.N = 0;
  return m;
}
bool passes_fit(int n, int precision) { return line_passes(n, precision).N > 0; }
constexpr long long kMaxLine = 1 << 17;   // eight blocks of 8192 points (512 threads)

// the pass twiddles W_{Ns R}^{r k}, [r - 1][k], k < Ns, as interleaved (re, im)
std::vector<double> line_tables(const LinePlan& m) {
  std::vector<double> t;
  int ns = m.r0;
  for (int p = 0; p < m.np; ++p, ns *= m.R)
    if (ns > 1)
      for (int r = 1; r < m.R; ++r)
        for (int k = 0; k < ns; ++k) {
          const double th = 6.283185307179586476925286766559 * (double)(r * k) / ((double)ns * m.R);
          t.push_back(std::cos(th));
          t.push_back(-std::sin(th));
        }
  return t;
}

// Blocks a transform is split over: the fewest that give kLineBlocks blocks (every block reads
// the whole sequence, so S multiplies the reads from L2), more where the sub-transform would
// not fit a block, fewer where it would drop below 64 points.  40 FP32 sequences of 32768 (N = 1e5, four
// right-hand sides) take S = 4, 36 us forward and 34 back; with S = 8 30 and 29; 40 of 16384 S = 4, 19
// and 18 (S = 8 19 and 16); 80 of 32768 S = 4, 50 and 47.
int line_split(const Plan& plan, int CR) {
  const int h = (int)(plan.geom.nf / 2);
  int S = 1;
  while (S < kMaxSplit && (!passes_fit(h / S, plan.precision) || ((long long)CR * S < kLineBlocks && h / S >= 128)))
    S *= 2;
  return S;
}

template <typename T, bool INV, int S>
void line_launch(const LineArgs<T>& a, const LinePlan& m, int CR, cudaStream_t st) {
  const size_t smem = sizeof(cpx<T>) * ((size_t)a.N + a.N / (sizeof(T) == 4 ? 16 : 8) + 1);
  void (*k)(LineArgs<T>) = nullptr;
  if constexpr (sizeof(T) == 4)
    k = m.R == 4 ? k_line<T, INV, S, 4, 1> : (m.NB == 1 ? k_line<T, INV, S, 8, 1> : k_line<T, INV, S, 8, 2>);
  else
    k = m.NB == 1 ? k_line<T, INV, S, 4, 1> : k_line<T, INV, S, 4, 4>;
  GPN_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k<<<dim3(S, (unsigned)CR), m.N / (m.R * m.NB), smem, st>>>(a);
}

template <typename T, bool INV>
void line_run(Plan& plan, int R, cudaStream_t st) {
  const int CR = plan.geom.C * R, S = line_split(plan, CR);
  int si = 0;
  while ((1 << si) < S) ++si;
  LineArgs<T> a{};
  a.h = (int)(plan.geom.nf / 2);
  a.in = (const cpx<T>*)(INV ? plan.line_spec : plan.grid);
  a.out = (cpx<T>*)(INV ? plan.grid_out : plan.line_spec);
  a.tw = (const cpx<T>*)plan.line_tw;
  a.ptw = (const cpx<T>*)plan.line_ptw[si];
  const LinePlan m = line_passes(a.h / S, plan.precision);
  a.N = m.N;
  a.r0 = m.r0;
  a.np = m.np;
  a.lo = plan.line_lo / 2;
  a.hi = (plan.line_hi + 1) / 2;
  switch (S) {
    case 1: line_launch<T, INV, 1>(a, m, CR, st); break;
    case 2: line_launch<T, INV, 2>(a, m, CR, st); break;
    case 4: line_launch<T, INV, 4>(a, m, CR, st); break;
    default: line_launch<T, INV, 8>(a, m, CR, st);
  }
  GPN_CUDA(cudaGetLastError());
}

template <typename T>
void line_diag_impl(Plan& plan, int R, cudaStream_t st) {
  LineDiagArgs<T> a{};
  a.Z = (cpx<T>*)plan.line_spec;
  a.tw = (const cpx<T>*)plan.line_tw;
  a.A = (const T*)plan.a_tensor;
  a.n_freq = plan.n_freq;
  a.h = (int)(plan.geom.nf / 2);
  a.M = (int)plan.geom.M;
  a.C = plan.geom.C;
  const size_t smem = 2 * sizeof(cpx<T>) * kDiagK * a.C;
  k_line_diag<T><<<dim3((unsigned)(a.h / 2 / kDiagK + 1), (unsigned)R), dim3(kDiagK, a.C), smem, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

template <typename T>
void* upload(Plan& plan, const std::vector<double>& v) {
  const std::vector<T> f(v.begin(), v.end());
  void* dst = plan.alloc(std::max<size_t>(f.size(), 2) * sizeof(T));
  if (!f.empty()) GPN_CUDA(cudaMemcpy(dst, f.data(), f.size() * sizeof(T), cudaMemcpyHostToDevice));
  return dst;
}

}  // namespace

// Plans whose transforms run here: nf = 2^a whose eighth fits a block.  `pitch`: complex
// values per channel of the buffer the spectra can live in.
bool line_supported(int d, long long nf, int precision, long long pitch) {
  if (d != 1 || nf < 64 || (nf & (nf - 1)) || nf / 2 > pitch || precision == GP_DF64) return false;
  return nf <= kMaxLine && passes_fit((int)(nf / 2 / kMaxSplit), precision);
}

// the cells the points reach and, with the spare tables, where each cell's points start (every 1-D
// plan spreads with k_spread1d)
void line_points_setup(Plan& plan, cudaStream_t st) {
  const PointSet& ps = plan.pts;
  const int n = (int)ps.n, cells = (int)plan.geom.nf;
  int first = 0, last = 0;
  GPN_CUDA(cudaMemcpyAsync(&first, ps.cell0[0], sizeof(int), cudaMemcpyDeviceToHost, st));
  GPN_CUDA(cudaMemcpyAsync(&last, ps.cell0[0] + n - 1, sizeof(int), cudaMemcpyDeviceToHost, st));
  if (plan.spare) {
    plan.line_start = (int*)plan.alloc(sizeof(int) * ((size_t)cells + 1));
    k_line_start<<<blocks_for(cells + 1, 256), 256, 0, st>>>(ps.cell0[0], n, cells, plan.line_start);
    GPN_CUDA(cudaGetLastError());
  }
  GPN_CUDA(cudaStreamSynchronize(st));
  plan.line_cell0 = first;
  plan.line_cell1 = last + plan.geom.width;   // at most nf: no support leaves the grid
  size_t sums = 0;   // the most that the parts of any number of right-hand sides hold
  for (int R = 1; R <= plan.grid_rhs; ++R) {
    const size_t parts = spread_parts(plan, R);
    if (parts > 1) sums = std::max(sums, parts * R * plan.geom.C * (plan.line_cell1 - plan.line_cell0));
  }
  if (sums) plan.line_scratch = plan.alloc(sums * plan.real_size);
}

// twiddles, pass tables of every split, and the cells the transforms read and write (the
// support of any point or query of the plan's box); spec: [r][C][nf/2] complex
void line_setup(Plan& plan, void* spec) {
  const Hyper& h = plan.h;
  plan.line = true;
  plan.line_spec = spec;
  const double half = 0.5 * (h.box_hi[0] - h.box_lo[0]) * h.nf * h.dw;
  const long long lo = (long long)std::ceil(0.5 * h.nf - half - 0.5 * h.width) - 1;
  const long long hi = (long long)std::ceil(0.5 * h.nf + half - 0.5 * h.width) + h.width + 1;
  plan.line_lo = (int)std::max(0ll, lo);
  plan.line_hi = (int)std::min(h.nf, hi);
  std::vector<double> tw;
  for (long long k = 0; k < h.nf; ++k) {
    const double th = 6.283185307179586476925286766559 * (double)k / (double)h.nf;
    tw.push_back(std::cos(th));
    tw.push_back(-std::sin(th));
  }
  const bool f32 = plan.precision == GP_FP32;
  plan.line_tw = f32 ? upload<float>(plan, tw) : upload<double>(plan, tw);
  for (int si = 0; si < 4; ++si) {
    const int n = (int)(h.nf / 2) >> si;
    if (n < 4 || !passes_fit(n, plan.precision)) continue;
    const std::vector<double> t = line_tables(line_passes(n, plan.precision));
    plan.line_ptw[si] = f32 ? upload<float>(plan, t) : upload<double>(plan, t);
  }
}

void line_forward(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    line_run<float, false>(plan, R, st);
  else
    line_run<double, false>(plan, R, st);
}

void line_inverse(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    line_run<float, true>(plan, R, st);
  else
    line_run<double, true>(plan, R, st);
}

void line_diag(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    line_diag_impl<float>(plan, R, st);
  else
    line_diag_impl<double>(plan, R, st);
}

void launch_spread1d(Plan& plan, const double* alpha, const int* perm, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    spread_impl<float>(plan, alpha, perm, R, st);
  else
    spread_impl<double>(plan, alpha, perm, R, st);
}

void launch_interp1d(Plan& plan, const PointSet& ps, const double* alpha, double shift, double* out, const int* perm,
                     int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    interp_impl<float>(plan, ps, alpha, shift, out, perm, R, st);
  else
    interp_impl<double>(plan, ps, alpha, shift, out, perm, R, st);
}

}  // namespace gpn
