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
// a group of 32 cells are one contiguous run.
#include <algorithm>
#include <cmath>
#include <type_traits>
#include <vector>

#include "fft_mixed.h"
#include "kernels.h"

namespace gpn {

namespace {

using fft::cpx;
using fft::MixedPlan;

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

// ---- spreading --------------------------------------------------------------------------

constexpr int kCells = 32;      // cells a block
constexpr int kWarps = 8;

template <typename T>
struct Spread1Args {
  const int* l0;
  const T* xi;
  const T* psi;          // tabulated kernel values [n][width] (null: evaluate)
  const T* wk;           // [n][C]
  const int* start;      // per cell group: first point reaching it, first point past it
  int group0;            // first cell group launched
  const double* alpha;   // sorted order, n x R column-major
  long long n;
  T* grid;               // [r][k][nf]
  long long nf;
  int width, C;
  T beta, inv_halfw;
};

template <typename T>
__host__ __device__ constexpr int wk_pitch(int nc) {
  return (nc + (int)(16 / sizeof(T)) - 1) / (int)(16 / sizeof(T)) * (int)(16 / sizeof(T));
}

// One block takes 32 cells, one a lane, and all channels in registers (NC = C, or 32 with the
// extra ones zero).  The points that reach the group are dealt to the warps in runs of up to 32:
// a warp tabulates its run's kernel values and w_k alpha in shared memory, then walks the run,
// every lane adding the point's value at its cell.  The warps' sums are added in order (results
// do not depend on scheduling) and every cell is written, so the grid needs no clearing.
template <typename T, int NC>
__global__ void __launch_bounds__(32 * kWarps) k_spread1d(Spread1Args<T> a) {
  constexpr int WP = wk_pitch<T>(NC), VW = (int)(16 / sizeof(T));
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  const int W = a.width, PS = W | 1, C = a.C, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, r = blockIdx.y;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* s_wk = reinterpret_cast<T*>(smem_raw) + warp * 32 * (WP + PS + VW);   // [32][WP], then [32][PS]
  T* s_psi = s_wk + 32 * WP;
  const int g = a.group0 + blockIdx.x, cell = g * kCells + lane;
  const int p0 = a.start[2 * g], p1 = a.start[2 * g + 1];
  // points a warp takes at a time: an even share, so that short runs occupy every warp
  const int run = min(32, (p1 - p0 + kWarps - 1) / kWarps);
  const double* alpha = a.alpha + (size_t)r * a.n;
  T acc[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) acc[k] = T(0);
  for (int q0 = p0 + warp * run; q0 < p1; q0 += kWarps * run) {
    const int m = min(run, p1 - q0);
    const int l0 = lane < m ? a.l0[q0 + lane] : 0;
    for (int i = lane; i < m * W; i += 32) {
      const int q = i / W, j = i - q * W;
      s_psi[q * PS + j] =
          a.psi ? a.psi[(size_t)q0 * W + i] : psi_at<T>(j, a.xi[q0 + q], a.beta, a.inv_halfw);
    }
    for (int i = lane; i < m * C; i += 32) {
      const int q = i / C, k = i - q * C;
      s_wk[q * WP + k] = a.wk[(size_t)q0 * C + i] * (T)alpha[q0 + q];
    }
    if (C < NC)
      for (int q = lane; q < m; q += 32)
        for (int k = C; k < NC; ++k) s_wk[q * WP + k] = T(0);
    __syncwarp();
    for (int q = 0; q < m; ++q) {
      const int j = cell - __shfl_sync(0xffffffffu, l0, q);
      const T ps = (unsigned)j < (unsigned)W ? s_psi[q * PS + j] : T(0);
      T w[WP];
#pragma unroll
      for (int v = 0; v < WP / VW; ++v) {
        const V u = reinterpret_cast<const V*>(s_wk + q * WP)[v];
        w[VW * v] = u.x;
        w[VW * v + 1] = u.y;
        if constexpr (VW == 4) {
          w[VW * v + 2] = u.z;
          w[VW * v + 3] = u.w;
        }
      }
#pragma unroll
      for (int k = 0; k < NC; ++k) acc[k] += ps * w[k];
    }
    __syncwarp();
  }
  __syncthreads();
  T* red = reinterpret_cast<T*>(smem_raw);   // [warp][NC][32]
#pragma unroll
  for (int k = 0; k < NC; ++k) red[(warp * NC + k) * 32 + lane] = acc[k];
  __syncthreads();
  if (cell >= a.nf) return;
  for (int k = warp; k < C; k += kWarps) {
    T s = T(0);
#pragma unroll
    for (int q = 0; q < kWarps; ++q) s += red[(q * NC + k) * 32 + lane];
    a.grid[((size_t)r * C + k) * a.nf + cell] = s;
  }
}

template <typename T, int NC>
void spread_launch(const Spread1Args<T>& a, dim3 grid, cudaStream_t st) {
  const size_t tab = 32 * (size_t)(wk_pitch<T>(NC) + (a.width | 1) + (int)(16 / sizeof(T)));
  const size_t smem = kWarps * sizeof(T) * std::max<size_t>(tab, 32 * NC);
  GPN_CUDA(cudaFuncSetAttribute(k_spread1d<T, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_spread1d<T, NC><<<grid, 32 * kWarps, smem, st>>>(a);
}

template <typename T, int NC>
void spread_dispatch(const Spread1Args<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 16) {
    spread_launch<T, 32>(a, grid, st);
  } else {
    if (a.C == NC)
      spread_launch<T, NC>(a, grid, st);
    else
      spread_dispatch<T, NC + 1>(a, grid, st);
  }
}

template <typename T>
void spread_impl(Plan& plan, const double* alpha_sorted, int R, cudaStream_t st) {
  const GridGeom& g = plan.geom;
  const PointSet& ps = plan.pts;
  Spread1Args<T> a{ps.cell0[0],      (const T*)ps.xi[0], (const T*)ps.psi[0], (const T*)ps.wk,
                   plan.line_start,  plan.line_group0,   alpha_sorted,        ps.n,
                   (T*)plan.grid,    g.nf,               g.width,             g.C,
                   es_beta_arg<T>(g.beta), (T)(2.0 / g.width)};
  spread_dispatch<T, 1>(a, dim3((unsigned)plan.line_groups, (unsigned)R), st);
  GPN_CUDA(cudaGetLastError());
}

// start[2g], start[2g + 1]: the sorted points whose support meets cells [32 g, 32 g + 32)
__global__ void k_line_start(const int* __restrict__ l0, int n, int W, int groups, int* __restrict__ start) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= 2 * groups) return;
  const int c = (i / 2) * kCells + (i % 2 ? kCells : 1 - W);   // first l0 past the group / reaching it
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (l0[mid] < c)
      lo = mid + 1;
    else
      hi = mid;
  }
  start[i] = lo;
}

// ---- interpolation ------------------------------------------------------------------------

template <typename T>
struct Interp1Args {
  const int* l0;
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
  if (a.alpha) res += (a.dcorr ? a.shift + a.dcorr[p] : a.shift) * a.alpha[(size_t)r * a.n + p];
  a.out[(size_t)r * a.n + p] = res;
}

// Sixteen lanes a point: lane j holds psi(j), lane k sums channel k (k + 16, ...) over the W
// cells; the products w_k beta_k are added in float64.  For point sets too small to fill the
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
  double part = 0.0;
  for (int k0 = 0; k0 < a.C; k0 += 16) {
    const bool in = k0 + gl < a.C;
    const int k = in ? k0 + gl : a.C - 1;
    const T* gk = g + (size_t)k * a.nf;
    T s = T(0);
#pragma unroll 4
    for (int j = 0; j < W; ++j) s += __shfl_sync(0xffffffffu, pj, j, 16) * __ldg(gk + j);
    if (in) part += (double)(a.wk[q * a.C + k] * s);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o, 16);
  if (on && gl == 0) finish_point(a, p, r, part);
}

// A thread a point, NC = C channels in registers (32 with the extra ones unused): neighbouring
// points read neighbouring cells.
template <typename T, int NC>
__global__ void __launch_bounds__(128) k_interp1d(Interp1Args<T> a) {
  const long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int r = blockIdx.y, W = a.width, C = NC <= 16 ? NC : a.C;
  if (p >= a.n) return;
  const T* g = a.grid + (size_t)r * C * a.nf + a.l0[p];
  const T x = a.xi[p];
  T acc[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) acc[k] = T(0);
  for (int j = 0; j < W; ++j) {
    const T ps = a.psi ? a.psi[p * W + j] : psi_at<T>(j, x, a.beta, a.inv_halfw);
#pragma unroll
    for (int k = 0; k < NC; ++k)
      if (NC <= 16 || k < C) acc[k] += ps * __ldg(g + (size_t)k * a.nf + j);
  }
  double res = 0.0;
#pragma unroll
  for (int k = 0; k < NC; ++k)
    if (NC <= 16 || k < C) res += (double)a.wk[p * C + k] * (double)acc[k];
  finish_point(a, p, r, res);
}

template <typename T, int NC>
void interp_dispatch(const Interp1Args<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 16) {
    k_interp1d<T, 32><<<grid, 128, 0, st>>>(a);
  } else {
    if (a.C == NC)
      k_interp1d<T, NC><<<grid, 128, 0, st>>>(a);
    else
      interp_dispatch<T, NC + 1>(a, grid, st);
  }
}

template <typename T>
void interp_impl(Plan& plan, const PointSet& ps, const double* alpha_sorted, double shift, double* out_sorted, int R,
                 cudaStream_t st) {
  const GridGeom& g = plan.geom;
  Interp1Args<T> a{ps.cell0[0],
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
                   alpha_sorted,
                   shift,
                   (&ps == &plan.pts) ? plan.dcorr : nullptr,
                   out_sorted};
  // a thread a point once the points fill half of the chip's threads (152 SMs x 1024)
  if (ps.n * R >= 152ll * 1024)
    interp_dispatch<T, 1>(a, dim3((unsigned)((ps.n + 127) / 128), (unsigned)R), st);
  else
    k_interp1d_lanes<T><<<dim3((unsigned)((ps.n + 7) / 8), (unsigned)R), 128, 0, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

// ---- transforms -----------------------------------------------------------------------------

// threads a block: 128 registers a thread in FP32, 255 in float64
template <typename T>
constexpr int kLineThreads = sizeof(T) == 4 ? 512 : 256;
constexpr int kMaxSplit = 8;
// blocks of a launch: at most four an SM
constexpr int kLineBlocks = 4 * 152;

template <typename T>
struct LineArgs {
  const cpx<T>* in;      // forward: grid rows as pairs [cr][h]; inverse: spectra [cr][h]
  cpx<T>* out;
  const cpx<T>* tw;      // exp(-2 pi i k / nf), k < nf
  const cpx<T>* ptw;     // pass twiddles of the h / S point transform
  MixedPlan m;
  int h;
  int lo, hi;            // pairs of the row that hold data or are read by the interpolation
};

// a * exp(-+ 2 pi i q / 4)
template <bool INV, typename T>
__device__ __forceinline__ cpx<T> quarter_turns(cpx<T> a, int q) {
  if (q & 1) a = fft::rot90<INV>(a);
  return q & 2 ? cpx<T>{-a.x, -a.y} : a;
}

template <bool INV, bool HELD, typename T, typename In, typename Out, typename Sync>
__device__ __forceinline__ void line_pass(int R, int N, int J, int Ns, int jl, const cpx<T>* tw, In in, Out out,
                                          Sync sync) {
  switch (R) {
    case 16: fft::mixed_pass<16, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 8: fft::mixed_pass<8, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 4: fft::mixed_pass<4, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    default: fft::mixed_pass<2, INV, HELD>(N, J, Ns, jl, tw, in, out, sync);
  }
}

// blockIdx = (output residue q, channel and right-hand side)
template <typename T, bool INV, int S>
__global__ void __launch_bounds__(kLineThreads<T>, 1) k_line(LineArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.m.N, J = a.m.J, jl = threadIdx.x, q = blockIdx.x;
  const cpx<T>* src = a.in + (size_t)blockIdx.y * a.h;
  cpx<T>* dst = a.out + (size_t)blockIdx.y * a.h;
  auto twid = [&](int i) {
    cpx<T> w = load_c(a.tw + i);
    if (INV) w.y = -w.y;
    return w;
  };
  auto at = [&](int j) {
    return INV || (j >= a.lo && j < a.hi) ? load_c(src + j) : cpx<T>{T(0), T(0)};
  };
  const cpx<T> w8 = S == 8 ? twid(q * (a.h / 4)) : cpx<T>{T(1), T(0)};   // W_8^q
  auto sums = [&](int n) -> cpx<T> {
    if constexpr (S == 1) return at(n);
    cpx<T> z[S], u;
#pragma unroll
    for (int i = 0; i < S; ++i) z[i] = at(n + i * N);
    // W_S^{i q}: the halves pair up with the sign (-1)^q, the quarters with quarter turns
#pragma unroll
    for (int i = 0; i < S / 2; ++i) z[i] = q & 1 ? z[i] - z[i + S / 2] : z[i] + z[i + S / 2];
    if constexpr (S == 2) u = z[0];
    if constexpr (S == 4) u = z[0] + quarter_turns<INV>(z[1], q & 3);
    if constexpr (S == 8) {
      const cpx<T> u0 = z[0] + quarter_turns<INV>(z[2], q & 3), u1 = z[1] + quarter_turns<INV>(z[3], q & 3);
      u = u0 + (q & 1 ? fft::cmul(u1, w8) : quarter_turns<INV>(u1, q / 2));
    }
    return q == 0 ? u : fft::cmul(u, twid(2 * n * q));
  };
  auto put = [&](int k, cpx<T> v) {
    const int j = q + S * k;
    if (!INV || (j >= a.lo && j < a.hi)) store_c(dst + j, v);
  };
  line_pass<INV, false, T>(a.m.R[0], N, J, 1, jl, a.ptw, sums, [&](int n, cpx<T> v) { store_c(s + n, v); }, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int p = 1; p + 1 < a.m.np; ++p) {
    line_pass<INV, true, T>(a.m.R[p], N, J, ns, jl, a.ptw + a.m.tw[p], [&](int n) { return load_c(s + n); },
                            [&](int n, cpx<T> v) { store_c(s + n, v); }, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[p];
  }
  if (a.m.np == 1) {
    for (int n = jl; n < N; n += blockDim.x) put(n, load_c(s + n));
    return;
  }
  line_pass<INV, false, T>(a.m.R[a.m.np - 1], N, J, ns, jl, a.ptw + a.m.tw[a.m.np - 1],
                           [&](int n) { return load_c(s + n); }, put, [] {});
}

// ---- step 3 on the pairs (k, h - k) -----------------------------------------------------------

constexpr int kDiagK = 16;   // pairs a block

template <typename T>
struct LineDiagArgs {
  cpx<T>* Z;             // [r][C][h], in place
  const cpx<T>* tw;      // exp(-2 pi i k / nf)
  const T* A;            // packed upper triangle [p][f], f = 0..M
  long long n_freq;
  int h, M, C, R;
};

// blockDim = (kDiagK pairs, C channels)
template <typename T>
__global__ void __launch_bounds__(1024) k_line_diag(LineDiagArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s_lo = reinterpret_cast<cpx<T>*>(smem_raw);   // [C][kDiagK]: X[k]
  const int C = a.C, tx = threadIdx.x, c = threadIdx.y, h = a.h;
  cpx<T>* s_hi = s_lo + C * kDiagK;                     // X[h - k]
  const int k = blockIdx.x * kDiagK + tx, kn = h - k;
  const bool on = k <= h / 2, lo = on && k <= a.M, hi = on && kn <= a.M;
  const cpx<T> w = on ? load_c(a.tw + k) : cpx<T>{T(1), T(0)}, wn{-w.x, w.y};   // W_nf^{h-k} = -conj W_nf^k
  const int rowp = c * C - c * (c - 1) / 2;
  for (int r = 0; r < a.R; ++r) {
    cpx<T>* Z = a.Z + ((size_t)r * C + c) * h;
    cpx<T> zk{T(0), T(0)}, zn{T(0), T(0)};
    if (lo) {
      zk = load_c(Z + k);
      zn = load_c(Z + (kn & (h - 1)));
    }
    store_c(s_lo + c * kDiagK + tx, fft::r2c_split(zk, zn, w));
    if (hi) store_c(s_hi + c * kDiagK + tx, fft::r2c_split(zn, zk, wn));
    __syncthreads();
    cpx<T> a0{T(0), T(0)}, a1{T(0), T(0)};
    if (lo) {
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
      store_c(Z + k, fft::c2r_merge(a0, a1, w));
      if (k != 0 && kn != k) store_c(Z + kn, fft::c2r_merge(a1, a0, wn));
    }
    __syncthreads();   // the next right-hand side refills the modes
  }
}

// the passes of the h / S point transform: radix 8 (16 for long ones) and a last 4 or 2
MixedPlan line_passes(int n) {
  MixedPlan m;
  m.N = n;
  const int big = n >= 2048 ? 16 : 8;
  for (int rest = n; rest > 1; ++m.np) {
    int r = big;
    while (rest % r) r /= 2;
    if (m.np == fft::kMaxPasses) return MixedPlan{};
    m.R[m.np] = r;
    rest /= r;
  }
  m.J = std::max(1, n / big);
  int off = 0, ns = 1;
  for (int p = 0; p < m.np; ++p) {
    m.tw[p] = off;
    if (p > 0) off += (m.R[p] - 1) * ns;
    ns *= m.R[p];
  }
  return m;
}

template <typename T>
bool passes_fit(int n) {
  const MixedPlan m = line_passes(n);
  return m.np > 0 && m.J <= kLineThreads<T> && sizeof(cpx<T>) * (size_t)n <= (size_t(128) << 10);
}
bool passes_fit(int n, int precision) { return precision == GP_FP32 ? passes_fit<float>(n) : passes_fit<double>(n); }

// blocks a transform is split over: as many as keep the launch within kLineBlocks, more where
// the sub-transform would not fit a block, fewer where it would drop below 64 points
int line_split(const Plan& plan, int CR) {
  const int h = (int)(plan.geom.nf / 2);
  int S = kMaxSplit;
  while (S > 1 && ((long long)CR * S > kLineBlocks || h / S < 64) && passes_fit(h / (S / 2), plan.precision)) S /= 2;
  return S;
}

template <typename T, bool INV, int S>
void line_launch(const LineArgs<T>& a, int CR, cudaStream_t st) {
  const size_t smem = sizeof(cpx<T>) * (size_t)a.m.N;
  GPN_CUDA(cudaFuncSetAttribute(k_line<T, INV, S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_line<T, INV, S><<<dim3(S, (unsigned)CR), a.m.J, smem, st>>>(a);
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
  a.m = line_passes(a.h / S);
  a.lo = plan.line_lo / 2;
  a.hi = (plan.line_hi + 1) / 2;
  switch (S) {
    case 1: line_launch<T, INV, 1>(a, CR, st); break;
    case 2: line_launch<T, INV, 2>(a, CR, st); break;
    case 4: line_launch<T, INV, 4>(a, CR, st); break;
    default: line_launch<T, INV, 8>(a, CR, st);
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
  a.R = R;
  const size_t smem = 2 * sizeof(cpx<T>) * kDiagK * a.C;
  k_line_diag<T><<<(unsigned)(a.h / 2 / kDiagK + 1), dim3(kDiagK, a.C), smem, st>>>(a);
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
  if (d != 1 || nf < 16 || (nf & (nf - 1)) || nf / 2 > pitch || precision == GP_DF64) return false;
  return nf / 2 / kMaxSplit <= (1 << 20) && passes_fit((int)std::max<long long>(2, nf / 2 / kMaxSplit), precision);
}

// the cell groups the points reach (every 1-D plan spreads with k_spread1d)
void line_points_setup(Plan& plan, cudaStream_t st) {
  const PointSet& ps = plan.pts;
  const int n = (int)ps.n, W = plan.geom.width;
  int first = 0, last = 0;
  GPN_CUDA(cudaMemcpyAsync(&first, ps.cell0[0], sizeof(int), cudaMemcpyDeviceToHost, st));
  GPN_CUDA(cudaMemcpyAsync(&last, ps.cell0[0] + n - 1, sizeof(int), cudaMemcpyDeviceToHost, st));
  const int groups = (int)((plan.geom.nf + kCells - 1) / kCells);
  plan.line_start = (int*)plan.alloc(sizeof(int) * 2 * groups);
  k_line_start<<<blocks_for(2 * groups, 256), 256, 0, st>>>(ps.cell0[0], n, W, groups, plan.line_start);
  GPN_CUDA(cudaGetLastError());
  GPN_CUDA(cudaStreamSynchronize(st));
  plan.line_group0 = first / kCells;
  plan.line_groups = (last + W - 1) / kCells - plan.line_group0 + 1;
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
    if (n < 2 || !passes_fit(n, plan.precision)) continue;
    const std::vector<double> t = fft::mixed_tables(line_passes(n));
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

void launch_spread1d(Plan& plan, const double* alpha_sorted, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    spread_impl<float>(plan, alpha_sorted, R, st);
  else
    spread_impl<double>(plan, alpha_sorted, R, st);
}

void launch_interp1d(Plan& plan, const PointSet& ps, const double* alpha_sorted, double shift, double* out_sorted,
                     int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    interp_impl<float>(plan, ps, alpha_sorted, shift, out_sorted, R, st);
  else
    interp_impl<double>(plan, ps, alpha_sorted, shift, out_sorted, R, st);
}

}  // namespace gpn
