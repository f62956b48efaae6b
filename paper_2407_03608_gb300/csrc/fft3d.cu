// 3-D transforms over the occupied box of the fine grid (d = 3): the uniform FFTs of the
// type-1 and type-2 NUFFTs (App. D) with step (3) of Sec. 4.2 between them.
//
// The points' support covers only a box of E_0 x E_1 x E_2 cells of the nf^3 grid (about
// 0.53 nf per axis on the uniform unit cube), and only the modes |n_a| <= M are used (the
// restriction Pi of Sec. 3.4).  So the grids hold the box alone, every axis is transformed
// on its own, from its E input cells to its 2M + 1 modes (or back), and the rest of the
// nf^3 grid is never touched.  The channels are innermost in every array: a cell or mode
// of all channels is contiguous, so a transform along any axis runs over adjacent columns,
// and the x transform takes two real channels as one complex sequence.
//   grid  [r][z][y][x][Cp]     box cells (real), Cp = C rounded up to even
//   X1    [r][z][y][q]         after the x transform, q = m_x Cs + k, pitch Qp
//   X2    [r][z][n_y + M][q]   after y
//   X3    [r][n_z + M][n_y + M][q]   after z: the mode box step 3 works on in place
// and the same arrays backwards.  X1 and X3 share one buffer, X2 is the other.  The spectra
// are made of 16-byte elements: one complex float64 value, or in FP32 those of two adjacent
// channels, {re, re, im, im} (Cs = C rounded up to even), which the passes transform with
// packed instructions (fft_mixed.h).
//
// Each block transforms B adjacent columns through shared memory, [n][b] with b fastest,
// with the mixed-radix passes of fft_mixed.h: the first pass reads its inputs straight from
// global memory and the last one writes straight to it, so a three-pass length exchanges
// through shared memory twice.
//
// Bound: issue and the shared-memory exchanges (FP32), the FP64 pipe (float64).  Forward /
// inverse, ms, full-cube cuFFT -> here: FP32 nf 512 C 8 6.18 / 6.28 -> 1.87 / 1.92, FP32 nf 864
// C 10 59.4 / 64.0 -> 14.7 / 14.3, float64 nf 256 C 7 12.0 / 12.1 -> 4.17 / 4.08.  The first of
// these with radices up to 16 and 128 registers 2.10, with four adjacent columns instead of
// eight 1.95, with scalar instead of packed FP32 arithmetic 2.47.  Step 3: 1.56 -> 0.72 ms with
// A', 42.6 -> 7.44 memory-lean (nf 864).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "fft_mixed.h"
#include "kernels.h"

namespace gpn {

namespace {

using fft::cv;
using fft::f2;
using fft::MixedPlan;
using fft::Span;
using fft::vset;

// threads of a transform block: two blocks an SM keep 64 registers a thread (up to 10 elements
// of four words in flight)
constexpr int kBoxThreads = 512;

// the element type of a plan's arithmetic, and the values it holds
template <typename T>
using VecOf = typename std::conditional<sizeof(T) == 4, f2, double>::type;
template <typename T>
constexpr int kLanes = fft::Elem<VecOf<T>>::lanes;

template <typename V>
__device__ __forceinline__ cv<V> load_v(const cv<V>* p) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  cv<V> v;
  memcpy(&v, &u, 16);
  return v;
}
template <typename V>
__device__ __forceinline__ void store_v(cv<V>* p, cv<V> v) {
  float4 u;
  memcpy(&u, &v, 16);
  *reinterpret_cast<float4*>(p) = u;
}
template <typename V>
__device__ __forceinline__ cv<V> zero_v() {
  return {vset<V>(0), vset<V>(0)};
}

template <typename V>
struct BoxColsArgs {
  const cv<V>* in;
  cv<V>* out;
  const cv<V>* tw;
  MixedPlan m;
  int B;                                  // columns a block
  int lo, ext, M;                         // box window along the axis, modes
  long long in_r, in_o, in_s;             // strides: right-hand side, outer index, element
  long long out_r, out_o, out_s;
};

// Transforms along y and z.  Forward: box cells [lo, lo + ext) to the modes -M..M; inverse
// back.  blockIdx = (column group, outer index, right-hand side).
template <typename V, bool INV>
__global__ void __launch_bounds__(kBoxThreads, 2) k_box_cols(BoxColsArgs<V> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int B = a.B, jl = threadIdx.x / B, b = threadIdx.x - jl * B, N = a.m.N, J = a.m.J, M = a.M;
  const long long col = blockIdx.x * (long long)B + b;
  const cv<V>* src = a.in + blockIdx.z * a.in_r + blockIdx.y * a.in_o + col;
  cv<V>* dst = a.out + blockIdx.z * a.out_r + blockIdx.y * a.out_o + col;
  cv<V>* sb = reinterpret_cast<cv<V>*>(smem_raw) + b;
  // element n of the sequence: its place along the axis in the window or mode array, or -1
  auto window = [&](int n) { return (unsigned)(n - a.lo) < (unsigned)a.ext ? n - a.lo : -1; };
  auto mode = [&](int n) { return n <= M ? n + M : (n >= N - M ? n - N + M : -1); };
  const long long in_s = a.in_s, out_s = a.out_s;
  const auto from_smem = [&](int n) { return load_v(sb + n * B); };
  const auto to_smem = [&](int n, cv<V> v) { store_v(sb + n * B, v); };
  fft::mixed_pass_any<INV, false, V>(
      a.m.R[0], N, J, jl, Span<V>{1, 0, a.tw},
      [&](int n) {
        const int i = INV ? mode(n) : window(n);
        return i >= 0 ? load_v(src + i * in_s) : zero_v<V>();
      },
      to_smem, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int p = 1; p + 1 < a.m.np; ++p) {
    fft::mixed_pass_any<INV, true, V>(a.m.R[p], N, J, jl, Span<V>{ns, a.m.inv_ns[p], a.tw + a.m.tw[p]}, from_smem,
                                      to_smem, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[p];
  }
  const int p = a.m.np - 1;
  fft::mixed_pass_any<INV, false, V>(
      a.m.R[p], N, J, jl, Span<V>{ns, a.m.inv_ns[p], a.tw + a.m.tw[p]}, from_smem,
      [&](int n, cv<V> v) {
        const int i = INV ? window(n) : mode(n);
        if (i >= 0) store_v(dst + i * out_s, v);
      },
      [] {});
}

template <typename T>
struct BoxRowsArgs {
  T* grid;                // box cells [row][x][Cp]
  cv<VecOf<T>>* X;        // [row][q / lanes]
  const cv<VecOf<T>>* tw;
  MixedPlan m;
  int YB, PB;             // rows and channel groups a block
  int pitch;              // shared-memory elements per sequence element
  int lo, ext, M;
  int Cp;                 // channel pitch of the grid
  int Ce;                 // elements per mode of X (Cs / lanes)
  long long Qe;           // elements per row of X
  long long nrows;        // E_0 E_1
};

// the channels of group p at a cell: 2 lanes of them, the first half as real parts, the second
// (zero past the pitch) as imaginary parts
template <typename T>
__device__ __forceinline__ cv<VecOf<T>> load_group(const T* cell, int p, int Cp) {
  using V = VecOf<T>;
  constexpr int L = kLanes<T>;
  const V* c = reinterpret_cast<const V*>(cell) + 2 * p;
  return {c[0], (2 * p + 1) * L < Cp ? c[1] : vset<V>(0)};
}
template <typename T>
__device__ __forceinline__ void store_group(T* cell, int p, int Cp, cv<VecOf<T>> v) {
  using V = VecOf<T>;
  constexpr int L = kLanes<T>;
  V* c = reinterpret_cast<V*>(cell) + 2 * p;
  c[0] = v.x;
  if ((2 * p + 1) * L < Cp) c[1] = v.y;
}

// Transforms along x.  A sequence takes channel group p of one row: with lanes L, channels
// 2 L p .. as real parts and the L after them as imaginary parts, so that one complex transform
// Z serves 2 L real rows: X_a[m] = (Z[m] + conj Z[N-m]) / 2 for the first channels and
// X_b[m] = (Z[m] - conj Z[N-m]) / 2i for the second.  blockIdx = (row group, channel groups).
template <typename T>
__global__ void __launch_bounds__(kBoxThreads, 2) k_box_rows_fwd(BoxRowsArgs<T> a) {
  using V = VecOf<T>;
  constexpr int L = kLanes<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cv<V>* s = reinterpret_cast<cv<V>*>(smem_raw);
  const int PB = a.PB, B = a.YB * PB, jl = threadIdx.x / B, b = threadIdx.x - jl * B;
  const int N = a.m.N, J = a.m.J, M = a.M, Cp = a.Cp, pitch = a.pitch;
  const int yb = b / PB, p = blockIdx.y * PB + (b - yb * PB);
  const long long row = blockIdx.x * (long long)a.YB + yb;
  const bool valid = row < a.nrows && 2 * p * L < Cp;
  const T* src = a.grid + (valid ? row : 0) * (long long)a.ext * Cp;
  cv<V>* sb = s + b;
  const auto from_smem = [&](int n) { return load_v(sb + n * pitch); };
  const auto to_smem = [&](int n, cv<V> v) { store_v(sb + n * pitch, v); };
  fft::mixed_pass_any<false, false, V>(
      a.m.R[0], N, J, jl, Span<V>{1, 0, a.tw},
      [&](int n) {
        const int i = n - a.lo;
        return valid && (unsigned)i < (unsigned)a.ext ? load_group(src + i * Cp, p, Cp) : zero_v<V>();
      },
      to_smem, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int q = 1; q < a.m.np; ++q) {
    fft::mixed_pass_any<false, true, V>(a.m.R[q], N, J, jl, Span<V>{ns, a.m.inv_ns[q], a.tw + a.m.tw[q]}, from_smem,
                                        to_smem, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[q];
  }
  // the two elements of every (row, mode, group), groups fastest: adjacent in X
  const int m0 = threadIdx.x / PB, pc = threadIdx.x - m0 * PB, mstep = blockDim.x / PB;
  const int e = 2 * (blockIdx.y * PB + pc);
  if (e >= a.Ce || m0 >= mstep) return;
  const V half = vset<V>(T(0.5));
  for (int y = 0; y < a.YB; ++y) {
    const long long r = blockIdx.x * (long long)a.YB + y;
    if (r >= a.nrows) break;
    cv<V>* dst = a.X + r * a.Qe + e;
    const cv<V>* sy = s + y * PB + pc;
    for (int m = m0; m <= M; m += mstep) {
      const cv<V> z = load_v(sy + m * pitch), w = load_v(sy + (m == 0 ? 0 : N - m) * pitch);
      cv<V>* o = dst + m * a.Ce;
      store_v(o, {fft::vmul(half, fft::vadd(z.x, w.x)), fft::vmul(half, fft::vsub(z.y, w.y))});
      if (e + 1 < a.Ce) store_v(o + 1, {fft::vmul(half, fft::vadd(z.y, w.y)), fft::vmul(half, fft::vsub(w.x, z.x))});
    }
  }
}

// The inverse: Z[m] = X_a[m] + i X_b[m], Z[N-m] = conj(X_a[m]) + i conj(X_b[m]) (the imaginary
// part of mode 0 is dropped, as a C2R transform does), zero elsewhere.
template <typename T>
__global__ void __launch_bounds__(kBoxThreads, 2) k_box_rows_inv(BoxRowsArgs<T> a) {
  using V = VecOf<T>;
  constexpr int L = kLanes<T>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cv<V>* s = reinterpret_cast<cv<V>*>(smem_raw);
  const int PB = a.PB, B = a.YB * PB, jl = threadIdx.x / B, b = threadIdx.x - jl * B;
  const int N = a.m.N, J = a.m.J, M = a.M, Cp = a.Cp, pitch = a.pitch;
  const int yb = b / PB, p = blockIdx.y * PB + (b - yb * PB);
  const long long row = blockIdx.x * (long long)a.YB + yb;
  const bool valid = row < a.nrows && 2 * p * L < Cp, two = 2 * p + 1 < a.Ce;
  const cv<V>* src = a.X + (valid ? row : 0) * a.Qe + 2 * p;
  T* dst = a.grid + (valid ? row : 0) * (long long)a.ext * Cp;
  cv<V>* sb = s + b;
  const auto from_smem = [&](int n) { return load_v(sb + n * pitch); };
  const auto to_smem = [&](int n, cv<V> v) { store_v(sb + n * pitch, v); };
  fft::mixed_pass_any<true, false, V>(
      a.m.R[0], N, J, jl, Span<V>{1, 0, a.tw},
      [&](int n) {
        const bool up = n <= M, down = n >= N - M;
        if (!valid || !(up || down)) return zero_v<V>();
        const cv<V>* x = src + (up ? n : N - n) * a.Ce;
        const cv<V> u = load_v(x), v = two ? load_v(x + 1) : zero_v<V>();
        if (n == 0) return cv<V>{u.x, v.x};
        return up ? fft::add_turn<true>(v, u) : cv<V>{fft::vadd(u.x, v.y), fft::vsub(v.x, u.y)};
      },
      to_smem, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int q = 1; q + 1 < a.m.np; ++q) {
    fft::mixed_pass_any<true, true, V>(a.m.R[q], N, J, jl, Span<V>{ns, a.m.inv_ns[q], a.tw + a.m.tw[q]}, from_smem,
                                       to_smem, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[q];
  }
  const int q = a.m.np - 1;
  fft::mixed_pass_any<true, false, V>(
      a.m.R[q], N, J, jl, Span<V>{ns, a.m.inv_ns[q], a.tw + a.m.tw[q]}, from_smem,
      [&](int n, cv<V> v) {
        const int i = n - a.lo;
        if (valid && (unsigned)i < (unsigned)a.ext) store_group(dst + i * Cp, p, Cp, v);
      },
      [] {});
}

// ---- step 3 on the mode box -----------------------------------------------------------
//
// a_k[n] = sum_l A'_kl[|n|] b_l[n], in place.  A' depends on |n_z|, |n_y| and m_x alone, so a
// block takes (|n_z|, |n_y|) and kDiagM adjacent m_x, and serves the four (two, one) sign
// combinations from the same entries: the tensor is stored on the octant only, a quarter of
// the half box.  The block stages the channel-innermost data in shared memory by coalesced
// copies (odd pitch: the threads' rows fall in different banks); thread t owns m_x = m0 + t.
//
// LEAN: the entries are formed in registers from the per-dimension factors,
// A'_kl = sum_j g_kj g_lj with g_kj = sqrt(v~_j) E'_kj(|n_z|) E'_kj(|n_y|) E'_kj(m_x): C(C+1)/2
// multiply-adds a node, shared by the four sign combinations and every right-hand side (the
// form that applies g_j twice to each spectrum value costs 4 C a node for each of them).

constexpr int kDiagM = 64;

template <typename T>
struct BoxDiagArgs {
  cv<VecOf<T>>* X;        // [r][nz + M][ny + M][q / lanes]
  const T* A;             // [pair][|nz|][|ny|][m], the octant (null: lean)
  const T* tab;           // lean factors [j][m][CP]
  const T* sqv;           // sqrt(v~_j)
  long long n_freq;       // (M + 1)^3
  long long Qe, xr;       // row pitch and right-hand-side stride of X, in elements
  int M, C, CP, J, R;
};

// channel k of the elements at e: its real and imaginary part
template <typename T>
__device__ __forceinline__ T& re_of(cv<VecOf<T>>* e, int k) {
  return reinterpret_cast<T*>(e)[kLanes<T> == 2 ? k / 2 * 4 + k % 2 : 2 * k];
}
template <typename T>
__device__ __forceinline__ T& im_of(cv<VecOf<T>>* e, int k) {
  return reinterpret_cast<T*>(e)[kLanes<T> == 2 ? k / 2 * 4 + 2 + k % 2 : 2 * k + 1];
}

// rows of the sign combinations of (|nz|, |ny|); returns their number
__device__ __forceinline__ int sign_rows(int nz, int ny, int M, long long (&row)[4]) {
  int c = 0;
  const long long W = 2 * M + 1;
#pragma unroll
  for (int sz = 0; sz < 2; ++sz)
#pragma unroll
    for (int sy = 0; sy < 2; ++sy)
      if (!(sz && nz == 0) && !(sy && ny == 0)) row[c++] = (long long)(sz ? M - nz : M + nz) * W + (sy ? M - ny : M + ny);
  return c;
}

// the shared factors sqrt(v~_j) E'_kj(|nz|) E'_kj(|ny|) of a block, [j][CP]
template <typename T>
__device__ __forceinline__ void stage_factors(const BoxDiagArgs<T>& a, T* s_em, int nz, int ny) {
  const long long Mp = a.M + 1;
  for (int i = threadIdx.x; i < a.J * a.CP; i += blockDim.x) {
    const int j = i / a.CP, k = i - j * a.CP;
    s_em[i] = k < a.C ? a.sqv[j] * a.tab[(j * Mp + nz) * a.CP + k] * a.tab[(j * Mp + ny) * a.CP + k] : T(0);
  }
}

// NC = C <= 12 channels: the C(C+1)/2 entries in registers
template <typename T, int NC, bool LEAN>
__global__ void __launch_bounds__(kDiagM) k_box_diag(BoxDiagArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using V = VecOf<T>;
  constexpr int L = kLanes<T>, NE = (NC + L - 1) / L, PITCH = NE | 1, NP = NC * (NC + 1) / 2;
  cv<V>* s_b = reinterpret_cast<cv<V>*>(smem_raw);             // [4][kDiagM][PITCH]
  const int ny = blockIdx.y, nz = blockIdx.z, m0 = blockIdx.x * kDiagM, t = threadIdx.x;
  const int Mp = a.M + 1, nm = min(kDiagM, Mp - m0);
  long long row[4];
  const int ns = sign_rows(nz, ny, a.M, row);
  T av[NP];
  const int m = m0 + min(t, nm - 1);
  if constexpr (LEAN) {
    constexpr int VW = (int)(16 / sizeof(T)), CP = (NC + VW - 1) / VW * VW;
    T* s_em = reinterpret_cast<T*>(s_b);                       // staged before the data
    stage_factors(a, s_em, nz, ny);
    __syncthreads();
#pragma unroll
    for (int p = 0; p < NP; ++p) av[p] = T(0);
    const T* tm = a.tab + (size_t)m * CP;
    const size_t jstride = (size_t)Mp * CP;
#pragma unroll 1
    for (int j = 0; j < a.J; ++j) {
      T g[CP];
#pragma unroll
      for (int v = 0; v < CP / VW; ++v) {
        if constexpr (VW == 4) {
          const float4 x = __ldg(reinterpret_cast<const float4*>(tm + j * jstride) + v);
          const float4 e = reinterpret_cast<const float4*>(s_em + j * CP)[v];
          g[4 * v] = x.x * e.x, g[4 * v + 1] = x.y * e.y, g[4 * v + 2] = x.z * e.z, g[4 * v + 3] = x.w * e.w;
        } else {
          const double2 x = __ldg(reinterpret_cast<const double2*>(tm + j * jstride) + v);
          const double2 e = reinterpret_cast<const double2*>(s_em + j * CP)[v];
          g[2 * v] = x.x * e.x, g[2 * v + 1] = x.y * e.y;
        }
      }
      int p = 0;
#pragma unroll
      for (int k = 0; k < NC; ++k)
#pragma unroll
        for (int l = k; l < NC; ++l, ++p) av[p] += g[k] * g[l];
    }
    __syncthreads();
  } else {
    const T* Am = a.A + ((size_t)nz * Mp + ny) * Mp + m;
#pragma unroll
    for (int p = 0; p < NP; ++p) av[p] = __ldg(Am + (size_t)p * a.n_freq);
  }
  for (int r = 0; r < a.R; ++r) {
    cv<V>* Xr = a.X + r * a.xr + (size_t)m0 * NE;
    for (int s = 0; s < ns; ++s)
      for (int e = t; e < nm * NE; e += kDiagM) {
        const int f = e / NE;
        store_v(s_b + (s * kDiagM + f) * PITCH + (e - f * NE), load_v(Xr + row[s] * a.Qe + e));
      }
    __syncthreads();
    if (t < nm) {
      for (int s = 0; s < ns; ++s) {
        cv<V>* sb = s_b + (s * kDiagM + t) * PITCH;
        T bx[NE * L], by[NE * L];
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          cv<V> v = load_v(sb + e);
#pragma unroll
          for (int l = 0; l < L; ++l) {
            bx[e * L + l] = re_of<T>(&v, l);
            by[e * L + l] = im_of<T>(&v, l);
          }
        }
#pragma unroll
        for (int e = 0; e < NE; ++e) {
          cv<V> o = zero_v<V>();
#pragma unroll
          for (int q = 0; q < L; ++q) {
            const int k = e * L + q;
            T ox = T(0), oy = T(0);
            if (k < NC) {
#pragma unroll
              for (int l = 0; l < NC; ++l) {
                const int lo = k < l ? k : l, hi = k < l ? l : k;
                const T w = av[lo * NC - lo * (lo - 1) / 2 + (hi - lo)];
                ox += w * bx[l];
                oy += w * by[l];
              }
            }
            re_of<T>(&o, q) = ox;
            im_of<T>(&o, q) = oy;
          }
          store_v(sb + e, o);
        }
      }
    }
    __syncthreads();
    for (int s = 0; s < ns; ++s)
      for (int e = t; e < nm * NE; e += kDiagM) {
        const int f = e / NE;
        store_v(Xr + row[s] * a.Qe + e, load_v(s_b + (s * kDiagM + f) * PITCH + (e - f * NE)));
      }
    __syncthreads();
  }
}

// more channels: inputs and sums in shared memory, the entries read (or the nodes walked)
// once per sign combination
template <typename T, bool LEAN>
__global__ void __launch_bounds__(kDiagM) k_box_diag_wide(BoxDiagArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using V = VecOf<T>;
  constexpr int L = kLanes<T>;
  const int C = a.C, E = (C + L - 1) / L, PITCH = E | 1;
  cv<V>* s_b = reinterpret_cast<cv<V>*>(smem_raw);             // [kDiagM][PITCH]
  cv<V>* s_o = s_b + kDiagM * PITCH;                           // [kDiagM][PITCH]
  T* s_em = reinterpret_cast<T*>(s_o + kDiagM * PITCH);        // lean: [J][CP]
  const int ny = blockIdx.y, nz = blockIdx.z, m0 = blockIdx.x * kDiagM, t = threadIdx.x;
  const int Mp = a.M + 1, nm = min(kDiagM, Mp - m0);
  long long row[4];
  const int ns = sign_rows(nz, ny, a.M, row);
  if constexpr (LEAN) stage_factors(a, s_em, nz, ny);
  const int m = m0 + min(t, nm - 1);
  for (int r = 0; r < a.R; ++r)
    for (int s = 0; s < ns; ++s) {
      cv<V>* Xs = a.X + r * a.xr + row[s] * a.Qe + (size_t)m0 * E;
      for (int e = t; e < nm * E; e += kDiagM) store_v(s_b + e / E * PITCH + e % E, load_v(Xs + e));
      __syncthreads();
      cv<V>* b = s_b + t * PITCH;
      cv<V>* o = s_o + t * PITCH;
      if (t < nm) {
        for (int e = 0; e < E; ++e) store_v(o + e, zero_v<V>());
        if constexpr (LEAN) {
          for (int j = 0; j < a.J; ++j) {
            const T* tm = a.tab + ((size_t)j * Mp + m) * a.CP;
            const T* em = s_em + j * a.CP;
            T ux = T(0), uy = T(0);
            for (int l = 0; l < C; ++l) {
              const T g = em[l] * __ldg(tm + l);
              ux += g * re_of<T>(b, l);
              uy += g * im_of<T>(b, l);
            }
            for (int k = 0; k < C; ++k) {
              const T g = em[k] * __ldg(tm + k);
              re_of<T>(o, k) += g * ux;
              im_of<T>(o, k) += g * uy;
            }
          }
        } else {
          const T* Am = a.A + ((size_t)nz * Mp + ny) * Mp + m;
          for (int k = 0; k < C; ++k) {
            T vx = T(0), vy = T(0);
            for (int l = 0; l < C; ++l) {
              const int lo = k < l ? k : l, hi = k < l ? l : k;
              const T w = __ldg(Am + (size_t)(lo * C - lo * (lo - 1) / 2 + (hi - lo)) * a.n_freq);
              vx += w * re_of<T>(b, l);
              vy += w * im_of<T>(b, l);
            }
            re_of<T>(o, k) = vx;
            im_of<T>(o, k) = vy;
          }
        }
      }
      __syncthreads();
      for (int e = t; e < nm * E; e += kDiagM) store_v(Xs + e, load_v(s_o + e / E * PITCH + e % E));
      __syncthreads();
    }
}

// Memory-lean FP32 with more channels: NB >= C of them.  A node's factors and the sums stay in
// registers, the inputs in shared memory; the factors come as vectors.  (With factors, inputs and
// sums re-read from memory at every node, 15 channels at nf 128 took 1015 us, 25 channels 1520; the
// full-grid kernel 295 and 1001; this one 200 and 250.  Float64 keeps the form above: 3970 us
// against 6290 on the full grid.)
template <int NB>
__global__ void __launch_bounds__(kDiagM) k_box_lean_wide(BoxDiagArgs<float> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int C = a.C, E = (C + 1) / 2, PITCH = E | 1;
  cv<f2>* s_b = reinterpret_cast<cv<f2>*>(smem_raw);           // [kDiagM][PITCH]
  float* s_em = reinterpret_cast<float*>(s_b + kDiagM * PITCH);   // [J][CP]
  const int ny = blockIdx.y, nz = blockIdx.z, m0 = blockIdx.x * kDiagM, t = threadIdx.x;
  const int Mp = a.M + 1, nm = min(kDiagM, Mp - m0);
  long long row[4];
  const int ns = sign_rows(nz, ny, a.M, row);
  stage_factors(a, s_em, nz, ny);
  const float* tm = a.tab + (size_t)(m0 + min(t, nm - 1)) * a.CP;
  const size_t jstride = (size_t)Mp * a.CP;
  cv<f2>* b = s_b + t * PITCH;
  for (int r = 0; r < a.R; ++r)
    for (int s = 0; s < ns; ++s) {
      cv<f2>* Xs = a.X + r * a.xr + row[s] * a.Qe + (size_t)m0 * E;
      for (int e = t; e < nm * E; e += kDiagM) store_v(s_b + e / E * PITCH + e % E, load_v(Xs + e));
      __syncthreads();
      if (t < nm) {
        float ox[NB], oy[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) ox[k] = oy[k] = 0.f;
#pragma unroll 1
        for (int j = 0; j < a.J; ++j) {
          float g[NB];
#pragma unroll
          for (int v = 0; v < NB / 4; ++v) {
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), e = x;
            if (4 * v < a.CP) {
              x = __ldg(reinterpret_cast<const float4*>(tm + j * jstride) + v);
              e = reinterpret_cast<const float4*>(s_em + j * a.CP)[v];
            }
            g[4 * v] = x.x * e.x, g[4 * v + 1] = x.y * e.y, g[4 * v + 2] = x.z * e.z, g[4 * v + 3] = x.w * e.w;
          }
          float ux = 0.f, uy = 0.f;
#pragma unroll
          for (int e = 0; e < NB / 2; ++e)
            if (e < E) {
              const cv<f2> v = load_v(b + e);
              ux += g[2 * e] * v.x.x + g[2 * e + 1] * v.x.y;
              uy += g[2 * e] * v.y.x + g[2 * e + 1] * v.y.y;
            }
#pragma unroll
          for (int k = 0; k < NB; ++k) {
            ox[k] += g[k] * ux;
            oy[k] += g[k] * uy;
          }
        }
#pragma unroll
        for (int e = 0; e < NB / 2; ++e)
          if (e < E) store_v(b + e, cv<f2>{{ox[2 * e], ox[2 * e + 1]}, {oy[2 * e], oy[2 * e + 1]}});
      }
      __syncthreads();
      for (int e = t; e < nm * E; e += kDiagM) store_v(Xs + e, load_v(s_b + e / E * PITCH + e % E));
      __syncthreads();
    }
}

void lean_wide_launch(const BoxDiagArgs<float>& a, dim3 grid, cudaStream_t st) {
  void (*k)(BoxDiagArgs<float>) = a.C <= 16 ? k_box_lean_wide<16> : a.C <= 24 ? k_box_lean_wide<24> : k_box_lean_wide<32>;
  const size_t smem = 16 * kDiagM * (size_t)((a.C + 1) / 2 | 1) + sizeof(float) * a.J * a.CP;
  GPN_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k<<<grid, kDiagM, smem, st>>>(a);
}

template <typename T, int NC, bool LEAN>
void diag_launch(const BoxDiagArgs<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 12 && LEAN && sizeof(T) == 4) {
    lean_wide_launch(a, grid, st);
  } else if constexpr (NC > 12) {
    const int E = (a.C + kLanes<T> - 1) / kLanes<T>;
    const size_t smem = 2 * 16 * kDiagM * (E | 1) + (LEAN ? sizeof(T) * a.J * a.CP : 0);
    GPN_CUDA(cudaFuncSetAttribute(k_box_diag_wide<T, LEAN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_box_diag_wide<T, LEAN><<<grid, kDiagM, smem, st>>>(a);
  } else if (a.C == NC) {
    const int E = (NC + kLanes<T> - 1) / kLanes<T>;
    const size_t smem = std::max<size_t>(4 * 16 * kDiagM * (E | 1), LEAN ? sizeof(T) * a.J * a.CP : 0);
    GPN_CUDA(cudaFuncSetAttribute(k_box_diag<T, NC, LEAN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_box_diag<T, NC, LEAN><<<grid, kDiagM, smem, st>>>(a);
  } else {
    diag_launch<T, NC + 1, LEAN>(a, grid, st);
  }
}

template <typename T>
void box_diag_impl(Plan& plan, int R, cudaStream_t st) {
  const Box3& bx = plan.box3;
  BoxDiagArgs<T> a{};
  a.X = (cv<VecOf<T>>*)bx.buf_a;
  a.A = (const T*)plan.a_tensor;
  a.tab = (const T*)plan.lean_tab;
  a.sqv = (const T*)plan.lean_sqv;
  a.n_freq = plan.n_freq;
  a.Qe = bx.Qe;
  a.xr = bx.size_a;
  a.M = (int)plan.geom.M;
  a.C = plan.geom.C;
  a.CP = plan.lean_cp;
  a.J = plan.lean_J;
  a.R = R;
  const dim3 grid((unsigned)((a.M + kDiagM) / kDiagM), (unsigned)(a.M + 1), (unsigned)(a.M + 1));
  if (plan.lean)
    diag_launch<T, 1, true>(a, grid, st);
  else
    diag_launch<T, 1, false>(a, grid, st);
  GPN_CUDA(cudaGetLastError());
}

template <typename T, bool INV>
void box_cols(Plan& plan, int axis, int R, cudaStream_t st) {
  using V = VecOf<T>;
  const Box3& bx = plan.box3;
  const long long W = 2 * plan.geom.M + 1, Qe = bx.Qe;
  BoxColsArgs<V> a{};
  a.tw = (const cv<V>*)bx.tw;
  a.m = bx.fft;
  a.B = bx.cols;
  a.lo = bx.lo[axis];
  a.ext = bx.ext[axis];
  a.M = (int)plan.geom.M;
  long long ncols, outer;
  // forward strides (the inverse swaps in and out): y takes buf_a [z][y][q] to buf_b
  // [z][ny][q]; z takes buf_b [z][(ny, q)] to buf_a [nz][(ny, q)]
  if (axis == 1) {
    ncols = Qe;
    outer = bx.ext[0];
    a.in_o = (long long)bx.ext[1] * Qe;
    a.out_o = W * Qe;
    a.in_s = a.out_s = Qe;
    a.in = (const cv<V>*)bx.buf_a;
    a.out = (cv<V>*)bx.buf_b;
    a.in_r = bx.size_a;
    a.out_r = bx.size_b;
  } else {
    ncols = W * Qe;
    outer = 1;
    a.in_s = a.out_s = W * Qe;
    a.in = (const cv<V>*)bx.buf_b;
    a.out = (cv<V>*)bx.buf_a;
    a.in_r = bx.size_b;
    a.out_r = bx.size_a;
  }
  if (INV) {
    const cv<V>* in = a.in;
    a.in = a.out;
    a.out = const_cast<cv<V>*>(in);
    std::swap(a.in_o, a.out_o);
    std::swap(a.in_r, a.out_r);
  }
  const size_t smem = 16 * (size_t)a.m.N * a.B;
  GPN_CUDA(cudaFuncSetAttribute(k_box_cols<V, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_box_cols<V, INV><<<dim3((unsigned)(ncols / a.B), (unsigned)outer, (unsigned)R), a.m.J * a.B, smem, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

template <typename T, bool INV>
void box_rows(Plan& plan, int R, cudaStream_t st) {
  const Box3& bx = plan.box3;
  BoxRowsArgs<T> a{};
  a.tw = (const cv<VecOf<T>>*)bx.tw;
  a.m = bx.fft;
  a.YB = bx.rows;
  a.PB = bx.groups;
  const int B = a.YB * a.PB;
  // an odd multiple of the channel groups: the mode-by-mode reads of the split spread over the banks
  a.pitch = a.YB % 2 ? B : B + a.PB;
  a.lo = bx.lo[2];
  a.ext = bx.ext[2];
  a.M = (int)plan.geom.M;
  a.Cp = bx.Cp;
  a.Ce = (plan.geom.C + kLanes<T> - 1) / kLanes<T>;
  a.Qe = bx.Qe;
  a.nrows = (long long)bx.ext[0] * bx.ext[1];
  const size_t smem = 16 * (size_t)a.m.N * a.pitch;
  void (*k)(BoxRowsArgs<T>) = INV ? k_box_rows_inv<T> : k_box_rows_fwd<T>;
  GPN_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int ngroups = (bx.Cp + 2 * kLanes<T> - 1) / (2 * kLanes<T>);
  const dim3 grid((unsigned)((a.nrows + a.YB - 1) / a.YB), (unsigned)((ngroups + a.PB - 1) / a.PB));
  for (int r = 0; r < R; ++r) {
    a.grid = (T*)(INV ? plan.grid_out : plan.grid) + (size_t)r * plan.view.rstride;
    a.X = (cv<VecOf<T>>*)bx.buf_a + (size_t)r * bx.size_a;
    k<<<grid, a.m.J * B, smem, st>>>(a);
  }
  GPN_CUDA(cudaGetLastError());
}

template <typename T>
void forward_impl(Plan& plan, int R, cudaStream_t st) {
  box_rows<T, false>(plan, R, st);
  box_cols<T, false>(plan, 1, R, st);
  box_cols<T, false>(plan, 0, R, st);
}
template <typename T>
void inverse_impl(Plan& plan, int R, cudaStream_t st) {
  box_cols<T, true>(plan, 0, R, st);
  box_cols<T, true>(plan, 1, R, st);
  box_rows<T, true>(plan, R, st);
}

}  // namespace

// every grid size the plan chooses itself; longer ones need more passes than kMaxPasses or more
// shared memory than a block has
bool box3_supported(int d, long long nf) { return d == 3 && nf <= 2048 && fft::mixed_plan((int)nf).np > 0; }

// The box (the cells the support of any point or query of the plan's box can cover, and one
// more on either side), the transform schedule, and the layout of the arrays.
void box3_layout(Plan& plan) {
  const Hyper& h = plan.h;
  Box3& bx = plan.box3;
  const int C = plan.geom.C;
  const double inv_h = h.nf * h.dw;
  for (int q = 0; q < 3; ++q) {
    const double half = 0.5 * (h.box_hi[q] - h.box_lo[q]) * inv_h;
    const long long lo = (long long)std::ceil(0.5 * h.nf - half - 0.5 * h.width) - 1;
    const long long hi = (long long)std::ceil(0.5 * h.nf + half - 0.5 * h.width) + h.width + 1;
    bx.lo[q] = (int)std::max(0ll, lo);
    bx.ext[q] = (int)(std::min(h.nf, hi) - bx.lo[q]);
  }
  bx.Cp = (C + 1) / 2 * 2;
  const int lanes = plan.precision == GP_FP32 ? 2 : 1;
  bx.Qe = ((h.M + 1) * ((C + lanes - 1) / lanes) + 7) / 8 * 8;
  bx.fft = fft::mixed_plan((int)h.nf);
  const int J = bx.fft.J, groups = (bx.Cp + 2 * lanes - 1) / (2 * lanes);
  bx.cols = 8;                                // 128-byte segments of adjacent columns
  while (bx.cols > 1 && bx.cols * J > kBoxThreads) bx.cols /= 2;
  bx.groups = std::max(1, std::min(groups, kBoxThreads / J));
  bx.rows = std::max(1, std::min(8 / bx.groups, kBoxThreads / (J * bx.groups)));
  const long long W = 2 * h.M + 1;
  bx.size_a = std::max((long long)bx.ext[0] * bx.ext[1], W * W) * bx.Qe;
  bx.size_b = (long long)bx.ext[0] * W * bx.Qe;
  GridView& v = plan.view;
  v.cstride = 1;
  for (int q = 0; q < 3; ++q) {
    v.lo[q] = bx.lo[q];
    v.ext[q] = bx.ext[q];
  }
  v.stride[2] = bx.Cp;
  v.stride[1] = v.stride[2] * bx.ext[2];
  v.stride[0] = v.stride[1] * bx.ext[1];
  v.rstride = v.stride[0] * bx.ext[0];
}

// the buffers of the spectra and the twiddle tables
void box3_setup(Plan& plan) {
  Box3& bx = plan.box3;
  const bool f32 = plan.precision == GP_FP32;
  bx.buf_a = plan.alloc(16 * bx.size_a * plan.grid_rhs);
  bx.buf_b = plan.alloc(16 * bx.size_b * plan.grid_rhs);
  const std::vector<double> t = fft::mixed_tables(bx.fft);
  bx.tw = plan.alloc(std::max<size_t>(t.size() / 2, 1) * 16);
  if (f32) {
    // each twiddle part twice, once per lane
    std::vector<float> f;
    for (double v : t) f.insert(f.end(), 2, (float)v);
    GPN_CUDA(cudaMemcpy(bx.tw, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
  } else {
    GPN_CUDA(cudaMemcpy(bx.tw, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
  }
}

void box3_forward(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    forward_impl<float>(plan, R, st);
  else
    forward_impl<double>(plan, R, st);
}

void box3_inverse(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    inverse_impl<float>(plan, R, st);
  else
    inverse_impl<double>(plan, R, st);
}

void box3_diag(Plan& plan, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    box_diag_impl<float>(plan, R, st);
  else
    box_diag_impl<double>(plan, R, st);
}

}  // namespace gpn
