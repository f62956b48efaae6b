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
//   X1    [r][z][y][q]         after the x transform, q = m_x C + k, pitch Qp
//   X2    [r][z][n_y + M][q]   after y
//   X3    [r][n_z + M][n_y + M][q]   after z: the mode box step 3 works on in place
// and the same arrays backwards.  X1 and X3 share one buffer, X2 is the other.
//
// Each block transforms B adjacent columns through shared memory, [n][b] with b fastest,
// with the mixed-radix passes of fft_mixed.h: the first pass reads its inputs straight from
// global memory and the last one writes straight to it, so a three-pass length exchanges
// through shared memory twice.
#include <algorithm>
#include <cmath>
#include <vector>

#include "fft_mixed.h"
#include "kernels.h"

namespace gpn {

namespace {

using fft::cpx;
using fft::MixedPlan;

// threads of a transform block: two blocks an SM keep 64 registers a thread in FP32 (16
// values in flight) and 128 in float64
template <typename T>
constexpr int kBoxThreads = sizeof(T) == 4 ? 512 : 256;

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

template <typename T>
struct BoxColsArgs {
  const cpx<T>* in;
  cpx<T>* out;
  const cpx<T>* tw;
  MixedPlan m;
  int B;                                  // columns a block
  int lo, ext, M;                         // box window along the axis, modes
  long long in_r, in_o, in_s;             // strides: right-hand side, outer index, element
  long long out_r, out_o, out_s;
};

// Transforms along y and z.  Forward: box cells [lo, lo + ext) to the modes -M..M; inverse
// back.  blockIdx = (column group, outer index, right-hand side).
template <typename T, bool INV>
__global__ void __launch_bounds__(kBoxThreads<T>, 2) k_box_cols(BoxColsArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s = reinterpret_cast<cpx<T>*>(smem_raw);
  const int B = a.B, b = threadIdx.x % B, jl = threadIdx.x / B, N = a.m.N, J = a.m.J, M = a.M;
  const long long col = blockIdx.x * (long long)B + b;
  const cpx<T>* src = a.in + blockIdx.z * a.in_r + blockIdx.y * a.in_o + col;
  cpx<T>* dst = a.out + blockIdx.z * a.out_r + blockIdx.y * a.out_o + col;
  cpx<T>* sb = s + b;
  // element n of the sequence: its place along the axis in the window or mode array, or -1
  auto window = [&](int n) { return (unsigned)(n - a.lo) < (unsigned)a.ext ? n - a.lo : -1; };
  auto mode = [&](int n) { return n <= M ? n + M : (n >= N - M ? n - N + M : -1); };
  const long long in_s = a.in_s, out_s = a.out_s;
  fft::mixed_pass_any<INV, false, T>(
      a.m.R[0], N, J, 1, jl, a.tw,
      [&](int n) {
        const int i = INV ? mode(n) : window(n);
        return i >= 0 ? load_c(src + i * in_s) : cpx<T>{T(0), T(0)};
      },
      [&](int n, cpx<T> v) { store_c(sb + n * B, v); }, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int p = 1; p + 1 < a.m.np; ++p) {
    fft::mixed_pass_any<INV, true, T>(
        a.m.R[p], N, J, ns, jl, a.tw + a.m.tw[p], [&](int n) { return load_c(sb + n * B); },
        [&](int n, cpx<T> v) { store_c(sb + n * B, v); }, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[p];
  }
  fft::mixed_pass_any<INV, false, T>(
      a.m.R[a.m.np - 1], N, J, ns, jl, a.tw + a.m.tw[a.m.np - 1], [&](int n) { return load_c(sb + n * B); },
      [&](int n, cpx<T> v) {
        const int i = INV ? window(n) : mode(n);
        if (i >= 0) store_c(dst + i * out_s, v);
      },
      [] {});
}

template <typename T>
struct BoxRowsArgs {
  T* grid;                // box cells [row][x][Cp]
  cpx<T>* X;              // [row][q]
  const cpx<T>* tw;
  MixedPlan m;
  int YB, PB;             // rows and channel pairs a block
  int pitch;              // shared-memory elements per sequence element
  int lo, ext, M;
  int C, Cp;
  long long Qp;
  long long nrows;        // R E_0 E_1
};

// Transforms along x.  A sequence is the pair of channels (2p, 2p + 1) of one row as real and
// imaginary part; its transform Z gives X_2p[m] = (Z[m] + conj Z[N-m]) / 2 and
// X_2p+1[m] = (Z[m] - conj Z[N-m]) / 2i.  blockIdx = (row group, pair group).
template <typename T>
__global__ void __launch_bounds__(kBoxThreads<T>, 2) k_box_rows_fwd(BoxRowsArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s = reinterpret_cast<cpx<T>*>(smem_raw);
  const int PB = a.PB, B = a.YB * PB, b = threadIdx.x % B, jl = threadIdx.x / B;
  const int N = a.m.N, J = a.m.J, M = a.M, P = a.Cp / 2;
  const int yb = b / PB, p = blockIdx.y * PB + (b - yb * PB);
  const long long row = blockIdx.x * (long long)a.YB + yb;
  const bool valid = row < a.nrows && p < P;
  const cpx<T>* src = reinterpret_cast<const cpx<T>*>(a.grid) + (valid ? row : 0) * (long long)a.ext * P + p;
  cpx<T>* sb = s + b;
  const int pitch = a.pitch;
  fft::mixed_pass_any<false, false, T>(
      a.m.R[0], N, J, 1, jl, a.tw,
      [&](int n) {
        const int i = n - a.lo;
        return valid && (unsigned)i < (unsigned)a.ext ? load_c(src + (long long)i * P) : cpx<T>{T(0), T(0)};
      },
      [&](int n, cpx<T> v) { store_c(sb + n * pitch, v); }, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int q = 1; q < a.m.np; ++q) {
    fft::mixed_pass_any<false, true, T>(
        a.m.R[q], N, J, ns, jl, a.tw + a.m.tw[q], [&](int n) { return load_c(sb + n * pitch); },
        [&](int n, cpx<T> v) { store_c(sb + n * pitch, v); }, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[q];
  }
  // the two channels of every (row, mode, pair), pairs fastest: adjacent in X
  const int pc = threadIdx.x % PB, m0 = threadIdx.x / PB, mstep = blockDim.x / PB;
  const int k = 2 * (blockIdx.y * PB + pc);
  if (k >= a.C || m0 >= mstep) return;
  for (int y = 0; y < a.YB; ++y) {
    const long long r = blockIdx.x * (long long)a.YB + y;
    if (r >= a.nrows) break;
    cpx<T>* dst = a.X + r * a.Qp + k;
    const cpx<T>* sy = s + y * PB + pc;
    for (int m = m0; m <= M; m += mstep) {
      const cpx<T> z = load_c(sy + m * pitch), w = load_c(sy + (m == 0 ? 0 : N - m) * pitch);
      cpx<T>* o = dst + (long long)m * a.C;
      store_c(o, {T(0.5) * (z.x + w.x), T(0.5) * (z.y - w.y)});
      if (k + 1 < a.C) store_c(o + 1, {T(0.5) * (z.y + w.y), T(0.5) * (w.x - z.x)});
    }
  }
}

// The inverse: Z[m] = X_2p[m] + i X_2p+1[m], Z[N-m] = conj(X_2p[m]) + i conj(X_2p+1[m]) (the
// imaginary part of mode 0 is dropped, as a C2R transform does), zero elsewhere.
template <typename T>
__global__ void __launch_bounds__(kBoxThreads<T>, 2) k_box_rows_inv(BoxRowsArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* s = reinterpret_cast<cpx<T>*>(smem_raw);
  const int PB = a.PB, B = a.YB * PB, b = threadIdx.x % B, jl = threadIdx.x / B;
  const int N = a.m.N, J = a.m.J, M = a.M, P = a.Cp / 2;
  const int yb = b / PB, p = blockIdx.y * PB + (b - yb * PB);
  const long long row = blockIdx.x * (long long)a.YB + yb;
  const bool valid = row < a.nrows && p < P, two = 2 * p + 1 < a.C;
  const cpx<T>* src = a.X + (valid ? row : 0) * a.Qp + 2 * p;
  cpx<T>* dst = reinterpret_cast<cpx<T>*>(a.grid) + (valid ? row : 0) * (long long)a.ext * P + p;
  cpx<T>* sb = s + b;
  const int pitch = a.pitch;
  fft::mixed_pass_any<true, false, T>(
      a.m.R[0], N, J, 1, jl, a.tw,
      [&](int n) {
        const bool up = n <= M, down = n >= N - M;
        if (!valid || !(up || down)) return cpx<T>{T(0), T(0)};
        const cpx<T>* x = src + (long long)(up ? n : N - n) * a.C;
        const cpx<T> u = load_c(x), v = two ? load_c(x + 1) : cpx<T>{T(0), T(0)};
        if (n == 0) return cpx<T>{u.x, v.x};
        return up ? cpx<T>{u.x - v.y, u.y + v.x} : cpx<T>{u.x + v.y, v.x - u.y};
      },
      [&](int n, cpx<T> v) { store_c(sb + n * pitch, v); }, [] {});
  __syncthreads();
  int ns = a.m.R[0];
  for (int q = 1; q + 1 < a.m.np; ++q) {
    fft::mixed_pass_any<true, true, T>(
        a.m.R[q], N, J, ns, jl, a.tw + a.m.tw[q], [&](int n) { return load_c(sb + n * pitch); },
        [&](int n, cpx<T> v) { store_c(sb + n * pitch, v); }, [] { __syncthreads(); });
    __syncthreads();
    ns *= a.m.R[q];
  }
  fft::mixed_pass_any<true, false, T>(
      a.m.R[a.m.np - 1], N, J, ns, jl, a.tw + a.m.tw[a.m.np - 1], [&](int n) { return load_c(sb + n * pitch); },
      [&](int n, cpx<T> v) {
        const int i = n - a.lo;
        if (valid && (unsigned)i < (unsigned)a.ext) store_c(dst + (long long)i * P, v);
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
  cpx<T>* X;              // [r][nz + M][ny + M][q]
  const T* A;             // [pair][|nz|][|ny|][m], the octant (null: lean)
  const T* tab;           // lean factors [j][m][CP]
  const T* sqv;           // sqrt(v~_j)
  long long n_freq;       // (M + 1)^3
  long long Qp, xr;       // row pitch and right-hand-side stride of X
  int M, C, CP, J, R;
};

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
  constexpr int PITCH = NC | 1, NP = NC * (NC + 1) / 2;
  cpx<T>* s_b = reinterpret_cast<cpx<T>*>(smem_raw);           // [4][kDiagM][PITCH]
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
    cpx<T>* Xr = a.X + r * a.xr + (size_t)m0 * NC;
    for (int s = 0; s < ns; ++s)
      for (int e = t; e < nm * NC; e += kDiagM) {
        const int f = e / NC;
        s_b[(s * kDiagM + f) * PITCH + (e - f * NC)] = load_c(Xr + row[s] * a.Qp + e);
      }
    __syncthreads();
    if (t < nm) {
      for (int s = 0; s < ns; ++s) {
        cpx<T>* sb = s_b + (s * kDiagM + t) * PITCH;
        cpx<T> b[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) b[k] = load_c(sb + k);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          cpx<T> o{T(0), T(0)};
#pragma unroll
          for (int l = 0; l < NC; ++l) {
            const int lo = k < l ? k : l, hi = k < l ? l : k;
            const T w = av[lo * NC - lo * (lo - 1) / 2 + (hi - lo)];
            o.x += w * b[l].x;
            o.y += w * b[l].y;
          }
          store_c(sb + k, o);
        }
      }
    }
    __syncthreads();
    for (int s = 0; s < ns; ++s)
      for (int e = t; e < nm * NC; e += kDiagM) {
        const int f = e / NC;
        store_c(Xr + row[s] * a.Qp + e, s_b[(s * kDiagM + f) * PITCH + (e - f * NC)]);
      }
    __syncthreads();
  }
}

// more channels: inputs and sums in shared memory, the entries read (or the nodes walked)
// once per sign combination
template <typename T, bool LEAN>
__global__ void __launch_bounds__(kDiagM) k_box_diag_wide(BoxDiagArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int C = a.C, PITCH = C | 1;
  cpx<T>* s_b = reinterpret_cast<cpx<T>*>(smem_raw);           // [kDiagM][PITCH]
  cpx<T>* s_o = s_b + kDiagM * PITCH;                          // [kDiagM][PITCH]
  T* s_em = reinterpret_cast<T*>(s_o + kDiagM * PITCH);        // lean: [J][CP]
  const int ny = blockIdx.y, nz = blockIdx.z, m0 = blockIdx.x * kDiagM, t = threadIdx.x;
  const int Mp = a.M + 1, nm = min(kDiagM, Mp - m0);
  long long row[4];
  const int ns = sign_rows(nz, ny, a.M, row);
  if constexpr (LEAN) stage_factors(a, s_em, nz, ny);
  const int m = m0 + min(t, nm - 1);
  for (int r = 0; r < a.R; ++r)
    for (int s = 0; s < ns; ++s) {
      cpx<T>* Xs = a.X + r * a.xr + row[s] * a.Qp + (size_t)m0 * C;
      for (int e = t; e < nm * C; e += kDiagM) s_b[e / C * PITCH + e % C] = load_c(Xs + e);
      __syncthreads();
      const cpx<T>* b = s_b + t * PITCH;
      cpx<T>* o = s_o + t * PITCH;
      if (t < nm) {
        if constexpr (LEAN) {
          for (int k = 0; k < C; ++k) store_c(o + k, {T(0), T(0)});
          for (int j = 0; j < a.J; ++j) {
            const T* tm = a.tab + ((size_t)j * Mp + m) * a.CP;
            const T* em = s_em + j * a.CP;
            cpx<T> u{T(0), T(0)};
            for (int l = 0; l < C; ++l) {
              const T g = em[l] * __ldg(tm + l);
              u.x += g * b[l].x;
              u.y += g * b[l].y;
            }
            for (int k = 0; k < C; ++k) {
              const T g = em[k] * __ldg(tm + k);
              o[k].x += g * u.x;
              o[k].y += g * u.y;
            }
          }
        } else {
          const T* Am = a.A + ((size_t)nz * Mp + ny) * Mp + m;
          for (int k = 0; k < C; ++k) {
            cpx<T> v{T(0), T(0)};
            for (int l = 0; l < C; ++l) {
              const int lo = k < l ? k : l, hi = k < l ? l : k;
              const T w = __ldg(Am + (size_t)(lo * C - lo * (lo - 1) / 2 + (hi - lo)) * a.n_freq);
              v.x += w * b[l].x;
              v.y += w * b[l].y;
            }
            store_c(o + k, v);
          }
        }
      }
      __syncthreads();
      for (int e = t; e < nm * C; e += kDiagM) store_c(Xs + e, s_o[e / C * PITCH + e % C]);
      __syncthreads();
    }
}

template <typename T, int NC, bool LEAN>
void diag_launch(const BoxDiagArgs<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 12) {
    const size_t smem = 2 * sizeof(cpx<T>) * kDiagM * (a.C | 1) + (LEAN ? sizeof(T) * a.J * a.CP : 0);
    GPN_CUDA(cudaFuncSetAttribute(k_box_diag_wide<T, LEAN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_box_diag_wide<T, LEAN><<<grid, kDiagM, smem, st>>>(a);
  } else if (a.C == NC) {
    const size_t smem =
        std::max<size_t>(4 * sizeof(cpx<T>) * kDiagM * (NC | 1), LEAN ? sizeof(T) * a.J * a.CP : 0);
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
  a.X = (cpx<T>*)bx.buf_a;
  a.A = (const T*)plan.a_tensor;
  a.tab = (const T*)plan.lean_tab;
  a.sqv = (const T*)plan.lean_sqv;
  a.n_freq = plan.n_freq;
  a.Qp = bx.Qp;
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
  const Box3& bx = plan.box3;
  const long long W = 2 * plan.geom.M + 1, Qp = bx.Qp;
  BoxColsArgs<T> a{};
  a.tw = (const cpx<T>*)bx.tw;
  a.m = bx.fft;
  a.B = bx.cols;
  a.lo = bx.lo[axis];
  a.ext = bx.ext[axis];
  a.M = (int)plan.geom.M;
  long long ncols, outer;
  // forward strides (the inverse swaps in and out): y takes buf_a [z][y][q] to buf_b
  // [z][ny][q]; z takes buf_b [z][(ny, q)] to buf_a [nz][(ny, q)]
  if (axis == 1) {
    ncols = Qp;
    outer = bx.ext[0];
    a.in_o = (long long)bx.ext[1] * Qp;
    a.out_o = W * Qp;
    a.in_s = a.out_s = Qp;
    a.in = (const cpx<T>*)bx.buf_a;
    a.out = (cpx<T>*)bx.buf_b;
    a.in_r = bx.size_a;
    a.out_r = bx.size_b;
  } else {
    ncols = W * Qp;
    outer = 1;
    a.in_s = a.out_s = W * Qp;
    a.in = (const cpx<T>*)bx.buf_b;
    a.out = (cpx<T>*)bx.buf_a;
    a.in_r = bx.size_b;
    a.out_r = bx.size_a;
  }
  if (INV) {
    const cpx<T>* in = a.in;
    a.in = a.out;
    a.out = const_cast<cpx<T>*>(in);
    std::swap(a.in_o, a.out_o);
    std::swap(a.in_r, a.out_r);
  }
  const size_t smem = sizeof(cpx<T>) * (size_t)a.m.N * a.B;
  GPN_CUDA(cudaFuncSetAttribute(k_box_cols<T, INV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_box_cols<T, INV><<<dim3((unsigned)(ncols / a.B), (unsigned)outer, (unsigned)R), a.m.J * a.B, smem, st>>>(a);
  GPN_CUDA(cudaGetLastError());
}

template <typename T, bool INV>
void box_rows(Plan& plan, int R, cudaStream_t st) {
  const Box3& bx = plan.box3;
  BoxRowsArgs<T> a{};
  a.tw = (const cpx<T>*)bx.tw;
  a.m = bx.fft;
  a.YB = bx.rows;
  a.PB = bx.pairs;
  const int B = a.YB * a.PB;
  // an odd multiple of the pair group: the mode-by-mode reads of the split spread over the banks
  a.pitch = a.YB % 2 ? B : B + a.PB;
  a.lo = bx.lo[2];
  a.ext = bx.ext[2];
  a.M = (int)plan.geom.M;
  a.C = plan.geom.C;
  a.Cp = bx.Cp;
  a.Qp = bx.Qp;
  a.nrows = (long long)bx.ext[0] * bx.ext[1];
  const size_t smem = sizeof(cpx<T>) * (size_t)a.m.N * a.pitch;
  void (*k)(BoxRowsArgs<T>) = INV ? k_box_rows_inv<T> : k_box_rows_fwd<T>;
  GPN_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const dim3 grid((unsigned)((a.nrows + a.YB - 1) / a.YB), (unsigned)((bx.Cp / 2 + a.PB - 1) / a.PB));
  for (int r = 0; r < R; ++r) {
    a.grid = (T*)(INV ? plan.grid_out : plan.grid) + (size_t)r * plan.view.rstride;
    a.X = (cpx<T>*)bx.buf_a + (size_t)r * bx.size_a;
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

bool box3_supported(int d, long long nf) { return d == 3 && nf <= 2048 && fft::mixed_plan((int)nf).np > 0; }

// The box (the cells the support of any point or query of the plan's box can cover, and one
// more on either side), the transform schedule and its tables, and the buffers.
void box3_setup(Plan& plan) {
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
  const bool f32 = plan.precision == GP_FP32;
  bx.Cp = (C + 1) / 2 * 2;
  bx.Qp = ((h.M + 1) * C + 15) / 16 * 16;
  bx.fft = fft::mixed_plan((int)h.nf);
  const int tmax = f32 ? kBoxThreads<float> : kBoxThreads<double>, J = bx.fft.J;
  bx.cols = f32 ? 16 : 8;                     // 128-byte segments of adjacent columns
  while (bx.cols > 1 && bx.cols * J > tmax) bx.cols /= 2;
  bx.pairs = std::max(1, std::min(bx.Cp / 2, tmax / J));
  bx.rows = std::max(1, std::min((f32 ? 16 : 8) / bx.pairs, tmax / (J * bx.pairs)));
  const long long W = 2 * h.M + 1;
  bx.size_a = std::max((long long)bx.ext[0] * bx.ext[1], W * W) * bx.Qp;
  bx.size_b = (long long)bx.ext[0] * W * bx.Qp;
  const size_t cs = 2 * plan.real_size;
  bx.buf_a = plan.alloc(cs * bx.size_a * plan.grid_rhs);
  bx.buf_b = plan.alloc(cs * bx.size_b * plan.grid_rhs);
  const std::vector<double> t = fft::mixed_tables(bx.fft);
  bx.tw = plan.alloc(t.size() * plan.real_size);
  if (f32) {
    const std::vector<float> f(t.begin(), t.end());
    GPN_CUDA(cudaMemcpy(bx.tw, f.data(), f.size() * sizeof(float), cudaMemcpyHostToDevice));
  } else {
    GPN_CUDA(cudaMemcpy(bx.tw, t.data(), t.size() * sizeof(double), cudaMemcpyHostToDevice));
  }
  // the grids' layout
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
