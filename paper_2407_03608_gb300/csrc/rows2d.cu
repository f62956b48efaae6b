// FP32 inverse row transforms of the pruned 2-D path (fft2d.cu has the layout and the other
// stages).
//
// Rows y and y + 1 are transformed as one sequence of packed values (fft_mixed.h): a thread
// holds 16 complex values of both rows, every sum and product is one packed instruction, one
// 16-byte shared-memory access moves a value of both rows, and they share the twiddles and the
// address arithmetic.  A block takes PK = 2 such pairs, so that what it reads of a mode's column
// is one whole 32-byte sector (with one pair, half of every sector is fetched for nothing:
// measured 1.58 ms against 1.19 ms at nf = 8192), and loads several pairs of modes before it
// uses the first, merging them into the half-length input on their way to shared memory.
//
// Bound: latency of the sector-sized column reads and the shared-memory exchanges (neither fewer
// instructions nor more warps helped further: radix 8 at 64 registers and 32 warps 1.31 ms).
// Against one row at a time: nf 2048 with 30 grids .288 -> .169 ms, nf 4096 1.94 -> 1.80 (64
// grids), nf 8192 1.22 -> 1.21 (9 grids).  The forward rows in this form: 1.06 -> 1.17 ms at
// nf = 8192, so they stay as they were.
#include "fft2d.h"
#include "fft_mixed.h"

namespace gpn {

namespace {

using fft::cv;
using fft::f2;
using fft::vset;

// shared-memory elements of a pair of rows (one spare per 16, and the slot N2)
__host__ __device__ constexpr int pair_buf(int n2) { return n2 + n2 / 16 + 1; }
// twiddles staged: the two-level table of the real split ([hi][lo]), then the pass tables (they
// follow the two-level table of the length-N2 FFT in global memory)
__host__ __device__ constexpr int pair_tw(int L) { return tw_hi(1 << L) + 64 + fft::pass_table_size(L); }
constexpr size_t pair_smem(int L, int pk) { return (size_t)pk * pair_buf(1 << L) * 16 + (size_t)pair_tw(L) * 8; }

__device__ __forceinline__ cv<f2> ld_pair(const cv<f2>* p) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  return {{u.x, u.y}, {u.z, u.w}};
}
__device__ __forceinline__ void st_pair(cv<f2>* p, cv<f2> v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.x.x, v.x.y, v.y.x, v.y.y);
}
__device__ __forceinline__ cv<f2> both(cpx<float> w) { return {vset<f2>(w.x), vset<f2>(w.y)}; }

// twiddles and the DFT of a radix-16 butterfly j at span Ns (pass table tw)
template <bool INV>
__device__ __forceinline__ int pair_butterfly(cv<f2> (&v)[16], int j, int Ns, const cpx<float>* tw) {
  const int k = j & (Ns - 1);
  if (Ns > 1) {
#pragma unroll
    for (int r = 1; r < 16; ++r) v[r] = fft::twiddle<INV>(v[r], both(tw[(r - 1) * Ns + k]));
  }
  fft::vdft<INV, 16>(v);
  return (j - k) * 16 + k;
}

// The transform of length 2^L from the registers x[u] = element t + u N/16, in the buffer b;
// the last pass hands element n to out(n, v).  No barrier follows.
template <bool INV, int L, typename Out>
__device__ __forceinline__ void pair_fft(cv<f2>* b, cv<f2> (&x)[16], const cpx<float>* ptab, int t, Out out) {
  constexpr int N = 1 << L, NT = N / 16, R0 = (L % 4 == 0) ? 16 : (1 << (L % 4)), NB = 16 / R0;
  constexpr int S = (L % 4 == 0) ? L / 4 - 1 : L / 4;   // radix-16 passes after the first
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    cv<f2> v[R0];
#pragma unroll
    for (int r = 0; r < R0; ++r) v[r] = x[c + r * NB];
    fft::vdft<INV, R0>(v);
#pragma unroll
    for (int r = 0; r < R0; ++r) {
      const int n = (t + c * NT) * R0 + r;
      if constexpr (S == 0)
        out(n, v[r]);
      else
        st_pair(b + fft::pad(n), v[r]);
    }
  }
  int Ns = R0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 16; ++r) x[r] = ld_pair(b + fft::pad(t + r * NT));
    const int base = pair_butterfly<INV>(x, t, Ns, ptab + fft::pass_table_offset(L, Ns));
    if (s + 1 < S) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 16; ++r) st_pair(b + fft::pad(base + r * Ns), x[r]);
    } else {
#pragma unroll
      for (int r = 0; r < 16; ++r) out(base + r * Ns, x[r]);
    }
    Ns *= 16;
  }
}

template <int L, int PK>
constexpr int kPairThreads = PK * (1 << L) / 16;
// 128 registers a thread: 512 threads an SM
template <int L, int PK>
constexpr int kPairBlocks = kPairThreads<L, PK> >= 512 ? 1 : kPairThreads<L, PK> < 32 ? 1 : 512 / kPairThreads<L, PK>;

__device__ __forceinline__ void stage_pair_twiddles(cpx<float>* s_tw, const cpx<float>* __restrict__ g, int L) {
  const cpx<float>* src = g + tw_hi(1 << L) + 64;
  for (int i = threadIdx.x; i < pair_tw(L); i += blockDim.x) s_tw[i] = src[i];
}

// inverse: modes 0..M of 2 PK rows (zero above M; the imaginary part of mode 0 is dropped, as a
// C2R transform does) to the grid columns [col_lo, col_hi)
template <int L, int PK>
__global__ void __launch_bounds__((kPairThreads<L, PK>), (kPairBlocks<L, PK>)) k_pairs_inv(RowsArgs<float> a) {
  constexpr int N2 = 1 << L, NT = N2 / 16, BUF = pair_buf(N2);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cv<f2>* buf = reinterpret_cast<cv<f2>*>(smem_raw);
  cpx<float>* s_tw = reinterpret_cast<cpx<float>*>(buf + PK * BUF);
  const int q = threadIdx.x / NT, t = threadIdx.x - q * NT;
  cv<f2>* b = buf + q * BUF;
  const long long item = blockIdx.x;
  const int cr = (int)(item / a.npairs);
  const long long y0 = a.row0 + (item - (long long)cr * a.npairs) * (2 * PK), y = y0 + 2 * q;
  stage_pair_twiddles(s_tw, a.tw, L);
  const fft::Twiddle2<float> wn{s_tw, s_tw + tw_hi(N2)};
  const float* src = reinterpret_cast<const float*>(a.X + (size_t)cr * (a.M + 1) * a.nf + y0);
  __syncthreads();
  // merge the modes (k, N2 - k) (fft_core.h's c2r_merge; one product serves both) into the
  // half-length input
  constexpr int NTH = kPairThreads<L, PK>, U = 4;   // U pairs of modes loaded before the first is used
  for (int k0 = threadIdx.x; k0 <= N2 / 2; k0 += U * NTH) {
    float4 u[U][PK], v[U][PK];
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int k = k0 + i * NTH, kn = N2 - k;
#pragma unroll
      for (int r = 0; r < PK; ++r) {
        u[i][r] = v[i][r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k <= N2 / 2 && k <= a.M) u[i][r] = *reinterpret_cast<const float4*>(src + (size_t)k * a.nf * 2 + 4 * r);
        if (k <= N2 / 2 && kn <= a.M) v[i][r] = *reinterpret_cast<const float4*>(src + (size_t)kn * a.nf * 2 + 4 * r);
      }
    }
#pragma unroll
    for (int i = 0; i < U; ++i) {
      const int k = k0 + i * NTH, kn = N2 - k;
      if (k > N2 / 2) break;
      const cv<f2> w = both(wn(k));
#pragma unroll
      for (int r = 0; r < PK; ++r) {
        float4 p0 = u[i][r];
        const float4 p1 = v[i][r];
        if (k == 0) p0.y = p0.w = 0.f;
        const cv<f2> xk{{p0.x, p0.z}, {p0.y, p0.w}}, xn{{p1.x, p1.z}, {p1.y, p1.w}};
        const cv<f2> e{fft::vadd(xk.x, xn.x), fft::vsub(xk.y, xn.y)}, o{fft::vsub(xk.x, xn.x), fft::vadd(xk.y, xn.y)};
        const cv<f2> p = fft::twiddle<true>(o, w);
        st_pair(buf + r * BUF + fft::pad(k), {fft::vsub(e.x, p.y), fft::vadd(e.y, p.x)});
        if (k != 0 && kn != k) st_pair(buf + r * BUF + fft::pad(kn), {fft::vadd(e.x, p.y), fft::vsub(p.x, e.y)});
      }
    }
  }
  __syncthreads();
  cv<f2> x[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) x[u] = ld_pair(b + fft::pad(t + u * NT));
  __syncthreads();   // the first pass rewrites the buffer
  float* dst = a.gout + (size_t)cr * a.G + y * a.nf;
  const bool in0 = y < a.row_hi, in1 = y + 1 < a.row_hi;
  pair_fft<true, L>(b, x, s_tw + tw_hi(N2) + 64, t, [&](int n, cv<f2> v) {
    if (2 * n + 1 >= a.col_lo && 2 * n < a.col_hi) {
      if (in0) *reinterpret_cast<float2*>(dst + 2 * n) = make_float2(v.x.x, v.y.x);
      if (in1) *reinterpret_cast<float2*>(dst + a.nf + 2 * n) = make_float2(v.x.y, v.y.y);
    }
  });
}

// pairs of rows a block takes: two where they fit one block of 512 threads
constexpr int row_pairs(int L) { return L <= 12 ? 2 : 1; }

template <int L>
void pairs_launch(RowsArgs<float> a, int row_lo, int grids, cudaStream_t st) {
  constexpr int PK = row_pairs(L);
  constexpr size_t smem = pair_smem(L, PK);
  a.row0 = row_lo / (2 * PK) * (2 * PK);
  a.npairs = (a.row_hi - a.row0 + 2 * PK - 1) / (2 * PK);
  a.nitems = a.npairs * grids;
  GPN_CUDA(cudaFuncSetAttribute(k_pairs_inv<L, PK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_pairs_inv<L, PK><<<(unsigned)a.nitems, kPairThreads<L, PK>, smem, st>>>(a);
}

}  // namespace

void rows_pairs_inv(int L, const RowsArgs<float>& a, int row_lo, int grids, cudaStream_t st) {
  switch (L) {
    case 4: pairs_launch<4>(a, row_lo, grids, st); break;
    case 5: pairs_launch<5>(a, row_lo, grids, st); break;
    case 6: pairs_launch<6>(a, row_lo, grids, st); break;
    case 7: pairs_launch<7>(a, row_lo, grids, st); break;
    case 8: pairs_launch<8>(a, row_lo, grids, st); break;
    case 9: pairs_launch<9>(a, row_lo, grids, st); break;
    case 10: pairs_launch<10>(a, row_lo, grids, st); break;
    case 11: pairs_launch<11>(a, row_lo, grids, st); break;
    case 12: pairs_launch<12>(a, row_lo, grids, st); break;
    default: pairs_launch<13>(a, row_lo, grids, st);
  }
}

}  // namespace gpn
