// Mixed-radix building blocks of the 3-D box transforms (App. D's uniform FFT stage):
// DFTs of 2, 3, 4, 5, 6, 7, 8, 9, 10 and 16 points in registers, the factorisation of a
// 7-smooth length into two to four such radices, and the pass twiddles.  Everything here
// is __host__ __device__, so that the schedule the kernels run is checked on the CPU.
//
// The element type V is one value (float64) or two values of adjacent sequences side by side
// (FP32, struct f2), whose sums and products are single packed instructions: the passes are
// bound by instruction issue, and a packed complex value costs the address arithmetic, loads,
// stores and twiddles of one.
//
// Conventions as in fft_core.h: forward e^{-2 pi i jk/N}, inverse e^{+2 pi i jk/N},
// nothing normalised, Stockham order (natural in, natural out).
#pragma once

#include <algorithm>
#include <vector>

#include "fft_core.h"

namespace gpn {
namespace fft {

// two FP32 values of adjacent sequences
struct alignas(8) f2 {
  float x, y;
};

// the scalar type of an element, and the values it holds
template <typename V>
struct Elem {
  using scalar = V;
  static constexpr int lanes = 1;
};
template <>
struct Elem<f2> {
  using scalar = float;
  static constexpr int lanes = 2;
};

template <typename V>
GPN_HD V vset(typename Elem<V>::scalar a) { return a; }
template <>
GPN_HD f2 vset<f2>(float a) { return {a, a}; }

// a + b, a - b, a b, a b + c
GPN_HD double vadd(double a, double b) { return a + b; }
GPN_HD double vsub(double a, double b) { return a - b; }
GPN_HD double vmul(double a, double b) { return a * b; }
GPN_HD double vfma(double a, double b, double c) { return a * b + c; }
#ifdef __CUDA_ARCH__
GPN_HD float2 as_float2(f2 a) { return make_float2(a.x, a.y); }
GPN_HD f2 as_f2(float2 a) { return {a.x, a.y}; }
GPN_HD f2 vadd(f2 a, f2 b) { return as_f2(__fadd2_rn(as_float2(a), as_float2(b))); }
GPN_HD f2 vmul(f2 a, f2 b) { return as_f2(__fmul2_rn(as_float2(a), as_float2(b))); }
GPN_HD f2 vfma(f2 a, f2 b, f2 c) { return as_f2(__ffma2_rn(as_float2(a), as_float2(b), as_float2(c))); }
// one packed instruction, the same rounding as a - b
GPN_HD f2 vsub(f2 a, f2 b) { return vfma(b, f2{-1.0f, -1.0f}, a); }
#else
GPN_HD f2 vadd(f2 a, f2 b) { return {a.x + b.x, a.y + b.y}; }
GPN_HD f2 vsub(f2 a, f2 b) { return {a.x - b.x, a.y - b.y}; }
GPN_HD f2 vmul(f2 a, f2 b) { return {a.x * b.x, a.y * b.y}; }
GPN_HD f2 vfma(f2 a, f2 b, f2 c) { return {__builtin_fmaf(a.x, b.x, c.x), __builtin_fmaf(a.y, b.y, c.y)}; }
#endif
// a + s b
template <typename V>
GPN_HD V vaxpy(typename Elem<V>::scalar s, V b, V a) { return vfma(b, vset<V>(s), a); }

// a complex element: 16 bytes (one float64 value or two FP32 values), one vector access
template <typename V>
struct alignas(16) cv {
  V x, y;
};

template <typename V>
GPN_HD cv<V> operator+(cv<V> a, cv<V> b) { return {vadd(a.x, b.x), vadd(a.y, b.y)}; }
template <typename V>
GPN_HD cv<V> operator-(cv<V> a, cv<V> b) { return {vsub(a.x, b.x), vsub(a.y, b.y)}; }
// a + s b
template <typename V>
GPN_HD cv<V> axpy(typename Elem<V>::scalar s, cv<V> b, cv<V> a) { return {vaxpy(s, b.x, a.x), vaxpy(s, b.y, a.y)}; }
template <typename V>
GPN_HD cv<V> scaled(typename Elem<V>::scalar s, cv<V> a) { return {vmul(a.x, vset<V>(s)), vmul(a.y, vset<V>(s))}; }
// a + s t b with t = -i (forward) or +i (inverse); s = -1 subtracts the turned value
template <bool INV, typename V>
GPN_HD cv<V> add_turned(typename Elem<V>::scalar s, cv<V> b, cv<V> a) {
  return INV ? cv<V>{vaxpy(-s, b.y, a.x), vaxpy(s, b.x, a.y)} : cv<V>{vaxpy(s, b.y, a.x), vaxpy(-s, b.x, a.y)};
}
template <bool INV, typename V>
GPN_HD cv<V> add_turn(cv<V> b, cv<V> a) {
  return INV ? cv<V>{vsub(a.x, b.y), vadd(a.y, b.x)} : cv<V>{vadd(a.x, b.y), vsub(a.y, b.x)};
}
template <bool INV, typename V>
GPN_HD cv<V> sub_turn(cv<V> b, cv<V> a) { return add_turn<!INV>(b, a); }
// a w (forward) or a conj(w) (inverse), w = {cos, -sin} broadcast to the lanes
template <bool INV, typename V>
GPN_HD cv<V> twiddle(cv<V> a, cv<V> w) {
  const V m = vmul(w.y, vset<V>(-1));
  return INV ? cv<V>{vfma(a.y, w.y, vmul(a.x, w.x)), vfma(a.x, m, vmul(a.y, w.x))}
             : cv<V>{vfma(a.y, m, vmul(a.x, w.x)), vfma(a.x, w.y, vmul(a.y, w.x))};
}

// cos and sin of 2 pi i / R, folded at compile time (Taylor series: |x| <= pi, 30 terms)
GPN_HDC double series_cos(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k <= 30; ++k) {
    term *= -x * x / ((2.0 * k - 1.0) * (2.0 * k));
    sum += term;
  }
  return sum;
}
GPN_HDC double series_sin(double x) {
  double term = x, sum = x;
  for (int k = 1; k <= 30; ++k) {
    term *= -x * x / ((2.0 * k) * (2.0 * k + 1.0));
    sum += term;
  }
  return sum;
}
template <int R, int I>
struct Root {
  // the angle 2 pi i / R in (-pi, pi]
  static constexpr int i = I % R;
  static constexpr double angle = 6.283185307179586476925286766559 * (2 * i > R ? i - R : i) / R;
  static constexpr double c = series_cos(angle), s = series_sin(angle);
};

// a + b W_R^I and a - b W_R^I (W_R^-I inverse), products folded into the sums
template <bool INV, int R, int I, typename V>
GPN_HD void rotate_pair(cv<V> a, cv<V> b, cv<V>& plus, cv<V>& minus) {
  using T = typename Elem<V>::scalar;
  const T c = (T)Root<R, I>::c, s = INV ? (T)Root<R, I>::s : -(T)Root<R, I>::s;
  plus = {vaxpy(c, b.x, vaxpy(-s, b.y, a.x)), vaxpy(s, b.x, vaxpy(c, b.y, a.y))};
  minus = {vaxpy(-c, b.x, vaxpy(s, b.y, a.x)), vaxpy(-s, b.x, vaxpy(-c, b.y, a.y))};
}

template <bool INV, typename V, int S = 1>
GPN_HD void vdft4(cv<V>* v) {
  const cv<V> a0 = v[0] + v[2 * S], a1 = v[0] - v[2 * S], b0 = v[S] + v[3 * S], d = v[S] - v[3 * S];
  v[0] = a0 + b0;
  v[2 * S] = a0 - b0;
  v[S] = add_turn<INV>(d, a1);
  v[3 * S] = sub_turn<INV>(d, a1);
}

// radix-8 = 2 x 4 at stride S: the odd half's eighth turns are folded into the last sums
template <bool INV, typename V, int S = 1>
GPN_HD void vdft8(cv<V>* v) {
  using T = typename Elem<V>::scalar;
  const T q = (T)kS45;
  vdft4<INV, V, 2 * S>(v);
  vdft4<INV, V, 2 * S>(v + S);
  const cv<V> o0 = v[S], o1 = v[3 * S], o2 = v[5 * S], o3 = v[7 * S];
  const cv<V> e0 = v[0], e1 = v[2 * S], e2 = v[4 * S], e3 = v[6 * S];
  v[0] = e0 + o0;
  v[4 * S] = e0 - o0;
  v[2 * S] = add_turn<INV>(o2, e2);
  v[6 * S] = sub_turn<INV>(o2, e2);
  // o1 W_8 = (x + t y, y - t x) / sqrt 2 and o3 W_8^3 = (t y - x, -y - t x) / sqrt 2 with t = 1
  // forward, -1 inverse
  const cv<V> u1 = add_turn<INV>(o1, o1);
  const V d3 = vsub(o3.y, o3.x), s3 = vadd(o3.x, o3.y);
  v[S] = axpy(q, u1, e1);
  v[5 * S] = axpy(-q, u1, e1);
  v[3 * S] = INV ? cv<V>{vaxpy(-q, s3, e3.x), vaxpy(-q, d3, e3.y)} : cv<V>{vaxpy(q, d3, e3.x), vaxpy(-q, s3, e3.y)};
  v[7 * S] = INV ? cv<V>{vaxpy(q, s3, e3.x), vaxpy(q, d3, e3.y)} : cv<V>{vaxpy(-q, d3, e3.x), vaxpy(q, s3, e3.y)};
}

// radix-16 = 2 x 8
template <bool INV, typename V>
GPN_HD void vdft16(cv<V>* v) {
  vdft8<INV, V, 2>(v);
  vdft8<INV, V, 2>(v + 1);
  cv<V> e[8], o[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    e[k] = v[2 * k];
    o[k] = v[2 * k + 1];
  }
  v[0] = e[0] + o[0];
  v[8] = e[0] - o[0];
  rotate_pair<INV, 16, 1>(e[1], o[1], v[1], v[9]);
  rotate_pair<INV, 16, 2>(e[2], o[2], v[2], v[10]);
  rotate_pair<INV, 16, 3>(e[3], o[3], v[3], v[11]);
  v[4] = add_turn<INV>(o[4], e[4]);
  v[12] = sub_turn<INV>(o[4], e[4]);
  rotate_pair<INV, 16, 5>(e[5], o[5], v[5], v[13]);
  rotate_pair<INV, 16, 6>(e[6], o[6], v[6], v[14]);
  rotate_pair<INV, 16, 7>(e[7], o[7], v[7], v[15]);
}

template <bool INV, typename V>
GPN_HD void vdft3(cv<V>* v) {
  using T = typename Elem<V>::scalar;
  const T s = (T)Root<3, 1>::s;
  const cv<V> t = v[1] + v[2], d = v[1] - v[2], m = axpy((T)-0.5, t, v[0]);
  v[0] = v[0] + t;
  v[1] = add_turned<INV>(s, d, m);
  v[2] = add_turned<INV>(-s, d, m);
}

template <bool INV, typename V>
GPN_HD void vdft5(cv<V>* v) {
  using T = typename Elem<V>::scalar;
  const T c1 = (T)Root<5, 1>::c, c2 = (T)Root<5, 2>::c, s1 = (T)Root<5, 1>::s, s2 = (T)Root<5, 2>::s;
  const cv<V> t1 = v[1] + v[4], t2 = v[2] + v[3], d1 = v[1] - v[4], d2 = v[2] - v[3];
  const cv<V> a1 = axpy(c2, t2, axpy(c1, t1, v[0])), a2 = axpy(c1, t2, axpy(c2, t1, v[0]));
  const cv<V> b1 = axpy(s2, d2, scaled(s1, d1)), b2 = axpy(-s1, d2, scaled(s2, d1));
  v[0] = v[0] + t1 + t2;
  v[1] = add_turn<INV>(b1, a1);
  v[4] = sub_turn<INV>(b1, a1);
  v[2] = add_turn<INV>(b2, a2);
  v[3] = sub_turn<INV>(b2, a2);
}

template <bool INV, typename V>
GPN_HD void vdft7(cv<V>* v) {
  using T = typename Elem<V>::scalar;
  const T c1 = (T)Root<7, 1>::c, c2 = (T)Root<7, 2>::c, c3 = (T)Root<7, 3>::c;
  const T s1 = (T)Root<7, 1>::s, s2 = (T)Root<7, 2>::s, s3 = (T)Root<7, 3>::s;
  const cv<V> t1 = v[1] + v[6], t2 = v[2] + v[5], t3 = v[3] + v[4];
  const cv<V> d1 = v[1] - v[6], d2 = v[2] - v[5], d3 = v[3] - v[4];
  const cv<V> a1 = axpy(c3, t3, axpy(c2, t2, axpy(c1, t1, v[0])));
  const cv<V> a2 = axpy(c1, t3, axpy(c3, t2, axpy(c2, t1, v[0])));
  const cv<V> a3 = axpy(c2, t3, axpy(c1, t2, axpy(c3, t1, v[0])));
  const cv<V> b1 = axpy(s3, d3, axpy(s2, d2, scaled(s1, d1)));
  const cv<V> b2 = axpy(-s1, d3, axpy(-s3, d2, scaled(s2, d1)));
  const cv<V> b3 = axpy(s2, d3, axpy(-s1, d2, scaled(s3, d1)));
  v[0] = v[0] + t1 + t2 + t3;
  v[1] = add_turn<INV>(b1, a1);
  v[6] = sub_turn<INV>(b1, a1);
  v[2] = add_turn<INV>(b2, a2);
  v[5] = sub_turn<INV>(b2, a2);
  v[3] = add_turn<INV>(b3, a3);
  v[4] = sub_turn<INV>(b3, a3);
}

template <bool INV, int R, typename V>
GPN_HD void vdft(cv<V>* v);

// the twiddles W_R^{n2 k1} of row n2 (k1 = 1 .. A-1)
template <bool INV, int A, int B, int N2, int K1, typename V>
GPN_HD void comp_twiddles(cv<V> (&u)[A]) {
  if constexpr (K1 < A) {
    using T = typename Elem<V>::scalar;
    const T c = (T)Root<A * B, N2 * K1>::c, s = INV ? (T)Root<A * B, N2 * K1>::s : -(T)Root<A * B, N2 * K1>::s;
    const cv<V> a = u[K1];
    u[K1] = {vaxpy(-s, a.y, vmul(a.x, vset<V>(c))), vaxpy(s, a.x, vmul(a.y, vset<V>(c)))};
    comp_twiddles<INV, A, B, N2, K1 + 1>(u);
  }
}
template <bool INV, int A, int B, int N2, typename V>
GPN_HD void comp_rows(const cv<V>* v, cv<V> (&w)[B][A]) {
  if constexpr (N2 < B) {
#pragma unroll
    for (int a = 0; a < A; ++a) w[N2][a] = v[B * a + N2];
    vdft<INV, A>(w[N2]);
    if constexpr (N2 > 0) comp_twiddles<INV, A, B, N2, 1>(w[N2]);
    comp_rows<INV, A, B, N2 + 1>(v, w);
  }
}
// radix A B: sample n = B n1 + n2, output k = k1 + A k2
template <bool INV, int A, int B, typename V>
GPN_HD void vdft_comp(cv<V>* v) {
  cv<V> w[B][A];
  comp_rows<INV, A, B, 0>(v, w);
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    cv<V> u[B];
#pragma unroll
    for (int b = 0; b < B; ++b) u[b] = w[b][k1];
    vdft<INV, B>(u);
#pragma unroll
    for (int b = 0; b < B; ++b) v[k1 + A * b] = u[b];
  }
}

template <bool INV, int R, typename V>
GPN_HD void vdft(cv<V>* v) {
  if constexpr (R == 2) {
    const cv<V> a = v[0];
    v[0] = a + v[1];
    v[1] = a - v[1];
  }
  if constexpr (R == 3) vdft3<INV>(v);
  if constexpr (R == 4) vdft4<INV>(v);
  if constexpr (R == 5) vdft5<INV>(v);
  if constexpr (R == 6) vdft_comp<INV, 3, 2>(v);
  if constexpr (R == 7) vdft7<INV>(v);
  if constexpr (R == 8) vdft8<INV>(v);
  if constexpr (R == 9) vdft_comp<INV, 3, 3>(v);
  if constexpr (R == 10) vdft_comp<INV, 5, 2>(v);
  if constexpr (R == 16) vdft16<INV>(v);
}

// Butterflies a thread holds at once in a pass done in place (all reads before any write): at
// most 10 elements of four words, so that a thread keeps to 64 registers.
GPN_HDC int held(int R) { return R == 2 ? 4 : R == 3 ? 3 : R <= 5 ? 2 : 1; }

constexpr int kMaxPasses = 4;

// The passes of a length-N transform: radices in order, the lanes J a column needs so that
// every pass fits its butterflies, and where each pass's twiddles start in the table.
struct MixedPlan {
  int N = 0;
  int np = 0;
  int R[kMaxPasses] = {0, 0, 0, 0};
  int J = 0;
  int tw[kMaxPasses] = {0, 0, 0, 0};   // offset of pass p: [r - 1][k], k < Ns
  unsigned inv_ns[kMaxPasses] = {0, 0, 0, 0};   // ceil(2^32 / Ns): j / Ns = mulhi(j, inv_ns)
};

// The factorisation into 2 to 4 ordered radices with the fewest passes, then the fewest
// lanes (every pass but the first is done in place and fits its butterflies), then the fewest
// idle butterfly slots; np = 0 when N is not 7-smooth or too short.
inline MixedPlan mixed_plan(int N) {
  static const int kRadix[] = {10, 9, 8, 7, 6, 5, 4, 3, 2};
  MixedPlan best;
  long long best_cost = -1;
  int r[kMaxPasses];
  auto search = [&](auto&& self, int np, int rest) -> void {
    if (rest == 1 && np >= 2) {
      int J = (N + 9) / 10;
      for (int p = 1; p < np; ++p) J = std::max(J, (N + r[p] * held(r[p]) - 1) / (r[p] * held(r[p])));
      long long work = 0;
      for (int p = 0; p < np; ++p) work += ((N / r[p] + J - 1) / J) * r[p];
      const long long cost = ((long long)np * 100000 + J) * 1000 + work;
      if (best_cost < 0 || cost < best_cost) {
        best_cost = cost;
        best.N = N;
        best.np = np;
        best.J = J;
        for (int p = 0; p < np; ++p) best.R[p] = r[p];
      }
      return;
    }
    if (np == kMaxPasses) return;
    for (int q : kRadix)
      if (rest % q == 0) {
        r[np] = q;
        self(self, np + 1, rest / q);
      }
  };
  if (N >= 4) search(search, 0, N);
  int off = 0, ns = 1;
  for (int p = 0; p < best.np; ++p) {
    best.tw[p] = off;
    best.inv_ns[p] = (unsigned)(((1ull << 32) + ns - 1) / ns);   // (ns > 1: used for p > 0)
    if (p > 0) off += (best.R[p] - 1) * ns;
    ns *= best.R[p];
  }
  return best;
}

// The pass twiddles W_{Ns R}^{r k} as interleaved (re, im) float64 values.
inline std::vector<double> mixed_tables(const MixedPlan& m) {
  std::vector<double> t;
  int ns = 1;
  for (int p = 0; p < m.np; ++p) {
    if (p > 0)
      for (int r = 1; r < m.R[p]; ++r)
        for (int k = 0; k < ns; ++k) {
          const double th = 6.283185307179586476925286766559 * (double)(r * k) / ((double)ns * m.R[p]);
          t.push_back(std::cos(th));
          t.push_back(-std::sin(th));
        }
    ns *= m.R[p];
  }
  return t;
}

GPN_HD int mulhi(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  return (int)__umulhi(a, b);
#else
  return (int)(((unsigned long long)a * b) >> 32);
#endif
}

// the span of a pass: product of the earlier radices, its twiddles, and 2^32 / Ns
template <typename V>
struct Span {
  int Ns;
  unsigned inv;
  const cv<V>* tw;
};

// twiddles and the DFT of one butterfly j, then its outputs
template <int R, bool INV, typename V, typename Out>
GPN_HD void butterfly(cv<V> (&v)[R], int j, const Span<V>& sp, Out out) {
  int base = j * R;
  if (sp.Ns > 1) {
    const int k = j - mulhi((unsigned)j, sp.inv) * sp.Ns;
    const cv<V>* tw = sp.tw + k;
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = twiddle<INV>(v[r], tw[(r - 1) * sp.Ns]);
    base = (j - k) * R + k;
  }
  vdft<INV, R>(v);
#pragma unroll
  for (int r = 0; r < R; ++r) out(base + r * sp.Ns, v[r]);
}

// One Stockham pass of radix R of the transforms a block holds: lane jl of J takes the
// butterflies jl, jl + J, ...  in(n) gives element n of the lane's column, out(n, v) takes
// element n of the result.  HELD: the pass is done in place, every butterfly is read before
// sync() and the first write (at most held(R) a lane); otherwise in and out are different
// places and the butterflies follow one another.
template <int R, bool INV, bool HELD, typename V, typename In, typename Out, typename Sync>
GPN_HD void mixed_pass(int N, int J, int jl, const Span<V>& sp, In in, Out out, Sync sync) {
  const int nbf = N / R;
  if constexpr (HELD) {
    constexpr int NB = held(R);
    cv<V> v[NB][R];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = jl + b * J;
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = j < nbf ? in(j + r * nbf) : cv<V>{vset<V>(0), vset<V>(0)};
    }
    sync();
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = jl + b * J;
      if (j < nbf) butterfly<R, INV>(v[b], j, sp, out);
    }
  } else {
#pragma unroll 1
    for (int j = jl; j < nbf; j += J) {
      cv<V> v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = in(j + r * nbf);
      butterfly<R, INV>(v, j, sp, out);
    }
  }
}

// the pass of a radix known at run time (the same for a whole block)
template <bool INV, bool HELD, typename V, typename In, typename Out, typename Sync>
GPN_HD void mixed_pass_any(int R, int N, int J, int jl, const Span<V>& sp, In in, Out out, Sync sync) {
  switch (R) {
    case 10: mixed_pass<10, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 9: mixed_pass<9, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 8: mixed_pass<8, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 7: mixed_pass<7, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 6: mixed_pass<6, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 5: mixed_pass<5, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 4: mixed_pass<4, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    case 3: mixed_pass<3, INV, HELD>(N, J, jl, sp, in, out, sync); break;
    default: mixed_pass<2, INV, HELD>(N, J, jl, sp, in, out, sync);
  }
}

}  // namespace fft
}  // namespace gpn
