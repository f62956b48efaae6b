// Mixed-radix building blocks of the 3-D box transforms (App. D's uniform FFT stage):
// DFTs of 2, 3, 4, 5, 6, 7, 8, 9, 10 and 16 points in registers, the factorisation of a
// 7-smooth length into two to four such radices, and the pass twiddles.  Everything here
// is __host__ __device__, so that the schedule the kernels run is checked on the CPU.
//
// Conventions as in fft_core.h: forward e^{-2 pi i jk/N}, inverse e^{+2 pi i jk/N},
// nothing normalised, Stockham order (natural in, natural out).
#pragma once

#include <algorithm>
#include <vector>

#include "fft_core.h"

namespace gpn {
namespace fft {

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

template <typename T>
GPN_HD cpx<T> scale(T a, cpx<T> v) { return {a * v.x, a * v.y}; }

template <bool INV, typename T>
GPN_HD void dft3(cpx<T>* v) {
  const cpx<T> t = v[1] + v[2], m = v[0] - scale((T)0.5, t);
  const cpx<T> d = rot90<INV>(scale((T)Root<3, 1>::s, v[1] - v[2]));
  v[0] = v[0] + t;
  v[1] = m + d;
  v[2] = m - d;
}

template <bool INV, typename T>
GPN_HD void dft5(cpx<T>* v) {
  const T c1 = (T)Root<5, 1>::c, c2 = (T)Root<5, 2>::c, s1 = (T)Root<5, 1>::s, s2 = (T)Root<5, 2>::s;
  const cpx<T> t1 = v[1] + v[4], t2 = v[2] + v[3], d1 = v[1] - v[4], d2 = v[2] - v[3];
  const cpx<T> a1 = v[0] + scale(c1, t1) + scale(c2, t2), a2 = v[0] + scale(c2, t1) + scale(c1, t2);
  const cpx<T> b1 = rot90<INV>(scale(s1, d1) + scale(s2, d2)), b2 = rot90<INV>(scale(s2, d1) - scale(s1, d2));
  v[0] = v[0] + t1 + t2;
  v[1] = a1 + b1;
  v[4] = a1 - b1;
  v[2] = a2 + b2;
  v[3] = a2 - b2;
}

template <bool INV, typename T>
GPN_HD void dft7(cpx<T>* v) {
  const T c1 = (T)Root<7, 1>::c, c2 = (T)Root<7, 2>::c, c3 = (T)Root<7, 3>::c;
  const T s1 = (T)Root<7, 1>::s, s2 = (T)Root<7, 2>::s, s3 = (T)Root<7, 3>::s;
  const cpx<T> t1 = v[1] + v[6], t2 = v[2] + v[5], t3 = v[3] + v[4];
  const cpx<T> d1 = v[1] - v[6], d2 = v[2] - v[5], d3 = v[3] - v[4];
  const cpx<T> a1 = v[0] + scale(c1, t1) + scale(c2, t2) + scale(c3, t3);
  const cpx<T> a2 = v[0] + scale(c2, t1) + scale(c3, t2) + scale(c1, t3);
  const cpx<T> a3 = v[0] + scale(c3, t1) + scale(c1, t2) + scale(c2, t3);
  const cpx<T> b1 = rot90<INV>(scale(s1, d1) + scale(s2, d2) + scale(s3, d3));
  const cpx<T> b2 = rot90<INV>(scale(s2, d1) - scale(s3, d2) - scale(s1, d3));
  const cpx<T> b3 = rot90<INV>(scale(s3, d1) - scale(s1, d2) + scale(s2, d3));
  v[0] = v[0] + t1 + t2 + t3;
  v[1] = a1 + b1;
  v[6] = a1 - b1;
  v[2] = a2 + b2;
  v[5] = a2 - b2;
  v[3] = a3 + b3;
  v[4] = a3 - b3;
}

template <bool INV, int R, typename T>
GPN_HD void dft_any(cpx<T>* v);

// the twiddles W_R^{n2 k1} of row n2 (k1 = 1 .. A-1), then the row moves on
template <bool INV, int A, int B, int N2, int K1, typename T>
GPN_HD void comp_twiddles(cpx<T> (&u)[A]) {
  if constexpr (K1 < A) {
    const T c = (T)Root<A * B, N2 * K1>::c, s = (T)Root<A * B, N2 * K1>::s;
    u[K1] = cmul(u[K1], cpx<T>{c, INV ? s : -s});
    comp_twiddles<INV, A, B, N2, K1 + 1>(u);
  }
}
template <bool INV, int A, int B, int N2, typename T>
GPN_HD void comp_rows(const cpx<T>* v, cpx<T> (&w)[B][A]) {
  if constexpr (N2 < B) {
#pragma unroll
    for (int a = 0; a < A; ++a) w[N2][a] = v[B * a + N2];
    dft_any<INV, A>(w[N2]);
    if constexpr (N2 > 0) comp_twiddles<INV, A, B, N2, 1>(w[N2]);
    comp_rows<INV, A, B, N2 + 1>(v, w);
  }
}
// radix A B: sample n = B n1 + n2, output k = k1 + A k2
template <bool INV, int A, int B, typename T>
GPN_HD void dft_comp(cpx<T>* v) {
  cpx<T> w[B][A];
  comp_rows<INV, A, B, 0>(v, w);
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) {
    cpx<T> u[B];
#pragma unroll
    for (int b = 0; b < B; ++b) u[b] = w[b][k1];
    dft_any<INV, B>(u);
#pragma unroll
    for (int b = 0; b < B; ++b) v[k1 + A * b] = u[b];
  }
}

template <bool INV, int R, typename T>
GPN_HD void dft_any(cpx<T>* v) {
  if constexpr (R == 2 || R == 4 || R == 8 || R == 16) dft<INV, R>(v);
  if constexpr (R == 3) dft3<INV>(v);
  if constexpr (R == 5) dft5<INV>(v);
  if constexpr (R == 6) dft_comp<INV, 3, 2>(v);
  if constexpr (R == 7) dft7<INV>(v);
  if constexpr (R == 9) dft_comp<INV, 3, 3>(v);
  if constexpr (R == 10) dft_comp<INV, 5, 2>(v);
}

// Butterflies a thread holds at once in a pass done in place (all reads before any write):
// at most 18 values, fewer where the radix needs many temporaries of its own.
GPN_HDC int held(int R) { return R == 2 ? 8 : R == 3 ? 6 : R == 4 ? 4 : R <= 6 ? 3 : R <= 8 ? 2 : 1; }

constexpr int kMaxPasses = 4;

// The passes of a length-N transform: radices in order, the lanes J a column needs so that
// every pass fits its butterflies, and where each pass's twiddles start in the table.
struct MixedPlan {
  int N = 0;
  int np = 0;
  int R[kMaxPasses] = {0, 0, 0, 0};
  int J = 0;
  int tw[kMaxPasses] = {0, 0, 0, 0};   // offset of pass p: [r - 1][k], k < Ns
};

// The factorisation into 2 to 4 ordered radices with the fewest passes, then the fewest
// lanes (every pass but the first is done in place and fits its butterflies), then the fewest
// idle butterfly slots; np = 0 when N is not 7-smooth or too short.
inline MixedPlan mixed_plan(int N) {
  static const int kRadix[] = {16, 10, 9, 8, 7, 6, 5, 4, 3, 2};
  MixedPlan best;
  long long best_cost = -1;
  int r[kMaxPasses];
  auto search = [&](auto&& self, int np, int rest) -> void {
    if (rest == 1 && np >= 2) {
      int J = (N + 17) / 18;
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

// twiddles and the DFT of one butterfly j, then its outputs
template <int R, bool INV, typename T, typename Out>
GPN_HD void butterfly(cpx<T> (&v)[R], int j, int Ns, const cpx<T>* tw, Out out) {
  const int k = Ns == 1 ? 0 : (int)((unsigned)j % (unsigned)Ns);
  if (Ns > 1) {
#pragma unroll
    for (int r = 1; r < R; ++r) {
      cpx<T> w = tw[(r - 1) * Ns + k];
      if (INV) w.y = -w.y;
      v[r] = cmul(v[r], w);
    }
  }
  dft_any<INV, R>(v);
  const int base = (j - k) * R + k;
#pragma unroll
  for (int r = 0; r < R; ++r) out(base + r * Ns, v[r]);
}

// One Stockham pass of radix R at span Ns of the transforms a block holds: lane jl of J
// takes the butterflies jl, jl + J, ...  in(n) gives element n of the lane's column, out(n, v)
// takes element n of the result.  HELD: the pass is done in place, every butterfly is read
// before sync() and the first write (at most held(R) a lane); otherwise in and out are
// different places and the butterflies follow one another.
template <int R, bool INV, bool HELD, typename T, typename In, typename Out, typename Sync>
GPN_HD void mixed_pass(int N, int J, int Ns, int jl, const cpx<T>* tw, In in, Out out, Sync sync) {
  const int nbf = N / R;
  if constexpr (HELD) {
    constexpr int NB = held(R);
    cpx<T> v[NB][R];
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = jl + b * J;
#pragma unroll
      for (int r = 0; r < R; ++r) v[b][r] = j < nbf ? in(j + r * nbf) : cpx<T>{T(0), T(0)};
    }
    sync();
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int j = jl + b * J;
      if (j < nbf) butterfly<R, INV>(v[b], j, Ns, tw, out);
    }
  } else {
#pragma unroll 1
    for (int j = jl; j < nbf; j += J) {
      cpx<T> v[R];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = in(j + r * nbf);
      butterfly<R, INV>(v, j, Ns, tw, out);
    }
  }
}

// the pass of a radix known at run time (the same for a whole block)
template <bool INV, bool HELD, typename T, typename In, typename Out, typename Sync>
GPN_HD void mixed_pass_any(int R, int N, int J, int Ns, int jl, const cpx<T>* tw, In in, Out out, Sync sync) {
  switch (R) {
    case 16: mixed_pass<16, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 10: mixed_pass<10, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 9: mixed_pass<9, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 8: mixed_pass<8, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 7: mixed_pass<7, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 6: mixed_pass<6, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 5: mixed_pass<5, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 4: mixed_pass<4, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    case 3: mixed_pass<3, INV, HELD>(N, J, Ns, jl, tw, in, out, sync); break;
    default: mixed_pass<2, INV, HELD>(N, J, Ns, jl, tw, in, out, sync);
  }
}

}  // namespace fft
}  // namespace gpn
