// Host program for tests/test_fft_mixed.py: the mixed-radix passes of csrc/fft_mixed.h with
// the kernels' schedule (lanes 0..J-1 of a column, reads of a pass before its writes).
// stdin: N, then 2 N reals; stdout: np J, then the forward and the inverse transform (in
// float64, then in float).
#include <cstdio>
#include <cstdlib>

#include "fft_mixed.h"

using namespace gpn::fft;

template <bool INV, typename V>
void transform(const MixedPlan& m, const std::vector<double>& x) {
  using T = typename Elem<V>::scalar;
  std::vector<cv<V>> buf(m.N), next(m.N), tw;
  for (int i = 0; i < m.N; ++i) buf[i] = {vset<V>((T)x[2 * i]), vset<V>((T)x[2 * i + 1])};
  const std::vector<double> t = mixed_tables(m);
  for (size_t i = 0; i < t.size(); i += 2) tw.push_back({vset<V>((T)t[i]), vset<V>((T)t[i + 1])});
  int ns = 1;
  for (int p = 0; p < m.np; ++p) {
    const auto in = [&](int n) { return buf[n]; };
    const auto out = [&](int n, cv<V> v) { next[n] = v; };
    const Span<V> sp{ns, m.inv_ns[p], tw.data() + m.tw[p]};
    for (int jl = 0; jl < m.J; ++jl) {
      if (p == 0)
        mixed_pass_any<INV, false, V>(m.R[p], m.N, m.J, jl, sp, in, out, [] {});
      else
        mixed_pass_any<INV, true, V>(m.R[p], m.N, m.J, jl, sp, in, out, [] {});
    }
    buf.swap(next);
    ns *= m.R[p];
  }
  for (const auto& v : buf) {
    double re, im;
    if constexpr (Elem<V>::lanes == 2) {
      if (v.x.x != v.x.y || v.y.x != v.y.y) std::exit(2);   // both lanes hold the same sequence
      re = v.x.x, im = v.y.y;
    } else {
      re = v.x, im = v.y;
    }
    std::printf("%.17g %.17g\n", re, im);
  }
}

int main() {
  int N;
  if (std::scanf("%d", &N) != 1) return 1;
  std::vector<double> x(2 * N);
  for (double& v : x)
    if (std::scanf("%lf", &v) != 1) return 1;
  const MixedPlan m = mixed_plan(N);
  std::printf("%d %d\n", m.np, m.J);
  if (m.np == 0) return 0;
  transform<false, double>(m, x);
  transform<true, double>(m, x);
  transform<false, f2>(m, x);
  return 0;
}
