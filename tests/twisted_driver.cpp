// Host driver of the twisted eigenvector of a tridiagonal
// (paper_1905_01331_gb300/csrc/tridiag_df.cuh), in the order of the Lanczos kernel.
// stdin: cases "m th al_0 .. al_{m-1} be_0 .. be_{m-2}"; stdout per case: the
// unnormalised vector in pair arithmetic, then in FP64 (2 m numbers).
#include <cstdio>
#include <vector>

#include "../paper_1905_01331_gb300/csrc/tridiag_df.cuh"

using namespace ttn::tdf;

template <typename A>
static void vector(const std::vector<double>& al, const std::vector<double>& be, double th) {
  const int m = (int)al.size();
  std::vector<typename A::T> ms(m), b2(m), dp(m), dm(m);
  for (int i = 0; i < m; ++i) twist_row<A>(al.data(), be.data(), m, th, i, ms.data(), b2.data());
  twist_pivots<A>(ms.data(), b2.data(), m, true, dp.data());
  twist_pivots<A>(ms.data(), b2.data(), m, false, dm.data());
  double best = 1e300;
  int r = 0;
  for (int i = 0; i < m; ++i) {
    const double g = twist_gap<A>(ms.data(), dp.data(), dm.data(), i);
    if (g < best) { best = g; r = i; }
  }
  for (int i = 0; i + 1 < m; ++i) b2[i] = twist_multiplier<A>(be.data(), dp.data(), dm.data(), r, i);
  dp[r] = A::one();
  twist_outwards<A>(b2.data(), m, r, true, dp.data());
  twist_outwards<A>(b2.data(), m, r, false, dp.data());
  for (int i = 0; i < m; ++i) std::printf("%.17g ", A::to(dp[i]));
}

int main() {
  int m;
  double th;
  while (std::scanf("%d %lf", &m, &th) == 2) {
    std::vector<double> al(m), be(m, 0.0);
    bool ok = true;
    for (double& x : al) ok = ok && std::scanf("%lf", &x) == 1;
    for (int i = 0; i + 1 < m; ++i) ok = ok && std::scanf("%lf", &be[i]) == 1;
    if (!ok) return 1;
    vector<ArithDF>(al, be, th);
    vector<ArithD>(al, be, th);
    std::printf("\n");
  }
  return 0;
}
