// CPU check of the fixed-point entropy functions of fx64.cuh against extended
// precision libm: 2^-z over [0, 64), log1p over [0, 1], both as absolute
// errors, and the sums of log cosh u and u e^{-u^2/2} over runs of samples
// (light and heavy tails, one sample beyond the functions' range), as absolute
// errors per sample.  Prints one line per function: "<name> <max error>"; the
// last lines check samples that are not finite.
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>
#include <vector>

#include "fx64.cuh"

using namespace vl::fx;
typedef long double LD;

int main() {
  std::vector<u64> e(EXP_N), l(LOG_N);
  std::vector<u32> r(LOG_N);
  for (int j = 0; j < EXP_N; ++j) e[j] = exp_entry(j);
  for (int j = 0; j < LOG_N; ++j) {
    l[j] = kLog[j];
    r[j] = log_recip(j);
  }
  const Tab T{e.data(), l.data(), r.data()};
  std::mt19937_64 g(2409);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  std::normal_distribution<double> N(0.0, 1.0);
  LD ee = 0, el = 0;
  for (int k = 0; k < 400000; ++k) {
    const double z = k & 1 ? 64.0 * U(g) : U(g);
    const u32 n = (u32)z;
    const u64 F = (u64)ldexpl((LD)z - n, 63);
    ee = fmaxl(ee, fabsl((LD)exp2neg(n, F, T) * 0x1p-63L - exp2l(-(LD)z)));
    u64 y = (u64)ldexpl((LD)U(g), 63) >> (k % 5 ? 0 : k % 60);
    if (k < 2) y = k ? (1ull << 63) - 1 : 0;
    el = fmaxl(el, fabsl((LD)(long long)log1p_fx(y, T) * 0x1p-63L - log1pl((LD)y * 0x1p-63L)));
  }
  std::printf("exp %.6e\nlog1p %.6e\n", (double)ee, (double)el);
  LD ea = 0, eb = 0;
  const LD kappa = 2.0L / 0.693147180559945309417232121458L;
  for (int rep = 0; rep < 2000; ++rep) {
    const int len = 1 + (int)(g() % 200);
    Moments M;
    LD A = 0, B = 0, mag = 0;
    for (int t = 0; t < len; ++t) {
      double u = N(g);
      if (rep % 3 == 1) u /= std::sqrt(0.01 + N(g) * N(g));
      if (rep % 3 == 2) u = std::sqrt(12.0) * (U(g) - 0.5);
      if (rep % 10 == 0 && t == 0) u = -40.0 - 100.0 * U(g);
      const double w = (double)(kappa * u);
      moments_add(M, w, T);
      const LD x = (LD)w / kappa, a = fabsl(x);
      A += a + log1pl(expl(-2 * a)) - 0.693147180559945309417232121458L;
      B += x * expl(-x * x / 2);
      mag += a;
    }
    double a, b;
    moments_sums(M, len, a, b);
    // the results are rounded to doubles (2^-53 of the sums, with one more
    // rounding where a sample beyond the range was added in FP64)
    ea = fmaxl(ea, fmaxl(0.0L, fabsl(a - A) - mag * 0x1p-52L) / len);
    eb = fmaxl(eb, fmaxl(0.0L, fabsl(b - B) - fabsl(B) * 0x1p-52L) / len);
  }
  std::printf("logcosh %.6e\ngauss %.6e\n", (double)ea, (double)eb);
  const double inf = std::numeric_limits<double>::infinity();
  const double bad[3] = {inf, -inf, std::nan("")};
  int ok = 1;
  for (double w : bad) {
    Moments M;
    moments_add(M, w, T);
    moments_add(M, 0.5, T);
    double a, b;
    moments_sums(M, 2, a, b);
    ok &= !std::isfinite(a) && std::isnan(b);
  }
  std::printf("nonfinite %d\n", ok);
  return 0;
}
