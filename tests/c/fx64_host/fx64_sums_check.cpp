// CPU check of the sums of the fixed-point entropy functions (fx64.cuh) before
// and after their conversion to doubles.  The accumulators are compared with sums
// in units of 2^-100 (128-bit integers, each term from extended precision), so
// that nothing is rounded away: errors per sample of the sums of |u| and of
// log1p(e^{-2|u|}).  Then moments_sums' doubles against the
// accumulators' own values: the error beyond two units of 2^-52 of the result, per
// run.  "beyond" is the same with a sample outside the functions' range, whose
// excess is added in FP64.  One line each: "<name> <max error>".
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "fx64.cuh"

using namespace vl::fx;
typedef long double LD;
typedef __int128 I;

static I value(const Acc& a) {  // 96 bits, two's complement
  return ((I)(int)a.w2 << 64) | (I)(((u64)a.w1 << 32) | a.w0);
}
static I fixed100(LD x) { return (I)floorl(ldexpl(x, 100)); }
static LD real(I x, int bits) { return ldexpl((LD)x, -bits); }

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
  const LD ln2 = 0.693147180559945309417232121458L;
  LD ew = 0, ef = 0, ea = 0, eb = 0, far = 0;
  for (int rep = 0; rep < 4000; ++rep) {
    const int len = 1 + (int)(g() % 200);
    const bool beyond = rep % 8 == 7;
    Moments M;
    I W = 0, F = 0;
    LD excess = 0;
    for (int t = 0; t < len; ++t) {
      double u = N(g);
      if (rep % 4 == 1) u /= std::sqrt(0.02 + N(g) * N(g));
      if (rep % 4 == 2) u = std::sqrt(12.0) * (U(g) - 0.5);
      if (rep % 4 == 3) u *= std::exp2(-60.0 * U(g));
      double w = std::fmin(std::fmax(2.0 / (double)ln2 * u, -63.9), 63.9);
      if (beyond && t == 0) {
        w = -64.0 - 300.0 * U(g);
        excess = -(LD)w - 64;
      }
      moments_add(M, w, T);
      const LD x = w, a = fabsl(x) < 64 ? fabsl(x) : 64;
      W += fixed100(a);
      F += fixed100(log1pl(exp2l(-a)));
    }
    const I dw = (value(M.w) << 43) - W, df = (value(M.f) << 37) - F;
    ew = fmaxl(ew, fabsl(real(dw, 100)) * ln2 / 2 / len);
    ef = fmaxl(ef, fabsl(real(df, 100)) / len);
    double a, b;
    moments_sums(M, len, a, b);
    const LD A = (real(value(M.w), 57) + excess) * ln2 / 2 + real(value(M.f), 63) - len * ln2;
    const LD B = real(value(M.g), 57) * ln2 / 2;
    const LD da = fabsl(a - A) - fabsl(A) * 0x1p-51L, db = fabsl(b - B) - fabsl(B) * 0x1p-51L;
    LD& worst = beyond ? far : ea;
    worst = fmaxl(worst, da);
    eb = fmaxl(eb, db);
  }
  std::printf("abs %.6e\nlog1p %.6e\n", (double)ew, (double)ef);
  std::printf("convert_logcosh %.6e\nconvert_gauss %.6e\nbeyond %.6e\n", (double)ea, (double)eb,
              (double)far);
  return 0;
}
