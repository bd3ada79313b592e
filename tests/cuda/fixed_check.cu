// Host check of the block fixed point of fr_fixed.cuh (its functions compile for both sides) against
// long double, on operands drawn with splitmix64.  For every term count n given on the command line:
// the worst ratio of the error of a contraction to its bound
//   (1 + 0.5625 n) 2^-56 sum|c| max|x| + 2^-53 |result|
// (truncated operands: 1/2 unit of the sum; rounded entries: n/16; the products of low limbs left
// out: n/2; rounding of the sum: 1/2; a unit is at most 2^-56 sum|c| max|x|; then one rounding to
// double), and the worst error in ulps of fx_double against the integer it is given.
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "fr_fixed.cuh"

using namespace frg;

static uint64_t ctr = 0;
static uint64_t rnd() {
  uint64_t z = ++ctr * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
// sign, random significand, exponent in [lo, hi]
static double draw(int lo, int hi) {
  const uint64_t r = rnd();
  const int e = lo + int((rnd() >> 20) % uint64_t(hi - lo + 1));
  return fx_from_bits((r & 0x800FFFFFFFFFFFFFull) | (uint64_t(e + 1023) << 52));
}

int main(int argc, char** argv) {
  for (int a = 1; a < argc; ++a) {
    const int n = atoi(argv[a]);
    double worst = 0.0;
    for (int t = 0; t < 20000; ++t) {
      // every magnitude from the smallest normal group up; within a group up to 2^80 apart; zeros
      const int top = t % 3 == 0 ? 0 : int(rnd() % 1800) - 900, spread = int(rnd() % 80);
      double x[32], c[32], sum = 0.0;
      uint32_t w = 0;
      long double exact = 0.0L, big = 0.0L;
      for (int j = 0; j < n; ++j) {
        x[j] = rnd() % 16 == 0 ? 0.0 : draw(top - spread, top);
        c[j] = draw(-6, 4);
        sum += std::fabs(c[j]);
        if (fx_mag(x[j]) > w) w = fx_mag(x[j]);
        exact += (long double)(x[j]) * c[j];
        if (std::fabs(x[j]) > big) big = std::fabs(x[j]);
      }
      const int k = fx_scale(sum), E = int(w >> 20) < FX_E_MIN ? FX_E_MIN : int(w >> 20);
      FxAcc acc{0, 0};
      for (int j = 0; j < n; ++j) fx_mac(acc, fx_limbs(x[j], E), fx_coef(c[j], k));
      const double got = fx_double(fx_sum(acc), fx_unit(E, k), E >= FX_E_BAD);
      const long double err = fabsl((long double)got - exact);
      const long double bound = (1.0L + 0.5625L * n) * sum * big * 0x1p-56L + 0x1p-53L * fabsl(exact);
      if (bound > 0.0L && double(err / bound) > worst) worst = double(err / bound);
      if (bound == 0.0L && got != 0.0) worst = 1e30;
    }
    printf("n%d %.6f\n", n, worst);
  }
  // sums of products (two, and the exact difference of the first factors with a third) and of squares:
  // operands cut at their last bit and the rounding, each a unit of 2^-58 (2^-57) 2^(Ev - 1022)
  // 2^(Ew - 1022) at most, two units for a square and for the difference; then one rounding to double
  double dot = 0.0, sq = 0.0;
  for (int t = 0; t < 200000; ++t) {
    const int ta = int(rnd() % 800) - 400, tb = int(rnd() % 800) - 400, spread = int(rnd() % 70);
    double x[4], y[3];
    for (int k = 0; k < 4; ++k) x[k] = rnd() % 16 == 0 ? 0.0 : draw(ta - spread, ta);
    for (int k = 0; k < 3; ++k) y[k] = draw(tb - spread, tb);
    const int Ex = fx_pexp(std::max(fx_mag(x[0]), fx_mag(x[1])));
    const int Ey = fx_pexp(std::max(fx_mag(y[0]), std::max(fx_mag(y[1]), fx_mag(y[2]))));
    const long long a = fx_value(x[0], Ex), b = fx_value(x[1], Ex);
    const double got = fx_double(fx_dot3(fx_split(a), fx_split(fx_value(y[0], Ey)), fx_split(b), fx_split(fx_value(y[1], Ey)),
                                         fx_diff(fx_split(a), fx_split(b)), fx_split(fx_value(y[2], Ey))),
                                 fx_punit(Ex, Ey, FX_PK3), fx_pbad(Ex, Ey));
    const long double want = (long double)x[0] * y[0] + (long double)x[1] * y[1] + ((long double)x[0] - x[1]) * y[2];
    const long double bd = 9.0L * ldexpl(1.0L, Ex + Ey - 2102 - FX_PK3) + 0x1p-53L * fabsl(want);
    dot = std::max(dot, double(fabsl(got - want) / bd));
    const int Es = fx_pexp(std::max(fx_mag(x[1]), std::max(fx_mag(x[2]), fx_mag(x[3]))));
    const int2 l[3] = {fx_split(fx_value(x[1], Es)), fx_split(fx_value(x[2], Es)), fx_split(fx_value(x[3], Es))};
    const double gs = fx_double(fx_sum_sq<3>(l), fx_punit(Es, Es, FX_PK), fx_pbad(Es, Es));
    const long double ws = (long double)x[1] * x[1] + (long double)x[2] * x[2] + (long double)x[3] * x[3];
    const long double bs = 7.0L * ldexpl(1.0L, 2 * Es - 2102 - FX_PK) + 0x1p-53L * ws;
    sq = std::max(sq, double(fabsl(gs - ws) / bs));
  }
  printf("dot %.6f\nsquares %.6f\n", dot, sq);
  double ulps = 0.0;
  for (int t = 0; t < 200000; ++t) {
    const int sh = int(rnd() % 63);
    const long long v = (long long)(rnd()) >> sh;
    const double want = ldexp(double(v), 10), got = fx_double(v, 1023 + 10, false);
    const double d = std::fabs(double((long long)(fx_bits(want) - fx_bits(got))));
    if (d > ulps) ulps = d;
  }
  printf("double %.1f\nzero %.1f\nnan %d\n", ulps, fx_double(0, 900, false), fx_double(5, 900, true) != fx_double(5, 900, true));
  return 0;
}
