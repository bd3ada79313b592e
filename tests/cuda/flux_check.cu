// Host check of the FP64 form's interface flux (rusanov2_fx of fr_kernels.cuh, which compiles for both
// sides) against the same flux in long double, F2 = f(qL) + f(qR) - lambda (qR - qL) with
// lambda = max(|u_n| + c), where a wave speed that is not a number loses to one that is (as in fmax).
// For every kind of state it prints the worst ratio of the error to its bound
//   (6 kappa + 16) 2^-53 S_v,   kappa = max (E + |m|^2 / 2 rho) / |E - |m|^2 / 2 rho| of the two sides,
//   S_v = 2 s (|Q_L| + |Q_R|) + pressure terms, s = max(lambda, |v_L|, |v_R|), Q the largest magnitude of
//   v's group (density, momenta, energy) on a side
// (in units of 2^-53: 1/rho 4, |m|^2 2, so 6 of the kinetic energy and 2 more of the pressure; half of
// that, the root, the product and the sum 3 kappa + 8 for lambda; 5 for a velocity; less than 1 for the cut
// operands; the sum's and the pressure's roundings).
// Special values: 0 if every result is non-finite where the FP64 formula is.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <limits>

#include "fr_kernels.cuh"

using namespace frg;
typedef long double LD;

static uint64_t ctr = 0;
static double rnd() {  // splitmix64, uniform in [0, 1)
  uint64_t z = ++ctr * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return double((z ^ (z >> 31)) >> 11) * 0x1p-53;
}
static const double GAM = 1.4;

template <class T>
static T max_num(T a, T b) {
  return std::isnan(a) ? b : (std::isnan(b) ? a : (a > b ? a : b));
}
// the flux in T; scale (nullable): S_v / (sum of the groups' magnitudes) parts for the bound
template <int DIM, class T>
static void flux(const double* qL, const double* qR, int axis, T* F, T* S, T* kappa) {
  constexpr int NV = DIM + 2;
  const T gm1 = T(GAM - 1.0);
  T v[2], p[2], c[2];
  *kappa = 1;
  for (int s = 0; s < 2; ++s) {
    const double* q = s ? qR : qL;
    T m2 = 0;
    for (int b = 0; b < DIM; ++b) m2 += T(q[1 + b]) * q[1 + b];
    const T ke = m2 / (2 * T(q[0]));
    p[s] = gm1 * (q[NV - 1] - ke);
    v[s] = T(q[1 + axis]) / q[0];
    c[s] = std::sqrt(T(GAM) * p[s] / q[0]);
    const T k = (std::fabs(T(q[NV - 1])) + ke) / std::fabs(q[NV - 1] - ke);
    if (k > *kappa) *kappa = k;
  }
  const T lam = max_num(std::fabs(v[0]) + c[0], std::fabs(v[1]) + c[1]);
  T s = lam;
  for (int k = 0; k < 2; ++k)
    if (std::fabs(v[k]) > s) s = std::fabs(v[k]);
  for (int w = 0; w < NV; ++w) {
    F[w] = qL[w] * v[0] + qR[w] * v[1] + lam * (T(qL[w]) - qR[w]);
    T mag = 0;
    for (int side = 0; side < 2; ++side) {
      const double* q = side ? qR : qL;
      T m = 0;
      for (int x = 0; x < NV; ++x)
        if (fx_group(x, NV) == fx_group(w, NV) && std::fabs(T(q[x])) > m) m = std::fabs(T(q[x]));
      mag += m;
    }
    S[w] = 2 * s * mag;
    if (w == 1 + axis) {
      F[w] += p[0] + p[1];
      S[w] += std::fabs(p[0]) + std::fabs(p[1]);
    }
    if (w == NV - 1) {
      F[w] += p[0] * v[0] + p[1] * v[1];
      S[w] += (std::fabs(p[0]) + std::fabs(p[1])) * s;
    }
  }
}

// a state of scale `a` (density, momenta and energy alike), speeds of O(1)
template <int DIM>
static void state(double a, double p, double* q) {
  q[0] = a * (0.5 + rnd());
  double ke = 0;
  for (int b = 0; b < DIM; ++b) {
    const double v = 2.0 * rnd() - 1.0;
    q[1 + b] = q[0] * v;
    ke += 0.5 * q[0] * v * v;
  }
  q[DIM + 1] = a * p / (GAM - 1.0) + ke;
}

template <int DIM>
static double ratio(const double* qL, const double* qR, int axis) {
  constexpr int NV = DIM + 2;
  double F[NV];
  LD W[NV], S[NV], k;
  rusanov2_fx<DIM>(qL, qR, axis, std::sqrt(GAM), GAM - 1.0, F);
  flux<DIM, LD>(qL, qR, axis, W, S, &k);
  double worst = 0;
  for (int v = 0; v < NV; ++v) {
    const LD b = (6 * k + 16) * 0x1p-53L * S[v], e = std::fabs(LD(F[v]) - W[v]);
    const double r = std::isnan(F[v]) ? 1e300 : double(e / b);
    if (r > worst) worst = r;
  }
  return worst;
}

template <int DIM>
static void kinds() {
  constexpr int NV = DIM + 2;
  double qL[NV], qR[NV], worst;
  auto line = [&](const char* name) { printf("%s%d %.3e\n", name, DIM, worst); };
  worst = 0;
  for (int t = 0; t < 20000; ++t) {
    state<DIM>(1.0, 0.1 + rnd(), qL);
    state<DIM>(1.0, 0.1 + rnd(), qR);
    worst = fmax(worst, ratio<DIM>(qL, qR, t % DIM));
  }
  line("plain");
  // units in which all values are tiny or huge
  for (int e : {-470, -440, 440}) {
    worst = 0;
    for (int t = 0; t < 5000; ++t) {
      state<DIM>(std::ldexp(1.0, e), 0.1 + rnd(), qL);
      state<DIM>(std::ldexp(1.0, e), 0.1 + rnd(), qR);
      worst = fmax(worst, ratio<DIM>(qL, qR, t % DIM));
    }
    line(e == -470 ? "smallest" : (e < 0 ? "tiny" : "huge"));
  }
  // one side 10 to 1e8 times as dense as the other at the same speeds and temperatures
  worst = 0;
  for (int t = 0; t < 20000; ++t) {
    const double f = std::pow(10.0, 1.0 + 7.0 * rnd());
    state<DIM>(t & 1 ? f : 1.0, 0.1 + rnd(), qL);
    state<DIM>(t & 1 ? 1.0 : f, 0.1 + rnd(), qR);
    worst = fmax(worst, ratio<DIM>(qL, qR, t % DIM));
  }
  line("jump");
  // one side's pressure negative: its wave speed is not a number, the other side's counts; its own
  // speed is up to 100 times that
  worst = 0;
  for (int t = 0; t < 20000; ++t) {
    state<DIM>(1.0, 0.1 + rnd(), qL);
    state<DIM>(1.0, 0.1 + rnd(), qR);
    const double f = std::pow(100.0, rnd());
    for (int b = 0; b < DIM; ++b) qL[1 + b] = qL[0] * f * (rnd() < 0.5 ? -1.0 : 1.0) * (0.5 + rnd());
    qL[NV - 1] *= 0.2 * rnd();
    if (t & 1) worst = fmax(worst, ratio<DIM>(qL, qR, t % DIM));
    else worst = fmax(worst, ratio<DIM>(qR, qL, t % DIM));
  }
  line("negative_pressure");
  // NaN (either sign) or infinity in one entry of one side: non-finite wherever the FP64 formula is
  int lost = 0;
  const double inf = std::numeric_limits<double>::infinity();
  const double sp[4] = {std::copysign(std::nan(""), 1.0), std::copysign(std::nan(""), -1.0), inf, -inf};
  for (int t = 0; t < 20000; ++t) {
    state<DIM>(1.0, 0.1 + rnd(), qL);
    state<DIM>(1.0, 0.1 + rnd(), qR);
    ((t & 1) ? qL : qR)[(t >> 1) % NV] = sp[(t / (2 * NV)) % 4];
    double F[NV], W[NV], S[NV], k;
    const int axis = int(rnd() * DIM);
    rusanov2_fx<DIM>(qL, qR, axis, std::sqrt(GAM), GAM - 1.0, F);
    flux<DIM, double>(qL, qR, axis, W, S, &k);
    for (int v = 0; v < NV; ++v) lost += std::isfinite(F[v]) && !std::isfinite(W[v]);
  }
  printf("special%d %d\n", DIM, lost);
}

int main() {
  kinds<2>();
  kinds<3>();
  // the larger of two wave speeds: a NaN of either sign loses to a number on either side
  const double pn = std::copysign(std::nan(""), 1.0), nn = std::copysign(std::nan(""), -1.0);
  const double inf = std::numeric_limits<double>::infinity();
  int bad = 0;
  for (double n : {pn, nn}) bad += !(fmax_num(n, 2.0) == 2.0) + !(fmax_num(2.0, n) == 2.0) + !(fmax_num(n, 0.0) == 0.0) + !std::isnan(fmax_num(n, nn));
  bad += !(fmax_num(1.0, 2.0) == 2.0) + !(fmax_num(2.0, 1.0) == 2.0) + !(fmax_num(inf, 1e308) == inf) + !(fmax_num(0.0, 5e-324) == 5e-324);
  printf("larger %d\n", bad);
  return 0;
}
