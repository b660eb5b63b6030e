// Host check of the entropy-variable increment w(u + e) - w(u) (csrc/es_prep_fx.cuh) against long double
// for changes of 1e-13 to 1e-2 of the state, u + e not rounded: per range the largest error of a component in units of
// 2^-53 of its terms beyond the result's own rounding, and the mean error relative to the component
// (momentum: to the vector) beside that of the same formula in double.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "es_prep_fx.cuh"

using namespace es;
typedef long double L;

static L log1(L z) { return log1pl(z); }
static double log1(double z) { return log1p(z); }

// size: the sum of the magnitudes of each component's terms
template <typename T>
static void increment(const T u[5], const T e[5], T gam, T dw[5], T size[5]) {
  const T gm1 = gam - 1, rho = u[0], rho1 = rho + e[0];
  const T m2 = u[1] * u[1] + u[2] * u[2] + u[3] * u[3], Pr = gm1 * (rho * u[4] - m2 / 2);
  const T x = e[0] / rho, ip = rho / Pr, beta = rho * ip, v2s = m2 / (rho * rho);
  T v[3], d[3], vd = 0, d2 = 0, ve = 0, vmax = 0, emax = 0;
  for (int k = 0; k < 3; ++k) {
    v[k] = u[1 + k] / rho;
    d[k] = (e[1 + k] - v[k] * e[0]) / rho1;
    vd += v[k] * d[k];
    d2 += d[k] * d[k];
    ve += v[k] * e[1 + k];
    vmax = std::max(vmax, std::fabs(v[k]));
    emax = std::max(emax, std::fabs(e[1 + k]));
  }
  const T y = gm1 * (e[4] - ve + v2s / 2 * e[0] - rho1 * d2 / 2) * ip, biy = beta / (1 + y);
  const T ds = log1(y) - gam * log1(x), xy = x - y;
  dw[0] = -ds / gm1 - biy / 2 * (xy * v2s + (1 + x) * (2 * vd + d2));
  for (int k = 0; k < 3; ++k) dw[1 + k] = biy * (xy * v[k] + (1 + x) * d[k]);
  dw[4] = -biy * xy;
  // eta = change of rho p relative to itself, a = d_1 - z1 eta relative to z1
  const T K = 3 * (vmax * rho + emax) * emax / Pr;
  const T eta = gm1 * (std::fabs(rho * e[4]) / Pr + std::fabs(u[4] * e[0]) / Pr + K), a = std::fabs(x) + eta;
  size[0] = 2 * (gam + 1) / gm1 * std::fabs(x) + 2 / gm1 * eta + K + m2 / Pr * eta;
  for (int k = 0; k < 3; ++k) size[1 + k] = rho * emax / Pr + beta * vmax * a;
  size[4] = beta * (std::fabs(x) + a);
  // rho p itself is a difference: its terms against it
  for (int k = 0; k < 5; ++k) size[k] *= gm1 * (rho * u[4] + m2 / 2) / Pr;
}

int main() {
  std::mt19937_64 R(7);
  std::uniform_real_distribution<double> U(-1, 1);
  for (double gam : {1.4, 5.0 / 3.0, 1.1, 2.5, 6.0})
    for (double mach : {0.0, 1e-6, 0.01, 0.3, 1.0, 3.0})
      for (double del : {1e-13, 1e-9, 1e-6, 1e-3, 8e-3, 0.019}) {
        const L g = gam, c = 2 * (g + 1) / (g - 1);
        int ktg = 0, eg;
        while (ldexpl(1, ktg) <= c) ++ktg;
        const fx C1 = llrintl(ldexpl(c, 62 - ktg)), g1 = llrintl(ldexpl(frexpl(1 / (g - 1), &eg), 62));
        L worst = 0, mean[5] = {}, mean64[5] = {};
        int out = 0, n = 0;
        for (int it = 0; it < 4000; ++it) {
          double rho = exp(5 * U(R)), p = exp(5 * U(R));
          if (it % 4 == 1) rho = ldexp(1.0, it % 7 - 3) * (1 - 1e-13 * (it % 3) * U(R));  // next to powers of two
          if (it % 4 == 2) p = ldexp(1.0, it % 5 - 2) / rho;
          const double a = sqrt(gam * p / rho);
          double u[5], e[5], v[3], k2 = 0;
          for (int k = 0; k < 3; ++k) {
            v[k] = mach * a * 0.57 * U(R);
            k2 += v[k] * v[k];
            u[1 + k] = rho * v[k];
          }
          u[0] = rho;
          u[4] = p / (gam - 1) + rho * k2 / 2;
          const double x = it % 9 == 8 ? 0 : del * U(R);
          e[0] = rho * x;
          e[4] = p * (1 + x) / (gam - 1) * (it % 11 == 10 ? 0 : del * U(R) / 2);
          for (int k = 0; k < 3; ++k) {
            const double dv = it % 13 == 12 ? 0 : a * del * U(R);
            e[1 + k] = rho * (1 + x) * dv + v[k] * e[0];
            e[4] += rho * x * v[k] * v[k] / 2 + rho * (1 + x) * (v[k] * dv + dv * dv / 2);
          }
          double dw[5], f[5], fs[5];
          if (!fx_increment(u, e, C1, ktg, g1, eg, dw)) {
            ++out;
            continue;
          }
          L lu[5], le[5], t[5], s[5];
          for (int k = 0; k < 5; ++k) lu[k] = u[k], le[k] = e[k];
          increment<L>(lu, le, g, t, s);
          increment<double>(u, e, gam, f, fs);
          const L tv = sqrtl(t[1] * t[1] + t[2] * t[2] + t[3] * t[3]);
          ++n;
          for (int k = 0; k < 5; ++k) {
            if (s[k] == 0) {
              if (dw[k] != 0) worst = 1e9L;
              continue;
            }
            worst = std::max(worst, (fabsl(dw[k] - t[k]) - ldexpl(fabsl(t[k]), -53)) / s[k]);
            const L r = k >= 1 && k < 4 ? tv : fabsl(t[k]);
            if (r == 0) continue;
            mean[k] += fabsl(dw[k] - t[k]) / r;
            mean64[k] += fabsl(f[k] - t[k]) / r;
          }
        }
        printf("increment %g %g %g out %d units %.3Lf mean", gam, mach, del, out, ldexpl(worst, 53));
        for (int k = 0; k < 5; ++k) printf(" %.3Lf %.3Lf", ldexpl(mean[k] / std::max(n, 1), 53), ldexpl(mean64[k] / std::max(n, 1), 53));
        puts("");
      }
  // changes that must be left to FP64
  const double inf = INFINITY, nan = NAN, u[5] = {1, 0.1, 0, 0, 2};
  const double bad[][5] = {{0.03, 0, 0, 0, 0}, {-0.03, 0, 0, 0, 0}, {0, 0, 0, 0, 0.2}, {nan, 0, 0, 0, 0}, {0, nan, 0, 0, 0},
                           {0, 0, 0, 0, nan},  {inf, 0, 0, 0, 0},   {0, 0, -inf, 0, 0}, {0, 0, 0, 0, inf}, {1e200, 0, 0, 0, 0},
                           {-2, 0, 0, 0, 0},   {0, 1, 0, 0, 0}};
  double dw[5];
  for (auto& e : bad) printf("bad %d\n", fx_increment(u, e, fx(3) << 60, 4, fx(5) << 59, 2, dw));
  int taken = 0;
  for (double x = 0.0205; x < 4; x *= 1.01)
    for (int k : {0, 4})
      for (double sign : {-1.0, 1.0}) {
        double e[5] = {};
        e[k] = sign * x * u[k] * (k ? 1.01 : 1.0);
        taken += fx_increment(u, e, fx(3) << 60, 4, fx(5) << 59, 2, dw);
      }
  printf("wide %d\n", taken);
  const double zero[5] = {};
  const bool ok = fx_increment(u, zero, fx(3) << 60, 4, fx(5) << 59, 2, dw);
  printf("zero %d %g %g %g %g %g\n", ok, dw[0], dw[1], dw[2], dw[3], dw[4]);
  return 0;
}
