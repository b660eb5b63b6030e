// Host check of csrc/es_relax_fx.cuh: the root of one element's relaxation function against long double
// (Newton on the node sums with log1p), per size of the increment, Mach number and gas constant.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "es_relax_fx.cuh"

using namespace es;
typedef long double L;

// gamma of the element in fixed point; 0: outside the range
static double root_fx(int n, const double (*u)[5], const double (*d)[5], const double* w, double J, double A, fx g1, int eg) {
  static FxRelaxNode nd[216];
  static FxRelaxTerm t[216];
  static FxRelaxSeries s[216];
  static FxRelaxSeriesF f[216];
  int bits = kRelaxNone, er = kRelaxNone, ex[216];
  fx cd[216];
  for (int i = 0; i < n; ++i) {
    if (!fx_relax_node(u[i], d[i], nd[i])) return 0;
    bits = std::max(bits, fx_relax_bits(nd[i]));
    er = std::max(er, nd[i].er);
  }
  const int E = bits + 2;
  if (E > kRelaxMaxE || E < kRelaxMinE) return 0;
  float est = 0;
  for (int i = 0; i < n; ++i) {
    t[i] = fx_relax_term(nd[i], E, er, 0.125 * w[i]);
    cd[i] = fx_relax_d2(nd[i], t[i], fx_relax_bits(nd[i]), E, g1, eg, ex + i);
    est += fx_relax_estimate(cd[i], ex[i]);
  }
  fx a = 0, T[kRelaxOrders + 1];
  float Tf[kRelaxOrders + 1];
  const int unit = fx_relax_unit(est);
  for (int i = 0; i < n; ++i) {
    a += fx_shift(cd[i], ex[i] + unit);
    s[i] = fx_relax_series(t[i], unit);
  }
  const int kl = fx_relax_last(E), kf = fx_relax_first_f(E);
  const fx gp1 = fx_relax_gp1(g1, eg);
  for (int k = 3; k < kf; ++k) {
    fx sp = 0, sm = 0, sx = 0;
    for (int i = 0; i < n; ++i) fx_relax_next(s[i], sp, sm, sx);
    T[k] = fx_relax_coefficient(k, sp, sm, sx, gp1);
    Tf[k] = fx_fraction(T[k]);
  }
  for (int i = 0; i < n; ++i) f[i] = fx_relax_series_f(s[i]);
  for (int k = kf; k <= kl; ++k) {
    float sp = 0, sm = 0, sx = 0;
    for (int i = 0; i < n; ++i) fx_relax_next_f(f[i], sp, sm, sx);
    Tf[k] = fx_relax_coefficient_f(k, sp, sm, sx, gp1);
  }
  return ldexp((double)fx_relax_root(a, unit, E, er, kf, kl, T, Tf, A, J, g1, eg), -61);
}

// r(g)/g - A and its derivative in long double
static L sum_ld(int n, const double (*u)[5], const double (*d)[5], const double* w, L J, L gam, L g) {
  L r = 0;
  for (int i = 0; i < n; ++i) {
    const double *a = u[i], *b = d[i];
    const L v[3] = {a[1] / (L)a[0], a[2] / (L)a[0], a[3] / (L)a[0]};
    const L e = a[4] - (a[1] * v[0] + a[2] * v[1] + a[3] * v[2]) / 2;
    L W = 0, Y = b[4];
    for (int k = 0; k < 3; ++k) {
      const L q = b[1 + k] - v[k] * b[0];
      W += q * q / (2 * a[0] * e);
      Y -= v[k] * (b[1 + k] + q) / 2;
    }
    Y /= e;
    const L X = b[0] / (L)a[0], x = g * X, al = X + Y, be = X * Y - W;
    // (1 + x) ((gam+1) l(x) - l(w)) + second-order terms, l(z) = log1p(z) - z
    auto l = [](L z) {
      if (fabsl(z) > 0.02L) return log1pl(z) - z;
      L s = 0;
      for (int k = 14; k >= 2; --k) s = s * z + (k % 2 ? 1.0L : -1.0L) / k;
      return s * z * z;
    };
    const L om = g * al + g * g * be;
    r += w[i] * J * a[0] / (gam - 1) * ((1 + x) * ((gam + 1) * l(x) - l(om)) + (gam + 1) * x * x - x * om - g * g * be);
  }
  return r / g;
}

int main() {
  std::mt19937_64 R(5);
  std::uniform_real_distribution<double> U(-1, 1);
  for (double gam : {1.4, 5.0 / 3.0, 1.1})
    for (double mach : {1e-4, 0.1, 1.0, 4.0})
      for (double del : {1e-9, 1e-6, 1e-4, 1e-3, 6e-3, 2e-2})
        for (int p : {2, 3, 5}) {
          int eg, out = 0;
          const fx g1 = llrintl(ldexpl(frexpl((L)gam - 1, &eg), 63));
          const int n = (p + 1) * (p + 1) * (p + 1);
          const double w3[6][6] = {{0}, {0}, {1. / 3, 4. / 3, 1. / 3}, {1. / 6, 5. / 6, 5. / 6, 1. / 6}, {0},
                                   {1. / 15, 0.37847495629784698, 0.55485837703548635, 0.55485837703548635,
                                    0.37847495629784698, 1. / 15}};
          L worst = 0, mean = 0;
          int cnt = 0;
          for (int it = 0; it < 60; ++it) {
            static double u[216][5], d[216][5], w[216];
            const double rho = exp(5 * U(R)), pr = exp(5 * U(R)), c = sqrt(gam * pr / rho), J = exp(3 * U(R));
            for (int i = 0; i < n; ++i) {
              w[i] = w3[p][i % (p + 1)] * w3[p][i / (p + 1) % (p + 1)] * w3[p][i / (p + 1) / (p + 1)];
              const double r = rho * (1 + 0.2 * U(R)), P = pr * (1 + 0.2 * U(R));
              double v[3], k2 = 0, dE;
              for (int k = 0; k < 3; ++k) v[k] = mach * c * U(R), u[i][1 + k] = r * v[k], k2 += v[k] * v[k];
              u[i][0] = r;
              u[i][4] = P / (gam - 1) + r * k2 / 2;
              // kinds: independent, acoustic, shear, one large node
              const int kind = it % 4;
              const double big = kind == 3 && i ? 0.05 * del : del;
              const double dr = (kind == 2 ? 0 : big) * r * U(R), dp = kind == 1 ? gam * P / r * dr : (kind == 2 ? 0 : big * P * U(R));
              d[i][0] = dr;
              dE = dp / (gam - 1) + dr * k2 / 2;
              for (int k = 0; k < 3; ++k) {
                const double dv = (kind == 1 ? 0.1 : 1.0) * big * c * U(R);
                d[i][1 + k] = v[k] * dr + r * dv;
                dE += r * v[k] * dv;
              }
              d[i][4] = dE;
            }
            const L gt = 1 + 0.1L * (L)U(R);
            const double A = -(double)sum_ld(n, u, d, w, J, gam, gt);
            L g = gt;  // root for the rounded A: the sum is close to linear in g
            for (int k = 0; k < 60; ++k) {
              const L step = g * (sum_ld(n, u, d, w, J, gam, g) + A) / A;
              g += step;
              if (fabsl(step) < 1e-19L) break;
            }
            const double f = root_fx(n, u, d, w, J, A, g1, eg);
            if (f == 0) {
              ++out;
              continue;
            }
            worst = std::max(worst, fabsl(f - g) / g);
            mean += fabsl(f - g) / g;
            ++cnt;
          }
          printf("root %g %g %g %d out %d ulps %.2Lf mean %.2Lf\n", gam, mach, del, p, out, ldexpl(worst, 53),
                 ldexpl(mean / std::max(cnt, 1), 53));
        }
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double ok[5] = {1, 0.1, 0, 0, 2.5};
  const double bad[][5] = {{nan, 0, 0, 0, 0}, {0, nan, 0, 0, 0}, {0, 0, inf, 0, 0}, {0, 0, 0, 0, nan}, {inf, 0, 0, 0, 1}};
  const double badu[][5] = {{-1, 0, 0, 0, 1}, {1, 0, 0, 0, -1}, {1, 2, 0, 0, 1}, {nan, 0, 0, 0, 1}, {1, nan, 0, 0, 1},
                            {1, 0, 0, 0, inf}, {0, 0, 0, 0, 1}, {1, 0, inf, 0, inf}};
  FxRelaxNode nd;
  for (auto& d : bad) printf("outd %d\n", fx_relax_node(ok, d, nd));
  for (auto& u : badu) printf("outu %d\n", fx_relax_node(u, ok, nd));
  return 0;
}
