// Host check of the relaxation's early decisions (csrc/es_relax_fx.cuh) against long double: an element
// taken for unconstrained by its largest increment alone, and a root kept from the series.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "es_relax_fx.cuh"

using namespace es;
typedef long double L;

int main() {
  std::mt19937_64 R(3);
  std::uniform_real_distribution<double> U(-1, 1);
  for (double gam : {1.0626, 1.4, 5.0 / 3.0, 2.9}) {
    int wrong = 0, below = 0;
    for (int it = 0; it < 40000; ++it) {
      // a node: X, Y, W of its increment, and a floor about its RMS change
      const double rho = exp(3 * U(R)), p = exp(3 * U(R)), size = ldexp(1.0, -56 - it % 500);
      double u[5], d[5], v[3];
      u[0] = rho;
      u[4] = p / (gam - 1);
      for (int k = 0; k < 3; ++k) {
        v[k] = 0.5 * U(R) * sqrt(p / rho);
        u[1 + k] = rho * v[k];
        u[4] += rho * v[k] * v[k] / 2;
      }
      d[0] = rho * size * U(R);
      for (int k = 0; k < 3; ++k) d[1 + k] = rho * sqrt(p / rho) * size * U(R);
      d[4] = u[4] * size * U(R);
      FxRelaxNode n;
      if (!fx_relax_node(u, d, n)) continue;
      L W = 0, Y = d[4];
      const L e = (L)u[4] - ((L)u[1] * u[1] + (L)u[2] * u[2] + (L)u[3] * u[3]) / (2 * (L)rho);
      for (int k = 0; k < 3; ++k) {
        const L vk = (L)u[1 + k] / u[0], q = d[1 + k] - vk * d[0];
        W += q * q / (2 * (L)rho * e);
        Y -= vk * (d[1 + k] + q) / 2;
      }
      Y /= e;
      const L X = (L)d[0] / rho, change = sqrtl(X * X + ((X - Y) * (X - Y) + 2 * W) / (gam - 1));
      const double floor = it % 3 == 2 ? (it % 2 ? 1e-8 : 1e-160) : (double)(change * (1 + 20 * fabs(U(R)) * (it % 3)));
      if (!fx_relax_below_floor(fx_relax_bits(n), floor, 1 / (gam - 1))) continue;
      ++below;
      wrong += change > (L)floor;
    }
    const double zero[5] = {}, u[5] = {1, 0, 0, 0, 2};
    FxRelaxNode n;
    const bool ok = fx_relax_node(u, zero, n) && fx_relax_below_floor(fx_relax_bits(n), 1e-140, 1 / (gam - 1)) &&
                    fx_relax_below_floor(fx_relax_bits(n), INFINITY, 1 / (gam - 1));
    printf("floor %g below %d wrong %d unchanged %d\n", gam, below, wrong, ok);
    // the root's q from the sum's estimate: inside 0.5 .. 1.5 never refused, outside 0.498 .. 1.502 always
    int eg, refused = 0, kept = 0, in = 0;
    const fx g1 = llrintl(ldexpl(frexpl((L)gam - 1, &eg), 63));
    for (int it = 0; it < 200000; ++it) {
      const int E = -2 - it % 49, er = it % 61 - 30;
      const double J = exp(20 * U(R)), want = it % 2 ? 1 + 0.6 * U(R) : exp(80 * U(R));
      const float est = ldexpf(1 + fabsf(U(R)), it % 90 - 60);
      const double A = -(double)(want * (L)J * est / ((L)gam - 1) * ldexpl(1, 2 * E + er + 4));
      const bool near = fx_relax_near_one(est, E, er, A, J, g1, eg);
      if (want >= 0.5 && want <= 1.5) {
        ++in;
        refused += !near;
      }
      kept += near && (want < 0.498 || want > 1.502);
    }
    printf("near %g in %d refused %d kept %d\n", gam, in, refused, kept);
  }
  return 0;
}
