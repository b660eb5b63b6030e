// Host check of csrc/es_fx.cuh against the same formulas in long double: prints, per range of
// states, the largest deviation of the five flux components in units of the result's last bit
// beyond 2^-53 of the component (the near branch's correction is good to 2^-54), and the branch
// taken for states outside the fixed-point range.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "es_fx.cuh"

using namespace es;
typedef long double L;

static void flux(const L* a, const L* b, L gam, L f[5]) {  // z1, z_m, z_a, z_b, z5
  const L s1 = a[0] + b[0], s5 = a[4] + b[4];
  auto F = [](L r) {
    if (fabsl(r) > 0.05L) return atanhl(r) / r;
    L s = 0;
    for (int k = 12; k >= 0; --k) s = s * r * r + 1.0L / (2 * k + 1);
    return s;
  };
  const L f1 = F((a[0] - b[0]) / s1), g = 1 / F((a[4] - b[4]) / s5);
  const L u = (a[1] + b[1]) / s1, v = (a[2] + b[2]) / s1, w = (a[3] + b[3]) / s1, p1 = s5 / s1;
  const L m = s1 * s5 * g / 4 * u;
  const L p2 = p1 * ((gam + 1) / (2 * gam) * g * f1 + (gam - 1) / (2 * gam));
  f[0] = m;
  f[1] = m * u + p1;
  f[2] = m * v;
  f[3] = m * w;
  f[4] = u * gam / (gam - 1) * p2 + m * (u * u + v * v + w * w) / 2;
}

static FxScale scale_of(const double z[][5], int n, fx C1, int ktg) {
  int mx1 = 0, mn1 = 0x7fffffff, mx5 = 0, mn5 = 0x7fffffff, mxv = 0;
  for (int i = 0; i < n; ++i) {
    mx1 = std::max(mx1, fx_hi_word(z[i][0]));
    mn1 = std::min(mn1, fx_hi_word(z[i][0]));
    mx5 = std::max(mx5, fx_hi_word(z[i][4]));
    mn5 = std::min(mn5, fx_hi_word(z[i][4]));
    for (int k = 1; k < 4; ++k) mxv = std::max(mxv, fx_hi_word(z[i][k]) & 0x7fffffff);
  }
  return fx_scale(mx1, mn1, mx5, mn5, mxv, C1, ktg);
}

int main() {
  std::mt19937_64 R(20);
  std::uniform_real_distribution<double> U(-1, 1);
  for (double gam : {1.4, 5.0 / 3.0, 1.1, 4.0}) {
    const L c = 2 * ((L)gam + 1) / ((L)gam - 1);
    int ktg = 0;
    while (ldexpl(1, ktg) <= c) ++ktg;
    const fx C1 = llrintl(ldexpl(c, 62 - ktg));
    for (double var : {0.0, 1e-12, 1e-6, 1e-3, 9.9e-3, 0.05, 0.19})
      for (double mach : {1e-7, 1e-3, 0.3, 1.2, 3.0}) {
        L worst[3] = {0, 0, 0};
        int slow = 0;
        for (int it = 0; it < 400; ++it) {
          double z[2][5];
          double z1 = exp(6 * U(R)), z5 = exp(6 * U(R));
          if (it % 4 == 1) z1 = 1 - 1e-11 * fabs(U(R));  // just below powers of two
          if (it % 4 == 2) z5 = 2 * (1 - 1e-13 * fabs(U(R)));
          for (auto& n : z) {
            n[0] = z1 * (1 - var * fabs(U(R)));
            n[4] = z5 * (1 - var * fabs(U(R)));
            for (int k = 1; k < 4; ++k) n[k] = mach * U(R);
          }
          const FxScale s = scale_of(z, 2, C1, ktg);
          if (s.tier == kFxSlow) {
            ++slow;
            continue;
          }
          fx a[2][5];
          FxPair p[2][2];
          L l[2][5], f[5];
          for (int i = 0; i < 2; ++i) {
            for (int k = 0; k < 5; ++k) l[i][k] = z[i][k];
            a[i][0] = fx_from_positive(z[i][0], s.e1);
            a[i][4] = fx_from_positive(z[i][4], s.e5);
            for (int k = 1; k < 4; ++k) a[i][k] = fx_from_double(z[i][k], s.ev);
            p[i][0] = fx_pair(a[i][0]);
            p[i][1] = fx_pair(a[i][4]);
          }
          const fx Q = fx(ldexp(0.17 * U(R), 62)) * 8;
          fx g[5];
          if (s.tier == kFxNear) fx_flux<kFxNear>(a[0], p[0], a[1], p[1], Q, s, g);
          else fx_flux<kFxFar>(a[0], p[0], a[1], p[1], Q, s, g);
          flux(l[0], l[1], gam, f);
          for (int v = 0; v < 5; ++v) {
            const L e = f[v] * ldexpl((L)Q, -65) * 8;
            const L d = fabsl(ldexpl((L)g[v], fx_unit(s, v)) - e) - ldexpl(fabsl(e), -53);
            const int t = v == 0 ? 0 : (v == 4 ? 2 : 1);
            worst[t] = std::max(worst[t], ldexpl(d, -fx_unit(s, v)));
            const double back = fx_to_double(g[v], fx_unit(s, v));
            if (fabsl(back - ldexpl((L)g[v], fx_unit(s, v))) > ldexpl(fabsl((L)back), -53)) worst[t] = 1e9L;
          }
        }
        printf("pair %g %g %g slow %d units %.1Lf %.1Lf %.1Lf\n", gam, var, mach, slow, worst[0], worst[1], worst[2]);
      }
  }
  const double inf = std::numeric_limits<double>::infinity(), nan = std::numeric_limits<double>::quiet_NaN();
  const double bad[][2][5] = {{{1, .1, 0, 0, 1}, {1, .1, 0, 0, nan}},    {{inf, .1, 0, 0, 1}, {1, .1, 0, 0, 1}},
                              {{1, .1, 0, 0, 1}, {-1, .1, 0, 0, 1}},     {{1, nan, 0, 0, 1}, {1, .1, 0, 0, 1}},
                              {{1, .1, 0, 0, 1}, {1.6, .1, 0, 0, 1}},    {{1, .1, 0, 0, 1}, {1, .1, 0, 0, 0.6}},
                              {{1, 5, 0, 0, 1}, {1, .1, 0, 0, 1}},       {{1, 1e-12, 0, 0, 1}, {1, 0, 0, 0, 1}},
                              {{1e-80, .1, 0, 0, 1}, {1e-80, .1, 0, 0, 1}}, {{1, .1, 0, 0, 0}, {1, .1, 0, 0, 0}},
                              {{-nan, .1, 0, 0, 1}, {1, .1, 0, 0, 1}},   {{1, -inf, 0, 0, 1}, {1, .1, 0, 0, 1}}};
  for (auto& z : bad) printf("bad %d\n", scale_of(z, 2, fx(3) << 60, 4).tier);
  return 0;
}
