// Host check of csrc/es_fx.cuh against the same formulas in long double: prints, per range of
// states, the largest deviation of the five flux components in units of the result's last bit
// beyond 2^-53 of the component (the near branch's correction is good to 2^-54), and the branch
// taken for states outside the fixed-point range.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>
#include <random>

#include "es_face_fx.cuh"
#include "es_prep_fx.cuh"

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
  for (double gam : {1.4, 5.0 / 3.0, 1.1}) {
    const L g = gam, c = 2 * (g + 1) / (g - 1);
    int ktg = 0, eg;
    while (ldexpl(1, ktg) <= c) ++ktg;
    const fx C1 = llrintl(ldexpl(c, 62 - ktg)), g1 = llrintl(ldexpl(frexpl(g - 1, &eg), 63));
    for (double mach : {1e-6, 0.1, 1.0, 3.0})
      for (double del : {1e-9, 1e-5, 8e-3}) {
        L wz = 0, ww = 0;
        int out = 0;
        for (int it = 0; it < 1000; ++it) {
          double rho = exp(5 * U(R)), p = exp(5 * U(R));
          if (it % 4 == 1) {  // rho p at and next to powers of two
            rho = ldexp(1.0, it % 7 - 3) * (1 - 1e-13 * (it % 3) * U(R));
            p = ldexp(1.0, it % 5 - 2) / rho;
          }
          const double a = sqrt(gam * p / rho);
          double q[2][5];
          L z[2][6];
          for (int i = 0; i < 2; ++i) {
            const double r = rho * (1 + i * del * U(R)), pr = p * (1 + i * del * U(R));
            double v[3], k2 = 0;
            for (int k = 0; k < 3; ++k) {
              v[k] = i ? q[0][1 + k] / rho + a * del * U(R) : mach * a * 0.57 * U(R);
              q[i][1 + k] = r * v[k];
              k2 += v[k] * v[k];
            }
            q[i][0] = r;
            q[i][4] = pr / (gam - 1) + 0.5 * r * k2;
            const double* y = q[i];
            const L Pr = (g - 1) * ((L)y[0] * y[4] - ((L)y[1] * y[1] + (L)y[2] * y[2] + (L)y[3] * y[3]) / 2);
            for (int k = 0; k < 4; ++k) z[i][k] = y[k] / sqrtl(Pr);
            z[i][4] = sqrtl(Pr);
            z[i][5] = 1 / z[i][0];
          }
          FxState s[2];
          double o[6], dw[5];
          if (!fx_state(q[0], g1, eg, s[0]) || !fx_state(q[1], g1, eg, s[1]) || !fx_increment(s[0], s[1], C1, ktg, dw)) {
            ++out;
            continue;
          }
          fx_state_planes(s[1], o);
          const L zv = std::max(fabsl(z[1][1]), std::max(fabsl(z[1][2]), fabsl(z[1][3])));
          L t[5] = {(g + 1) / (g - 1) * logl(z[1][0] / z[0][0]) + logl(z[1][4] / z[0][4])};
          for (int k = 1; k < 4; ++k) {
            t[0] -= (z[1][k] * z[1][k] - z[0][k] * z[0][k]) / 2;
            t[k] = z[1][0] * z[1][k] - z[0][0] * z[0][k];
          }
          t[4] = z[0][0] * z[0][0] - z[1][0] * z[1][0];
          for (int k = 0; k < 6; ++k)
            wz = std::max(wz, fabsl(o[k] - z[1][k]) / (k >= 1 && k < 4 ? zv : z[1][k]));
          // scales of the components: C1x + |z_v|^2, z1 (1 + |z_v|), z1^2
          for (int k = 0; k < 5; ++k)
            ww = std::max(ww, fabsl(dw[k] - t[k]) / (k == 0 ? c + zv * zv : z[0][0] * (k < 4 ? 1 + zv : 2 * z[0][0])));
        }
        printf("state %g %g %g out %d ulps %.2Lf %.3Lf\n", gam, mach, del, out, ldexpl(wz, 53), ldexpl(ww, 53));
      }
  }
  for (double gam : {1.4, 5.0 / 3.0, 1.1}) {
    const L c = 2 * ((L)gam + 1) / ((L)gam - 1);
    int ktg = 0;
    while (ldexpl(1, ktg) <= c) ++ktg;
    const fx C1 = llrintl(ldexpl(c, 62 - ktg));
    for (int diss : {0, 1})
      for (double var : {0.0, 1e-6, 9e-3, 0.18})
        for (double mach : {1e-4, 0.1, 1.0, 2.5}) {
          L worst = 0;
          int out = 0;
          for (int it = 0; it < 600; ++it) {
            const double z1 = it % 4 == 1 ? 1 - 1e-14 * (it % 5) : exp(5 * U(R)), z5 = it % 4 == 2 ? 1 - 1e-14 : exp(5 * U(R));
            double z[2][5], f[5];
            for (int i = 0; i < 2; ++i) {
              z[i][0] = z1 * (1 - (i ? var * fabs(U(R)) : 0.0));
              z[i][4] = z5 * (1 - (i ? 0.0 : var * fabs(U(R))));
              for (int k = 1; k < 4; ++k) z[i][k] = i ? z[0][k] + mach * sqrt(var) * U(R) : mach * U(R);
            }
            const int m = it % 3;
            if (!fx_face_flux(z[0], z[1], m, C1, ktg, sqrt(gam), diss, f)) {
              ++out;
              continue;
            }
            L l[2][5], w[5], q[2][5], lam = 0;  // rotated: z1, z_m, the next two, z5
            for (int i = 0; i < 2; ++i) {
              const int at[5] = {0, 1 + m, 1 + (m + 1) % 3, 1 + (m + 2) % 3, 4};
              for (int k = 0; k < 5; ++k) l[i][k] = z[i][at[k]];
              q[i][0] = l[i][0] * l[i][4];
              q[i][4] = l[i][4] / l[i][0] * (1 / ((L)gam - 1) + (l[i][1] * l[i][1] + l[i][2] * l[i][2] + l[i][3] * l[i][3]) / 2);
              for (int k = 1; k < 4; ++k) q[i][k] = l[i][4] * l[i][k];
              lam = std::max(lam, (fabsl(l[i][1]) + sqrtl(gam)) / l[i][0]);
            }
            flux(l[0], l[1], gam, w);
            for (int k = 0; k < 5; ++k) w[k] -= diss * lam / 2 * (q[1][k] - q[0][k]);
            const L p = (L)z5 / z1, rate = (diss ? sqrtl(gam) : 0) + mach;
            const L sc[5] = {(L)z5 * rate, p * (1 + mach * rate), p * (1 + mach * rate), p * (1 + mach * rate),
                             p / z1 * rate * (1 / ((L)gam - 1) + 1 + mach * mach / 2)};
            const int to[5] = {0, 1 + m, 1 + (m + 1) % 3, 1 + (m + 2) % 3, 4};
            for (int k = 0; k < 5; ++k) worst = std::max(worst, fabsl(f[to[k]] - w[k]) / sc[k]);
          }
          printf("face %g %d %g %g out %d ulps %.2Lf\n", gam, diss, var, mach, out, ldexpl(worst, 53));
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
  const double badq[][5] = {{-1, 0, 0, 0, 1}, {1, 0, 0, 0, -1}, {1, 2, 0, 0, 1},    {nan, 0, 0, 0, 1}, {1, nan, 0, 0, 1},
                            {1, 0, 0, 0, inf}, {0, 0, 0, 0, 1}, {1, inf, 0, 0, inf}, {1e-200, 0, 0, 0, 1}, {1, 0, 0, 1.5, 1.1}};
  FxState st;
  for (auto& q : badq) printf("outq %d\n", fx_state(q, fx(0x6666666666666666ll), -1, st));
  return 0;
}
