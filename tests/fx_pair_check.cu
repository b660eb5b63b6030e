// Host check of the fixed-point two-point flux (csrc/es_fx.cuh) at the edges of its range.
//   slow  gas slower than the velocities' other scales: mass and energy flux relative to themselves
//   room  the room that fluxes beyond an element's scales are given
//   near  the logarithmic-mean correction and the flux up to the limit of the near tier
//   sums  sums along a line with the operators' own Q_ij, states at the corners of the range: a sum that leaves
//         2^61 is seen, though it may wrap past 2^63
//   metrics  rates of an element with anisotropic metrics, flow along the coarse direction
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include "es_fx.cuh"

using namespace es;
typedef long double L;

static L series(L r) {
  L s = 0;
  for (int k = 14; k >= 0; --k) s = s * r * r + 1.0L / (2 * k + 1);
  return s;
}
static void flux(const double* p, const double* q, L gam, L f[5]) {  // z1, z_m, z_a, z_b, z5
  L a[5], b[5];
  for (int k = 0; k < 5; ++k) a[k] = p[k], b[k] = q[k];
  const L s1 = a[0] + b[0], s5 = a[4] + b[4];
  const L f1 = series((a[0] - b[0]) / s1), g = 1 / series((a[4] - b[4]) / s5);
  const L u = (a[1] + b[1]) / s1, v = (a[2] + b[2]) / s1, w = (a[3] + b[3]) / s1, p1 = s5 / s1;
  const L m = s1 * s5 * g / 4 * u;
  f[0] = m;
  f[1] = m * u + p1;
  f[2] = m * v;
  f[3] = m * w;
  f[4] = u * gam / (gam - 1) * p1 * ((gam + 1) / (2 * gam) * g * f1 + (gam - 1) / (2 * gam)) + m * (u * u + v * v + w * w) / 2;
}

// the FP64 kernels' form of it
static void flux_double(const double* a, const double* b, double g, double f[5]) {
  const double S1 = a[0] + b[0], S5 = a[4] + b[4], P15 = S1 * S5, inv = 1 / P15, inv1 = S5 * inv;
  const double r1 = (a[0] - b[0]) * inv1, r5 = (a[4] - b[4]) * (S1 * inv), u1 = r1 * r1, u5 = r5 * r5;
  const double f1 = 1 + u1 * (1.0 / 3 + u1 * (1.0 / 5 + u1 * (1.0 / 7)));
  const double g5 = 0.25 - u5 * (1.0 / 12 + u5 * (1.0 / 45 + u5 * (11.0 / 945)));
  const double rho = P15 * g5, u = (a[1] + b[1]) * inv1, v = (a[2] + b[2]) * inv1, w = (a[3] + b[3]) * inv1;
  const double p1 = S5 * inv1, mass = rho * u;
  const double p2 = p1 * (2 * (g + 1) / (g - 1) * (g5 * f1) + 0.5);
  f[0] = mass;
  f[4] = u * p2 + 0.5 * mass * (u * u + v * v + w * w);
}

struct Gas {
  fx C1;
  int kt = 0;
  explicit Gas(double gam) {
    const L c = 2 * ((L)gam + 1) / ((L)gam - 1);
    while (ldexpl(1, kt) <= c) ++kt;
    C1 = llrintl(ldexpl(c, 62 - kt));
  }
};

// |difference| of the pair's flux from long double beyond the result's rounding, Q |Q_ij|/4 with 65 bits;
// false outside the range
static bool pair(const double a[5], const double b[5], double gam, const Gas& gas, fx Q, L diff[5], L want[5], FxScale& s) {
  int mxv = 0;
  for (int k = 1; k < 4; ++k)
    mxv = std::max({mxv, fx_hi_word(a[k]) & 0x7fffffff, fx_hi_word(b[k]) & 0x7fffffff});
  s = fx_scale(std::max(fx_hi_word(a[0]), fx_hi_word(b[0])), std::min(fx_hi_word(a[0]), fx_hi_word(b[0])),
               std::max(fx_hi_word(a[4]), fx_hi_word(b[4])), std::min(fx_hi_word(a[4]), fx_hi_word(b[4])), mxv, gas.C1, gas.kt);
  if (s.tier == kFxSlow) return false;
  fx x[2][5], g[5];
  FxPair p[2][2];
  for (int i = 0; i < 2; ++i) {
    const double* z = i ? b : a;
    x[i][0] = fx_from_positive(z[0], s.e1);
    x[i][4] = fx_from_positive(z[4], s.e5);
    for (int k = 1; k < 4; ++k) x[i][k] = fx_from_double(z[k], s.ev);
    p[i][0] = fx_pair(x[i][0]);
    p[i][1] = fx_pair(x[i][4]);
  }
  if (s.tier == kFxNear) fx_flux<kFxNear>(x[0], p[0], x[1], p[1], Q, s, g);
  else fx_flux<kFxFar>(x[0], p[0], x[1], p[1], Q, s, g);
  flux(a, b, gam, want);
  for (int v = 0; v < 5; ++v) {
    want[v] *= ldexpl((L)Q, -65) * 8;
    diff[v] = fabsl(ldexpl((L)g[v], fx_unit(s, v)) - want[v]) - ldexpl(fabsl(want[v]), -53);
  }
  return true;
}

// LGL nodes, and per degree Q_ij = omega_i D_ij, 1/omega_i
struct Line {
  int n;
  L x[6], w[6], Q[6][6];
  explicit Line(int p) : n(p + 1) {
    L P[6];
    for (int i = 0; i < n; ++i) {
      x[i] = -cosl(3.14159265358979323846264338327950288L * i / p);
      for (int it = 0; it < 60; ++it) {
        L a = 1, b = x[i];
        for (int k = 1; k < p; ++k) {
          const L c = ((2 * k + 1) * x[i] * b - k * a) / (k + 1);
          a = b;
          b = c;
        }
        P[i] = b;
        if (i > 0 && i < p) x[i] += (a - x[i] * b) / ((p + 1) * b);
      }
      w[i] = 2 / (p * (p + 1) * P[i] * P[i]);
    }
    for (int i = 0; i < n; ++i)
      for (int j = 0; j < n; ++j) Q[i][j] = i == j ? 0 : w[i] * P[i] / (P[j] * (x[i] - x[j]));
  }
  fx q(int i, int j) const { return i == j ? 0 : llrintl(ldexpl(Q[i][j], 63)); }
};

// the line sums of n nodes (component order z1, z_m, the others, z5), exact
static void line_sums(const Line& l, const double (*z)[5], const FxScale& s, __int128 r[6][5]) {
  fx x[6][5];
  FxPair p[6][2];
  for (int i = 0; i < l.n; ++i) {
    x[i][0] = fx_from_positive(z[i][0], s.e1);
    x[i][4] = fx_from_positive(z[i][4], s.e5);
    for (int k = 1; k < 4; ++k) x[i][k] = fx_from_double(z[i][k], s.ev);
    p[i][0] = fx_pair(x[i][0]);
    p[i][1] = fx_pair(x[i][4]);
    for (int c = 0; c < 5; ++c) r[i][c] = 0;
  }
  for (int i = 0; i < l.n; ++i)
    for (int j = i + 1; j < l.n; ++j) {
      fx g[5];
      if (s.tier == kFxNear) fx_flux<kFxNear>(x[i], p[i], x[j], p[j], l.q(i, j), s, g);
      else fx_flux<kFxFar>(x[i], p[i], x[j], p[j], l.q(i, j), s, g);
      for (int c = 0; c < 5; ++c) {
        r[i][c] += g[c];
        r[j][c] -= g[c];
      }
    }
}
static FxScale scale(const double (*z)[5], int n, const Gas& gas) {
  int mx1 = 0, mn1 = 0x7fffffff, mx5 = 0, mn5 = 0x7fffffff, mxv = 0;
  for (int i = 0; i < n; ++i) {
    mx1 = std::max(mx1, fx_hi_word(z[i][0]));
    mn1 = std::min(mn1, fx_hi_word(z[i][0]));
    mx5 = std::max(mx5, fx_hi_word(z[i][4]));
    mn5 = std::min(mn5, fx_hi_word(z[i][4]));
    for (int k = 1; k < 4; ++k) mxv = std::max(mxv, fx_hi_word(z[i][k]) & 0x7fffffff);
  }
  return fx_scale(mx1, mn1, mx5, mn5, mxv, gas.C1, gas.kt);
}

int main(int argc, char** argv) {
  std::mt19937_64 R(31);
  std::uniform_real_distribution<double> U(-1, 1);
  L diff[5], want[5];
  FxScale s;
  if (!strcmp(argv[1], "slow"))
    for (double gam : {1.4, 5.0 / 3.0, 1.1, 4.0})
      for (double speed : {1e-3, 1e-5, 1e-6, 1e-7, 1e-8, 2e-9})
        for (double var : {0.0, 1e-4, 0.1}) {
          const Gas gas(gam);
          L mass = 0, energy = 0;
          int out = 0;
          for (int it = 0; it < 4000; ++it) {
            double z[2][5];
            const double z1 = exp(6 * U(R)), z5 = exp(6 * U(R)), v = speed * (1 + fabs(U(R)));
            for (auto& n : z) {
              n[0] = z1 * (1 - var * fabs(U(R)));
              n[4] = z5 * (1 - var * fabs(U(R)));
              n[1] = v * (1 + var * U(R));  // along the line
              n[2] = v * U(R);
              n[3] = v * U(R);
            }
            const fx Q = fx(ldexp(0.25 * (0.25 + 0.7 * fabs(U(R))), 62)) * 8 * (it % 2 ? 1 : -1);
            if (!pair(z[0], z[1], gam, gas, Q, diff, want, s)) {
              ++out;
              continue;
            }
            mass = std::max(mass, diff[0] / fabsl(want[0]));
            energy = std::max(energy, diff[4] / fabsl(want[4]));
          }
          printf("slow %g %g %g out %d mass %.2Lf energy %.2Lf\n", gam, speed, var, out, ldexpl(mass, 53), ldexpl(energy, 53));
        }
  if (!strcmp(argv[1], "room")) {
    int wrong = 0, fp64 = 0, taken = 0;
    for (int Ev = -29; Ev <= 2; ++Ev)
      for (int first = 0; first < 6; ++first)
        for (int dm = 0; dm < 12; ++dm)
          for (int de = 0; de < 45; ++de) {
            const int one = 1023 << 20, mxv = (1022 + Ev) << 20;  // z1 = z5 = 1, |z_v| = 2^(Ev - 1)
            FxScale a = fx_scale(one, one, one, one, mxv - (1 << 20) + 1, fx(3) << 60, 4);
            if (a.tier == kFxSlow) continue;
            a.se += first;
            FxScale b = a;
            fx_widen(b, dm, de);
            const int um = fx_unit(b, 1) - fx_unit(a, 1), ue = fx_unit(b, 4) - fx_unit(a, 4);
            const bool fits = dm <= 6 && first + de <= std::max(-(a.ev - 1022), 0) + 6;
            if (b.tier == kFxSlow) {
              ++fp64;
              wrong += fits;
            } else {
              ++taken;
              wrong += !fits || um < dm || ue < de || um > (dm ? dm + 3 : 0) || ue > (de ? de + 3 : 0);
            }
            wrong += b.sv < 0 || b.sv > 63 || b.se < 0 || b.se > 63;
          }
    printf("room wrong %d taken %d fp64 %d\n", wrong, taken, fp64);
  }
  if (!strcmp(argv[1], "near")) {
    // the correction alone, |r| up to 0.0101 by steps; the tier that the pair's high words give
    L worst = 0;
    int near = 0;
    for (int it = 0; it < 3000000; ++it) {
      const double r = 0.0101 * (it % 3 ? U(R) : (1 - 1e-3 * fabs(U(R))) * 0.5), b = it % 5 ? 1 + fabs(U(R)) : 2 - 1e-3 * fabs(U(R)), a = b * (1 + r) / (1 - r);
      const FxScale t = fx_scale(fx_hi_word(std::max(a, b)), fx_hi_word(std::min(a, b)), 1023 << 20, 1023 << 20, 1020 << 20, fx(3) << 60, 4);
      if (t.tier != kFxNear) continue;
      ++near;
      const FxPair x = fx_pair(fx_from_positive(a, t.e1)), y = fx_pair(fx_from_positive(b, t.e1));
      const float q = fx_rcpf(x.h + y.h);
      const L rr = ((L)a - b) / ((L)a + b), f = series(rr);
      worst = std::max(worst, fabsl(ldexpl((L)fx_near(x, y, q, 0.2f, 1.0f / 7.0f), -64) - (f - 1)));
      worst = std::max(worst, fabsl(ldexpl((L)fx_near(x, y, q, 4.0f / 45.0f, 44.0f / 945.0f), -64) - (1 - 1 / f)));
    }
    printf("correction %d units %.3Lf\n", near, ldexpl(worst, 53));
    // the flux relative to itself, and the FP64 formula's
    for (double gam : {1.4, 5.0 / 3.0, 1.1, 4.0})
      for (double mach : {1e-3, 0.3, 1.2, 3.0}) {
        const Gas gas(gam);
        L mean[2][2] = {}, most[2][2] = {};
        int n = 0;
        for (int it = 0; it < 60000; ++it) {
          double z[2][5], f[5];
          const double z1 = exp(6 * U(R)), z5 = exp(6 * U(R)), r = 0.0099 * (it % 2 ? 1 : fabs(U(R)));
          for (int i = 0; i < 2; ++i) {
            z[i][0] = z1 * (i ? (1 - r) / (1 + r) : 1);
            z[i][4] = z5 * (i ? 1 : (1 - r) / (1 + r));
            for (int k = 1; k < 4; ++k) z[i][k] = mach * (0.3 + 0.3 * fabs(U(R)));
          }
          if (!pair(z[0], z[1], gam, gas, 1ll << 62, diff, want, s) || s.tier != kFxNear) continue;
          flux_double(z[0], z[1], gam, f);
          ++n;
          for (int v : {0, 4}) {
            const L e[2] = {(diff[v] + ldexpl(fabsl(want[v]), -53)) / fabsl(want[v]), fabsl(f[v] / want[v] - 1)};
            for (int k = 0; k < 2; ++k) {
              mean[v / 4][k] += e[k];
              most[v / 4][k] = std::max(most[v / 4][k], e[k]);
            }
          }
        }
        printf("near %g %g pairs %d", gam, mach, n);
        for (auto& m : mean)
          for (L x : m) printf(" %.2Lf", ldexpl(x / n, 53));
        for (auto& m : most)
          for (L x : m) printf(" %.2Lf", ldexpl(x, 53));
        puts("");
      }
  }
  if (!strcmp(argv[1], "sums"))
    for (int p = 2; p <= 5; ++p) {
      const Line l(p);
      L largest = 0, q = 0;
      int missed = 0, beyond = 0, out = 0, n = 0;
      for (int i = 0; i <= p; ++i)
        for (int j = 0; j <= p; ++j) q = std::max(q, fabsl(l.Q[i][j]));
      for (double gam : {1.4, 5.0 / 3.0 + 1e-6, 1.1, 4.0})
        for (int it = 0; it < 30000; ++it) {
          // z1 and z5 at the ends of a factor 1.498 (near: 1.0098), from a power of two up or just below one
          const Gas gas(gam);
          const double f = it % 3 ? 1 / 1.498 : 1 / 1.0098, v = it % 2 ? 0.99999 : (it % 4 ? 1.99 : 3.99);
          const double lo1 = it % 5 ? 1.0000001 : 1.9999, lo5 = it % 7 ? 1.9999 : 1.0000001;
          double z[7][5];
          __int128 r[6][5];
          for (int i = 0; i < 7; ++i) {  // (node 7: elsewhere in the element, holds the scales)
            z[i][0] = i == 6 ? lo1 : lo1 * (U(R) > 0 ? 1 : f);
            z[i][4] = i == 6 ? lo5 : lo5 * (U(R) > 0 ? 1 : f);
            for (int k = 1; k < 4; ++k) z[i][k] = v * (i == 6 ? 1 : (it % 11 ? (U(R) > 0 ? 1 : -1) : U(R)));
          }
          const FxScale t = scale(z, 7, gas);
          if (t.tier == kFxSlow) {
            ++out;
            continue;
          }
          ++n;
          line_sums(l, z, t, r);
          for (int i = 0; i <= p; ++i)
            for (int c = 0; c < 5; ++c)
              for (int side = -1; side < 2; ++side) {  // with the largest face flux that is taken, or none
                const __int128 e = r[i][c] + (i == 0 || i == p ? (__int128)side << (t.tier == kFxNear ? 61 : 60) : 0);
                const fx w = fx(e);
                const bool seen = ((fx_hi(w) + 0x20000000) & 0xc0000000) != 0;
                largest = std::max(largest, fabsl((L)e));
                const bool big = e >= ((__int128)1 << 61) || e < -((__int128)1 << 61);
                beyond += big;
                missed += big != seen;
              }
        }
      printf("sums %d out %d beyond %d missed %d largest %.3Lf Q %.3Lf\n", p, out, beyond, missed, ldexpl(largest, -63), q);
    }
  if (!strcmp(argv[1], "metrics"))
    for (int p = 2; p <= 5; ++p)
      for (double ratio : {1.0, 3.9, 7.9, 15.9, 16.5, 17.5, 33.0, 1e3}) {
        // sums of the coarse direction, as the kernel joins them: r (1/omega) metric in units of the largest metric
        const Line l(p);
        const Gas gas(1.4);
        const double metric[3] = {1.9, 1.9 * ratio, 1.9 * ratio};
        L err[5] = {}, err64[5] = {}, top[5] = {};
        for (int it = 0; it < 300; ++it) {
          double z[6][5];
          const double a = 3 * U(R);
          for (int i = 0; i <= p; ++i) {
            const double x = (double)l.x[i];
            z[i][0] = 1.1 + 0.01 * sin(x + a);
            z[i][4] = 1.3 + 0.01 * cos(x - a);
            z[i][1] = 0.3 + 0.1 * sin(x + 2 * a);
            z[i][2] = 0.2 * cos(x + a);
            z[i][3] = 0;
          }
          const FxScale t = scale(z, p + 1, gas);
          __int128 r[6][5];
          line_sums(l, z, t, r);
          const int em = (fx_hi_word(metric[1])) >> 20;
          int kw = 0;
          while ((1 << kw) <= p * (p + 1) / 2) ++kw;
          for (int i = 0; i <= p; ++i) {
            const fx w = fx_mul63(llrintl(ldexpl(1 / l.w[i], 63 - kw)), fx_from_double(metric[0], em));
            L k[5] = {}, f[5];
            double k64[5] = {};
            for (int j = 0; j <= p; ++j) {
              if (j == i) continue;
              flux(z[i], z[j], 1.4, f);
              const double d = (double)(2 * l.Q[i][j] / l.w[i]);
              for (int c = 0; c < 5; ++c) {
                k[c] += 2 * l.Q[i][j] / l.w[i] * metric[0] * f[c];
                k64[c] = fma(d, (double)f[c], k64[c]);
              }
            }
            for (int c = 0; c < 5; ++c) {
              const L got = ldexpl((L)fx_mul63(fx(r[i][c]), w), fx_unit(t, c) + em - 1022 + kw + 1);
              top[c] = std::max(top[c], fabsl(k[c]));
              err[c] = std::max(err[c], fabsl(got - k[c]));
              err64[c] = std::max(err64[c], fabsl(metric[0] * k64[c] - k[c]));
            }
          }
        }
        printf("metrics %d %g taken %d", p, ratio, fx_metrics_close(metric));
        for (int c : {0, 1, 4}) printf(" %.2Le %.2Le", err[c] / top[c], err64[c] / top[c]);
        puts("");
      }
  return 0;
}
