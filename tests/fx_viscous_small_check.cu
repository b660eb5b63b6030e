// Host check of csrc/es_viscous_fx.cuh: the viscous flux of a node whose gradients are far below the largest that
// the element's scales hold, against long double, in units of 2^-53 of the flux that the node's own
// largest gradient gives.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>

#include "es_viscous_fx.cuh"

using namespace es;
typedef long double L;

int main() {
  std::mt19937_64 R(11);
  std::uniform_real_distribution<double> U(-1, 1);
  for (double mach : {1e-5, 0.1, 1.0, 3.0})
    for (double size : {0.5, 0.05, 1e-3, 1e-6}) {
      L wt = 0, wh = 0;
      for (int it = 0; it < 4000; ++it) {
        const double z1 = exp(8 * U(R)), mu = exp(20 * U(R)), kap = exp(20 * U(R)), iz1 = 1 / z1;
        // e1: the element's largest z1, up to 8 times this node's; ev: the largest |z_v|
        int e1 = ilogb(z1) + 1 + it % 3, ev = std::max(ilogb(mach) + 1 + it % 2, -100);
        const int ut = int(30 * U(R)) - 40;
        fx t[3][4], nz[3];
        L th[3][4], v[3], f[3][4];
        for (int m = 0; m < 3; ++m)
          for (int c = 0; c < 4; ++c) {
            t[m][c] = fx(U(R) * size * 0x1p62);
            th[m][c] = ldexpl((L)t[m][c], c < 3 ? ut : ut - ev + e1);
          }
        L big = 0;  // as a fraction of 2^62
        for (int m = 0; m < 3; ++m)
          for (int c = 0; c < 4; ++c) big = std::max(big, ldexpl(fabsl((L)t[m][c]), -62));
        for (int k = 0; k < 3; ++k) {
          const double z = mach * (it % 5 == 4 ? 0.999 : U(R));
          nz[k] = fx_from_double(z, ev + 1022);
          v[k] = (L)z * iz1;
        }
        FxViscous V;
        V.emu = ilogb(mu) + 1;
        V.ekap = ilogb(kap) + 1;
        V.mu = fx_from_positive(mu, V.emu + 1022);
        V.kap = fx_from_positive(kap, V.ekap + 1022);
        double o[3][4];
        fx_viscous_flux(t, nz, iz1, e1, ev, ut, V, o);
        const L a = (L)iz1 * iz1, st = mu * a * big * ldexpl(1, 62 + ut), sh = kap * a * a * big * ldexpl(1, 62 + ut - ev + e1);
        L b[3][3];
        for (int m = 0; m < 3; ++m)
          for (int k = 0; k < 3; ++k) b[m][k] = th[m][k] - v[k] * th[m][3];
        const L tr = b[0][0] + b[1][1] + b[2][2];
        for (int m = 0; m < 3; ++m) {
          f[m][3] = -kap * a * a * th[m][3];
          for (int k = 0; k < 3; ++k) {
            f[m][k] = mu * a * (b[m][k] + b[k][m] - (m == k ? tr * 2 / 3 : 0));
            f[m][3] += f[m][k] * v[k];
            wt = std::max(wt, (fabsl(o[m][k] - f[m][k]) - ldexpl(fabsl(f[m][k]), -53)) / st);
          }
          const L vm = ldexpl(1, ev) * iz1;
          wh = std::max(wh, (fabsl(o[m][3] - f[m][3]) - ldexpl(fabsl(f[m][3]), -53)) / (sh + st * vm));
        }
      }
      printf("viscous %g %g ulps %.2Lf %.2Lf\n", mach, size, ldexpl(wt, 53), ldexpl(wh, 53));
    }
  return 0;
}
