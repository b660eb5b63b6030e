// The FP64 mode's interface flux in 64-bit fixed point (es_fx.cuh): the two-point flux of a pair
// of face nodes in the scales of that pair, and the Rusanov dissipation lambda/2 [[q]] from the
// same fractions.  An FP64 face node takes 42 + 44 FP64 instructions, each the time of ~76 of one
// scheduler's; this takes about 900 integer and FP32 ones.  Taylor--Green 32^3 p = 3: k_face
// 244 -> 101 us per launch, with the launch shape of k_face_fp64.
#pragma once
#include "es_fx.cuh"

namespace es {

// a b 2^ex 2^64 rounded to a double, b of any magnitude below 2^62
ES_HD double fx_product(fx a, fx b, int ex) {
  const fx n = b < 0 ? -b : b;
  const int sh = n ? fx_clz(uint64_t(n)) - 2 : 0;
  return fx_to_double(fx_mul(a, b << sh), ex - sh);
}

// f_num(L, R) along x_m: the EC flux, with diss = 1 less lambda/2 (q_R - q_L); a, b: z1..z5 of the
// two sides.  False where the pair is outside the fixed-point range (fx_scale).
//
// Dissipation, in fractions x of the scales A1, Av, A5 = 2^(E + 1):
//   rho = x1 x5, m_k = x5 x_k, E = (x5/x1) e, e = 1/(gam-1) + |z_v|^2/2 (scaled by 2^-kt),
//   lambda = max (sqrt(gam) + |z_m|)/z1 (the numerator scaled by 1/8).
// The jumps are differences of 60..62-bit products, so that a jump keeps its leading bits; flux and
// dissipation are rounded once each and joined by one FP64 subtraction.
ES_HD bool fx_face_flux(const double a[5], const double b[5], int m, fx C1, int ktg, double sqrt_gam, int diss,
                        double f[5]) {
  const int h1a = fx_hi_word(a[0]), h1b = fx_hi_word(b[0]), h5a = fx_hi_word(a[4]), h5b = fx_hi_word(b[4]);
  int mxv = 0;
#pragma unroll
  for (int k = 1; k < 4; ++k) {
    const int ha = fx_hi_word(a[k]) & 0x7fffffff, hb = fx_hi_word(b[k]) & 0x7fffffff;
    mxv = mxv > ha ? mxv : ha;
    mxv = mxv > hb ? mxv : hb;
  }
  const FxScale sc = fx_scale(h1a > h1b ? h1a : h1b, h1a < h1b ? h1a : h1b, h5a > h5b ? h5a : h5b,
                              h5a < h5b ? h5a : h5b, mxv, C1, ktg);
  if (sc.tier == kFxSlow || !(sqrt_gam < 3.0)) return false;
  // component order z1, z_m, the other two, z5
  fx x[2][5];
  FxPair p[2][2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const double* z = s ? b : a;
    const double z0 = m == 0 ? z[1] : (m == 1 ? z[2] : z[3]), z1 = m == 0 ? z[2] : (m == 1 ? z[3] : z[1]),
                 z2 = m == 0 ? z[3] : (m == 1 ? z[1] : z[2]);
    x[s][0] = fx_from_positive(z[0], sc.e1);
    x[s][1] = fx_from_double(z0, sc.ev);
    x[s][2] = fx_from_double(z1, sc.ev);
    x[s][3] = fx_from_double(z2, sc.ev);
    x[s][4] = fx_from_positive(z[4], sc.e5);
    p[s][0] = fx_pair(x[s][0]);
    p[s][1] = fx_pair(x[s][4]);
  }
  const fx Q = 1ll << 62;  // 2 Q = 1
  fx g[5];
  if (sc.tier == kFxNear) fx_flux<kFxNear>(x[0], p[0], x[1], p[1], Q, sc, g);
  else fx_flux<kFxFar>(x[0], p[0], x[1], p[1], Q, sc, g);
  double D[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (diss == 1) {
    const int Ev = sc.ev - 1022, E5 = sc.e5 - 1022, E1 = sc.e1 - 1022;
    const fx c0 = sc.C - (1ll << (64 - sc.kt));  // 4/(gam-1) = C1x - 2
    const fx sg = fx(sqrt_gam * 0x1p60);
    fx lam = 0, rho[2], en[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const fx t = x[s][0] * 2;  // z1 as a fraction in [1/3, 1)
      const fx r = fx_rcp(t, fx_rcpf(float(unsigned(fx_hi(t))) * 0x1p-31f));           // 60 fractional bits
      const fx v = x[s][1] < 0 ? -x[s][1] : x[s][1];
      const fx l = fx_mul(sg + (v >> (2 - Ev)), r);                                    // 59
      lam = lam > l ? lam : l;
      rho[s] = fx_mul(x[s][0], x[s][4]);                                               // 62
      const uint64_t v2 = uint64_t(fx_sqr(x[s][1])) + uint64_t(fx_sqr(x[s][2])) + uint64_t(fx_sqr(x[s][3]));
      en[s] = fx_mul(fx_mul(x[s][4], r) * 8, c0 + fx(v2 >> (sc.ss - 2)));              // 60 of 4 e x5/x1
    }
    lam *= 4;                                                                          // 61
    D[0] = fx_product(lam, rho[1] - rho[0], E5 - 55);
#pragma unroll
    for (int k = 1; k < 4; ++k)
      D[k] = fx_product(lam, fx_mul(x[1][4], x[1][k]) - fx_mul(x[0][4], x[0][k]), E5 - E1 + Ev - 55);
    D[4] = fx_product(lam, en[1] - en[0], E5 - 2 * E1 + sc.kt - 57);
  }
  double h[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) h[k] = fx_to_double(g[k], fx_unit(sc, k)) - D[k];
  f[0] = h[0];
  f[1] = m == 0 ? h[1] : (m == 1 ? h[3] : h[2]);
  f[2] = m == 0 ? h[2] : (m == 1 ? h[1] : h[3]);
  f[3] = m == 0 ? h[3] : (m == 1 ? h[2] : h[1]);
  f[4] = h[4];
  return true;
}

}  // namespace es
