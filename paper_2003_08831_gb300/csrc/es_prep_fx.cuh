// The stage preparation's thermodynamics in 64-bit fixed point (es_fx.cuh): the parameter vector
// of a state (ES_FP64) and the entropy-variable increment of a state change (ES_FP64, and the estimate
// of ES_MIXED).
//
// With Pr = rho p = (gam-1)(rho E - |m|^2/2) and rs = 1/sqrt(Pr):
//   z1 = rho rs, z_v = m rs, z5 = Pr rs,
// all carried with 58..60 significant bits (a double: 53); the increment is formed from the change of
// the state, never as a difference of two parameter vectors (which would keep 2^-58 of w instead of the
// increment).
//
// Each operation here takes 7-25 integer instructions where an FP64 one holds its pipe for the
// time of 76 (es_fx.cuh); a node needs about 25 FP64 operations less in the first stage and 110
// less in the later ones.  k_prep, mean of a step's three launches: Taylor--Green 32^3 p = 3 369 -> 126 us; Navier--
// Stokes p = 4 705 -> 243 us, and with ES_MIXED, whose increment alone is FP64, 510 -> 243 us.
#pragma once
#include "es_fx.cuh"

namespace es {

ES_HD uint64_t fx_umulhi(uint64_t a, uint64_t b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return uint64_t((unsigned __int128)a * b >> 64);
#endif
}
ES_HD unsigned fx_round_u(float a) {
#ifdef __CUDA_ARCH__
  return __float2uint_rn(a);
#else
  return unsigned(a + 0.5f);
#endif
}
ES_HD float fx_rsqrtf(float a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
#else
  return 1.0f / __builtin_sqrtf(a);
#endif
}

// 1/sqrt(f) for 1/4 <= f < 1 (63 fractional bits), result with 61: the FP32 approximation R
// refined by R (1 + e/2 + 3 e^2/8), e = 1 - f R^2 below 2^-20
ES_HD fx fx_rsqrt(fx f) {
  unsigned r0 = fx_round_u(fx_rsqrtf(float(unsigned(fx_hi(f))) * 0x1p-31f) * 0x1p30f);
  r0 = r0 < 0x7fffffffu ? r0 : 0x7fffffffu;
  const fx t = fx(fx_umulhi(uint64_t(f), fx_mulwu(r0, r0)));  // 59 fractional bits
  const fx e = (1ll << 59) - t;                               // |e| < 2^40
  const int eh = int(e >> 10);
  const fx h = (e >> 1) + (fx(fx_hi(fx_mulw(eh, eh)) >> 7) * 3 >> 3);
  // r0 h 2^-28, h in limbs of 32 and 10 bits
  const fx c = fx_madw(int(r0), int(h >> 10), fx(fx_mulwu(r0, unsigned(fx_lo(h)) << 22) >> 32)) >> 18;
  return (fx(r0) << 31) + c;
}

// z1, z_v, z5 as n 2^(s - 60)
struct FxState {
  fx z1, zv[3], z5;
  int s1, sv, s5;
};

// A state (rho, m, E) as fractions: rho = nr 2^(Er - 62), E = nE 2^(EE - 62), m = nm 2^(Em - 62), |m|^2/2 =
// q2 2^(2 Em - 61), and P = rho E - |m|^2/2 = rho p/(gam-1) = P 2^uP with 2^61 <= P < 2^62.
struct FxBase {
  fx nr, nE, nm[3], q2, P;
  int Er, EE, Em, uP;
};
// False where the state is not physical or its exponents or its internal energy (Mach number
// beyond ~1000) leave the fixed-point range: the caller then works in FP64.
ES_HD bool fx_base(const double q[5], FxBase& b) {
  const int hr = fx_hi_word(q[0]), hE = fx_hi_word(q[4]);
  const int m0 = fx_hi_word(q[1]) & 0x7fffffff, m1 = fx_hi_word(q[2]) & 0x7fffffff, m2 = fx_hi_word(q[3]) & 0x7fffffff;
  const int mm = m0 > m1 ? (m0 > m2 ? m0 : m2) : (m1 > m2 ? m1 : m2);
  const int er = hr >> 20, eE = hE >> 20;
  int em = mm >> 20;
  if (er < 723 || er > 1323 || eE < 723 || eE > 1323 || em > 1323) return false;  // signs, NaN, infinities too
  em = em > 673 ? em : 673;
  b.nr = fx_from_positive(q[0], er);  // 2^61 .. 2^62
  b.nE = fx_from_positive(q[4], eE);
#pragma unroll
  for (int k = 0; k < 3; ++k) b.nm[k] = fx_from_double(q[1 + k], em);
  b.Er = er - 1022;
  b.EE = eE - 1022;
  b.Em = em - 1022;
  // rho E and |m|^2/2 in units of 2^(Er + EE - 60)
  const fx a = fx_mul(b.nr, b.nE);
  fx k2 = b.q2 = fx_sqr(b.nm[0]) + fx_sqr(b.nm[1]) + fx_sqr(b.nm[2]);
  const int s = b.Er + b.EE - 2 * b.Em + 1;
  if (s >= 0) {
    k2 >>= s < 63 ? s : 63;
  } else {
    if (s < -4 || (k2 >> (61 + s)) != 0) return false;
    k2 <<= -s;
  }
  fx P = a - k2;
  if (P < (1ll << 40)) return false;
  const int lp = fx_clz(uint64_t(P)) - 2;
  b.P = P << lp;
  b.uP = b.Er + b.EE - 60 - lp;
  return true;
}
// its parameter vector; g1, eg: gam - 1 = g1 2^(eg - 63), 2^62 <= g1 < 2^63
ES_HD void fx_parameters(const FxBase& b, fx g1, int eg, FxState& z) {
  // (unsigned products: factors up to 2^63, where fx_mul's upper limb would overflow)
  fx X = fx(fx_umulhi(uint64_t(b.P), uint64_t(g1)));  // 2^59 .. 2^61
  // Pr = X 2^ex = f 2^(2 h), f = X 2^-63 after the shift that makes the exponent even
  int ex = b.uP + eg + 1;
  int sh = fx_clz(uint64_t(X)) - 2;
  sh += (ex - sh + 63) & 1;
  X <<= sh;
  const int h = (ex - sh + 63) >> 1;
  const fx rs = fx_rsqrt(X);
  z.z1 = fx_mul(b.nr, rs);
#pragma unroll
  for (int k = 0; k < 3; ++k) z.zv[k] = fx_mul(b.nm[k], rs);
  z.z5 = fx(fx_umulhi(uint64_t(X), uint64_t(rs)));
  z.s1 = b.Er + 1 - h;
  z.sv = b.Em + 1 - h;
  z.s5 = h;
}
ES_HD bool fx_state(const double q[5], fx g1, int eg, FxState& z) {
  FxBase b;
  if (!fx_base(q, b)) return false;
  fx_parameters(b, g1, eg, z);
  return true;
}

// FP32 reciprocal of a fraction in [1/4, 1) (63 bits), below 4 so that it fits fx_rcp's 31 bits
ES_HD float fx_rcp_seed(fx f) {
  const float q = fx_rcpf(float(unsigned(fx_hi(f))) * 0x1p-31f);
  return q < 0x1.fffffep1f ? q : 0x1.fffffep1f;
}

// the six planes of the parameter vector in FP64
ES_HD void fx_state_planes(const FxState& z, double o[6]) {
  o[0] = fx_to_double(z.z1, z.s1 - 60);
#pragma unroll
  for (int k = 0; k < 3; ++k) o[1 + k] = fx_to_double(z.zv[k], z.sv - 60);
  o[4] = fx_to_double(z.z5, z.s5 - 60);
  const fx f = z.z1 << 3;  // 2^61 .. 2^63
  const fx inv = fx_rcp(f, fx_rcp_seed(f));
  o[5] = fx_to_double(inv, -z.s1 - 60);
}

// Correction of ln(1 + y)/2 = r (1 + del), r = y/(2 + y) with |r| <= 0.01: del = r^2/3 + r^4/5 + r^6/7 +
// r^8/9 with 64 fractional bits, good to 2^-57 (the next term: 2^-69); u = r^2, 64 fractional bits
ES_HD fx fx_log_correction(fx u) {
  const int uh = int(u >> 20);
  const int t = 0x1999999a + int(fx_mulw(uh, 0x12492492 + int(fx_mulw(uh, 0x0e38e38e) >> 44)) >> 44);  // 31
  const fx s = 0x0aaaaaaaaaaaaaabll + (fx_mulw(uh, t) >> 14);                                            // 61
  return fx_mul(u << 11, s) >> 8;
}
// x as n 2^-s with 2^61 <= |n| < 2^62 (|x| < 2^62; 0: s = 62)
ES_HD fx fx_normal(fx x, int& s) {
  s = x ? fx_clz(uint64_t(x < 0 ? -x : x)) - 2 : 62;
  return x << s;
}
// x 2^s for s <= 0
ES_HD fx fx_align(fx x, int s) { return x >> fx_min(-s, 63); }

// w(u + e) - w(u).  With P = rho E - |m|^2/2 = rho p/(gam-1) and r_1 = rho + e_rho, its relative change
//   eta = (r_1 e_E + rho E e_rho/rho - K)/P,  K = (m + e_m/2) . e_m,
// a = e_rho - rho eta and F = 1/((gam-1) P (1 + eta)),
//   dw_v = (r_1 e_m + a m) F,  dw5 = -(r_1 e_rho + a rho) F,
//   dw1 = C1x ln(1 + x)/2 - 2/(gam-1) ln(1 + eta)/2 - (K - eta |m|^2/2) F,  x = e_rho/rho.
// The increments keep exponents of their own and no difference of the two states is taken, so every
// term is good to about 2^-57 of itself, however small the change (the FP64 form: some 2^-53).
// C1, ktg: C1x = C1 2^(ktg - 62); IG, ei: 1/(gam-1) = IG 2^(ei - 62), 2^61 <= IG < 2^62.
// False where rho or P change by more than 2 % or an exponent leaves fx_base's range: the caller then works
// in FP64.
ES_HD bool fx_increment(const FxBase& b, const double e[5], fx C1, int ktg, fx IG, int ei, double dw[5]) {
  const int m0 = fx_hi_word(e[1]) & 0x7fffffff, m1 = fx_hi_word(e[2]) & 0x7fffffff, m2 = fx_hi_word(e[3]) & 0x7fffffff;
  const int ed0 = fx_max(m0, fx_max(m1, m2)) >> 20;
  const int e0 = (fx_hi_word(e[0]) & 0x7fffffff) >> 20, e4 = (fx_hi_word(e[4]) & 0x7fffffff) >> 20;
  if (ktg > 12 || ed0 > 1323 || e4 > 1323 || e0 >= b.Er + 1022) return false;  // (NaN and infinities too)
  const int Er = b.Er, EE = b.EE, Em = b.Em, uP = b.uP, Dm = fx_max(ed0, 523) - 1022;
  const int D0 = fx_max(e0, 523) - 1022, DE = fx_max(e4, 523) - 1022;
  const fx nr = b.nr, nE = b.nE, q2 = b.q2, P = b.P;
  const fx n0 = fx_from_double(e[0], D0 + 1022), n4 = fx_from_double(e[4], DE + 1022);
  const fx d = fx_align(n0, D0 - Er);
  if (((d < 0 ? -d : d) >> 6) * 50 > (nr >> 6)) return false;
  const fx r1 = nr + d;
  // K in units of 2^uK
  const int cm = fx_max(Em, Dm), uK = cm + Dm - 60;
  fx nd[3], K = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    nd[k] = fx_from_double(e[1 + k], Dm + 1022);
    K += fx_mul(fx_align(b.nm[k], Em - cm) + fx_align(nd[k], Dm - 1 - cm), nd[k]);
  }
  const fx iP = fx_rcp(P * 2, fx_rcp_seed(P * 2)) * 2;  // 1/P = iP 2^(-123 - uP)
  const int u1 = Er + DE - 61, u2 = EE + D0 - 61, c = fx_max(u1, fx_max(u2, uK));
  const fx S = fx_align(fx_mul63(r1, n4), u1 - c) + fx_align(fx_mul63(nE, n0), u2 - c) - fx_align(K, uK - c);
  int lz;
  const fx n = fx_normal(fx_mul63(S, iP), lz);  // eta = n 2^ue
  const int ue = c - 60 - uP - lz;
  if (ue > -67) return false;
  const fx h62 = fx_align(n, ue + 62);
  if ((h62 < 0 ? -h62 : h62) * 50 > (1ll << 62)) return false;
  const fx s1 = (1ll << 62) + h62, s2 = (1ll << 62) + (h62 >> 1);
  // (2 rho + e_rho)/4, doubled where it could fall below 1/4
  const int up = nr < (3ll << 60) ? 1 : 0;
  const fx s3 = (nr << up) + (d << up >> 1);
  const fx inv = fx_rcp(s1, fx_rcp_seed(s1)) * 2;  // 1/(1 + eta): 62 fractional bits
  // ln(1 + eta)/2 and ln(1 + x)/2 in units of 2^ue and 2^ux
  const int ux = D0 - Er - 61 + up;
  const fx re = fx_mul63(n, fx_rcp(s2, fx_rcp_seed(s2)) * 2), rx = fx_mul63(n0, fx_rcp(s3, fx_rcp_seed(s3)));
  const fx Le = re + fx_mul(re, fx_log_correction(fx_align(fx_sqr(re * 2), 126 + 2 * ue)));
  const fx Lx = rx + fx_mul(rx, fx_log_correction(fx_align(fx_sqr(rx * 2), 126 + 2 * ux)));
  // a (in halves, to be below 2^62) and F
  const int uz = Er + ue + 1;
  int ua = fx_max(D0 - 62, uz) + 1, la, lf;
  const fx a = fx_normal(fx_align(n0, D0 - 62 - ua) - fx_align(fx_mul63(nr, n), uz - ua), la);
  ua -= la;
  const fx F = fx_normal(fx_mul63(fx_mul63(iP, inv) * 2, IG), lf);  // units of 2^(ei - 122 - uP - lf)
  const int uF = ei - 59 - uP - lf;
  {
    const int v1 = Er + Dm - 61, v2 = Em + ua + 1, cv = fx_max(v1, v2);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      dw[1 + k] = fx_to_double(fx_mul63(fx_align(fx_mul63(r1, nd[k]), v1 - cv) + fx_align(fx_mul63(b.nm[k], a), v2 - cv), F),
                               cv + uF);
    const int w1 = Er + D0 - 61, w2 = Er + ua + 1, cw = fx_max(w1, w2);
    dw[4] = fx_to_double(-fx_mul63(fx_align(fx_mul63(r1, n0), w1 - cw) + fx_align(fx_mul63(nr, a), w2 - cw), F), cw + uF);
  }
  const int uq = 2 * Em + ue + 2, ck = fx_max(uK, uq), p1 = ktg + ux + 1, p2 = ei + 2 + ue;
  const fx kin = fx_mul63(fx_align(K, uK - ck) - fx_align(fx_mul63(q2, n), uq - ck), F);
  const int cp = fx_max(ck + uF, fx_max(p1, p2));
  dw[0] = fx_to_double(fx_align(fx_mul63(C1, Lx), p1 - cp) - fx_align(fx_mul63(IG, Le), p2 - cp) -
                           fx_align(kin, ck + uF - cp), cp);
  return true;
}

ES_HD bool fx_increment(const double u[5], const double e[5], fx C1, int ktg, fx IG, int ei, double dw[5]) {
  FxBase b;
  return fx_base(u, b) && fx_increment(b, e, C1, ktg, IG, ei, dw);
}

// ln(b/a)/2 with 65 fractional bits for |b - a| <= 0.01 (b + a); a, b < 2^60 in the same unit,
// their sum at least 2^59
ES_HD fx fx_half_log(fx a, fx b, bool& ok) {
  const fx d = b - a, sum = b + a;
  ok = ok && (d < 0 ? -d : d) * 100 <= sum && sum >= (1ll << 59);
  const fx s = sum << 2;
  const float q = fx_rcp_seed(s);
  const fx r = fx_mul(d << 8, fx_rcp(s, q));
  return r + fx_mul(r, fx_near(fx_pair(b << 2), fx_pair(a << 2), q, 0.2f, 1.0f / 7.0f));
}

// w(b) - w(a) from two states alone, good to 2^-58 of w whatever the change (the step has the change itself
// and takes the form above); C1, ktg: C1x = C1 2^(ktg - 62).  False where the states differ by more than 2 % in
// z1 or z5 (relative to the sum: 1 %), or their scales by more than the shifts below take, or |z_v|
// (by its exponents) reaches a limit between 1 and 4: for faster flows the kinetic difference would
// lose its digits.
ES_HD bool fx_increment(const FxState& a, const FxState& b, fx C1, int ktg, double dw[5]) {
  const int s1 = a.s1 > b.s1 ? a.s1 : b.s1, s5 = a.s5 > b.s5 ? a.s5 : b.s5, sv = a.sv > b.sv ? a.sv : b.sv;
  bool ok = s1 - a.s1 <= 1 && s1 - b.s1 <= 1 && s5 - a.s5 <= 1 && s5 - b.s5 <= 1 && sv <= 2 && ktg <= 12;
  const fx a1 = a.z1 >> ((s1 - a.s1) & 63), b1 = b.z1 >> ((s1 - b.s1) & 63);
  const fx a5 = a.z5 >> ((s5 - a.s5) & 63), b5 = b.z5 >> ((s5 - b.s5) & 63);
  const fx L1 = fx_half_log(a1, b1, ok), L5 = fx_half_log(a5, b5, ok);
  if (!ok) return false;
  const int ha = sv - a.sv < 63 ? sv - a.sv : 63, hb = sv - b.sv < 63 ? sv - b.sv : 63;
  const fx S1 = (a1 + b1) * 2, D1 = (b1 - a1) * 64;  // 61 and 66 fractional bits
  fx k2 = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx av = a.zv[k] >> ha, bv = b.zv[k] >> hb;
    const fx S = av + bv, D = (bv - av) * 2;  // 60, 61
    k2 += fx_mul63(D, S);                     // 58
    // z1' z_v' - z1 z_v = (D1 S + S1 D)/2: 62 and 58 fractional bits
    dw[1 + k] = fx_to_double((fx_mul(D1, S) >> 3) + fx_mul63(S1, D), s1 + sv - 60);
  }
  dw[4] = fx_to_double(-fx_mul(D1, S1), 2 * s1 - 63);
  // 63 - ktg fractional bits throughout; |z_v|^2/2 from 58 with the scale 2^(2 sv + 1)
  const int sh = ktg - 5 - 2 * sv + 1;
  if (sh < 0 && ((k2 < 0 ? -k2 : k2) >> (61 + sh)) != 0) return false;
  const fx kin = sh >= 0 ? k2 >> (sh < 63 ? sh : 63) : k2 << -sh;
  dw[0] = fx_to_double(fx_mul(C1, L1) + (L5 >> (ktg + 1)) - kin, ktg - 63);
  return true;
}

}  // namespace es
