// The stage preparation's thermodynamics in 64-bit fixed point (es_fx.cuh): the parameter vector
// of a state and the entropy-variable increment between two states, for the modes that hold them
// in FP64 (ES_FP64, and the estimate of ES_MIXED).
//
// With Pr = rho p = (gam-1)(rho E - |m|^2/2) and rs = 1/sqrt(Pr):
//   z1 = rho rs, z_v = m rs, z5 = Pr rs,
// all carried with 58..60 significant bits (a double: 53), so that the increment
//   dw1 = C1x L1 + 2 L5 - (|z_v'|^2 - |z_v|^2)/2,  dw_v = z1' z_v' - z1 z_v,  dw5 = z1^2 - z1'^2,
//   L = ln(z'/z)/2 = r F(r^2), r = (z' - z)/(z' + z),
// can be taken from the two states directly: of a relative change delta it keeps 2^-58/delta,
// against the 2^-53/delta that the right-hand side it is multiplied with keeps.
//
// Each operation here takes 7-25 integer instructions where an FP64 one holds its pipe for the
// time of 76 (es_fx.cuh); a node needs about 25 FP64 operations less in the first stage and 110
// less in the later ones.  Taylor--Green 32^3 p = 3: k_prep 369 -> 121 us per launch; Navier--Stokes
// p = 4 705 -> 213 us, and with ES_MIXED, whose increment alone is FP64, 510 -> 223 us.
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

// The parameter vector of (rho, m, E); g1, eg: gam - 1 = g1 2^(eg - 63), 2^62 <= g1 < 2^63.
// False where the state is not physical or its exponents or its internal energy (Mach number
// beyond ~1000) leave the fixed-point range: the caller then works in FP64.
ES_HD bool fx_state(const double q[5], fx g1, int eg, FxState& z) {
  const int hr = fx_hi_word(q[0]), hE = fx_hi_word(q[4]);
  const int m0 = fx_hi_word(q[1]) & 0x7fffffff, m1 = fx_hi_word(q[2]) & 0x7fffffff, m2 = fx_hi_word(q[3]) & 0x7fffffff;
  const int mm = m0 > m1 ? (m0 > m2 ? m0 : m2) : (m1 > m2 ? m1 : m2);
  const int er = hr >> 20, eE = hE >> 20;
  int em = mm >> 20;
  if (er < 723 || er > 1323 || eE < 723 || eE > 1323 || em > 1323) return false;  // signs, NaN, infinities too
  em = em > 673 ? em : 673;
  const fx nr = fx_from_positive(q[0], er), nE = fx_from_positive(q[4], eE);  // 2^61 .. 2^62
  fx nm[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) nm[k] = fx_from_double(q[1 + k], em);
  const int Er = er - 1022, EE = eE - 1022, Em = em - 1022;
  // rho E and |m|^2/2 in units of 2^(Er + EE - 60)
  const fx a = fx_mul(nr, nE);
  fx k2 = fx_sqr(nm[0]) + fx_sqr(nm[1]) + fx_sqr(nm[2]);
  const int s = Er + EE - 2 * Em + 1;
  if (s >= 0) {
    k2 >>= s < 63 ? s : 63;
  } else {
    if (s < -4 || (k2 >> (61 + s)) != 0) return false;
    k2 <<= -s;
  }
  fx P = a - k2;
  if (P < (1ll << 40)) return false;
  const int lz = fx_clz(uint64_t(P));
  // (unsigned products: factors up to 2^63, where fx_mul's upper limb would overflow)
  fx X = fx(fx_umulhi(uint64_t(P) << (lz - 2), uint64_t(g1)));  // 2^59 .. 2^61
  // Pr = X 2^ex = f 2^(2 h), f = X 2^-63 after the shift that makes the exponent even
  int ex = Er + EE + eg - lz - 57;
  int sh = fx_clz(uint64_t(X)) - 2;
  sh += (ex - sh + 63) & 1;
  X <<= sh;
  const int h = (ex - sh + 63) >> 1;
  const fx rs = fx_rsqrt(X);
  z.z1 = fx_mul(nr, rs);
#pragma unroll
  for (int k = 0; k < 3; ++k) z.zv[k] = fx_mul(nm[k], rs);
  z.z5 = fx(fx_umulhi(uint64_t(X), uint64_t(rs)));
  z.s1 = Er + 1 - h;
  z.sv = Em + 1 - h;
  z.s5 = h;
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

// w(b) - w(a); C1, ktg: C1x = C1 2^(ktg - 62).  False where the states differ by more than 2 % in
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
