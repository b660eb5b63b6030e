// 64-bit block fixed point for the FP64 mode's flux differencing.
//
// GB300 retires one FP64 warp instruction in about 19 cycles per SM (measured), the time of
// some 76 instructions of one of its four schedulers, while a 32 x 32 -> 64 bit multiply-add
// (IMAD.WIDE) takes 2.7 scheduler slots: a 62-bit product of two fixed-point numbers costs
// about 11 slots on the integer pipe, a seventh of one FP64 instruction.  Along an LGL line
// all quantities of the two-point flux have known magnitudes relative to the element's
// largest values, so a block exponent per element and variable replaces the floating
// exponents: every value carries 58..62 fractional bits of the block's scale, against the 53
// of a double, and the sums over a line are exact.
//
// A number with F fractional bits is an int64 x * 2^F.  fx_mul multiplies F1 and F2 fractional
// bits into F1 + F2 - 64 and keeps the upper 64 bits of the product (error below 2 units), from
// balanced 32-bit limbs x = h 2^32 + l, -2^31 <= l < 2^31: three signed 32 x 32 -> 64 bit
// multiply-adds, the upper word of the cross terms joins the product of the upper limbs.  One
// factor must be below 2^62.6 and the other below 2^63 in magnitude (the cross terms' sum stays
// below 2^63).  Written with PTX multiply-adds: from plain 64-bit C the compiler makes 18
// instructions of a product, from these 7 (measured).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "es_fx_tab.h"

namespace es {

typedef long long fx;

#define ES_HD __host__ __device__ __forceinline__

ES_HD int fx_max(int a, int b) { return a > b ? a : b; }
ES_HD int fx_min(int a, int b) { return a < b ? a : b; }
ES_HD int fx_lo(fx x) { return int(x); }
ES_HD int fx_hi(fx x) { return int(x >> 32); }
ES_HD fx fx_mulw(int a, int b) {
#ifdef __CUDA_ARCH__
  fx r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return fx(a) * b;
#endif
}
ES_HD fx fx_madw(int a, int b, fx c) {
#ifdef __CUDA_ARCH__
  fx r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return fx(a) * b + c;
#endif
}
ES_HD uint64_t fx_mulwu(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return uint64_t(a) * b;
#endif
}
ES_HD uint64_t fx_madwu(unsigned a, unsigned b, uint64_t c) {
#ifdef __CUDA_ARCH__
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return uint64_t(a) * b + c;
#endif
}
// x y 2^-64, rounded (a truncated product would bias all sums of an element the same way)
ES_HD fx fx_mul(fx x, fx y) {
  const int xl = fx_lo(x), yl = fx_lo(y);
  const int xh = fx_hi(x) - (xl >> 31), yh = fx_hi(y) - (yl >> 31);
  const fx c = fx_madw(xl, yh, fx_madw(xh, yl, 0x80000000ll));
  return fx_madw(xh, yh, fx(fx_hi(c)));
}
// x y 2^-63: one more bit of the product
ES_HD fx fx_mul63(fx x, fx y) {
  const int xl = fx_lo(x), yl = fx_lo(y);
  const int xh = fx_hi(x) - (xl >> 31), yh = fx_hi(y) - (yl >> 31);
  const fx c = fx_madw(xl, yh, fx_madw(xh, yl, 0x40000000ll));
  return fx_madw(xh, yh, fx_madw(xh, yh, c >> 31));
}
// x^2 2^-64, |x| < 2^63
ES_HD fx fx_sqr(fx x) {
  const int xl = fx_lo(x), xh = fx_hi(x) - (xl >> 31);
  return fx_madw(xh, xh, fx_mulw(xh, xl) >> 31);
}

ES_HD int fx_hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  int64_t b;
  __builtin_memcpy(&b, &x, 8);
  return int(b >> 32);
#endif
}
ES_HD unsigned fx_lo_word(double x) {
#ifdef __CUDA_ARCH__
  return unsigned(__double2loint(x));
#else
  int64_t b;
  __builtin_memcpy(&b, &x, 8);
  return unsigned(b);
#endif
}
ES_HD double fx_make_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(fx(b));
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
ES_HD int fx_clz(uint64_t n) {
#ifdef __CUDA_ARCH__
  return __clzll(fx(n));
#else
  return n ? __builtin_clzll(n) : 64;
#endif
}

// A finite double as a fixed-point fraction of 2^(E + 1), 63 fractional bits, where the block's
// largest biased exponent is emax (E = emax - 1022, so |x| < 2^E and the fraction is below 1/2):
// exact down to 2^-9 of the block's largest power of two, truncated below; subnormals read as 0.
ES_HD fx fx_from_double(double x, int emax) {
  const int h = fx_hi_word(x);
  const int e = (h >> 20) & 0x7ff;
  fx m = (fx((h & 0xfffff) | 0x100000) << 41) | (fx(fx_lo_word(x)) << 9);
  const unsigned sh = unsigned(emax - e);
  m >>= sh < 63u ? sh : 63u;
  if (e == 0) m = 0;
  return h < 0 ? -m : m;
}

// the same for positive normal values with exponents just below emax
ES_HD fx fx_from_positive(double x, int emax) {
  const int h = fx_hi_word(x);
  const unsigned l = fx_lo_word(x);
  const fx m = fx((uint64_t(unsigned((h & 0xfffff) | 0x100000) << 9 | l >> 23) << 32) | (l << 9));
  return m >> ((emax - (h >> 20)) & 63);
}

// n 2^ex as a double, rounded to nearest (ties away); the result is normal or zero for the
// exponents the block scales allow
ES_HD double fx_to_double(fx n, int ex) {
  const fx s = n >> 63;
  uint64_t a = uint64_t((n ^ s) - s);
  const int lz = fx_clz(a);
  if (lz >= 64) return 0.0;
  a <<= lz - 1;  // leading bit at 62
  const uint64_t m = (a + 0x200) >> 10;  // 2^52 <= m <= 2^53
  // value = a 2^(ex + 1 - lz): the leading bit's exponent enters, m carries into it
  const uint64_t b = m + (uint64_t(unsigned(63 + ex - lz + 1022) << 20) << 32);
  return fx_make_double(b | (uint64_t(s) << 63));
}

// 1/s for 0.25 <= s < 1 (63 fractional bits), result with 60: an FP32 reciprocal q (relative
// error e below 2^-20) refined by r (1 + e + e^2), e = 1 - s r exact to 2^-60
ES_HD fx fx_rcp(fx s, float q) {
#ifdef __CUDA_ARCH__
  const unsigned r0 = __float2uint_rn(q * 0x1p29f);
#else
  const unsigned r0 = unsigned(q * 0x1p29f + 0.5f);
#endif
  const uint64_t t = fx_madwu(unsigned(fx_hi(s)), r0, fx_mulwu(unsigned(fx_lo(s)), r0) >> 32);
  fx e = (1ll << 60) - fx(t);  // |e| < 2^40
  const int eh = int(e >> 10);
  e += fx(fx_hi(fx_mulw(eh, eh)) >> 8);
  // r0 e 2^-29, e in limbs of 32 and 10 bits
  const fx c = fx_madw(int(r0), int(e >> 10), fx(fx_mulwu(r0, unsigned(fx_lo(e)) << 22) >> 32)) >> 19;
  return (fx(r0) << 31) + c;
}

// Logarithmic-mean corrections from u = r^2, r = (a - b)/(a + b):
//   F(u) - 1 = u/3 + u^2/5 + ...  and  1 - 1/F(u) = u/3 + 4 u^2/45 + 44 u^3/945 + ...
// (F(u) = atanh(sqrt u)/sqrt u), with 64 fractional bits.
// kFxNear, |r| <= 0.01: three terms (truncation below 1.2e-17, as in the FP64 flux) on the FP32
// pipe, which the integer products leave idle: a and b as pairs of floats (23 + 24 bits of the
// block fraction, so that sum and difference of the upper parts are exact), r and u as pairs.  At the
// limit the dropped bits of a and b move r by up to 2^-46 and the correction by 2/3 |r| of it, 0.9 units
// of 2^-53, the FP32 roundings of the u^2 term (below 2^-28.9) by 2.6 and those of its sum by 1.5: five at
// most, 4.0 measured, and 0.6 at |r| = 0.005.  The flux is still closer than in FP64, whose every product rounds: up to
// the limit 0.17 units of itself in the mass and 0.4 in the energy on average (FP64: 1.0 and 2.1), 1.9 and 3.3 at
// worst (5.6 and 11).  The pair becomes an integer through two additions to powers of two.
// kFxFar, |r| <= 0.2: twelve terms in fixed point (truncation below 2^-59; the terms from u^6 on
// enter with a weight below 2^-23 and are summed in 32 bits); r with 61 fractional bits.
constexpr int kFxSlow = 0, kFxNear = 1, kFxFar = 2;
struct FxPair {
  float h, l;
};
// the upper 47 fractional bits of a fraction 0 <= x < 1/2 (63 bits)
ES_HD FxPair fx_pair(fx x) {
  FxPair p;
  p.h = float(int(x >> 40)) * 0x1p-23f;
  p.l = float(int(x >> 16) & 0xffffff) * 0x1p-47f;
  return p;
}
ES_HD float fx_fma(float a, float b, float c) {
#ifdef __CUDA_ARCH__
  return __fmaf_rn(a, b, c);
#else
  return __builtin_fmaf(a, b, c);
#endif
}
ES_HD float fx_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
ES_HD float fx_mulf(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
ES_HD int fx_bits(float a) {
#ifdef __CUDA_ARCH__
  return __float_as_int(a);
#else
  int i;
  __builtin_memcpy(&i, &a, 4);
  return i;
#endif
}
ES_HD float fx_rcpf(float a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
#else
  return 1.0f / a;
#endif
}
// q: 1/(a.h + b.h) approximately; c2, c3: second and third coefficient
ES_HD fx fx_near(FxPair a, FxPair b, float q, float c2, float c3) {
  const float sh = fx_add(a.h, b.h), sl = fx_add(a.l, b.l);
  const float d0 = fx_add(a.h, -b.h), d1 = fx_add(a.l, -b.l);
  const float dh = fx_add(d0, d1), dl = fx_add(d1, -fx_add(dh, -d0));
  const float r = fx_mulf(dh, q);
  const float rl = fx_mulf(fx_add(fx_fma(-r, sh, dh), fx_fma(-r, sl, dl)), q);
  const float u = fx_mulf(r, r);
  const float ul = fx_fma(fx_add(r, r), rl, fx_fma(r, r, -u));
  constexpr float th = float(1.0 / 3.0);
  constexpr float tl = float(1.0 / 3.0 - double(th));
  float p = fx_mulf(u, th);
  float e = fx_fma(u, tl, fx_fma(u, th, -p));
  e = fx_fma(ul, th, e);
  const float us = fx_add(u, ul);
  e = fx_fma(us, fx_mulf(us, fx_fma(us, c3, c2)), e);
  const float n = fx_add(p, e);
  e = fx_add(e, -fx_add(n, -p));
  p = n;
  // p in units of 2^-37, the rest (below 2^-37) in units of 2^-59
  const float wp = fx_add(p, 0x1p-14f);
  const float we = fx_add(fx_add(fx_add(p, -fx_add(wp, -0x1p-14f)), e), 0x1.8p-36f);
  constexpr fx zero = -(fx(0x38800000) << 27) - (fx(0x2dc00000) << 5);  // bits of the two powers
  return fx_madw(fx_bits(wp), 1 << 27, fx_madw(fx_bits(we), 32, zero));
}
template <int WHICH>
ES_HD fx fx_series_far(fx r) {
  constexpr FxSeries T{};
  const fx u = fx_sqr(r * 4) * 4;  // 64 fractional bits
  const int uh = int(u >> 33);     // 31
  int h = int(T.c[WHICH][kFxTerms - 1] >> 31);
#pragma unroll
  for (int k = kFxTerms - 2; k >= 5; --k) h = int(T.c[WHICH][k] >> 31) + int(fx_mulw(h, uh) >> 31);
  fx s = fx(h) << 31;
#pragma unroll
  for (int k = 4; k >= 0; --k) s = T.c[WHICH][k] + fx_mul(s, u);
  return fx_mul(s, u) * 4;
}

// Whether the fixed-point forms take a mesh: all directions of an element are summed in units of its largest
// metric 2/h, and a direction whose metric is 2^k smaller loses k bits of its derivative, of the about
// five that the sums have over a double's.  Flow along the coarse direction, nothing varying in the fine
// one, p = 3, error of the mass equation against the FP64 kernels' 7.8e-13: 0.8e-13 at ratio 1, 1.7e-13 at 8 and 15,
// 6.7e-13 at 32, 41e-13 at 256.  From an exponent difference of five on (ratios of 16 to 32) the element goes to
// FP64, in every kernel: behind the faces of a thin element also a velocity much smaller than the others counts.
ES_HD bool fx_metrics_close(const double metric[3]) {
  const int a = fx_hi_word(metric[0]) >> 20, b = fx_hi_word(metric[1]) >> 20, c = fx_hi_word(metric[2]) >> 20;
  return fx_max(a, fx_max(b, c)) - fx_min(a, fx_min(b, c)) <= 4;
}

// Block scales of one element: biased exponents of the largest z1, z5 and |z2..z4|, and what
// the flux derives from them.
struct FxScale {
  int tier;        // kFxSlow: outside the fixed-point range, FP64 flux
  int e1, e5, ev;  // largest biased exponents
  int sv, sp, se;  // right shifts of the convective and the pressure part of the momentum flux, of the energy flux
  int kt, ss;      // t < 2^kt; right shift of |S_v|^2
  fx C;            // C1x 2^-kt, 63 fractional bits
};

// The block's exponent from the high word of its largest value: one more where that value's upper
// 20 fraction bits are all ones, so that the sum of two fractions stays below 1 - 2^-20 (the upper
// limb of fx_mul rounds up)
ES_HD int fx_block_exponent(int mx) { return (mx + 1) >> 20; }
// (of the velocities down to the slowest block that is taken, |z_v| = 2^-30: a block exponent that
// stopped above it would cost the mass and energy flux, which are proportional to the velocity, their digits)
constexpr int kFxSlowest = 993;
ES_HD int fx_block_exponent_v(int mxv) {
  const int e = fx_block_exponent(mxv);
  return e > kFxSlowest ? e : kFxSlowest;
}

// From the high words of the element's largest and smallest z1 and z5 and largest |z2..z4|.
// Fast when z1 and z5 are positive and vary by less than a factor 1.5 (u <= 0.04 for every
// pair; NaN, infinities and signs fall through the comparisons of the high words), their
// exponents leave every product inside the double range, and |z_v| < 4 (Mach below ~3.4).  Gas at
// rest (|z_v| < 2^-30) stays in FP64: there the volume sums have to cancel the face fluxes' bits
// (what remains is all that an undisturbed element next to a discontinuity moves by).
ES_HD FxScale fx_scale(int mx1, int mn1, int mx5, int mn5, int mxv, fx C1, int ktg) {
  FxScale s;
  s.e1 = fx_block_exponent(mx1);
  s.e5 = fx_block_exponent(mx5);
  s.ev = fx_block_exponent_v(mxv);
  const bool ok = mn1 > 0 && mn5 > 0 && s.e1 > 822 && s.e1 < 1222 && s.e5 > 822 && s.e5 < 1222 && s.ev <= 1024 &&
                  (mxv >> 20) >= kFxSlowest && ktg <= 12 && (mx1 >> 20) - (mn1 >> 20) <= 1 && (mx5 >> 20) - (mn5 >> 20) <= 1;
  // 21 leading bits of largest and smallest: (max - min)/(max + min) <= 0.2 or 0.01
  const int a1 = (mx1 & 0xfffff) | 0x100000, b1 = ((mn1 & 0xfffff) | 0x100000) >> (((mx1 >> 20) - (mn1 >> 20)) & 1);
  const int a5 = (mx5 & 0xfffff) | 0x100000, b5 = ((mn5 & 0xfffff) | 0x100000) >> (((mx5 >> 20) - (mn5 >> 20)) & 1);
  const bool far = (a1 - b1 + 1) * 5 <= a1 + b1 && (a5 - b5 + 1) * 5 <= a5 + b5;
  const bool near = (a1 - b1 + 1) * 100 <= a1 + b1 && (a5 - b5 + 1) * 100 <= a5 + b5;
  s.tier = !(ok && far) ? kFxSlow : (near ? kFxNear : kFxFar);
  const int Ev = s.ev - 1022;
  s.sv = Ev < 0 ? -2 * Ev : 0;
  s.sp = Ev > 0 ? 2 * Ev : 0;
  s.se = 0;
  s.kt = (ktg > 2 * Ev + 3 ? ktg : 2 * Ev + 3) + 1;
  s.ss = fx_min(s.kt - 2 - 2 * Ev, 63);
  s.C = (C1 >> ((s.kt - 1 - ktg) & 63));
  return s;
}
// More room in the momentum and the energy sums, for an element whose face or viscous fluxes pass its
// scales by 2^dm and 2^de.  The room is taken from the last bits of all its sums: as much as those fluxes need, and
// kFxMargin bits beside it (of the five that the sums have over a double's), so that larger ones found later
// do not take another attempt.  Up to 2^6 times the pressure and the enthalpy flux at sound speed, else FP64.
constexpr int kFxMargin = 3;
ES_HD void fx_widen(FxScale& s, int dm, int de) {
  const int Ev = s.ev - 1022;
  if (dm > 0) dm = fx_max(dm, fx_min(dm + kFxMargin, (Ev > 0 ? 2 * Ev : 0) + 6 - s.sp));
  if (de > 0) de = fx_max(de, fx_min(de + kFxMargin, (Ev < 0 ? -Ev : 0) + 6 - s.se));
  s.sv = fx_min(s.sv + dm, 63);
  s.sp += dm;
  s.se += de;
  if (s.sp > (Ev > 0 ? 2 * Ev : 0) + 6 || s.se > (Ev < 0 ? -Ev : 0) + 6) s.tier = kFxSlow;
}
// exponents of the flux sums' units: 2 Q_ij times the flux is n 2^unit for mass, momentum and energy
ES_HD int fx_unit(const FxScale& s, int v) {
  const int E1 = s.e1 - 1022, E5 = s.e5 - 1022, Ev = s.ev - 1022;
  return v == 0 ? E5 + Ev - 59 : (v < 4 ? E5 - E1 + s.sp - 59 : E5 + Ev - 2 * E1 + s.kt - (s.tier == kFxNear ? 61 : 60) + s.se);
}

// Twice Q_ij = omega_i D_ij times the Ismail--Roe flux between two nodes, in units of 2^fx_unit
// (a, b: z1, z_m, two other z_v, z5 as fractions of the block scales, 63 fractional bits; fa, fb:
// z1 and z5 as float pairs; Q: Q_ij / 4 with 65, |Q_ij| < 0.98 for p = 2..5).  With S = a + b, 1/S1 = inv, g = 4 g5 = 1 - eps,
// f1 = 1 + del (see ec_flux):
//   pq = Q S5/S1, M = g pq S_m, mass flux M S1, momentum M S_k (+ pq for k = m),
//   energy u_m (g pq t + 2^(1-kt) pq), u_m = S_m/S1, t = C1x f1 + |S_v|^2/2 (scaled by 2^-kt).
// Every factor Q multiplies once, so the pair enters both nodes' sums with opposite signs.
// Bounds: 1/3 <= S1 < 1 (near: 0.49), so inv < 3 (2.05), pq < 0.74 (0.5), |u_m| < 3 (2.05), t < 0.95 (0.88, with
// 2^-kt <= 1/16 beside it, 0.82 with 1/8), so 4 y < 0.8 (8 y < 0.95) of 2^63.
template <int TIER>
ES_HD void fx_flux(const fx a[5], const FxPair fa[2], const fx b[5], const FxPair fb[2], fx Q, const FxScale& c,
                   fx g[5]) {
  const fx S1 = a[0] + b[0], Sm = a[1] + b[1], Sa = a[2] + b[2], Sb = a[3] + b[3], S5 = a[4] + b[4];
  const float q = fx_rcpf(fx_add(fa[0].h, fb[0].h)), q5 = fx_rcpf(fx_add(fa[1].h, fb[1].h));
  const fx inv = fx_rcp(S1, q);
  fx del, eps;
  if (TIER == kFxNear) {
    del = fx_near(fa[0], fb[0], q, 0.2f, 1.0f / 7.0f);
    eps = fx_near(fa[1], fb[1], q5, 4.0f / 45.0f, 44.0f / 945.0f);
  } else {
    del = fx_series_far<0>(fx_mul((a[0] - b[0]) * 4, inv));
    eps = fx_series_far<1>(fx_mul((a[4] - b[4]) * 4, fx_rcp(S5, q5)));
  }
  const fx pq = fx_mul(fx_mul(S5, inv) * 4, Q);                                        // 62 fractional bits
  const fx pg = pq - fx_mul(pq, eps);                                                  // 62
  const uint64_t ss = uint64_t(fx_sqr(Sm)) + uint64_t(fx_sqr(Sa)) + uint64_t(fx_sqr(Sb));
  const fx t = c.C + fx_mul(c.C, del) + fx(ss >> c.ss);                                // 63
  const fx M = fx_mul(pg, Sm) * 4, Ms = M >> c.sv;                                     // 63
  g[0] = fx_mul(M, S1);                                                                // 62
  g[1] = fx_mul(Ms, Sm) + (pq >> c.sp);
  g[2] = fx_mul(Ms, Sa);
  g[3] = fx_mul(Ms, Sb);
  const fx y = fx_mul(pg, t) + (pq >> c.kt);                                           // 61
  g[4] = fx_mul63(fx_mul(Sm, inv) * 4, y * (TIER == kFxNear ? 8 : 4)) >> c.se;         // 62, far: 61
}

}  // namespace es
