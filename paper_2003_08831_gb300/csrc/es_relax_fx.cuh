// The relaxation root of one element in 64-bit fixed point (es_fx.cuh), for increments below 1/16.
//
// With X = d_rho/rho, Y the linearised d_p/p, W = rho |d_v|^2/(2 e) (e: internal energy density) a
// node's state at gamma g has rho/rho_0 = 1 + g X and rho p/(rho_0 p_0) = 1 + w, w = alpha g + beta g^2,
// alpha = X + Y, beta = X Y - W, so that
//   (gam-1) D(g)/rho = (1 + g X) ((gam+1) log(1 + g X) - log(1 + w)) - gam g X + g Y.
// Its Taylor coefficients need no division and no logarithm: with m_1 = alpha, m_2 = 2 beta -
// alpha^2, m_k = -alpha m_{k-1} - beta m_{k-2} (k times the coefficients of log(1 + w)),
//   D_2 = ((gam-1) X^2 + (X - Y)^2)/2 + W,
//   D_k = (gam+1) (-X)^k/(k (k-1)) - m_k/k - X m_{k-1}/(k-1),
// and an element's r(g)/g = A + g (a + sum_{k>2} S_k g^{k-2}) is a polynomial: one pass over the
// nodes instead of one per Newton step.  X, Y, sqrt(W) and the sums are fractions of 2^E and its
// powers, E from the element's largest; order k weighs 2^(E (k-2)), and from 2^-32 on it is
// summed in FP32 (24 bits of it: 2^-56).  The series ends below 2^-56.
//
// An FP64 solve took about 60 FP64 instructions per node and 90 more per Newton step, each the
// time of 76 scheduler slots (es_fx.cuh); this takes about 1200 slots in all.  k_relax per launch:
// Taylor--Green 32^3 p = 3 471 -> 140 us, p = 4 1042 -> 285 us; 11 x 9 x 13 p = 5 90 -> 39 us; entry
// point with u_new, 17 x 13 x 19 p = 2 (two FP64 logarithms per node remain) 75 -> 43 us.  Against long
// double the root is 3 to 10 times closer than FP64's (tests/test_fx_relax.py).
#pragma once
#include "es_prep_fx.cuh"

namespace es {

// 2^63/k, k = 2 .. kRelaxOrders
constexpr int kRelaxOrders = 29;
constexpr int kRelaxMaxE = -2, kRelaxMinE = -50;
#define ES_FX_INV(k) fx((0x8000000000000000ull + (k) / 2) / (k))
#define ES_FX_INVERSES                                                                                         \
  {0, 0, ES_FX_INV(2), ES_FX_INV(3), ES_FX_INV(4), ES_FX_INV(5), ES_FX_INV(6), ES_FX_INV(7), ES_FX_INV(8),     \
  ES_FX_INV(9), ES_FX_INV(10), ES_FX_INV(11), ES_FX_INV(12), ES_FX_INV(13), ES_FX_INV(14), ES_FX_INV(15),      \
  ES_FX_INV(16), ES_FX_INV(17), ES_FX_INV(18), ES_FX_INV(19), ES_FX_INV(20), ES_FX_INV(21), ES_FX_INV(22),     \
  ES_FX_INV(23), ES_FX_INV(24), ES_FX_INV(25), ES_FX_INV(26), ES_FX_INV(27), ES_FX_INV(28), ES_FX_INV(29)}
static __constant__ fx kFxInvDevice[kRelaxOrders + 1] = ES_FX_INVERSES;
ES_HD fx fx_inv_table(int k) {
#ifdef __CUDA_ARCH__
  return kFxInvDevice[k];
#else
  const fx t[kRelaxOrders + 1] = ES_FX_INVERSES;
  return t[k];
#endif
}

ES_HD fx fx_abs(fx x) { return x < 0 ? -x : x; }
// x 2^s; to the left only where the result fits
ES_HD fx fx_shift(fx x, int s) {
  if (s >= 0) return fx(uint64_t(x) << fx_min(s, 63));
  return x >> fx_min(-s, 63);
}
// the same, rounded: truncation would bias a sum over the nodes
ES_HD fx fx_shift_round(fx x, int s) {
  if (s >= 0) return fx_shift(x, s);
  return ((x >> fx_min(-s - 1, 62)) + 1) >> 1;
}
// x^2 2^-64, rounded
ES_HD fx fx_sqr_round(fx x) {
  const int xl = fx_lo(x), xh = fx_hi(x) - (xl >> 31);
  return fx_madw(xh, xh, fx_madw(xh, xl, 0x40000000ll) >> 31);
}
// the float of a 64-bit fraction (64 fractional bits)
ES_HD float fx_fraction(fx x) {
#ifdef __CUDA_ARCH__
  return __ll2float_rn(x) * 0x1p-64f;
#else
  return float(x) * 0x1p-64f;
#endif
}

// X, Y, W of a node, each n 2^e, and its density nr 2^(er - 62)
struct FxRelaxNode {
  fx x, y, w, nr;
  int ex, ey, ew, er;
};
constexpr int kRelaxNone = -100000;
// a lane without a node
ES_HD FxRelaxNode fx_relax_empty() { return {0, 0, 0, 0, 0, 0, 0, kRelaxNone}; }

// From the state u and its increment d.  False outside the range (as fx_state).
//   W = |d_m - v d_rho|^2/(2 rho e),  Y = (d_E - v . (d_m + (d_m - v d_rho))/2)/e
ES_HD bool fx_relax_node(const double u[5], const double d[5], FxRelaxNode& o) {
  const int er = fx_hi_word(u[0]) >> 20, eE = fx_hi_word(u[4]) >> 20;
  const int em0 = fx_max(fx_max(fx_hi_word(u[1]) & 0x7fffffff, fx_hi_word(u[2]) & 0x7fffffff),
                         fx_hi_word(u[3]) & 0x7fffffff) >> 20;
  const int e0 = (fx_hi_word(d[0]) & 0x7fffffff) >> 20, e4 = (fx_hi_word(d[4]) & 0x7fffffff) >> 20;
  const int ed = fx_max(fx_max(fx_hi_word(d[1]) & 0x7fffffff, fx_hi_word(d[2]) & 0x7fffffff),
                        fx_hi_word(d[3]) & 0x7fffffff) >> 20;
  if (er < 723 || er > 1323 || eE < 723 || eE > 1323 || em0 > 1323 || e0 > 1323 || e4 > 1323 || ed > 1323) return false;
  const int Er = er - 1022, EE = eE - 1022, Em = fx_max(em0, 673) - 1022;
  const int D0 = fx_max(e0, 523) - 1022, DE = fx_max(e4, 523) - 1022, Dm = fx_max(ed, 523) - 1022;
  const fx nr = fx_from_positive(u[0], er);  // 2^61 .. 2^62
  const fx ri = fx_rcp(nr * 2, fx_rcp_seed(nr * 2)) * 2;  // 1/rho: 61 fractional bits of 2^-Er
  fx v[3], k2 = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx nm = fx_from_double(u[1 + k], Em + 1022);
    v[k] = fx_mul(nm, ri);  // 2^(Em - Er - 59)
    k2 += fx_mul(nm, v[k]);
    v[k] *= 4;
  }
  // e = E - |m|^2/(2 rho) in units of 2^(EE - 62)
  const int s = EE + Er - 2 * Em - 4;
  if (s < 0 && (s < -8 || (k2 >> (62 + s)) != 0)) return false;
  const fx ne = fx_from_positive(u[4], eE) - fx_shift(k2, -s);
  if (ne < (1ll << 50)) return false;
  const int lz = fx_clz(uint64_t(ne));
  const fx f = ne << (lz - 1);
  const int Ee = EE + 2 - lz;
  const fx ie = fx_rcp(f, fx_rcp_seed(f)) * 2;  // 1/e: 61 fractional bits of 2^-Ee
  const fx n0 = fx_from_double(d[0], D0 + 1022);
  // momentum increments and d_m - v d_rho in units of 2^(Q - 61)
  const int Q = fx_max(Dm, Em + D0 - Er);
  fx z2 = 0, S = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const fx dm = fx_from_double(d[1 + k], Q + 1 + 1022);
    const fx q = dm - fx_shift(fx_mul(v[k], n0) * 4, Em + D0 - Er - Q);
    z2 += fx_sqr_round(q);              // 2^(2 Q - 58)
    S += fx_mul(v[k], (dm + q) >> 1);   // 2^(Em - Er + Q - 58)
  }
  const int T = fx_max(DE, Em - Er + Q + 3);
  const fx num = fx_from_double(d[4], T + 1 + 1022) - fx_shift(S, Em - Er + Q + 3 - T);  // 2^(T - 61)
  o.x = fx_mul(n0, ri);
  o.ex = D0 - Er - 59;
  o.y = fx_mul(num, ie);
  o.ey = T - Ee - 58;
  o.w = fx_mul(z2, fx_mul(ri, ie) * 4);
  o.ew = 2 * Q - Er - Ee - 55;
  o.nr = nr;
  o.er = Er;
  return true;
}

// smallest s with |X|, |Y|, sqrt(W) < 2^s
ES_HD int fx_relax_bits(const FxRelaxNode& n) {
  const int bx = n.x ? n.ex + 64 - fx_clz(uint64_t(fx_abs(n.x))) : kRelaxNone;
  const int by = n.y ? n.ey + 64 - fx_clz(uint64_t(fx_abs(n.y))) : kRelaxNone;
  const int bw = n.w ? (n.ew + 65 - fx_clz(uint64_t(n.w))) >> 1 : kRelaxNone;
  return fx_max(fx_max(bx, by), bw);
}

// Whether |X|, |Y|, sqrt(W) < 2^bits alone keep the element's RMS change
//   2 a/sum c <= max (X^2 + ((X - Y)^2 + 2 W)/(gam-1)) < 2^(2 bits) (1 + 6/(gam-1))
// below the floor (a 1/1000 of room for the rounding of the FP64 form's sums; increments below 2^-499 read as 0)
ES_HD bool fx_relax_below_floor(int bits, double floor, double inv_gm1) {
  const double top = fx_make_double(uint64_t(1023 + 2 * fx_max(bits, -490)) << 52) * (1.001 + 6.006 * inv_gm1);
  return floor * floor >= top;
}

// The node's mass weight c = cn 2^ce, cn in 2^60 .. 2^62 (w8 = omega_i omega_j omega_k/8, er: the
// element's largest density exponent; c sums to less than 1/2), and X, Y as fractions of 2^E (E =
// s + 2: below 1/4), W of 2^2E, with 64 fractional bits.
struct FxRelaxTerm {
  fx x, y, w, cn;
  int ce;
};
ES_HD FxRelaxTerm fx_relax_term(const FxRelaxNode& n, int E, int er, double w8) {
  FxRelaxTerm t;
  t.x = fx_shift(n.x, n.ex - E + 64);
  t.y = fx_shift(n.y, n.ey - E + 64);
  t.w = fx_shift(n.w, n.ew - 2 * E + 64);
  const int ew = fx_hi_word(w8) >> 20;
  t.cn = fx_mul63(fx_from_positive(w8, ew), n.nr) * 2;
  t.ce = ew - 1022 - 63 + n.er - er;
  return t;
}
// cn D_2 (gam-1) < 2^62 in the node's own scale (s: its fx_relax_bits); c D_2 in the element's is
// 2^*ex times this
ES_HD fx fx_relax_d2(const FxRelaxNode& n, const FxRelaxTerm& t, int s, int E, fx g1, int eg, int* ex) {
  const int En = s > kRelaxNone ? s + 2 : E;
  const fx x = fx_shift(n.x, n.ex - En + 64), y = fx_shift(n.y, n.ey - En + 64);
  const fx D = fx_shift(fx_mul(g1, fx_sqr_round(x)), eg) + (fx_sqr_round(x - y) >> 1) +
               fx_shift(n.w, n.ew - 2 * En + 64);
  *ex = t.ce - 1 + 2 * (En - E);
  return fx_mul63(t.cn, D);
}
ES_HD float fx_int_float(int i) {
#ifdef __CUDA_ARCH__
  return __int_as_float(i);
#else
  float f;
  __builtin_memcpy(&f, &i, 4);
  return f;
#endif
}
// 2^n as a float, 0 below the normal range (n <= 127)
ES_HD float fx_pow2(int n) {
  if (n < -126) return 0.0f;
#ifdef __CUDA_ARCH__
  return __int_as_float((n + 127) << 23);
#else
  return __builtin_ldexpf(1.0f, n);
#endif
}
// The sums' unit: from an element's sum s of c D_2 in FP32, the exponent t for which 2^t s is in
// 2^60 .. 2^61 (the terms of D_2 are positive, so every one fits, whatever the weights), and for
// the higher orders kRelaxGap bits less: c (X^2 + Y^2 + 2 W) is below (6 + 6/(gam-1)) c D_2, 2^6.7
// of it for gam >= 17/16.
constexpr int kRelaxGap = 6;
ES_HD float fx_relax_estimate(fx cd, int ex) { return fx_fraction(cd) * fx_pow2(ex + 64); }
ES_HD int fx_relax_unit(float s) { return 60 - ((fx_bits(s) >> 23) - 127); }

// The recurrence of one node: p = c (-X)^k, m = c m_k, mb = -c beta m_{k-1} (units of 2^(k E)); from k = 2
struct FxRelaxSeries {
  fx x, al, be, p, m, mb;
};
ES_HD FxRelaxSeries fx_relax_series(const FxRelaxTerm& t, int unit) {
  FxRelaxSeries s;
  s.x = -t.x;
  s.al = -(t.x + t.y);
  s.be = t.w - fx_mul(t.x, t.y);
  const int sh = t.ce + unit - kRelaxGap;  // of fx_mul(cn, .): 64 + 64 - 64 fractional bits
  s.p = fx_shift_round(fx_mul(t.cn, fx_sqr_round(s.x)), sh);
  s.m = fx_shift_round(fx_mul(t.cn, -2 * s.be - fx_sqr_round(s.al)), sh);
  s.mb = -fx_shift_round(fx_mul(t.cn, fx_mul(s.al, s.be)), sh);
  return s;
}
// to the next order; adds p, m and -X m_{k-1} to the sums
ES_HD void fx_relax_next(FxRelaxSeries& s, fx& sp, fx& sm, fx& sx) {
  sx += fx_mul(s.m, s.x);
  const fx m = fx_mul(s.m, s.al) + s.mb;
  s.mb = fx_mul(s.m, s.be);
  s.m = m;
  s.p = fx_mul(s.p, s.x);
  sp += s.p;
  sm += m;
}
// gam + 1 with 61 fractional bits (gam < 3)
ES_HD fx fx_relax_gp1(fx g1, int eg) { return (g1 >> (2 - eg)) + (1ll << 62); }
// S_k from the sums
ES_HD fx fx_relax_coefficient(int k, fx sp, fx sm, fx sx, fx gp1) {
  const fx ik = fx_inv_table(k), i1 = fx_inv_table(k - 1);
  return fx_mul63(fx_mul(sp << 3, gp1), i1 - ik) - fx_mul63(sm, ik) + fx_mul63(sx, i1);
}
// Whether fx_relax_root's q, from the sum's FP32 estimate, can lie in its range 0.5 .. 1.5
ES_HD bool fx_relax_near_one(float est, int E, int er, double A, double J, fx g1, int eg) {
  const auto mantissa = [](int h) { return fx_int_float((h & 0xfffff) << 3 | 0x3f800000); };
  const int hA = fx_hi_word(A) & 0x7fffffff, hJ = fx_hi_word(J), he = fx_bits(est);
  const float f = fx_mulf(fx_mulf(mantissa(hA), fx_fraction(g1) * 4.0f), fx_rcpf(fx_mulf(mantissa(hJ), fx_int_float((he & 0x7fffff) | 0x3f800000))));
  const int n = (hA >> 20) - (hJ >> 20) - ((he >> 23) - 127) + eg - 1 - 2 * E - er - 4;  // q = f 2^n
  if (n < -4 || n > 4) return false;
  const float q = fx_mulf(f, fx_pow2(n));
  return q > 0.499f && q < 1.501f;
}
struct FxRelaxSeriesF {
  float x, al, be, p, m, mb;
};
ES_HD FxRelaxSeriesF fx_relax_series_f(const FxRelaxSeries& s) {
  return {fx_fraction(s.x), fx_fraction(s.al), fx_fraction(s.be), fx_fraction(s.p), fx_fraction(s.m), fx_fraction(s.mb)};
}
ES_HD void fx_relax_next_f(FxRelaxSeriesF& s, float& sp, float& sm, float& sx) {
  sx = fx_fma(s.m, s.x, sx);
  const float m = fx_fma(s.m, s.al, s.mb);
  s.mb = fx_mulf(s.m, s.be);
  s.m = m;
  s.p = fx_mulf(s.p, s.x);
  sp = fx_add(sp, s.p);
  sm = fx_add(sm, m);
}
ES_HD float fx_relax_coefficient_f(int k, float sp, float sm, float sx, fx gp1) {
  const float ik = fx_fraction(fx_inv_table(k)) * 2.0f, i1 = fx_fraction(fx_inv_table(k - 1)) * 2.0f;
  return sp * (fx_fraction(gp1) * 8.0f) * (i1 - ik) - sm * ik + sx * i1;
}
// last order and first FP32 order for the exponent E
ES_HD int fx_relax_last(int E) { return 1 + (55 - E) / -E; }
ES_HD int fx_relax_first_f(int E) { return fx_min(2 + (31 - E) / -E, fx_relax_last(E) + 1); }

// The root of g (1 + h(g)) = q near 1 with h = sum_{k>2} S_k (g 2^E)^{k-2}/a and q = -A (gam-1)
// 2^(-2 E - er - 4)/(J a), as n 2^-61; 0 where it is not found here (outside 0.5 .. 1.5, |h| >= 1/2,
// no convergence).  a: fx_relax_unit's bits; T: S_k below order kf (kRelaxGap bits less), Tf: all up to
// kl, as fractions of 2^64 of them; A < 0, J > 0.
// Newton steps in FP32, then steps whose residual is taken in fixed point: each of them gains
// 20 bits, so one that moved by less than 2^-38 was the last.
ES_HD fx fx_relax_root(fx a, int unit, int E, int er, int kf, int kl, const fx* T, const float* Tf, double A, double J,
                       fx g1, int eg) {
  const int eA = (fx_hi_word(A) & 0x7fffffff) >> 20, eJ = fx_hi_word(J) >> 20;
  if (a < (1ll << 40) || eA < 123 || eA > 1923 || eJ < 123 || eJ > 1923) return 0;
  const int lz = fx_clz(uint64_t(a)), room = lz - 1 + kRelaxGap;  // 2^room a of the orders' unit: na
  const fx na = a << (lz - 1), nJ = fx_from_positive(J, eJ) * 2;  // J = nJ 2^(eJ - 1085)
  const fx ia = fx_rcp(na, fx_rcp_seed(na)) * 2, iJ = fx_rcp(nJ, fx_rcp_seed(nJ)) * 2;  // 2^61 .. 2^62
  fx AG = fx_mul(fx_from_positive(-A, eA), g1), ii = fx_mul(ia, iJ);
  const int ca = fx_clz(uint64_t(AG)) - 2, ci = fx_clz(uint64_t(ii)) - 2;
  fx q = fx_mul(AG << ca, ii << ci);  // 2^58 .. 2^60
  const int up = eA - eJ + eg - 2 * E - er + unit + lz - 62 - ca - ci;
  if (up < 0 || up > 4) return 0;
  q <<= up;
  if (q < (1ll << 60) || q > (3ll << 60)) return 0;
  const float ra = fx_mulf(fx_rcpf(fx_fraction(na)), fx_pow2(room));  // 1/a
  const float qf = fx_fraction(q) * 8.0f, sE = fx_pow2(E);
  float g = qf, slope = 1.0f;
#pragma unroll 1
  for (int it = 0; it < 3; ++it) {
    const float u = fx_mulf(g, sE);
    float P = 0.0f, dP = 0.0f;
#pragma unroll 1
    for (int k = kl; k >= 3; --k) {
      dP = fx_fma(dP, u, P);
      P = fx_fma(P, u, Tf[k]);
    }
    const float h = fx_mulf(ra, fx_mulf(u, P));
    slope = fx_add(fx_add(1.0f, h), fx_mulf(ra, fx_mulf(u, fx_fma(u, dP, P))));
    if (!(slope > 0.25f)) return 0;
    g = fx_fma(-(fx_fma(g, h, fx_add(g, -qf))), fx_rcpf(slope), g);
  }
  if (!(g >= 0.5f && g <= 1.5f)) return 0;
  const float k1 = fx_rcpf(slope);
  float tail = 0.0f;
#pragma unroll 1
  for (int k = kl; k >= kf; --k) tail = fx_fma(tail, fx_mulf(g, sE), Tf[k]);
  if (!(tail > -0.5f && tail < 0.5f)) return 0;
  const fx tail64 = fx(int(tail * 0x1p31f)) * (1ll << 33);
  fx n = fx(int(g * 0x1p29f)) * (1ll << 32);
#pragma unroll 1
  for (int it = 0; it < 5; ++it) {
    const fx u = fx_shift(n, E + 3);
    fx h = tail64;
#pragma unroll 1
    for (int k = kf - 1; k >= 3; --k) h = T[k] + fx_mul(h, u);
    h = fx_mul(h, u);
    if ((fx_abs(h) >> (61 - room)) != 0) return 0;
    const fx res = q - n - fx_mul63(n, fx_mul(h * (1ll << room), ia) * 8);
    const fx step = fx(float(res) * k1);
    n += step;
    if (n < (1ll << 60) || n > (3ll << 60)) return 0;
    if (fx_abs(step) < (1ll << 23)) return n;
  }
  return 0;
}

}  // namespace es
