// The viscous flux of a node from the gradients of its entropy variables in 64-bit fixed point
// (es_grad_fx.cuh has the kernel and its figures).
#pragma once
#include "es_relax_fx.cuh"

namespace es {

// Exponents of the gas constants: x = n 2^(e - 62), n from fx_from_positive
struct FxViscous {
  fx mu, kap;  // mu; kappa/R
  int emu, ekap;
};

// The viscous flux of a node from t[m][c] = theta_m,c (c = 0..2: z1 z_v; 3: z1^2 = -w_5) in units
// of 2^(ut) for c < 3 and 2^(ut - ev + e1) for c = 3, |t| < 2^62; e1, ev: the element's exponents of
// z1 and z_v (z_k = nz_k 2^(ev - 62), |nz| < 2^62), iz1 = 1/z1 > 0 with z1 above an eighth of 2^e1.
//   b_mk = theta_m,k - v_k theta_m,3, tau_mk = mu a (b_mk + b_km - 2/3 delta_mk tr b), a = 1/z1^2
//   fV_m = (tau_m1, tau_m2, tau_m3, -kappa a^2/R theta_m,3 + sum_k tau_mk v_k)
// The gradients are brought to the top of their 62 bits first: along a line they are fractions of the largest that
// the element's w could have at its thinnest weight, some 2^8 above what they are, and six bits are room below.
ES_HD void fx_viscous_flux(const fx t0[3][4], const fx nz[3], double iz1, int e1, int ev, int ut, const FxViscous& V,
                           double f[3][4]) {
  int top = 1;
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int c = 0; c < 4; ++c) top |= fx_hi(t0[m][c]) ^ (fx_hi(t0[m][c]) >> 31);
  const int up = fx_clz(uint64_t(unsigned(top))) - 34;
  fx t[3][4];
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int c = 0; c < 4; ++c) t[m][c] = t0[m][c] << up;
  ut -= up;
  const int hi = fx_hi_word(iz1) >> 20, ei = hi - 1022;
  const fx ni = fx_from_positive(iz1, hi);  // 2^61 .. 2^62
  fx v[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) v[k] = fx_mul(nz[k], ni) * 4;  // 2^(ev + ei - 62), below 2^62
  fx b[3][3];  // 2^(ut + 6), below 2^61
  const int s = 2 + ei + e1 - 6;
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int k = 0; k < 3; ++k) b[m][k] = (t[m][k] >> 6) - fx_shift(fx_mul(v[k], t[m][3]), s);
  const fx tr = b[0][0] + b[1][1] + b[2][2];
  const fx third = fx_mul63(tr, 0x5555555555555555ll);  // 2/3 tr b
  const fx a = fx_sqr_round(ni * 2);                    // 1/z1^2: 2^(2 ei - 62), 2^60 .. 2^62
  const fx ma0 = fx_mul(V.mu, a);                       // 2^(emu + 2 ei - 60)
  const int ca = fx_clz(uint64_t(ma0)) - 2;
  const fx ma = ma0 << ca;
  fx tau[3][3];
  tau[0][1] = tau[1][0] = fx_mul63(b[0][1] + b[1][0], ma);
  tau[0][2] = tau[2][0] = fx_mul63(b[0][2] + b[2][0], ma);
  tau[1][2] = tau[2][1] = fx_mul63(b[1][2] + b[2][1], ma);
#pragma unroll
  for (int m = 0; m < 3; ++m) tau[m][m] = fx_mul63(2 * b[m][m] - third, ma);
  const int et = V.emu + 2 * ei + ut + 9 - ca;
  const fx kt0 = fx_mul(V.kap, fx_sqr_round(a * 2));  // 2^(ekap + 4 ei - 60)
  const int ck = fx_clz(uint64_t(kt0)) - 2;
  const fx kt = kt0 << ck;
  const int eh = V.ekap + 4 * ei + 4 - ck + ut - ev + e1, ew = et + ev + ei + 1, ec = fx_max(eh, ew);
#pragma unroll
  for (int m = 0; m < 3; ++m) {
    fx w = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      f[m][k] = fx_to_double(tau[m][k], et);
      w += fx_mul63(tau[m][k], v[k]);
    }
    f[m][3] = fx_to_double(fx_shift(w, ew - ec) - fx_shift(fx_mul(kt, t[m][3]), eh - ec), ec);
  }
}

}  // namespace es
