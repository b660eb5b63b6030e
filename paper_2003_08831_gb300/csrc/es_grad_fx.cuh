// k_grad of the FP64 mode in 64-bit block fixed point (es_fx.cuh): BR1 gradients theta_m of w_2..w_5
// and the viscous flux of every node.
//
// Bound: the FP64 form was held by the FP64 pipe (about 135 instructions per node at p = 4).  Here
// w = (z1 z_v, z1^2) are fractions of the element's largest values, the sums along a line are exact
// but for the products' last bits, and so are the face terms: with Q = omega D,
//   omega_i theta_i = sum_{j != i} Q_ij w_j + w_next/2 (i = p) - w_prev/2 (i = 0),
// the diagonal of D cancelling the interior half of the face terms.  The chain rule follows in the same
// units, so a node's flux carries 2^-56 of (its element's w) (2/h)/omega, against FP64's 2^-53 for
// every one of the sum's terms.
//
// Per launch: Navier--Stokes p = 4 32^3 1167 -> 525 us, viscous shock p = 3 25^3 267 -> 127 us
// (80, 96 and 168 registers per thread: within 3 % of 128).
#pragma once
#include "es_viscous_fx.cuh"

namespace es {

// a node of an element outside the fixed-point range (the arithmetic of k_grad)
template <int P1>
__device__ __noinline__ void grad_node_fp64(const Params& P, const double* __restrict__ aux, double* __restrict__ fV, int e,
                                            int n) {
  constexpr int Np = P1 * P1 * P1;
  const long long N = (long long)P.K * Np, g0 = (long long)e * Np, g = g0 + n;
  const InstGeom& G = geom_of(P, inst_of(P, e));
  const int ii[3] = {n % P1, (n / P1) % P1, n / (P1 * P1)};
  double th[3][4], w[4], wn[4];
  const auto load = [&](long long at, double* o) {
    const double z1 = aux[at];
    for (int c = 0; c < 3; ++c) o[c] = z1 * aux[(1 + c) * N + at];
    o[3] = -z1 * z1;
  };
  load(g, w);
#pragma unroll 1
  for (int m = 0; m < 3; ++m) {
    const int im = m == 0 ? ii[0] : (m == 1 ? ii[1] : ii[2]);
    const int a = m == 0 ? ii[1] : ii[0], b = m == 2 ? ii[1] : ii[2];
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int j = 0; j < P1; ++j) {
      load(g0 + line_node<P1>(m, a, b, j), wn);
      for (int c = 0; c < 4; ++c) acc[c] = fma(P.D[im * P1 + j], wn[c], acc[c]);
    }
    if (im == P1 - 1 || im == 0) {
      const bool right = im == P1 - 1;
      if (at_boundary(P, e, m, right ? 1 : 0)) {
        const double* bv = bc_values(P, m, right ? 1 : 0);
        for (int c = 0; c < 4; ++c) wn[c] = bv[6 + c];
      } else {
        load((long long)neighbour(P, e, m, right ? +1 : -1) * Np + line_node<P1>(m, a, b, right ? 0 : P1 - 1), wn);
      }
      const double sg = right ? 0.5 * P.inv_omega_end : -0.5 * P.inv_omega_end;
      for (int c = 0; c < 4; ++c) acc[c] += sg * (wn[c] - w[c]);
    }
    for (int c = 0; c < 4; ++c) th[m][c] = G.metric[m] * acc[c];
  }
  const double iz1 = aux[5 * N + g];
  const double v[3] = {aux[N + g] * iz1, aux[2 * N + g] * iz1, aux[3 * N + g] * iz1};
  const double a = iz1 * iz1, ma = P.mu * a, kt = P.kappa_heat * a * a * P.inv_R;
  double b[3][3];
  for (int m = 0; m < 3; ++m)
    for (int k = 0; k < 3; ++k) b[m][k] = th[m][k] + v[k] * th[m][3];
  const double dsum = (ma * (-2.0 / 3.0)) * (b[0][0] + b[1][1] + b[2][2]);
  for (int m = 0; m < 3; ++m) {
    double fe = kt * th[m][3];
    for (int k = 0; k < 3; ++k) {
      const double tau = m == k ? (ma + ma) * b[m][m] + dsum : ma * (b[m][k] + b[k][m]);
      fV[(long long)(m * 4 + k) * N + g] = tau;
      fe += tau * v[k];
    }
    fV[(long long)(m * 4 + 3) * N + g] = fe;
  }
}

// Tiles (elements per CTA), 128 threads: about two nodes per thread
template <int P1> struct GradFxCfg;
template <> struct GradFxCfg<3> { static constexpr int EPB = 8, THREADS = 128; };
template <> struct GradFxCfg<4> { static constexpr int EPB = 4, THREADS = 128; };
template <> struct GradFxCfg<5> { static constexpr int EPB = 2, THREADS = 128; };
template <> struct GradFxCfg<6> { static constexpr int EPB = 1, THREADS = 128; };
// largest high words of z1 and |z_v| and the smallest of z1, the element's faces' outer states included
enum { kGMx1, kGMn1, kGMxV, kGradMeta };

template <int P1, int EPB, int THREADS>
__global__ void __launch_bounds__(THREADS, 65536 / (THREADS * 128))
    k_grad_fx(const __grid_constant__ FxParams P, const double* __restrict__ aux, double* __restrict__ fV) {
  constexpr int P2 = P1 * P1, Np = P1 * P2, Nf = 6 * P2, ST = EPB * Np, SF = EPB * Nf;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx* ws = reinterpret_cast<fx*>(smem_raw);  // [4][ST] interior, [4][SF] outer states of the faces
  fx* wf = ws + 4 * ST;
  __shared__ int meta[kGradMeta][EPB];
  __shared__ fx sQ[P1 * P1];
  const long long N = (long long)P.K * Np;
  const int e0 = blockIdx.x * EPB, nel = min(EPB, P.K - e0), nn = nel * Np, nf = nel * Nf;
  for (int t = threadIdx.x; t < kGradMeta * EPB; t += THREADS) meta[t / EPB][t % EPB] = t / EPB == kGMn1 ? 0x7fffffff : 0;
  for (int t = threadIdx.x; t < P1 * P1; t += THREADS) {
    const int i = t / P1, j = t % P1;
    sQ[t] = i < j ? P.fxQ[i * P1 + j] : (i > j ? -P.fxQ[j * P1 + i] : 0);
  }
  // outer state of face node t: z1 and z_v, c = 0..3
  const auto outer = [&](int t, double z[4]) {
    const int e = e0 + t / Nf, f = t % Nf / P2, ab = t % P2, m = f >> 1, side = f & 1;
    if (at_boundary(P, e, m, side)) {
      const double* bv = bc_values(P, m, side);
#pragma unroll
      for (int c = 0; c < 4; ++c) z[c] = bv[c];
    } else {
      const double* src = aux + (long long)neighbour(P, e, m, side ? +1 : -1) * Np +
                          line_node<P1>(m, ab % P1, ab / P1, side ? 0 : P1 - 1);
#pragma unroll
      for (int c = 0; c < 4; ++c) z[c] = src[c * N];
    }
  };
  const auto inner = [&](int t, double z[4]) {
#pragma unroll
    for (int c = 0; c < 4; ++c) z[c] = aux[c * N + (long long)e0 * Np + t];
  };
  // (the high word of a negative or NaN z1 counts as beyond every exponent allowed)
  const auto extremes = [&](int el, const double z[4]) {
    const int h1 = __double2hiint(z[0]), hp = h1 < 0 ? 0x7fffffff : h1;
    const bool one = warp_uniform(el);
    fx_smem_max(&meta[kGMx1][el], hp, one);
    fx_smem_min(&meta[kGMn1][el], hp, one);
    fx_smem_max(&meta[kGMxV][el],
                max(max(__double2hiint(z[1]) & 0x7fffffff, __double2hiint(z[2]) & 0x7fffffff),
                    __double2hiint(z[3]) & 0x7fffffff), one);
  };
  __syncthreads();
  double z[4];
  // (threads beyond the tile repeat its last node)
  for (int t0 = 0; t0 < nn; t0 += THREADS) {
    const int t = min(t0 + int(threadIdx.x), nn - 1);
    inner(t, z);
    extremes(t / Np, z);
  }
  for (int t0 = 0; t0 < nf; t0 += THREADS) {
    const int t = min(t0 + int(threadIdx.x), nf - 1);
    outer(t, z);
    extremes(t / Nf, z);
  }
  __syncthreads();
  // w in fixed point: z1 z_v in units of 2^(e1 + ev - 62), z1^2 of 2^(2 e1 - 62)
  const auto put = [&](int el, const double z[4], fx* o, int stride) {
    const int e1 = fx_block_exponent(meta[kGMx1][el]), ev = max(fx_block_exponent(meta[kGMxV][el]), 922);
    const fx n1 = fx_from_positive(z[0], e1) * 2;
#pragma unroll
    for (int c = 0; c < 3; ++c) o[c * stride] = fx_mul63(n1, fx_from_double(z[1 + c], ev));
    o[3 * stride] = fx_sqr_round(n1);
  };
  for (int t = threadIdx.x; t < nn; t += THREADS) {
    inner(t, z);
    put(t / Np, z, ws + t, ST);
  }
  for (int t = threadIdx.x; t < nf; t += THREADS) {
    outer(t, z);
    put(t / Nf, z, wf + t, SF);
  }
  __syncthreads();

  const double kap = P.kappa_heat * P.inv_R;
  const int emu = __double2hiint(P.mu) >> 20, ekap = __double2hiint(kap) >> 20;
  FxViscous V;
  V.mu = fx_from_positive(P.mu, emu);
  V.kap = fx_from_positive(kap, ekap);
  V.emu = emu - 1022;
  V.ekap = ekap - 1022;
  const bool constants = emu > 922 && emu < 1122 && ekap > 922 && ekap < 1122;
  for (int t = threadIdx.x; t < nn; t += THREADS) {
    const int el = t / Np, n = t - el * Np, e = e0 + el;
    const InstGeom& G = geom_of(P, inst_of(P, e));
    const int mx1 = meta[kGMx1][el], mn1 = meta[kGMn1][el], mxv = meta[kGMxV][el];
    const int em = fx_metric_exponent(G);
    // z1 within a factor of two or so; exponents in +-100; NaN and signs fail the comparisons
    if (!constants || (mx1 >> 20) > 1121 || (mn1 >> 20) < 923 || (mx1 >> 20) - (mn1 >> 20) > 1 || (mxv >> 20) > 1121 ||
        em > 1121 || em < 923) {
      grad_node_fp64<P1>(P, aux, fV, e, n);
      continue;
    }
    const int e1 = fx_block_exponent(mx1) - 1022, ev = max(fx_block_exponent(mxv), 922) - 1022;
    const int ii[3] = {n % P1, (n / P1) % P1, n / P2};
    fx th[3][4];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int im = ii[m], a = m == 0 ? ii[1] : ii[0], b = m == 2 ? ii[1] : ii[2];
      const fx* line = ws + el * Np + line_node<P1>(m, a, b, 0);
      constexpr int step[3] = {1, P1, P2};
      fx r[4] = {0, 0, 0, 0};
#pragma unroll
      for (int j = 0; j < P1; ++j) {
        const fx q = sQ[im * P1 + j];
#pragma unroll
        for (int c = 0; c < 4; ++c) r[c] += fx_mul(q, line[c * ST + j * step[m]]);
      }
      if (im == 0 || im == P1 - 1) {
        const fx* o = wf + el * Nf + (2 * m + (im ? 1 : 0)) * P2 + a + P1 * b;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const fx h = o[c * SF] >> 2;
          r[c] += im ? h : -h;
        }
      }
      const fx w = fx_mul63(P.fxW[im], fx_from_double(G.metric[m], em));
#pragma unroll
      for (int c = 0; c < 4; ++c) th[m][c] = fx_mul63(r[c], w);
    }
    const long long g = (long long)e0 * Np + t;
    fx nz[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) nz[k] = fx_from_double(aux[(1 + k) * N + g], ev + 1022);
    double f[3][4];
    fx_viscous_flux(th, nz, aux[5 * N + g], e1, ev, e1 + ev - 62 + P.fxKw + (em - 1022) + 2, V, f);
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int c = 0; c < 4; ++c) fV[(long long)(m * 4 + c) * N + g] = f[m][c];
  }
}
}  // namespace es
