// k_volume of the FP64 mode: flux differencing, face terms and viscous divergence in 64-bit block
// fixed point on the integer pipe (es_fx.cuh), FP64 for d and the element sums.
//
// Bound: the FP64 form spent 84 % of its time on the FP64 pipe (52 FP64 instructions per pair of
// nodes, ~76 scheduler slots each).  A pair now takes about 230 integer and FP32 instructions, half
// of them on the half-rate ALU pipe, which sets the time.  Taylor--Green 32^3 p = 3, one stage's
// launch (mean of a step's three): 1089 us -> 254 us; p = 5, 11 x 9 x 13: 363 us -> 100 us.
// Accuracy against long double (right-hand side, 149 states, per variable): 0.29 of the FP64 form's
// error in the median, 1.06 at most; element sums equal to two digits.
#pragma once
#include "es_fx.cuh"

namespace es {

// High words of each element's extreme values: largest and smallest z1, z5, largest |z2..z4|.
// kBad: a face flux, viscous flux or sum beyond the element's scales (kFxMass: a mass flux).
// kRetry: the element is in its second attempt.  kMxT, kMxH: bits by which its momentum and energy fluxes pass
// the scales (before the lines, for Navier--Stokes: largest stress and viscous energy flux).
enum { kMx1, kMn1, kMx5, kMn5, kMxV, kBad, kRetry, kMxT, kMxH, kFxMeta };
constexpr int kFxWide = 1, kFxMass = 2;

template <int P1, int EPB>
struct VolFxSmem {
  static constexpr int Np = P1 * P1 * P1;
  static constexpr size_t red = 0;                                          // [2][EPB Np] doubles, over z
  static constexpr size_t z = 0;                                            // [5][EPB Np] fx
  static constexpr size_t acc = z + size_t(5) * EPB * Np * 8;               // [5][EPB Np] fx (slow elements: double)
  static constexpr size_t pair = acc + size_t(5) * EPB * Np * 8;            // [EPB Np] z1, z5 as float pairs
  static constexpr size_t w3 = pair + size_t(EPB) * Np * 16;                // [Np] omega_i omega_j omega_k
  static constexpr size_t scale = w3 + size_t(Np) * 8;                      // [EPB] FxScale
  static constexpr size_t meta = scale + EPB * sizeof(FxScale);             // [kFxMeta][EPB]
  static constexpr size_t bytes = meta + size_t(kFxMeta) * EPB * sizeof(int);
};

// Position of node n in the tile's shared-memory planes.  P1 = 4: a permutation within the
// element for which the 16 lines of any direction, at any position along the line, lie in 16
// different 8-byte banks (plain order: 4-way conflicts along x1 and x2).
template <int P1>
__device__ __forceinline__ int fx_pos(int n) {
  if (P1 != 4) return n;
  const int k = n >> 4, j = (n >> 2) & 3, i = n & 3;
  return (k << 4) | (((j + k) & 3) << 2) | ((i + k) & 3);
}

// Extremes per element in shared memory, one value of every lane (all lanes of the warp present): one
// atomic for a warp within one element, else one per lane (which are taken one by one where they
// meet at an address).  Taylor--Green 32^3 p = 3: k_volume_fx 265 -> 254 us per launch.
__device__ __forceinline__ void fx_smem_max(int* at, int v, bool one) {
  if (one) {
    v = __reduce_max_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMax(at, v);
  } else {
    atomicMax(at, v);
  }
}
__device__ __forceinline__ void fx_smem_min(int* at, int v, bool one) {
  if (one) {
    v = __reduce_min_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) atomicMin(at, v);
  } else {
    atomicMin(at, v);
  }
}
// whether all lanes of the warp hold the same value
__device__ __forceinline__ bool warp_uniform(int v) {
  return __all_sync(0xffffffffu, v == __shfl_sync(0xffffffffu, v, 0));
}

// largest biased exponent of the instance's metrics
__device__ __forceinline__ int fx_metric_exponent(const InstGeom& G) {
  return max(max(__double2hiint(G.metric[0]), __double2hiint(G.metric[1])), __double2hiint(G.metric[2])) >> 20;
}

// Whether an element's viscous fluxes could leave its scales, from exponents: stress below mu |v| (2/h)/omega
// 2^3, heat below kappa/R p/rho (2/h)/omega 2^1
__device__ __forceinline__ bool fx_viscous_element(const FxParams& P, const FxScale& sc, int em) {
  const int d = em - 1022 + P.fxKw, E1 = sc.e1 - 1022, v = sc.ev - 1022 - E1 + 1;
  const int t = (__double2hiint(P.mu) >> 20) + d + v + 3;
  const int h = (__double2hiint(P.kappa_heat * P.inv_R) >> 20) + 2 - 2 * E1 + d + 1;
  const int room = sc.tier == kFxNear ? 1081 : 1080;
  return t > room + fx_unit(sc, 1) || max(h, t + v) > room + fx_unit(sc, 4);
}

// An LGL line of an element outside the fixed-point range, in FP64 with its face terms (the
// arithmetic of volume_body), from the parameter vector in global memory; acc holds doubles
template <int P1, bool NS>
__device__ __noinline__ void volume_line_fp64(const Params& P, const double* __restrict__ aux,
                                              const double* __restrict__ F, const double* __restrict__ FL,
                                              const double* __restrict__ fV, int e, int m, int ab, double met,
                                              double* acc, int stride) {
  constexpr int P2 = P1 * P1, Np = P1 * P2;
  const long long N = (long long)P.K * Np, g0 = (long long)e * Np;
  const int a = ab % P1, b = ab / P1;
  Zstate<double> z[P1];
  double r[P1][5];
  for (int i = 0; i < P1; ++i) {
    const long long g = g0 + line_node<P1>(m, a, b, i);
    for (int c = 0; c < kAux; ++c) z[i].z[c] = aux[c * N + g];
    for (int v = 0; v < 5; ++v) r[i][v] = 0.0;
  }
  for (int i = 0; i < P1; ++i)
    for (int j = i + 1; j < P1; ++j) {
      double f[5];
      ec_flux(z[i], z[j], m, P.Cd, f);
      for (int v = 0; v < 5; ++v) {
        r[i][v] = fma(P.D2[i * P1 + j], f[v], r[i][v]);
        r[j][v] = fma(P.D2[j * P1 + i], f[v], r[j][v]);
      }
    }
  const bool lo_b = at_boundary(P, e, m, 0);
  const int em = lo_b ? e : neighbour(P, e, m, -1);
  const double* Fm = lo_b ? FL : F;
  for (int v = 0; v < 5; ++v) {
    r[P1 - 1][v] = fma(P.inv_omega_end, F[((long long)(m * 5 + v) * P.K + e) * P2 + ab], r[P1 - 1][v]);
    r[0][v] = fma(-P.inv_omega_end, Fm[((long long)(m * 5 + v) * P.K + em) * P2 + ab], r[0][v]);
  }
  if (NS) {
    const int ep = neighbour(P, e, m, +1);
    for (int c = 0; c < 4; ++c) {
      const double* fc = fV + (long long)(m * 4 + c) * N;
      double fl[P1];
      for (int j = 0; j < P1; ++j) fl[j] = fc[g0 + line_node<P1>(m, a, b, j)];
      const double f_next =
          at_boundary(P, e, m, 1) ? fl[P1 - 1] : fc[(long long)ep * Np + line_node<P1>(m, a, b, 0)];
      const double f_prev = lo_b ? fl[0] : fc[(long long)em * Np + line_node<P1>(m, a, b, P1 - 1)];
      for (int i = 0; i < P1; ++i) {
        double s = 0.0;
        for (int j = 0; j < P1; ++j) s = fma(P.D[i * P1 + j], fl[j], s);
        if (i == P1 - 1) s += 0.5 * P.inv_omega_end * (f_next - fl[P1 - 1]);
        if (i == 0) s -= 0.5 * P.inv_omega_end * (f_prev - fl[0]);
        r[i][1 + c] -= s;
      }
    }
  }
  for (int i = 0; i < P1; ++i) {
    const int n = fx_pos<P1>(line_node<P1>(m, a, b, i));
    for (int v = 0; v < 5; ++v) acc[v * stride + n] = fma(-met, r[i][v], m == 0 ? 0.0 : acc[v * stride + n]);
  }
}

// One LGL line in fixed point: every unordered pair once, both nodes' sums in registers, the
// face fluxes at both ends (f_hi, f_lo: plane stride fs), for Navier--Stokes the viscous
// divergence, then each node's sum times metric/omega_i into the element's accumulator.  Component order (z1, z_m, the other two, z5),
// so that the flux needs no selects on the direction.  Returns 0, or what does not
// fit the element's scales (kFxMass, kFxWide): a face flux (2^60, near: 2^61), a viscous flux (2^58, 2^59) or a sum
// (2^61: the weighted sums of three directions stay below 2^63).  States at the corners of the range bring
// the sums to 0.8 of 2^63, and one that wrapped would still be seen, being below 1.75 of it.  need[] takes the bits by which
// fluxes pass (kMxT, kMxH: momentum, energy); a sum that passes takes two of each.  check: only the fluxes.
// Viscous part: omega_i (D f + lifting)_i = sum_{j != i} Q_ij f_j + f_next/2 (i = p) - f_prev/2
// (i = 0), the diagonal of D cancelling the lifting's interior half (fv: planes of this direction,
// plane stride N; v_hi, v_lo: nodes whose values stand for f_next and f_prev).
template <int P1, int TIER, bool NS, int DIRS>
__device__ __forceinline__ int volume_line_fx(const FxParams& P, const FxScale& sc, int m, int a, int b, fx wm,
                                               const fx* __restrict__ z, const float4* __restrict__ zf,
                                               const double* __restrict__ f_hi, const double* __restrict__ f_lo,
                                               long long fs, const double* __restrict__ fv, long long g0,
                                               long long v_hi, long long v_lo, long long N, fx* __restrict__ acc,
                                               int stride, int* __restrict__ need, int need_stride, bool check) {
  const int c1 = m, c2 = m == 2 ? 0 : m + 1, c3 = m == 0 ? 2 : m - 1;
  const int comp[5] = {0, (1 + c1) * stride, (1 + c2) * stride, (1 + c3) * stride, 4 * stride};
  fx r[P1][5];
#pragma unroll
  for (int i = 0; i < P1; ++i)
#pragma unroll
    for (int c = 0; c < 5; ++c) r[i][c] = 0;
  int mass = 0, mom = 0, ener = 0;  // bits beyond the scales (0 or less: fits)
  {
    const int v[5] = {0, 1 + c1, 1 + c2, 1 + c3, 4};
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      const int emax = 1084 + fx_unit(sc, c == 0 ? 0 : (c == 4 ? 4 : 1));
      const double hi = f_hi[v[c] * fs], lo = f_lo[v[c] * fs];
      const int top = max(__double2hiint(hi) & 0x7fffffff, __double2hiint(lo) & 0x7fffffff) >> 20;
      int& over = c == 0 ? mass : (c == 4 ? ener : mom);
      over = max(over, top - (emax - (TIER == kFxNear ? 1 : 2)));
      r[P1 - 1][c] = fx_from_double(hi, emax);
      r[0][c] = -fx_from_double(lo, emax);
    }
    if constexpr (NS) {
#pragma unroll
      for (int c = 1; c < 5; ++c) {
        const int emax = 1083 + fx_unit(sc, c == 4 ? 4 : 1);  // twice the value: Q carries a factor 1/4 and 65 bits
        const double* f = fv + (long long)(c == 4 ? 3 : v[c] - 1) * N;
        double fl[P1];
#pragma unroll
        for (int j = 0; j < P1; ++j) fl[j] = f[g0 + line_node<P1>(m, a, b, j)];
        const double hi = f[v_hi], lo = f[v_lo];
        int top = max(__double2hiint(hi) & 0x7fffffff, __double2hiint(lo) & 0x7fffffff);
        fx n[P1];
#pragma unroll
        for (int j = 0; j < P1; ++j) {
          top = max(top, __double2hiint(fl[j]) & 0x7fffffff);
          n[j] = fx_from_double(fl[j], emax);
        }
        int& over = c == 4 ? ener : mom;
        over = max(over, (top >> 20) - (emax - (TIER == kFxNear ? 2 : 3)));
        r[P1 - 1][c] -= fx_from_double(hi, emax) >> 2;
        r[0][c] += fx_from_double(lo, emax) >> 2;
#pragma unroll
        for (int i = 0; i < P1; ++i)
#pragma unroll
          for (int j = i + 1; j < P1; ++j) {
            r[i][c] -= fx_mul(P.fxQ[i * P1 + j], n[j]);
            r[j][c] += fx_mul(P.fxQ[i * P1 + j], n[i]);
          }
      }
    }
  }
  // the element is done again in other scales, or in FP64: no pair of this line is formed (viscous
  // shock p = 3 25^3, where a band of elements needs the second attempt: 744 -> 693 us per launch)
  if ((mass | mom | ener) > 0) {
    atomicMax(need + kMxT * need_stride, mom);
    atomicMax(need + kMxH * need_stride, ener);
    return mass > 0 ? kFxMass : kFxWide;
  }
  if (check) return 0;
#pragma unroll
  for (int i = 0; i < P1 - 1; ++i) {
    fx si[5];
    const int ni = fx_pos<P1>(line_node<P1>(m, a, b, i));
#pragma unroll
    for (int c = 0; c < 5; ++c) si[c] = z[comp[c] + ni];
    const float4 qi = zf[ni];
    const FxPair fi[2] = {{qi.x, qi.y}, {qi.z, qi.w}};
#pragma unroll
    for (int j = i + 1; j < P1; ++j) {
      fx sj[5], g[5];
      const int nj = fx_pos<P1>(line_node<P1>(m, a, b, j));
#pragma unroll
      for (int c = 0; c < 5; ++c) sj[c] = z[comp[c] + nj];
      const float4 qj = zf[nj];
      const FxPair fj[2] = {{qj.x, qj.y}, {qj.z, qj.w}};
      fx_flux<TIER>(si, fi, sj, fj, P.fxQ[i * P1 + j], sc, g);
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        r[i][c] += g[c];
        r[j][c] -= g[c];
      }
    }
  }
  int over = 0;
#pragma unroll
  for (int i = 0; i < P1; ++i) {
    const int n = fx_pos<P1>(line_node<P1>(m, a, b, i));
    const fx w = fx_mul63(P.fxW[i], wm);
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      over |= fx_hi(r[i][c]) + 0x20000000;  // bits 30, 31 set unless |r| < 2^61
      const fx val = fx_mul63(r[i][c], w);
      if constexpr (DIRS == 3)  // integer sums: any order gives the same bits
        atomicAdd(reinterpret_cast<unsigned long long*>(acc) + comp[c] + n, (unsigned long long)val);
      else
        acc[comp[c] + n] = m == 0 ? val : acc[comp[c] + n] + val;
    }
  }
  if (!(over & 0xc0000000)) return 0;
  atomicMax(need + kMxT * need_stride, 2);
  atomicMax(need + kMxH * need_stride, 2);
  return kFxWide;
}

// Tiles (elements per CTA, threads) and register bounds, measured on GB300 (one right-hand side,
// tiles 0, 1 and 2, us): the kernel waits on the latency of its dependent integer products, so few
// registers pay until they spill into the sums.  Taylor--Green 48^3 p = 2: 297, 319, 318; 40^3 p = 3: 447, 416,
// 421; 32^3 p = 4: 565, 676, 668 (the second at 128 registers 698); 24^3 p = 5: 620, 633, 800; Navier--Stokes 24^3
// p = 4: 390, 471, 459 (the second at 128 registers 510).
// Variant 3 is for meshes of few elements, whatever tile is asked for (the bits are the same): one
// element per CTA and a thread for every line of its three directions.
constexpr int kVolFxSmall = 3;
template <int P1, int V> struct VolFxCfg;
template <> struct VolFxCfg<3, 0> { static constexpr int EPB = 16, THREADS = 160, REGS = 100; };
template <> struct VolFxCfg<3, 1> { static constexpr int EPB = 32, THREADS = 288, REGS = 100; };
template <> struct VolFxCfg<3, 2> { static constexpr int EPB = 3, THREADS = 32, REGS = 100; };
template <> struct VolFxCfg<3, kVolFxSmall> { static constexpr int EPB = 1, THREADS = 32, REGS = 168; };
template <> struct VolFxCfg<4, 0> { static constexpr int EPB = 4, THREADS = 64, REGS = 168; };
template <> struct VolFxCfg<4, 1> { static constexpr int EPB = 8, THREADS = 128, REGS = 128; };
template <> struct VolFxCfg<4, 2> { static constexpr int EPB = 2, THREADS = 32, REGS = 128; };
template <> struct VolFxCfg<4, kVolFxSmall> { static constexpr int EPB = 1, THREADS = 64, REGS = 168; };
template <> struct VolFxCfg<5, 0> { static constexpr int EPB = 5, THREADS = 128, REGS = 168; };
template <> struct VolFxCfg<5, 1> { static constexpr int EPB = 1, THREADS = 32, REGS = 168; };
template <> struct VolFxCfg<5, 2> { static constexpr int EPB = 2, THREADS = 64, REGS = 168; };
template <> struct VolFxCfg<5, kVolFxSmall> { static constexpr int EPB = 1, THREADS = 96, REGS = 168; };
template <> struct VolFxCfg<6, 0> { static constexpr int EPB = 2, THREADS = 96, REGS = 168; };
template <> struct VolFxCfg<6, 1> { static constexpr int EPB = 4, THREADS = 160, REGS = 128; };
template <> struct VolFxCfg<6, 2> { static constexpr int EPB = 1, THREADS = 64, REGS = 168; };
template <> struct VolFxCfg<6, kVolFxSmall> { static constexpr int EPB = 1, THREADS = 128, REGS = 168; };

// DIRS: directions worked on together, 1 (in turn, by the same threads) or 3 (small meshes)
template <int P1, int EPB, int THREADS, int REGS, bool NS, int DIRS = 1>
__global__ void __launch_bounds__(THREADS, 65536 / (THREADS * REGS)) k_volume_fx(const __grid_constant__ FxParams P,
                                                       const __grid_constant__ StageVol sv,
                                                       const double* __restrict__ aux, const double* __restrict__ F,
                                                       const double* __restrict__ FL,
                                                       const double* __restrict__ fV) {
  using S = VolFxSmem<P1, EPB>;
  constexpr int P2 = P1 * P1, Np = P1 * P2, ST = EPB * Np;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx* z = reinterpret_cast<fx*>(smem_raw + S::z);
  fx* acc = reinterpret_cast<fx*>(smem_raw + S::acc);
  double* w3 = reinterpret_cast<double*>(smem_raw + S::w3);
  FxScale* scale = reinterpret_cast<FxScale*>(smem_raw + S::scale);
  int* meta = reinterpret_cast<int*>(smem_raw + S::meta);
  float4* zf = reinterpret_cast<float4*>(smem_raw + S::pair);
  double* red = reinterpret_cast<double*>(smem_raw + S::red);
  const long long N = (long long)P.K * Np;
  const int e0 = blockIdx.x * EPB;
  const int nel = min(EPB, P.K - e0);
  const int nn = nel * Np;

  // the tile's parameter vector: each element's extreme values, then fixed point in their scales
  {
    constexpr int NT = (ST + THREADS - 1) / THREADS;
    double ld[NT][kAux];
    const double* __restrict__ src = aux + (long long)e0 * Np;
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int t = threadIdx.x + i * THREADS;
#pragma unroll
      for (int c = 0; c < kAux; ++c)
        ld[i][c] = src[c * N + min(t, nn - 1)];
    }
    for (int t = threadIdx.x; t < kFxMeta * EPB; t += THREADS) {
      const int k = t / EPB;
      meta[t] = k == kMn1 || k == kMn5 ? 0x7fffffff : 0;
    }
    for (int n = threadIdx.x; n < Np; n += THREADS)
      w3[n] = P.omega[n % P1] * P.omega[(n / P1) % P1] * P.omega[n / P2];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      // (threads beyond the tile repeat its last node)
      const int el = min(int(threadIdx.x) + i * THREADS, nn - 1) / Np;
      const int h1 = __double2hiint(ld[i][0]), h5 = __double2hiint(ld[i][4]);
      const int hv = max(max(__double2hiint(ld[i][1]) & 0x7fffffff, __double2hiint(ld[i][2]) & 0x7fffffff),
                         __double2hiint(ld[i][3]) & 0x7fffffff);
      const bool one = warp_uniform(el);
      fx_smem_max(meta + kMx1 * EPB + el, h1, one);
      fx_smem_min(meta + kMn1 * EPB + el, h1, one);
      fx_smem_max(meta + kMx5 * EPB + el, h5, one);
      fx_smem_min(meta + kMn5 * EPB + el, h5, one);
      fx_smem_max(meta + kMxV * EPB + el, hv, one);
    }
    __syncthreads();
    bool viscous = false;
    if (threadIdx.x < nel) {
      const int el = threadIdx.x;
      scale[el] = fx_scale(meta[kMx1 * EPB + el], meta[kMn1 * EPB + el], meta[kMx5 * EPB + el],
                           meta[kMn5 * EPB + el], meta[kMxV * EPB + el], P.fxC, P.fxKt);
      if (!fx_mesh(P, inst_of(P, e0 + el))) scale[el].tier = kFxSlow;
      // (heat conduction does not vanish with the velocity)
      if constexpr (NS) scale[el].se = min(max(1018 - scale[el].ev, 0), kFxMargin);
      if constexpr (NS) viscous = fx_viscous_element(P, scale[el], fx_metric_exponent(geom_of(P, inst_of(P, e0 + el))));
    }
    // Where the viscous fluxes may not fit: looked at before any pair is formed, and the room they need
    // given at once (an element that does not fit all the same is found below).
    // Viscous shock 25^3 p = 3 693 -> 540 us per launch (576 with the room that every element is given now,
    // three bits or what it needs); looked at without the estimate before it, Navier--Stokes p = 4 takes
    // 941 us (930 with, 924 with neither).
    if constexpr (NS) {
      if (__syncthreads_or(viscous)) {
#pragma unroll 1
        for (int t0 = 0; t0 < nn; t0 += THREADS) {
          const int t = min(t0 + int(threadIdx.x), nn - 1), el = t / Np;
          const double* f = fV + (long long)e0 * Np + t;
          int top[2] = {0, 0};
#pragma unroll
          for (int c = 0; c < 12; ++c) {
            int& h = top[(c & 3) == 3];
            h = max(h, __double2hiint(f[c * N]) & 0x7fffffff);
          }
          const bool one = warp_uniform(el);
          fx_smem_max(meta + kMxT * EPB + el, top[0], one);
          fx_smem_max(meta + kMxH * EPB + el, top[1], one);
        }
        __syncthreads();
        if (threadIdx.x < nel) {
          const int el = threadIdx.x, room = scale[el].tier == kFxNear ? 1081 : 1080;  // volume_line_fx's limits
          int &t = meta[kMxT * EPB + el], &h = meta[kMxH * EPB + el];
          fx_widen(scale[el], max((t >> 20) - room - fx_unit(scale[el], 1), 0), max((h >> 20) - room - fx_unit(scale[el], 4), 0));
          t = h = 0;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < NT; ++i) {
      const int t = threadIdx.x + i * THREADS;
      if (t < nn) {
        const int el = t / Np;
        const int ev = fx_block_exponent_v(meta[kMxV * EPB + el]);
        fx* zt = z + el * Np + fx_pos<P1>(t - el * Np);
        const fx z1 = fx_from_positive(ld[i][0], fx_block_exponent(meta[kMx1 * EPB + el]));
        const fx z5 = fx_from_positive(ld[i][4], fx_block_exponent(meta[kMx5 * EPB + el]));
        const FxPair p1 = fx_pair(z1), p5 = fx_pair(z5);
        zf[zt - z] = make_float4(p1.h, p1.l, p5.h, p5.l);
        zt[0] = z1;
        zt[ST] = fx_from_double(ld[i][1], ev);
        zt[2 * ST] = fx_from_double(ld[i][2], ev);
        zt[3 * ST] = fx_from_double(ld[i][3], ev);
        zt[4 * ST] = z5;
      }
    }
  }
  __syncthreads();

  // all three directions; elements whose fluxes did not fit their scales once more in coarser ones
  const int my = threadIdx.x;
#pragma unroll 1
  for (int attempt = 0; attempt < 2; ++attempt) {
    if constexpr (DIRS == 3) {
      for (int t = threadIdx.x; t < 5 * ST; t += THREADS)
        if (attempt == 0 || (t % ST < nn && meta[kRetry * EPB + t % ST / Np])) acc[t] = 0;
      __syncthreads();
    }
#pragma unroll 1
    for (int m0 = 0; m0 < 3; m0 += DIRS) {
      for (int l3 = threadIdx.x; l3 < DIRS * nel * P2; l3 += THREADS) {
        const int m = DIRS == 3 ? l3 / (nel * P2) : m0;
        const int l = DIRS == 3 ? l3 - m * (nel * P2) : l3;
        const int el = l / P2, ab = l % P2, e = e0 + el;
        const FxScale& sc = scale[el];
        if (sc.tier == kFxSlow || (attempt && !meta[kRetry * EPB + el])) continue;
        // (passed in an earlier direction: only how far this one's fluxes pass)
        const bool check = DIRS == 1 && m && meta[kBad * EPB + el];
        const InstGeom& G = geom_of(P, inst_of(P, e));
        const int em = fx_metric_exponent(G);
        const fx wm = fx_from_double(G.metric[m], em);
        // this element's +x_m flux and the -x_m neighbour's (the boundary flux in FL)
        const long long fs = (long long)P.K * P2;
        const bool lo_b = at_boundary(P, e, m, 0);
        const double* f_hi = F + m * 5 * fs + (long long)e * P2 + ab;
        const double* f_lo = (lo_b ? FL : F) + m * 5 * fs + (long long)(lo_b ? e : neighbour(P, e, m, -1)) * P2 + ab;
        const int a = ab % P1, b = ab / P1;
        const long long g0 = (long long)e * Np;
        long long v_hi = 0, v_lo = 0;
        if constexpr (NS) {  // boundary faces take the interior viscous flux
          v_hi = at_boundary(P, e, m, 1) ? g0 + line_node<P1>(m, a, b, P1 - 1)
                                         : (long long)neighbour(P, e, m, +1) * Np + line_node<P1>(m, a, b, 0);
          v_lo = lo_b ? g0 + line_node<P1>(m, a, b, 0)
                      : (long long)neighbour(P, e, m, -1) * Np + line_node<P1>(m, a, b, P1 - 1);
        }
        const double* fv = NS ? fV + (long long)(m * 4) * N : nullptr;
        int beyond;
        if (sc.tier == kFxNear)
          beyond = volume_line_fx<P1, kFxNear, NS, DIRS>(P, sc, m, a, b, wm, z + el * Np, zf + el * Np, f_hi, f_lo, fs, fv, g0,
                                                 v_hi, v_lo, N, acc + el * Np, ST, meta + el, EPB, check);
        else
          beyond = volume_line_fx<P1, kFxFar, NS, DIRS>(P, sc, m, a, b, wm, z + el * Np, zf + el * Np, f_hi, f_lo, fs, fv, g0,
                                                v_hi, v_lo, N, acc + el * Np, ST, meta + el, EPB, check);
        if (beyond) atomicOr(meta + kBad * EPB + el, beyond);
      }
      __syncthreads();
    }
    const bool bad = my < nel && scale[my].tier != kFxSlow && meta[kBad * EPB + my];
    if (attempt == 0 && bad) {
      fx_widen(scale[my], meta[kMxT * EPB + my], meta[kMxH * EPB + my]);
      if (meta[kBad * EPB + my] & kFxMass) scale[my].tier = kFxSlow;
      meta[kRetry * EPB + my] = 1;
      meta[kBad * EPB + my] = 0;
    }
    if (attempt == 1 && bad) scale[my].tier = kFxSlow;
    if (!__syncthreads_or(bad)) break;
  }
  // elements outside the fixed-point range, in FP64
  if (__syncthreads_or(my < nel && scale[my].tier == kFxSlow)) {
#pragma unroll 1
    for (int m = 0; m < 3; ++m) {
      for (int l = threadIdx.x; l < nel * P2; l += THREADS) {
        const int el = l / P2;
        if (scale[el].tier != kFxSlow) continue;
        volume_line_fp64<P1, NS>(P, aux, F, FL, fV, e0 + el, m, l % P2, geom_of(P, inst_of(P, e0 + el)).metric[m],
                                 reinterpret_cast<double*>(acc) + el * Np, ST);
      }
      __syncthreads();
    }
  }

  // node phase: k_i = volume sums + face terms; d in the last stage; element sums (z is dead)
  const bool wantE = sv.E != nullptr;
  const bool wantA = sv.dw != nullptr;
  for (int t = threadIdx.x; t < nn; t += THREADS) {
    const long long g = (long long)e0 * Np + t;
    const int el = t / Np, n = t % Np, e = e0 + el;
    const InstGeom& G = geom_of(P, inst_of(P, e));
    const FxScale& sc = scale[el];
    double k[5];
    const int at = el * Np + fx_pos<P1>(n);
    if (sc.tier == kFxSlow) {
#pragma unroll
      for (int v = 0; v < 5; ++v) k[v] = reinterpret_cast<const double*>(acc)[v * ST + at];
    } else {
      const int em = fx_metric_exponent(G) - 1022 + P.fxKw + 1;  // metric: fraction of 2^(E + 1)
#pragma unroll
      for (int v = 0; v < 5; ++v) k[v] = fx_to_double(-acc[v * ST + at], fx_unit(sc, v) + em);
    }
    if (sv.d_out) {
      const double cs = sv.dcoef_self * G.dt;
      double dv[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) dv[v] = cs * k[v];
      for (int j = 0; j < sv.nd; ++j) {
        const double cj = sv.dcoef[j] * G.dt;
#pragma unroll
        for (int v = 0; v < 5; ++v) dv[v] = fma(cj, static_cast<const double*>(sv.dk[j])[v * N + g], dv[v]);
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) sv.d_out[v * N + g] = dv[v];
    } else {
      double* ko = sv.kout64 ? sv.kout64 : static_cast<double*>(sv.kout);
#pragma unroll
      for (int v = 0; v < 5; ++v) ko[v * N + g] = k[v];
    }
    if (wantE) {
      Zstate<double> s;
#pragma unroll
      for (int c = 0; c < kAux; ++c) s.z[c] = aux[c * N + g];
      double w[5];
      z_to_w(s, P.Cd, w);
      double sum = 0.0;
#pragma unroll
      for (int v = 0; v < 5; ++v) sum = fma(w[v], k[v], sum);
      red[t] = w3[n] * sum;
    }
    if (wantA) {
      double sum = 0.0;
#pragma unroll
      for (int v = 0; v < 5; ++v) sum = fma(sv.dw[v * N + g], k[v], sum);
      red[ST + t] = w3[n] * sum;
    }
  }
  const bool doA = sv.A != nullptr && (wantA || sv.A_init);
  if (!wantE && !doA) return;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int el = warp; el < nel; el += THREADS >> 5) {
    const int e = e0 + el;
    const InstGeom& G = geom_of(P, inst_of(P, e));
    double sE = 0.0, sA = 0.0;
    for (int n = lane; n < Np; n += 32) {
      if (wantE) sE += red[el * Np + n];
      if (wantA) sA += red[ST + el * Np + n];
    }
    if (wantE) sE = warp_sum(sE);
    if (wantA) sA = warp_sum(sA);
    if (lane == 0) {
      if (wantE) sv.E[e] = G.J * sE;
      if (doA) sv.A[e] = (sv.A_init ? 0.0 : sv.A[e]) + (wantA ? sv.A_scale * (G.J * G.dt) * sA : 0.0);
    }
  }
}

}  // namespace es
