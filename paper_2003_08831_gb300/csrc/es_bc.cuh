// Exterior states of the Dirichlet-penalty boundaries.
#pragma once
#include "../../include/es.h"
#include "es_device.cuh"
#include "es_launch.h"

namespace es {

// Exterior values of the Dirichlet-penalty boundaries at time *t + t_off: a warp evaluates
// one (direction, side) i = 2 m + side.  ES_BC_VISCOUS_SHOCK evaluates the Section 4.1.2 profile: V in
// (V_f, 1) solves x - speed t = (alpha/2) [log((1-V)(V-V_f)) + (1+V_f)/(1-V_f)
// log((1-V)/(V-V_f))] (to the last bit), u = V, rho = 1/V, p from the constant
// total enthalpy H, lab velocity u + speed along the direction.
//
// The bracket is cut into 33 parts per round, one interior point per lane, so that eleven rounds
// reach the last bit of a double: an evaluation (two logarithms) is a chain of ~90 dependent FP64
// operations, 3 us for a warp, and bisection by one thread needed 55 and more of them (502 us a
// launch, four launches of an RK4 step; 25 us as a launch of its own).  It is the first block of
// k_prep, which reads nothing of it: the values are used from k_face on.  Viscous shock 25^3 p = 3: 4
// launches of 37 us gone, k_prep as before; shock tube, 128 elements: 40 launches of 8 us gone, k_prep
// 5.5 -> 9.5 us.
static __device__ __noinline__ void bc_eval_side(const BcEval& bc, int i, int lane) {
  const BcSpec& spec = bc.spec;
  const int m = i / 2, side = i % 2;
  if (spec.kind[m] == ES_BC_PERIODIC) return;
  const double g = spec.gam;
  double q[5];
  if (spec.kind[m] == ES_BC_STATE) {
    for (int v = 0; v < 5; ++v) q[v] = spec.q[m][side][v];
  } else {
    const double vf = spec.vs[m][0], alpha = spec.vs[m][1], H = spec.vs[m][2], speed = spec.vs[m][3];
    const double time = (bc.t ? bc.t[0] : 0.0) + bc.t_off;
    const double xi = spec.vs[m][4 + side] - speed * time;
    const double c = (1.0 + vf) / (1.0 - vf);
    // x(V) decreases; 2 (x(V) - xi)/alpha = (1 + c) log(1 - V) + (1 - c) log(V - V_f) - 2 xi/alpha
    const double rhs = 2.0 * xi / alpha;
    double lo = vf, hi = 1.0;
    for (int it = 0; it < 40; ++it) {
      const double mid = fma(hi - lo, (lane + 1) * (1.0 / 33.0), lo);
      const bool inside = mid > lo && mid < hi;
      const bool below = inside ? (1.0 + c) * log(1.0 - mid) + (1.0 - c) * log(mid - vf) > rhs : mid <= lo;
      const unsigned above = ~__ballot_sync(0xffffffffu, below);  // lanes right of the root
      const int first = above ? __ffs(above) - 1 : 32;
      const double l = __shfl_sync(0xffffffffu, mid, first ? first - 1 : 0);
      const double h = __shfl_sync(0xffffffffu, mid, first < 32 ? first : 31);
      const double nlo = first ? fmax(l, lo) : lo, nhi = first < 32 ? fmin(h, hi) : hi;
      if (nlo == lo && nhi == hi) break;  // neighbouring doubles
      lo = nlo;
      hi = nhi;
    }
    const double u = 0.5 * (lo + hi);
    const double rho = 1.0 / u;
    const double p = (g - 1.0) / g * rho * (H - 0.5 * u * u);
    const double ul = u + speed;
    for (int v = 0; v < 5; ++v) q[v] = 0.0;
    q[0] = rho;
    q[1 + m] = rho * ul;
    q[4] = p / (g - 1.0) + 0.5 * rho * ul * ul;
  }
  if (lane) return;
  const double rho = q[0];
  const double v0 = q[1] / rho, v1 = q[2] / rho, v2 = q[3] / rho;
  const double p = (g - 1.0) * (q[4] - 0.5 * rho * (v0 * v0 + v1 * v1 + v2 * v2));
  const double z1 = sqrt(rho / p);
  double* o = bc.out + i * kBcVals;
  o[0] = z1;
  o[1] = z1 * v0;
  o[2] = z1 * v1;
  o[3] = z1 * v2;
  o[4] = sqrt(rho * p);
  o[5] = sqrt(p / rho);
  o[6] = rho * v0 / p;
  o[7] = rho * v1 / p;
  o[8] = rho * v2 / p;
  o[9] = -rho / p;
}

}  // namespace es
