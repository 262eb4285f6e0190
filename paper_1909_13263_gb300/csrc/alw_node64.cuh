// The Hamiltonian, the node alpha and the RK combination of one node in double (1D and 2D).
#pragma once
#include "alw_device.cuh"

namespace alw {

// Largest of two non-negative doubles by their bit patterns (integer comparisons: FP64 ones run on the FP64
// pipe); a NaN counts as larger than everything, so it survives to the caller's check.
__device__ __forceinline__ double max_bits(double a, double b) {
  const unsigned long long x = double_to_bits(a), y = double_to_bits(b);
  return bits_to_double(x > y ? x : y);
}
__device__ __forceinline__ double min_bits(double a, double b) {
  const unsigned long long x = double_to_bits(a), y = double_to_bits(b);
  return bits_to_double(x < y ? x : y);
}

// H at the mean one-sided derivatives and the node alpha in double, sharing what they have in common.
// With c = (u^- + u^+ + v^- + v^+)/2 and e = (|u^+ - u^-| + |v^+ - v^-|)/2 the four corner sums u + v are
// c +- e and c +- |du - dv|/2.  `known` is a lower bound of the grid maximum the alphas are folded into:
// an alpha that cannot exceed it is returned as 0 (0 = evaluate always, for a flux that uses the node's own).
// The trigonometric kinds need sin and cos of c only: |cos(c +- d)| is at most |cos c| cos d + |sin c| sin d,
// attained by one of the two signs, with cos d and sin d by their series for small d.
__device__ __forceinline__ void ham_node64(int kind, double um, double up, double vm, double vp, double x, double y,
                                           double known, double &H, double &ax, double &ay) {
  const double su = up + um, du = up - um;
  switch (kind) {
    case H_BURGERS2D:
    case H_BURGERS1D: {
      const bool two = kind == H_BURGERS2D;
      const double c = fma(0.5, two ? su + (vp + vm) : su, 1.0);
      H = 0.5 * c * c;
      ax = fma(0.5, two ? fabs(du) + fabs(vp - vm) : fabs(du), fabs(c));
      ay = two ? ax : 0.0;
    } break;
    case H_NEGCOS2D:
    case H_NEGCOS1D:
    case H_SIN2D: {
      const bool two = kind != H_NEGCOS1D;
      const double s2 = two ? su + (vp + vm) : su;
      const double c = kind == H_SIN2D ? 0.5 * s2 : fma(0.5, s2, 1.0);
      double sn, cs;
      sincos(c, &sn, &cs);
      H = kind == H_SIN2D ? sn : -cs;
      const double a = fabs(kind == H_SIN2D ? cs : sn), b = fabs(kind == H_SIN2D ? sn : cs);
      const double dv = two ? vp - vm : 0.0;
      const double e = 0.5 * (fabs(du) + fabs(dv));
      ax = 0.0;
      if (!(fma(b, e, a) <= known)) {
        const double e2 = 0.5 * fabs(fabs(du) - fabs(dv));
        auto corner = [&](double d) {
          double sd, cd;
          if (d <= 0.015625) {
            const double q = d * d;
            cd = fma(q, fma(q, fma(q, -1.0 / 720.0, 1.0 / 24.0), -0.5), 1.0);
            sd = d * fma(q, fma(q, 1.0 / 120.0, -1.0 / 6.0), 1.0);
            return fma(a, cd, b * sd);
          }
          sincos(c + d, &sn, &cs);
          const double r1 = fabs(kind == H_SIN2D ? cs : sn);
          sincos(c - d, &sn, &cs);
          return max_bits(r1, fabs(kind == H_SIN2D ? cs : sn));
        };
        ax = corner(e);
        if (two) ax = max_bits(ax, corner(e2));
      }
      ay = two ? ax : 0.0;
    } break;
    case H_ADVECT1D: {
      H = 0.5 * su;
      ax = fabs(su) < INFINITY ? 1.0 : NAN;
      ay = 0.0;
    } break;
    case H_EIKONAL2D: {
      const double p = 0.5 * su, q = 0.5 * (vp + vm);
      H = sqrt(fma(p, p, fma(q, q, 1.0)));
      // |H_p| = |u| / sqrt(u^2 + v^2 + 1) grows with |u| and falls with |v|
      const double ul = min_bits(fabs(um), fabs(up)), uh = max_bits(fabs(um), fabs(up));
      const double vl = min_bits(fabs(vm), fabs(vp)), vh = max_bits(fabs(vm), fabs(vp));
      ax = uh * rsqrt(fma(uh, uh, fma(vl, vl, 1.0)));
      ay = vh * rsqrt(fma(vh, vh, fma(ul, ul, 1.0)));
    } break;
    default:
      H = ham_value<double>(kind, 0.5 * su, 0.5 * (vp + vm), x, y);
      node_alpha<double>(kind, um, up, vm, vp, x, y, ax, ay);
  }
}

// Step 5's combinations: stage `stage` from phi^n (base), the stage's input src and dt L.
__device__ __forceinline__ double rk_node64(int stage, double base, double src, double dt, double L) {
  if (stage == 1) return src + dt * L;
  if (stage == 2) return 0.75 * base + 0.25 * (src + dt * L);
  // (phi^n + 2 (phi_2 + dt L)) / 3, the division as a product with its remainder folded back
  const double z = fma(2.0, fma(dt, L, src), base), third = 1.0 / 3.0, q = z * third;
  return fma(fma(-3.0, q, z), third, q);
}

}  // namespace alw
