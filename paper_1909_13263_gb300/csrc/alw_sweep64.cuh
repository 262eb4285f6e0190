// One-direction FP64 sweep of the WENO reconstruction with its nonlinear weights formed in float pairs.
//
// GB300 runs FP64 at about 1/76 of its FP32 rate (1.67 against 127 fused multiply-adds per SM and clock), and
// the reconstruction with double-precision indicators (three square roots, three logarithms, three divided
// differences and two divisions per node and direction) needs several hundred FP64 operations per node.
// The one-sided derivatives split into the fifth-order linear scheme and a deviation,
//   phi^- = lin^- - dev^-,  lin^- = (v_2 + v_3)/2 - 3 d_2/20 + d_1/30 - d_3/20,
//   dev^- = [(6U - 2V) T_a + (7V - U) T_b] / (20 den),
// with v = Delta^+ phi / dx, s, d, T its first, second and third differences (T_a, T_b, T_c of
// alw_device.cuh's compact form), the weight products A0 = q1 q2, A1 = q0 q2, A2 = q0 q1, U = A0 - A1,
// V = A2 - A1 and den = A0 + 6 A1 + 3 A2.  The linear part, which carries the accuracy of phi, stays
// in double; the deviation is a weight error (w - d) times third differences T, and is formed in unevaluated
// float pairs (df).  Its error, measured against 128-bit arithmetic on smooth, kinked and noisy data, is at
// most 2^-46.5 |T|.  A node takes this form when |T| (in units of phi) times 2 n, n the nodes along the line (at least
// 128), is at most |phi|: the derivative's error, 2^-46.5 |T| / dx, is then at most 2^-47.5 of the slope |phi| over
// the line's length on every grid, and that of phi over a stage below 2^-55 |phi| / (n / 128).
// Next to a kink T is as large as the jump and that fails, but there the weights of the stencils that
// cross the kink nearly vanish.  The node is then expanded about its dominant candidate k,
//   phi^- = phi^{-,k} + sum over the others of w_l (phi^{-,l} - phi^{-,k}),
// with the candidate in double and the sum in pairs, if the terms of the sum meet the bound (their sizes
// times n, Jiang-Peng 2 n, at most |phi|).
// Nodes that fail both (noise, data the grid does not resolve) are computed in double, side by side or, where a
// tile holds many, segment by segment with each stencil's indicators shared by the two sides it serves.
// The error of the one-sided derivatives against extended precision, as a share of that with double-precision
// indicators (1000 lines of 40 to 1040 nodes each with sharp kinks, rounded corners or steep slopes): rms 0.68-0.79,
// largest 0.15-0.91; up to 4000 nodes rms 0.65-0.80, largest 0.61-1.4.  (With limits 2^8, 2^7 and 2^8 on every grid the
// largest were up to 4 and 14 times the double sweep's.  With 2^10, 2^9 and 2^10 they were as good up to 1040 nodes, but
// coarse grids paid: N = 320 through the kink 20.8 ms against 19.2, 16.7 with the first limits.)
//
// Arc-length indicators: with sigma = sqrt(1 + a^2) + sqrt(1 + b^2), h = b - a and t = h / sigma (= tanh of
// half the difference of asinh b and asinh a), the mean of sqrt(1 + u^2) over [a, b], (F(b) - F(a)) / (2 h)
// with F(u) = u sqrt(1 + u^2) + asinh u, is exactly
//   G = sigma/2 - B(t^2)/sigma,  B(x) = 1/(1 - x) - atanh(sqrt x)/sqrt x = sum_k x^k 2k/(2k + 1),
// a correction of the trapezoid value free of cancellation; the series is summed up to |t| <= 1/4 (eleven
// terms; the remainder is below 2^-48 of G).  Longer intervals take the equal form
//   2 G = sigma/2 + (a + b)^2/(2 sigma) + ln((sigma + h)/(sigma - h))/h  (h > 0; all terms positive).
//
// The loop over a segment's nodes is rolled and one code serves both directions: unrolled, the sweeps did not
// fit the instruction cache (2.1 stall cycles per issue waiting for instructions).
//
// Measured (GB300, RK3 steps of Example 3, against the sweep with double indicators): 2048^2 18.4 -> 1.47 ms per
// step, 400^2 1570 -> 97 us; Example 10 on 1024^2 (kinks, double sine and cosine) 8.33 -> 0.86 ms.  On smooth data
// (cosine, dx = 0.1 to 5e-4) the error of the one-sided derivatives is 0.9-1.3e-16 rms against 0.9-1.8e-16.  Noise on
// every node, where all of it ends in double: 2048^2 15.0 -> 16.6 ms (Jiang-Peng 5.0 -> 5.7), 512^2 the same.
// What bounds it: the FP64 pipe, 59-63 operations per node and stage (30 cycles of an SM; 84 % of its peak at 2048^2).
#pragma once
#include <string.h>

#include "alw_device.cuh"

namespace alw {

// ---- float pairs -----------------------------------------------------------------------
struct df {
  float h, l;  // value h + l, |l| at most a few units in the last place of h
};

// (the host forms serve checks of this arithmetic on the CPU)
#ifdef __CUDACC__
#define ALW_HD __host__ __device__ __forceinline__
#define ALW_NOINLINE static __host__ __device__ __noinline__
#else
#define ALW_HD inline
#define ALW_NOINLINE static
#endif
#ifdef __CUDA_ARCH__
#define ALW_DEV(device, host) device
#else
#define ALW_DEV(device, host) host
#endif

ALW_HD float fa_(float a, float b) { return ALW_DEV(__fadd_rn(a, b), a + b); }
ALW_HD float fm_(float a, float b) { return ALW_DEV(__fmul_rn(a, b), a * b); }
ALW_HD float ff_(float a, float b, float c) { return ALW_DEV(__fmaf_rn(a, b, c), fmaf(a, b, c)); }
ALW_HD float asf_(unsigned a) {
  float r;
  memcpy(&r, &a, sizeof r);
  return r;
}
ALW_HD unsigned asu_(float a) {
  unsigned r;
  memcpy(&r, &a, sizeof r);
  return r;
}
ALW_HD unsigned hi_(double a) {
  unsigned long long u;
  memcpy(&u, &a, sizeof u);
  return (unsigned)(u >> 32);
}
ALW_HD unsigned lo_(double a) {
  unsigned long long u;
  memcpy(&u, &a, sizeof u);
  return (unsigned)u;
}
ALW_HD double hilo_(unsigned h, unsigned l) {
  const unsigned long long u = ((unsigned long long)h << 32) | l;
  double r;
  memcpy(&r, &u, sizeof r);
  return r;
}
ALW_HD unsigned shl3_(unsigned l, unsigned h) { return ALW_DEV(__funnelshift_l(l, h, 3), (h << 3) | (l >> 29)); }
ALW_HD float rsq_(float a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
#else
  return (float)((1.0 + 1.4e-7) / sqrt((double)a));
#endif
}
ALW_HD float rcp_(float a) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
#else
  return (float)((1.0 + 1.0e-7) / (double)a);
#endif
}

ALW_HD constexpr df pair_const_(double c) { return {(float)c, (float)(c - (double)(float)c)}; }
ALW_HD df quick_(float a, float b) {  // |a| >= |b|
  const float s = fa_(a, b);
  return {s, fa_(b, -fa_(s, -a))};
}
ALW_HD df add_(df a, df b) {  // absolute error about 2^-48 (|a| + |b|)
  const float s = fa_(a.h, b.h), c = fa_(s, -a.h);
  const float e = fa_(fa_(a.h, -fa_(s, -c)), fa_(b.h, -c));
  return quick_(s, fa_(e, fa_(a.l, b.l)));
}
ALW_HD df sub_(df a, df b) { return add_(a, df{-b.h, -b.l}); }
ALW_HD df addq_(df a, df b) {  // |a.h| >= |b.h|
  const float s = fa_(a.h, b.h);
  const float e = fa_(b.h, -fa_(s, -a.h));
  return quick_(s, fa_(e, fa_(a.l, b.l)));
}
// Products are not renormalised: the low part may reach 2^-22 of the high part, and the product of two low
// parts that the next product leaves out 2^-44.  Differences, where the high parts cancel, are.
ALW_HD df mul_(df a, df b) {
  const float p = fm_(a.h, b.h);
  return {p, ff_(a.l, b.h, ff_(a.h, b.l, ff_(a.h, b.h, -p)))};
}
ALW_HD df sqr_(df a) {
  const float p = fm_(a.h, a.h);
  return {p, ff_(fa_(a.h, a.h), a.l, ff_(a.h, a.h, -p))};
}
ALW_HD df mulf_(df a, float k) {
  const float p = fm_(a.h, k);
  return {p, ff_(a.l, k, ff_(a.h, k, -p))};
}
ALW_HD df sqrt_(df a) {  // a >= 1; the approximate root rounded to float by one Newton step, the pair by another
  const float y = rsq_(a.h), y2 = fm_(0.5f, y), s0 = fm_(a.h, y);
  const float s = ff_(ff_(-s0, s0, a.h), y2, s0);
  return {s, fm_(y2, fa_(ff_(-s, s, a.h), a.l))};
}
ALW_HD df rcp_(df a) {
  const float r = rcp_(a.h);
  return {r, fm_(r, ff_(-a.l, r, ff_(-a.h, r, 1.0f)))};
}

// Double to pair and back by their bit patterns (the conversion instructions between the two widths run
// at the FP64 rate).  Pairs keep 46 bits; |x| below 2^-95 becomes zero and |x| beyond the float range (or
// not finite) NaN, which every test of a segment fails.
ALW_HD df split_(double x) {
  const unsigned h = hi_(x), l = lo_(x), ah = h & 0x7fffffffu, sg = h & 0x80000000u;
  const unsigned t = shl3_(l, ah - 0x38000000u);
  const unsigned eb = (t & 0x7f800000u) - (23u << 23);
  const float base = asf_(eb | sg), low = asf_(eb | ((l >> 6) & 0x7fffffu) | sg);
  df r = {asf_(t | sg), fa_(low, -base)};
  if (ah - 0x3a000000u >= 0x47e00000u - 0x3a000000u) {
    r.h = ah >= 0x47e00000u ? asf_(0x7fc00000u) : 0.0f;
    r.l = 0.0f;
  }
  return r;
}
ALW_HD double widen_(float f) {  // exact (subnormal floats become zero)
  const unsigned t = asu_(f);
  const bool normal = (t & 0x7f800000u) != 0;
  return hilo_(normal ? (((t & 0x7fffffffu) >> 3) + 0x38000000u) | (t & 0x80000000u) : 0u, normal ? t << 29 : 0u);
}

// ---- constants of a sweep along one direction --------------------------------------------
struct Sweep64 {
  double c0, c1, c2, c3;  // rdx / 2, rdx / 30, -3 rdx / 20, -rdx / 20 (linear part from raw differences)
  double cdev;            // 20 dev back in units of phi_x
  double rdx, dx, eps_d;  // for the double form and the dominant-candidate form
  df scale;               // second differences of phi to the units of the indicators
  df eps;                 // arc length: 4 eps / dx^2; Jiang-Peng: eps
  float t2phi;            // 2 n T in units of phi, n >= 128
};

template <int W>
inline Sweep64 make_sweep64(double dx, double eps, int n) {
  auto pair = [](double x) {
    df r;
    r.h = (float)x;
    r.l = (float)(x - (double)r.h);
    return r;
  };
  Sweep64 c;
  const double rdx = 1.0 / dx;
  c.c0 = 0.5 * rdx;
  c.c1 = rdx / 30.0;
  c.c2 = -3.0 * rdx / 20.0;
  c.c3 = -rdx / 20.0;
  c.rdx = rdx;
  c.dx = dx;
  c.eps_d = eps;
  const bool arc = W == W_ARCLEN;
  // Jiang-Peng: differences times 32, which centres the indicators (at least eps) in the float range
  c.cdev = arc ? dx / 20.0 : 0.05 / 32.0;
  c.scale = pair(arc ? rdx * rdx : 32.0 * rdx);
  c.eps = pair(arc ? 4.0 * eps * rdx * rdx : 1024.0 * eps);
  c.t2phi = (float)((n > 128 ? 2.0 * n : 256.0) * (arc ? dx * dx : dx / 32.0));
  return c;
}

ALW_HD df horner_(df x, df p, double c) {  // c + x p, |c| > |x p|
  const float ch = (float)c, cl = (float)(c - (double)(float)c);
  const float m = fm_(x.h, p.h);
  const float e = ff_(x.l, p.h, ff_(x.h, p.l, ff_(x.h, p.h, -m)));
  const float s = fa_(ch, m);
  return {s, fa_(fa_(m, -fa_(s, -ch)), fa_(e, cl))};
}

// ln y, y >= 1: exponent and mantissa, ln m = 2 atanh z with z = (m - 1)/(m + 1), |z| <= 0.1716, by its
// series (terms up to z^17; from z^9 on in float)
ALW_HD df log_(df y) {
  unsigned k = asu_(y.h) >> 23;
  if ((asu_(y.h) & 0x7fffffu) > 0x3504f3u) ++k;
  const float sc = asf_((254u - k) << 23);  // 2^(127 - k)
  const df m = {y.h * sc, y.l * sc};
  const df z = mul_(add_(m, df{-1.0f, 0.0f}), rcp_(add_(m, df{1.0f, 0.0f})));
  const df z2 = sqr_(z);
  float f = 1.0f / 17.0f;
  f = ff_(f, z2.h, 1.0f / 15.0f);
  f = ff_(f, z2.h, 1.0f / 13.0f);
  f = ff_(f, z2.h, 1.0f / 11.0f);
  f = ff_(f, z2.h, 1.0f / 9.0f);
  df p = horner_(z2, df{f, 0.0f}, 1.0 / 7.0);
  p = horner_(z2, p, 1.0 / 5.0);
  p = horner_(z2, p, 1.0 / 3.0);
  p = horner_(z2, p, 1.0);
  const df l = mul_(df{2.0f * z.h, 2.0f * z.l}, p);
  return add_(mulf_(pair_const_(0.69314718055994530942), (float)((int)k - 127)), l);
}

// 2 G of a long interval (|t| > 1/4; see the header comment)
ALW_HD df long_mean_(df a, df sa, df b, df sb) {
  if (a.h > b.h) {
    df u = a;
    a = b;
    b = u;
    u = sa;
    sa = sb;
    sb = u;
  }
  const df sg = add_(sa, sb), h = sub_(b, a), m = add_(a, b);
  // sigma - h = (sa + a) + (sb - b), each without cancellation
  const df na = {-a.h, -a.l}, nb = {-b.h, -b.l};
  const df t1 = a.h >= 0.0f ? add_(sa, a) : rcp_(add_(sa, na));
  const df t2 = b.h <= 0.0f ? add_(sb, nb) : rcp_(add_(sb, b));
  const df y = mul_(add_(sg, h), rcp_(add_(t1, t2)));
  const df half = {0.5f, 0.0f};
  return add_(mul_(half, add_(sg, mul_(sqr_(m), rcp_(sg)))), mul_(log_(y), rcp_(h)));
}

// 2 G of an interval of width h with s = sqrt(1 + u^2) at its ends; is_long: |t| > 1/4 (or NaN), not valid
ALW_HD df short_mean_(df sa, df sb, df h, bool &is_long) {
  const df sg = add_(sa, sb), r = rcp_(sg), t = mul_(h, r), x = sqr_(t);
  is_long = !(fabsf(t.h) <= 0.25f);
  // 2 B(x) / x = sum_k x^k 4 (k + 1) / (2 k + 3): k >= 5 in float, the rest in pairs
  float f = 44.0f / 23.0f;
  f = ff_(f, x.h, 40.0f / 21.0f);
  f = ff_(f, x.h, 36.0f / 19.0f);
  f = ff_(f, x.h, 32.0f / 17.0f);
  f = ff_(f, x.h, 28.0f / 15.0f);
  f = ff_(f, x.h, 24.0f / 13.0f);
  df p = horner_(x, df{f, 0.0f}, 20.0 / 11.0);
  p = horner_(x, p, 16.0 / 9.0);
  p = horner_(x, p, 12.0 / 7.0);
  p = horner_(x, p, 8.0 / 5.0);
  p = horner_(x, p, 4.0 / 3.0);
  const df c = mul_(mul_(x, p), r);
  return addq_(sg, df{-c.h, -c.l});
}

ALW_HD df root_(df u) { return sqrt_(add_(df{1.0f, 0.0f}, sqr_(u))); }  // sqrt(1 + u^2)

// The three indicators q of a stencil from its second differences D1 .. D4 and their widths w1 .. w3.  Arc
// length: S2 = root_(D2) on entry, root_(D3) on return.  Jiang-Peng: pairs (s_m, s_{m+1}) as (x, y).
template <int W>
ALW_HD void stencil_q(df D1, df D2, df D3, df D4, df w1, df w2, df w3, df &S2, const Sweep64 &c, df &q0, df &q1,
                      df &q2) {
  if (W == W_ARCLEN) {
    // intervals (D2, D2 + w1), (D2, D3), (D3 - w3, D3)
    const df S3 = root_(D3);
    bool l0, l1, l2;
    df g0 = short_mean_(S2, root_(add_(D2, w1)), w1, l0);
    df g1 = short_mean_(S2, S3, w2, l1);
    df g2 = short_mean_(root_(sub_(D3, w3)), S3, w3, l2);
    if (l0 || l1 || l2) {
      // one copy of the long form (coarse grids, kinks): a rolled loop over the intervals
#pragma unroll 1
      for (int k = 0; k < 3; ++k) {
        const df a = k < 2 ? D2 : sub_(D3, w3), b = k > 0 ? D3 : add_(D2, w1);
        const df g = long_mean_(a, k < 2 ? S2 : root_(a), b, k > 0 ? S3 : root_(b));
        if (k == 0 && l0) g0 = g;
        if (k == 1 && l1) g1 = g;
        if (k == 2 && l2) g2 = g;
      }
    }
    auto q = [&](df g) { return sqr_(add_(sqr_(g), c.eps)); };  // (eps4 + (2 G)^2)^2
    q0 = q(g0);
    q1 = q(g1);
    q2 = q(g2);
    S2 = S3;
  } else {
    auto q = [&](df dd, df e) {  // (eps + 13 d^2 + 3 e^2)^2
      return sqr_(add_(add_(mulf_(sqr_(dd), 13.0f), mulf_(sqr_(e), 3.0f)), c.eps));
    };
    q0 = q(w1, sub_(D1, mulf_(D2, 3.0f)));  // x - 3y
    q1 = q(w2, add_(D2, D3));               // x + y
    q2 = q(w3, sub_(mulf_(D3, 3.0f), D4));  // 3x - y
  }
}

// Scales a stencil's q's by the power of two that brings the largest to about one, so that their products
// stay in the float range; false when one of them (before scaling) is out of range: above 1e37 (or infinite), or
// below 1e-27, where the low parts of the pair arithmetic that formed it run out of exponents (a product's
// remainder, 2^-48 of it, must stay above 2^-149).  Arc length never goes below 16; Jiang-Peng does when eps and
// the differences are both tiny.  NaN fails the caller's tests of the denominators.
ALW_HD bool scale_q(df &q0, df &q1, df &q2) {
  const float qm = fmaxf(q0.h, fmaxf(q1.h, q2.h)), qn = fminf(q0.h, fminf(q1.h, q2.h));
  const float sc = asf_(0x7f000000u - (asu_(qm) & 0x7f800000u));
  q0 = {q0.h * sc, q0.l * sc};
  q1 = {q1.h * sc, q1.l * sc};
  q2 = {q2.h * sc, q2.l * sc};
  return qm < 1e37f && qn > 1e-27f;
}

// Both deviations of a stencil, "-" of its node and "+" of the node before (times 20); false: out of range.
ALW_HD bool stencil_devs(df q0, df q1, df q2, df T2, df T3, df &minus, df &plus) {
  const bool ok = scale_q(q0, q1, q2);
  const df U = mul_(q2, sub_(q1, q0)), V = mul_(q0, sub_(q1, q2)), A1 = mul_(q0, q2);
  const df base = add_(mulf_(A1, 10.0f), add_(U, V));
  const df U2 = {U.h + U.h, U.l + U.l}, V2 = {V.h + V.h, V.l + V.l};
  const df denA = add_(base, V2), denB = add_(base, U2);
  const df nm = add_(mul_(sub_(mulf_(U, 6.0f), V2), T2), mul_(sub_(mulf_(V, 7.0f), U), T3));
  const df np = add_(mul_(sub_(mulf_(V, 6.0f), U2), T3), mul_(sub_(mulf_(U, 7.0f), V), T2));
  minus = mul_(nm, rcp_(denA));
  plus = mul_(np, rcp_(denB));
  return ok && denA.h > 1e-30f && denB.h > 1e-30f;
}

// Magnitude of phi from the upper word of |phi|, 0 outside the float range
ALW_HD float phi_size(unsigned p) {
  return p >= 0x3a000000u && p < 0x47e00000u ? asf_((p - 0x38000000u) << 3) : 0.0f;
}

// ---- the same in double, with FP64 operations saved where they can be: roots and reciprocals refine the
// float approximation by Newton steps (7 and 4 operations), one logarithm per long interval only
ALW_HD bool narrows_(double a) { return (hi_(a) & 0x7fffffffu) - 0x3a000000u < 0x47e00000u - 0x3a000000u; }
ALW_HD float narrow_(double a) {  // towards zero, by bit patterns (the conversion instruction runs at the FP64 rate)
  return asf_(shl3_(lo_(a), (hi_(a) & 0x7fffffffu) - 0x38000000u) | (hi_(a) & 0x80000000u));
}
ALW_HD double rcp64_(double a) {
  if (!narrows_(a)) return 1.0 / a;
  const double f = widen_(rcp_(narrow_(a))), r = fma(f, fma(-a, f, 1.0), f);
  return fma(r, fma(-a, r, 1.0), r);
}
ALW_HD double sqrt64_(double a) {  // a >= 1
  if (!narrows_(a)) return sqrt(a);
  const double y = widen_(rsq_(narrow_(a)));
  double g = a * y, h = 0.5 * y;
  const double r = fma(-g, h, 0.5);
  g = fma(g, r, g);
  h = fma(h, r, h);
  return fma(h, fma(-g, g, a), g);
}
ALW_HD double log64_(double y) {  // y >= 1, as log_ (terms up to z^23)
  unsigned k = hi_(y) >> 20, m = hi_(y) & 0xfffffu;
  if (m > 0x6a09eu) ++k;
  const double x = y * hilo_((2046u - k) << 20, 0u);
  const double z = (x - 1.0) * rcp64_(x + 1.0), z2 = z * z;
  double p = 1.0 / 23.0;
  p = fma(p, z2, 1.0 / 21.0);
  p = fma(p, z2, 1.0 / 19.0);
  p = fma(p, z2, 1.0 / 17.0);
  p = fma(p, z2, 1.0 / 15.0);
  p = fma(p, z2, 1.0 / 13.0);
  p = fma(p, z2, 1.0 / 11.0);
  p = fma(p, z2, 1.0 / 9.0);
  p = fma(p, z2, 1.0 / 7.0);
  p = fma(p, z2, 1.0 / 5.0);
  p = fma(p, z2, 1.0 / 3.0);
  const double w = 2.0 * z;
  return fma((double)((int)k - 1023), 0.69314718055994530942, fma(w * z2, p, w));
}
// G: by its series (see the header comment) or, for long intervals, as (F(b) - F(a)) / (2 h) with asinh b - asinh a =
// ln((sigma + h)/(sigma - h)).  That cancels nothing that counts: (sigma - |h|)(sigma + |h|) >= 4 and |h| > sigma / 4,
// so the rounding of sigma - |h| moves G by at most 2^-51 of itself.
ALW_HD double mean64_(double a, double sa, double b, double sb) {
  const double h = b - a, sg = sa + sb, d = fabs(h);
  if (d <= 0.25 * sg) {
    const double r = rcp64_(sg), t = h * r, x = t * t;
    double p = 26.0 / 27.0;
#pragma unroll
    for (int k = 12; k >= 1; --k) p = fma(p, x, 2.0 * k / (2.0 * k + 1.0));
    return fma(-x * p, r, 0.5 * sg);
  }
  const bool up = h > 0.0;   // the same bits whichever end comes first
  const double n = fma(up ? b : a, up ? sb : sa, -((up ? a : b) * (up ? sa : sb)));
  double w = sg - d;
  if ((int)hi_(w) <= 0) w = hilo_(hi_(sg) - (53u << 20), 0u);   // rounded away (ends beyond 1e7: l does not count)
  const double i = rcp64_(w * d), l = log64_((sg + d) * (d * i));
  return 0.5 * (n + l) * (w * i);
}

// Squared indicators of a stencil in double from its second differences s (over dx).  S2 = sqrt(1 + (s2 / dx)^2) on
// entry, of s3 on return (arc length).
template <int W>
ALW_HD void stencil64_(double s1, double s2, double s3, double s4, double &S2, const Sweep64 &c, double (&q)[3]) {
  if (W == W_ARCLEN) {
    const double u1 = s1 * c.rdx, u2 = s2 * c.rdx, u3 = s3 * c.rdx, u4 = s4 * c.rdx;
    const double R = 2.0 * u2 - u1, L = 2.0 * u3 - u4, S3 = sqrt64_(fma(u3, u3, 1.0));
    q[0] = mean64_(u2, S2, R, sqrt64_(fma(R, R, 1.0)));
    q[1] = mean64_(u2, S2, u3, S3);
    q[2] = mean64_(L, sqrt64_(fma(L, L, 1.0)), u3, S3);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double b = c.dx * q[k], e = fma(b, b, c.eps_d);
      q[k] = e * e;
    }
    S2 = S3;
  } else {
    const double s[5] = {0.0, s1, s2, s3, s4};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double x = s[k + 1], y = s[k + 2], d = x - y, z = k == 0 ? x - 3.0 * y : (k == 1 ? x + y : 3.0 * x - y);
      const double e = c.eps_d + (13.0 * d * d + 3.0 * z * z);
      q[k] = e * e;
    }
  }
}

// w_0 2 T_a + w_2 T_b + d_2 of a side, so that phi^- = (v_2 + v_3)/2 - (...)/6; the "+" side is minus the mirrored
// one.  omega_0, omega_2 in product form, or by quotients when the products leave the range.
ALW_HD double side64_(double q0, double q1, double q2, double s1, double s2, double s3, double s4) {
  const double d2 = s3 - s2, Ta = (s1 + s3) - 2.0 * s2, Tb = (s2 + s4) - 2.0 * s3;
  const double n0 = 0.1 * (q1 * q2), n2 = 0.3 * (q0 * q1), den = fma(0.6, q0 * q2, n0 + n2);
  double w0, w2;
  if (den > 1e-290 && den < 1e290) {
    const double r = den > 1e-35 && den < 1e35 ? rcp64_(den) : 1.0 / den;
    w0 = n0 * r;
    w2 = n2 * r;
  } else {
    const double a0 = 0.1 / q0, a1 = 0.6 / q1, a2 = 0.3 / q2, sum = a0 + a1 + a2;
    w0 = a0 / sum;
    w2 = a2 / sum;
  }
  return fma(w0, 2.0 * Ta, fma(w2, Tb, d2));
}

ALW_HD double root64_(double s, const Sweep64 &c) { return sqrt64_(fma(s * c.rdx, s * c.rdx, 1.0)); }

// phi^- of the node at cell a + 3 step in double
template <int W>
ALW_HD double minus64_double(const double *a, int step, const Sweep64 &c) {
  double v[5], s[5], q[3];
#pragma unroll
  for (int k = 0; k < 5; ++k) v[k] = a[(k + 1) * step] - a[k * step];
#pragma unroll
  for (int k = 1; k < 5; ++k) s[k] = (v[k] - v[k - 1]) * c.rdx;   // (scaled last: the differences are nearly exact)
  double S = W == W_ARCLEN ? root64_(s[2], c) : 0.0;
  stencil64_<W>(s[1], s[2], s[3], s[4], S, c, q);
  return fma(-1.0 / 6.0, side64_(q[0], q[1], q[2], s[1], s[2], s[3], s[4]), c.c0 * (v[2] + v[3]));
}

// Both sides of the nodes `rare` of a segment in double, the bits of minus64_double's: the "-" side of node j and the
// "+" side of node j - 1 share stencil j's indicators.  (phi^-, phi^+) of node q go to o[2 q ostep], o[2 q ostep + 1].
template <int W>
ALW_NOINLINE void sweep64_double(const double *a, int step, const Sweep64 &c, unsigned rare, double *o, int ostep) {
  int j = 0, last = 0;
  while (!(rare >> j & 1u)) ++j;
  while (rare >> last) ++last;
  const double *p = a + j * step;
  double x = p[4 * step], v1 = p[2 * step] - p[step], v2 = p[3 * step] - p[2 * step], v3 = x - p[3 * step];
  double s1 = (v1 - (p[step] - p[0])) * c.rdx, s2 = (v2 - v1) * c.rdx, s3 = (v3 - v2) * c.rdx;
  double S = W == W_ARCLEN ? root64_(s2, c) : 0.0;
#pragma unroll 1
  for (; j <= last; ++j) {
    const double y = a[(j + 5) * step], v4 = y - x, s4 = (v4 - v3) * c.rdx;
    double q[3];
    stencil64_<W>(s1, s2, s3, s4, S, c, q);
    if (rare >> j & 1u)
      o[2 * j * ostep] = fma(-1.0 / 6.0, side64_(q[0], q[1], q[2], s1, s2, s3, s4), c.c0 * (v2 + v3));
    if (j > 0 && (rare >> (j - 1) & 1u))
      o[2 * (j - 1) * ostep + 1] = fma(1.0 / 6.0, side64_(q[2], q[1], q[0], s4, s3, s2, s1), c.c0 * (v1 + v2));
    x = y;
    v1 = v2;
    v2 = v3;
    v3 = v4;
    s1 = s2;
    s2 = s3;
    s3 = s4;
  }
}

// phi^- of the node at cell a + 3 step where the linear expansion does not serve: about the dominant candidate,
// or, where that fails too, in double.  (phi^+ is minus the phi^- of the mirrored cells.)  Out of line: rare.
template <int W>
ALW_NOINLINE double minus64_rare(const double *a, int step, const Sweep64 &c) {
  double v[5], s[5], d[4];
  unsigned p = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const unsigned q = hi_(a[k * step]) & 0x7fffffffu;
    p = q > p ? q : p;
    if (k < 5) v[k] = a[(k + 1) * step] - a[k * step];
  }
  df D[5], w[4];
#pragma unroll
  for (int k = 1; k < 5; ++k) {
    s[k] = v[k] - v[k - 1];
    D[k] = mul_(split_(s[k]), c.scale);
    if (k > 1) d[k - 1] = s[k] - s[k - 1];
    if (k > 1) w[k - 1] = sub_(D[k], D[k - 1]);
  }
  df S = {0.0f, 0.0f}, q0, q1, q2;
  if (W == W_ARCLEN) S = root_(D[2]);
  stencil_q<W>(D[1], D[2], D[3], D[4], w[1], w[2], w[3], S, c, q0, q1, q2);
  const bool ok = scale_q(q0, q1, q2);
  const df Ta = sub_(w[2], w[1]), Tb = sub_(w[3], w[2]);
  // phi^- = (v_2 + v_3)/2 - d_2/6 - (w0 2 T_a + w2 T_b)/6, the w_k proportional to n_k
  const df n0 = mul_(q1, q2), n1 = mulf_(mul_(q0, q2), 6.0f), n2 = mulf_(mul_(q0, q1), 3.0f);
  const df r = rcp_(add_(n0, add_(n1, n2)));
  const df Ta2 = {2.0f * Ta.h, 2.0f * Ta.l}, nTa2 = {-Ta2.h, -Ta2.l}, nTb = {-Tb.h, -Tb.l};
  df x, y;
  double k = 0.0;
  if (n1.h >= n0.h && n1.h >= n2.h) {
    x = mul_(n0, Ta2);
    y = mul_(n2, Tb);
  } else if (n0.h >= n2.h) {
    k = 2.0 * (d[2] - d[1]);
    x = mul_(n1, nTa2);
    y = mul_(n2, add_(Tb, nTa2));
  } else {
    k = d[3] - d[2];
    x = mul_(n1, nTb);
    y = mul_(n0, add_(Ta2, nTb));
  }
  if (!(ok && r.h < 1e30f && (fabsf(x.h) + fabsf(y.h)) * r.h * c.t2phi <= (W == W_ARCLEN ? 2.0f : 1.0f) * phi_size(p)))
    return minus64_double<W>(a, step, c);
  const df z = mul_(add_(x, y), r);
  const double six = 1.0 / 6.0, cz = c.cdev * (20.0 / 6.0);
  const double dev = fma(cz, widen_(z.h) + widen_(z.l), (c.rdx * six) * k);
  return fma(c.rdx, fma(-six, d[2], 0.5 * (v[2] + v[3])), -dev);
}

// Nodes 0 .. nv - 1 of a segment from the cells a, a + step, ... (a = first node - 3): emit(p, phi^-, phi^+) in
// order.  Returns the mask of the nodes that did not qualify: the caller replaces their values by minus64_rare's
// (after the loop, whose values would otherwise be live across the call).
template <int W, class Emit>
ALW_HD unsigned sweep64(const double *a, int step, const Sweep64 &c, int nv, Emit emit) {
  // window at stencil j: phi at j + 4 (newest + 1 loaded in the loop), v_{j+1..j+3}, d_{j..j+2}, second
  // difference s_{j+3} (raw) and D_{j+2}, D_{j+3} (in units), widths w_{j+1}, w_{j+2}, T_{j+2}
  double x0 = a[0], v1, v2, v3, d0 = 0.0, d1, d2, s3;
  df D1, D2, D3, w1, w2, T2, S2 = {0.0f, 0.0f};
  unsigned p0, p1, p2;  // upper words of |phi| at j + 2 .. j + 4
  {
    const double x1 = a[step], x2 = a[2 * step], x3 = a[3 * step], x4 = a[4 * step];
    const double v0 = x1 - x0;
    v1 = x2 - x1;
    v2 = x3 - x2;
    v3 = x4 - x3;
    const double s1 = v1 - v0, s2 = v2 - v1;
    s3 = v3 - v2;
    d1 = s2 - s1;
    d2 = s3 - s2;
    D1 = mul_(split_(s1), c.scale);
    D2 = mul_(split_(s2), c.scale);
    D3 = mul_(split_(s3), c.scale);
    w1 = sub_(D2, D1);
    w2 = sub_(D3, D2);
    T2 = sub_(w2, w1);
    p0 = hi_(x2) & 0x7fffffffu;
    p1 = hi_(x3) & 0x7fffffffu;
    p2 = hi_(x4) & 0x7fffffffu;
    x0 = x4;
  }
  if (W == W_ARCLEN) S2 = root_(D2);
  df minus = {0.0f, 0.0f}, Tm = {0.0f, 0.0f};
  bool okm = true;
  unsigned rare = 0;
#pragma unroll 1
  for (int j = 0; j <= nv; ++j) {
    const double x5 = a[(j + 5) * step];
    const unsigned p3 = hi_(x5) & 0x7fffffffu;
    const double v4 = x5 - x0, s4 = v4 - v3, d3 = s4 - s3;
    const df D4 = mul_(split_(s4), c.scale), w3 = sub_(D4, D3), T3 = sub_(w3, w2);
    df q0, q1, q2;
    stencil_q<W>(D1, D2, D3, D4, w1, w2, w3, S2, c, q0, q1, q2);
    df next, plus;
    const bool ok = stencil_devs(q0, q1, q2, T2, T3, next, plus);
    // the node's |T| against its |phi| (the largest of three of its cells; outside the float range: fail)
    const unsigned pb = p0 > p1 ? (p0 > p3 ? p0 : p3) : (p1 > p3 ? p1 : p3);
    if (j > 0) {
      const double am = c.c0 * (v1 + v2);
      const double lm = fma(c.c2, d1, fma(c.c1, d0, fma(c.c3, d2, am)));
      const double lp = fma(c.c2, d2, fma(c.c1, d3, fma(c.c3, d1, am)));
      const double dm = fma(-c.cdev, widen_(minus.h) + widen_(minus.l), lm);
      const double dp = fma(c.cdev, widen_(plus.h) + widen_(plus.l), lp);
      const float tm = fmaxf(fabsf(Tm.h), fmaxf(fabsf(T2.h), fabsf(T3.h)));
      if (!(ok && okm && tm * c.t2phi <= phi_size(pb))) rare |= 1u << (j - 1);
      emit(j - 1, dm, dp);
    }
    minus = next;
    okm = ok;
    // shift
    x0 = x5;
    v1 = v2;
    v2 = v3;
    v3 = v4;
    s3 = s4;
    d0 = d1;
    d1 = d2;
    d2 = d3;
    D1 = D2;
    D2 = D3;
    D3 = D4;
    w1 = w2;
    w2 = w3;
    Tm = T2;
    T2 = T3;
    p0 = p1;
    p1 = p2;
    p2 = p3;
  }
  return rare;
}

}  // namespace alw
