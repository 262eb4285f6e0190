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
// in double (11 operations per node); the deviation is a weight error (w - d) times third differences T, and
// is formed in unevaluated float pairs (df, at least 44 significant bits).  A segment takes this path only
// when the deviation's error stays below a quarter of the last place of phi itself -- its largest |T| (in
// units of phi) times 2^10 is at most its largest |phi|, so that 2^-44 |w - d| |T| cfl < 2^-55 |phi| --
// and otherwise (kinks, data that the grid does not resolve) the caller runs the sweep in double.
//
// Arc-length indicators without logarithms: with sigma = sqrt(1 + a^2) + sqrt(1 + b^2), h = b - a and
// t = h / sigma (= tanh of half the difference of asinh b and asinh a), the mean of sqrt(1 + u^2) over
// [a, b], (F(b) - F(a)) / (2 h) with F(u) = u sqrt(1 + u^2) + asinh u, is exactly
//   G = sigma/2 - B(t^2)/sigma,  B(x) = 1/(1 - x) - atanh(sqrt x)/sqrt x = sum_k x^k 2k/(2k + 1),
// a correction of the trapezoid value free of cancellation.  The series is summed up to |t| <= 1/4 (eleven
// terms; the remainder is below 2^-48 of G); segments with a longer interval take the double sweep.
//
// Measured (GB300, RK3 steps of Example 3): 2048^2 18.6 -> 2.0 ms per step, 400^2 1.57 -> 0.114 ms; Example 10
// on 1024^2 (kinks, double sine and cosine) 8.4 -> 1.23 ms.  The error of the one-sided derivatives against
// 128-bit arithmetic is the double sweep's or smaller (cosine data, dx = 0.1 to 5e-4: 1.0-1.4e-16 rms against
// 0.9-1.8e-16).
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
#else
#define ALW_HD inline
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
ALW_HD df mul_(df a, df b) {
  const float p = fm_(a.h, b.h);
  return quick_(p, ff_(a.l, b.h, ff_(a.h, b.l, ff_(a.h, b.h, -p))));
}
ALW_HD df sqr_(df a) {
  const float p = fm_(a.h, a.h);
  return quick_(p, ff_(fa_(a.h, a.h), a.l, ff_(a.h, a.h, -p)));
}
ALW_HD df mulf_(df a, float k) {  // small integers k: not renormalised
  const float p = fm_(a.h, k);
  return {p, ff_(a.l, k, ff_(a.h, k, -p))};
}
ALW_HD df sqrt_(df a) {  // a >= 1; one Newton step from the approximate reciprocal root
  const float y = rsq_(a.h), s = fm_(a.h, y);
  const float r = fa_(ff_(-s, s, a.h), a.l);
  return {s, fm_(fm_(0.5f, y), r)};
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
  double cdev;            // weight deviation back in units of phi_x
  df scale;               // second differences of phi to the units of the indicators
  df eps;                 // arc length: 4 eps / dx^2; Jiang-Peng: eps
  float t2phi;            // 2^10 T in units of phi
};

template <int W>
inline Sweep64 make_sweep64(double dx, double eps) {
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
  const bool arc = W == W_ARCLEN;
  // Jiang-Peng: differences times 32, so that the products of the q's (at least eps^4) stay normal floats
  c.cdev = arc ? dx / 20.0 : 0.05 / 32.0;
  c.scale = pair(arc ? rdx * rdx : 32.0 * rdx);
  c.eps = pair(arc ? 4.0 * eps * rdx * rdx : 1024.0 * eps);
  c.t2phi = (float)(1024.0 * (arc ? dx * dx : dx / 32.0));
  return c;
}

// q = (eps4 + (2 G)^2)^2 of the interval [a, a + h] with s = sqrt(1 + u^2) at its ends; ok: |t| <= 1/4
ALW_HD df q_arc64(df sa, df sb, df h, df eps4, bool &ok) {
  const df sg = add_(sa, sb), r = rcp_(sg), t = mul_(h, r), x = sqr_(t);
  ok = ok && fabsf(t.h) <= 0.25f;
  // 2 B(x) / x = sum_k x^k 4 (k + 1) / (2 k + 3): k >= 5 in float, the rest in pairs
  float f = 44.0f / 23.0f;
  f = ff_(f, x.h, 40.0f / 21.0f);
  f = ff_(f, x.h, 36.0f / 19.0f);
  f = ff_(f, x.h, 32.0f / 17.0f);
  f = ff_(f, x.h, 28.0f / 15.0f);
  f = ff_(f, x.h, 24.0f / 13.0f);
  df p = {f, 0.0f};
  auto step = [&](double c) {
    const float ch = (float)c, cl = (float)(c - (double)(float)c);
    const float m = fm_(x.h, p.h);
    const float e = ff_(x.l, p.h, ff_(x.h, p.l, ff_(x.h, p.h, -m)));
    const float s = fa_(ch, m);
    p = df{s, fa_(fa_(m, -fa_(s, -ch)), fa_(e, cl))};
  };
  step(20.0 / 11.0);
  step(16.0 / 9.0);
  step(12.0 / 7.0);
  step(8.0 / 5.0);
  step(4.0 / 3.0);
  const df b = mul_(mul_(x, p), r);
  const df g = addq_(sg, df{-b.h, -b.l});
  return sqr_(add_(sqr_(g), eps4));
}

// Nodes i0 .. i0 + K - 1 from phi_at(m) = phi at i0 - 3 + m (m = 0 .. K + 5); emit(p, phi^-, phi^+).
// nv: nodes of the segment that count (the rest lie beyond the grid).  Returns false when the segment
// does not qualify (its emitted values are then not to be used).
template <int K, int W, class Load, class Emit>
ALW_HD bool sweep64(Load phi_at, const Sweep64 &c, int nv, Emit emit) {
  double v[K + 5], s[K + 5], d[K + 5];
  df D[K + 5], w[K + 5], T[K + 5], S[K + 6], qX[K + 6], qY[K + 6], qZ[K + 6];
  bool ok = true;
  float tmax = 0.0f;
  unsigned pmax = 0;
  double prev = phi_at(0);

  auto pos = [&](int m) {  // everything up to difference m
    const double x = phi_at(m + 1);
    if (m < nv + 5) {
      const unsigned a = hi_(x) & 0x7fffffffu;
      pmax = a > pmax ? a : pmax;
    }
    v[m] = x - prev;
    prev = x;
    if (m >= 1) {
      s[m] = v[m] - v[m - 1];
      D[m] = mul_(split_(s[m]), c.scale);
    }
    if (m >= 2) {
      d[m - 1] = s[m] - s[m - 1];
      w[m - 1] = sub_(D[m], D[m - 1]);
    }
    if (m >= 3) {
      T[m - 1] = sub_(w[m - 1], w[m - 2]);
      if (m < nv + 5) tmax = fmaxf(tmax, fabsf(T[m - 1].h));
    }
  };
  // indicators of stencil j, (X_{j+2}, Y_{j+2}, Z_{j+3}) (Jiang-Peng: (X_{j+1}, Y_{j+2}, Z_{j+3}))
  auto root = [&](df u) { return sqrt_(add_(df{1.0f, 0.0f}, sqr_(u))); };
  auto arc = [&](int j) {
    bool in = true;
    if (j == 0) S[2] = root(D[2]);
    S[j + 3] = root(D[j + 3]);
    qX[j] = q_arc64(S[j + 2], root(add_(D[j + 2], w[j + 1])), w[j + 1], c.eps, in);
    qY[j] = q_arc64(S[j + 2], S[j + 3], w[j + 2], c.eps, in);
    qZ[j] = q_arc64(root(sub_(D[j + 3], w[j + 3])), S[j + 3], w[j + 3], c.eps, in);
    ok = ok && (in || j > nv);
  };
  auto jp = [&](int j) {
    auto q = [&](df dd, df a) {  // (eps + 13 d^2 + 3 a^2)^2
      const df e = add_(add_(mulf_(sqr_(dd), 13.0f), mulf_(sqr_(a), 3.0f)), c.eps);
      return sqr_(e);
    };
    // pairs (s_m, s_{m+1}): X: x - 3y, Y: x + y, Z: 3x - y
    qX[j] = q(w[j + 1], sub_(D[j + 1], mulf_(D[j + 2], 3.0f)));
    qY[j] = q(w[j + 2], add_(D[j + 2], D[j + 3]));
    qZ[j] = q(w[j + 3], sub_(mulf_(D[j + 3], 3.0f), D[j + 4]));
  };
  // both corrections of stencil j: "-" of node j, "+" of node j - 1, 20 dev as pairs
  auto devs = [&](int j, df &minus, df &plus) {
    const df g0 = qX[j], g1 = qY[j], g2 = qZ[j];
    const df U = mul_(g2, sub_(g1, g0)), V = mul_(g0, sub_(g1, g2)), A1 = mul_(g0, g2);
    const df base = add_(mulf_(A1, 10.0f), add_(U, V));
    const df U2 = {U.h + U.h, U.l + U.l}, V2 = {V.h + V.h, V.l + V.l};
    const df dm = add_(base, V2), dp = add_(base, U2);
    // the products' range (NaN fails); den >= A0, A2 > 0
    ok = ok && ((dm.h < 1e30f && dp.h < 1e30f && dm.h > 1e-26f && dp.h > 1e-26f) || j > nv);
    const df U6 = mulf_(U, 6.0f), V6 = mulf_(V, 6.0f), U7 = mulf_(U, 7.0f), V7 = mulf_(V, 7.0f);
    const df nm = add_(mul_(sub_(U6, V2), T[j + 2]), mul_(sub_(V7, U), T[j + 3]));
    const df np = add_(mul_(sub_(V6, U2), T[j + 3]), mul_(sub_(U7, V), T[j + 2]));
    minus = mul_(nm, rcp_(dm));
    plus = mul_(np, rcp_(dp));
  };

  df minus, plus, dummy;
#pragma unroll
  for (int m = 0; m <= 4; ++m) pos(m);
  if (W == W_ARCLEN) arc(0);
  else jp(0);
  devs(0, minus, dummy);
#pragma unroll
  for (int p = 0; p < K; ++p) {
    df next;
    // stencil p + 1 reads differences up to p + 5 - (arc length: one less than the window holds)
    pos(p + 5 <= K + 4 ? p + 5 : K + 4);
    if (W == W_ARCLEN) arc(p + 1);
    else jp(p + 1);
    devs(p + 1, next, plus);
    const double a = c.c0 * (v[p + 2] + v[p + 3]);
    const double lm = fma(c.c2, d[p + 2], fma(c.c1, d[p + 1], fma(c.c3, d[p + 3], a)));
    const double lp = fma(c.c2, d[p + 3], fma(c.c1, d[p + 4], fma(c.c3, d[p + 2], a)));
    emit(p, fma(-c.cdev, widen_(minus.h) + widen_(minus.l), lm), fma(c.cdev, widen_(plus.h) + widen_(plus.l), lp));
    minus = next;
  }
  // pmax holds the upper word of the largest |phi|; below the float range (all phi tiny) no segment qualifies
  const float pm = pmax >= 0x3a000000u && pmax < 0x47e00000u ? asf_((pmax - 0x38000000u) << 3) : 0.0f;
  return ok && tmax * c.t2phi <= pm;
}

}  // namespace alw
