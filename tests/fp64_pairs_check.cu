// Host check of csrc/alw_sweep64.cuh: errors of its one-sided derivatives and of the same formulas with
// double-precision indicators, both against extended precision, on lines with sharp kinks, rounded corners and steep
// slopes (random place, strength and grid of 40 to 1040 nodes).  Prints per family and kind of weights: the largest
// and the rms error of either.
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

#include "alw_sweep64.cuh"

using namespace alw;

// F(u) = u sqrt(1 + u^2) + asinh u with double: its divided difference (a series for short intervals)
template <class T>
static T mean(T a, T b) {
  const T h = b - a, sa = std::sqrt(T(1) + a * a), sb = std::sqrt(T(1) + b * b);
  if (sizeof(T) > sizeof(double)) {
    const T sg = sa + sb, t = h / sg, x = t * t;
    if (std::fabs(t) < T(0.1)) {
      T c = 0;
      for (int k = 12; k >= 1; --k) c = c * x + T(2 * k) / T(2 * k + 1);
      return sg / 2 - c * x / sg;
    }
  } else if (std::fabs(h) <= T(5e-4) * (sa + sb)) {
    const T m = (a + b) / 2, r = T(1) / (T(1) + m * m), s = std::sqrt(T(1) + m * m), h2 = h * h, m2 = m * m;
    const T f4 = (12 * m2 - 3) * r * r * r / s, f6 = (45 - 540 * m2 + 360 * m2 * m2) * r * r * r * r * r / s;
    return s + h2 * (r / s / 24 + h2 * (f4 / 1920 + h2 * f6 / 322560));
  }
  return (b * sb + std::asinh(b) - a * sa - std::asinh(a)) / (2 * h);
}

// phi^- of the node at cell a + 3 step, all in T
template <int W, class T>
static T minus_plain(const double *a, int step, T dx, T eps) {
  T v[5], s[5], q[3];
  for (int k = 0; k < 5; ++k) v[k] = (T(a[(k + 1) * step]) - T(a[k * step])) / dx;
  for (int k = 1; k < 5; ++k) s[k] = v[k] - v[k - 1];
  for (int k = 0; k < 3; ++k) {
    T e;
    if (W == W_ARCLEN) {
      const T u[5] = {0, s[1] / dx, s[2] / dx, s[3] / dx, s[4] / dx};
      const T b = dx * (k == 0 ? mean(u[2], 2 * u[2] - u[1]) : k == 1 ? mean(u[2], u[3]) : mean(2 * u[3] - u[4], u[3]));
      e = eps + b * b;
    } else {
      const T x = s[k + 1], y = s[k + 2], z = k == 0 ? x - 3 * y : (k == 1 ? x + y : 3 * x - y);
      e = eps + (13 * (x - y) * (x - y) + 3 * z * z);
    }
    q[k] = e * e;
  }
  const T n0 = q[1] * q[2], n1 = 6 * q[0] * q[2], n2 = 3 * q[0] * q[1], den = n0 + n1 + n2;
  const T c = (7 * (v[2] + v[3]) - v[1] - v[4]) / 12, ta = (s[1] + s[3]) - 2 * s[2], tb = (s[2] + s[4]) - 2 * s[3];
  return c - n0 / den * ta / 3 - (n2 / den - T(0.5)) * tb / 6;
}

struct Sum {
  double largest[2] = {0, 0}, squares[2] = {0, 0};
  long n = 0;
};

template <int W>
static void line(const std::vector<double> &p, double dx, double eps, Sum &r) {
  typedef long double L;
  const Sweep64 c = make_sweep64<W>(dx, eps, (int)p.size() - 6);
  for (int i = 0; i + 6 < (int)p.size(); ++i) {
    double d[2] = {0, 0};
    const double *a = &p[i];
    if (sweep64<W>(a, 1, c, 1, [&](int, double m, double q) { d[0] = m, d[1] = q; })) {
      d[0] = minus64_rare<W>(a, 1, c);
      d[1] = -minus64_rare<W>(a + 6, -1, c);
    }
    const L ref[2] = {minus_plain<W, L>(a, 1, dx, eps), -minus_plain<W, L>(a + 6, -1, dx, eps)};
    const double plain[2] = {minus_plain<W, double>(a, 1, dx, eps), -minus_plain<W, double>(a + 6, -1, dx, eps)};
    for (int k = 0; k < 2; ++k) {
      const double e[2] = {(double)std::fabs(d[k] - ref[k]), (double)std::fabs(plain[k] - ref[k])};
      for (int j = 0; j < 2; ++j) {
        r.largest[j] = std::fmax(r.largest[j], e[j]);
        r.squares[j] += e[j] * e[j];
      }
    }
    r.n += 2;
  }
}

int main() {
  std::mt19937_64 gen(7);
  auto u = [&] { return (double)(gen() >> 11) * (1.0 / 9007199254740992.0); };
  const double pi = 3.14159265358979323846;
  for (int family = 0; family < 3; ++family)
    for (int w = 0; w < 2; ++w) {
      Sum r;
      for (int t = 0; t < 1000; ++t) {
        const int n = (int)(40 * std::pow(26.0, u()));
        const double x0 = u() - 0.5, s = 2 * u() + 0.05, th = 2 * pi * u(), b = std::pow(10.0, -6 * u()), dx = 2.0 / n;
        std::vector<double> p(n + 6);
        for (int i = 0; i < n + 6; ++i) {
          const double x = -1 + dx * (i - 3), y = x - x0;
          p[i] = family == 0 ? s * std::fabs(y) - std::cos(pi * x + th)
                 : family == 1 ? s * std::sqrt(y * y + b) + 0.3 * std::cos(pi * x + th)
                               : s * std::tanh(y / (3 * std::sqrt(b))) - std::cos(pi * x + th);
        }
        if (w) line<W_JP>(p, dx, 1e-6, r);
        else line<W_ARCLEN>(p, dx, 1e-6, r);
      }
      std::printf("%d %d %.6e %.6e %.6e %.6e\n", family, w, r.largest[0], r.largest[1], std::sqrt(r.squares[0] / r.n),
                  std::sqrt(r.squares[1] / r.n));
    }
}
