// unit_circle.cuh -- cos and sin of 2 pi p / n at compile time, to the nearest double: the constants of the
// transforms in registers.  (A Taylor series in plain doubles was off by up to 1.6 units of the last place, 0.67 in the
// mean square, and put FP64 transforms of 64 and 128 samples 8 to 12 % further off than those with sincospi.)
// Standard C++, so that a host program can check them.
#pragma once

namespace tsvd {
namespace ct {

// unevaluated sums of two doubles; TwoSum (Knuth) and TwoProduct by splitting (Dekker)
struct dd {
  double h, l;
};
constexpr dd two_sum(double a, double b) {
  const double s = a + b, bb = s - a;
  return dd{s, (a - (s - bb)) + (b - bb)};
}
constexpr dd two_prod(double a, double b) {
  const double p = a * b, s = 134217729.0;  // 2^27 + 1
  const double ca = s * a, ah = ca - (ca - a), al = a - ah;
  const double cb = s * b, bh = cb - (cb - b), bl = b - bh;
  return dd{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr dd norm(double h, double l) {
  const double s = h + l;
  return dd{s, l - (s - h)};
}
constexpr dd add(dd a, dd b) {
  const dd s = two_sum(a.h, b.h);
  return norm(s.h, s.l + (a.l + b.l));
}
constexpr dd mul(dd a, dd b) {
  const dd p = two_prod(a.h, b.h);
  return norm(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr dd div(dd a, double b) {
  const double q = a.h / b;
  const dd p = two_prod(q, b);
  return norm(q, (((a.h - p.h) - p.l) + a.l) / b);
}

// sum of (-1)^k x^(2k + odd) / (2k + odd)! for 0 <= x <= pi / 4 (twelve terms: below 2^-100)
constexpr double series(dd x, int odd) {
  const dd x2 = mul(x, x);
  dd t = odd ? x : dd{1.0, 0.0}, s = t;
  for (int k = 1; k < 13; ++k) {
    t = div(mul(dd{-t.h, -t.l}, x2), (2.0 * k + odd) * (2.0 * k + odd - 1.0));
    s = add(s, t);
  }
  return s.h;
}
// 2 pi p / n
constexpr dd angle(long p, long n) {
  const dd tau{6.283185307179586476925286766559, 2.4492935982947064e-16};
  return div(mul(tau, dd{(double)p, 0.0}), (double)n);
}
// cos and sin of 2 pi p / n (the series on the first octant; exact on the axes)
constexpr double cos2pi(long p, long n) {
  p %= n;
  if (2 * p > n) p = n - p;
  if (4 * p == n) return 0.0;
  if (4 * p > n) return -cos2pi(n - 2 * p, 2 * n);
  if (8 * p > n) return series(angle(n - 4 * p, 4 * n), 1);
  return series(angle(p, n), 0);
}
constexpr double sin2pi(long p, long n) {  // cos(theta - pi/2)
  return cos2pi(((4 * p - n) % (4 * n) + 4 * n) % (4 * n), 4 * n);
}

}  // namespace ct
}  // namespace tsvd
