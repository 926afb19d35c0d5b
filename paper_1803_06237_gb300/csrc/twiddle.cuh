// exp(-2 pi i k / L) as compile-time constants, correctly rounded to double.
// No CUDA in here: the constants are also checked by a host program.
//
// The angle is reduced to [0, pi / 4] with integers and its sine and cosine
// are summed as Taylor series in pairs of doubles (Knuth's exact sum, Dekker's
// exact product).  In plain double, with the angle only reduced to [-pi, pi],
// the rounding of the angle and the cancellation in the series left up to
// 9e-16 in the constants (L = 22, 30), where complex128 operands carry 1e-16.
#pragma once

namespace vie {

// unevaluated sum of two doubles
struct TwPair {
  double h, l;
};
constexpr TwPair tw_sum(double a, double b) {
  const double s = a + b, t = s - a;
  return TwPair{s, (a - (s - t)) + (b - t)};
}
constexpr TwPair tw_product(double a, double b) {
  const double ca = 134217729.0 * a, cb = 134217729.0 * b;   // 2^27 + 1: halves of 26 bits
  const double ah = ca - (ca - a), bh = cb - (cb - b), al = a - ah, bl = b - bh;
  const double p = a * b;
  return TwPair{p, ((ah * bh - p) + ah * bl + al * bh) + al * bl};
}
constexpr TwPair tw_add(TwPair a, TwPair b) {
  const TwPair s = tw_sum(a.h, b.h);
  return tw_sum(s.h, s.l + (a.l + b.l));
}
constexpr TwPair tw_mul(TwPair a, TwPair b) {
  const TwPair p = tw_product(a.h, b.h);
  return tw_sum(p.h, p.l + (a.h * b.l + a.l * b.h));
}
constexpr TwPair tw_div(TwPair a, double n) {
  const double q = a.h / n;
  const TwPair p = tw_product(q, n);
  return tw_sum(q, ((a.h - p.h) - p.l + a.l) / n);
}

// sin or cos of (pi / 2) num / den in [0, pi / 4]
constexpr double tw_series(int num, int den, bool want_sin) {
  const TwPair half_pi{1.5707963267948966, 6.123233995736766e-17};
  const TwPair x = tw_div(tw_mul(half_pi, TwPair{(double)num, 0.0}), (double)den);
  const TwPair x2 = tw_mul(x, x), minus{-x2.h, -x2.l};
  TwPair term = want_sin ? x : TwPair{1.0, 0.0}, sum = term;
  for (int n = want_sin ? 1 : 0; n < 26; n += 2) {   // the next term is below 1e-29
    term = tw_div(tw_mul(term, minus), (double)((n + 1) * (n + 2)));
    sum = tw_add(sum, term);
  }
  return sum.h;
}

template <int L, int K>
struct TwConst {
  static constexpr int k = ((K % L) + L) % L;
  static constexpr bool below = 2 * k > L;                 // angle past pi: its mirror image, sin changes sign
  static constexpr int a = below ? L - k : k;              // angle 2 pi a / L <= pi
  static constexpr bool left = 4 * a > L;                  // past pi / 2: cos changes sign
  static constexpr int b = left ? 2 * L - 4 * a : 4 * a;   // angle (pi / 2) b / L <= pi / 2
  static constexpr bool steep = 2 * b > L;                 // past pi / 4: sin and cos change places
  static constexpr int r = steep ? L - b : b;
  static constexpr double c = left ? -tw_series(r, L, steep) : tw_series(r, L, steep);
  static constexpr double s = below ? tw_series(r, L, !steep) : -tw_series(r, L, !steep);   // of exp(-i angle)
};

}  // namespace vie
