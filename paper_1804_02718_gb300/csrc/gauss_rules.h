// Gauss-Legendre rules of the element and pyramid integrals, on [0, 1], weights summing to 1 (plain C++).
#pragma once

#include <cmath>

namespace frlap {

// The orders, one rule after another.
constexpr int kNumQ = 6;
constexpr int rule_q(int r) { return r == 0 ? 4 : r == 1 ? 5 : r == 2 ? 8 : r == 3 ? 14 : r == 4 ? 20 : 32; }
constexpr int rule_off(int r) { return r == 0 ? 0 : rule_off(r - 1) + rule_q(r - 1); }
constexpr int kQTotal = rule_off(kNumQ);
struct GaussRules {
  double x[kQTotal], w[kQTotal];
};

// p = P_q(x) and dp = P_q'(x) (|x| < 1), by the three-term recurrence
template <typename R>
inline void legendre(int q, R x, R& p, R& dp) {
  R p0 = R(1), p1 = x;
  for (int k = 2; k <= q; ++k) {
    const R t = x * p1, p2 = t + (t - p0) * R(k - 1) / R(k);
    p0 = p1;
    p1 = p2;
  }
  p = p1;
  dp = R(q) * (x * p1 - p0) / (x * x - R(1));
}

// An error of a rule is one of every element's integral alike, so the last steps run in the type R, longer than
// double.  Where R is 128-bit software arithmetic an operation of it takes some 16 ns, so there are few: Newton's
// method (quadratic) reaches double's rounding in double, one step in R then squares that error, a second evaluation
// gives the weights, and the nodes' symmetry halves both: 9 200 operations for the six rules.
// A process's first 512^2 plan 3.7 -> 1.6 ms against twelve steps in R at every node (later ones 0.7).
template <typename R>
GaussRules make_gauss_rules() {
  GaussRules g;
  for (int r = 0; r < kNumQ; ++r) {
    const int q = rule_q(r), at = rule_off(r);
    for (int i = 0; 2 * i < q; ++i) {
      double x0 = std::cos(3.14159265358979323846 * (i + 0.75) / (q + 0.5)), p0, dp0;
      for (int it = 0; it < 5; ++it) {
        legendre(q, x0, p0, dp0);
        x0 -= p0 / dp0;
      }
      R x = R(x0), p, dp;
      legendre(q, x, p, dp);
      x = x - p / dp;
      legendre(q, x, p, dp);
      const R one = R(1), half = R(0.5);
      const int a = at + i, b = at + q - 1 - i;
      g.x[a] = (double)(half * (one - x));
      g.x[b] = (double)(half * (one + x));
      g.w[a] = g.w[b] = (double)(one / ((one - x * x) * dp * dp));  // (2 / ((1 - x^2) P'^2)) / 2
    }
  }
  return g;
}

}  // namespace frlap
