// The rotary frequencies theta_i = rope_base^(-2i/D), i < D/2, on the host (plain C++).
#pragma once

#include <math.h>

// An unevaluated sum hi + lo, |lo| <= ulp(hi) / 2: about 106 bits.
struct AdsDd {
  double hi, lo;
};
static inline AdsDd ads_dd_sum(double hi, double lo) {        // |hi| >= |lo|
  const double s = hi + lo;
  return AdsDd{s, lo - (s - hi)};
}

// Every call of the library forms the table anew, so it has to be cheap: base^(-2i/D) is the product of the repeated square roots
// of 1 / base that i's bits name, one multiplication per entry, in twice the precision, so that what is rounded in the end is
// good to some 2^-100 (pow: half an ulp and a little more).  D = 128 on one x86 core: 0.27 us; 64 calls of pow take 0.9.
static inline void ads_rope_theta(double base, int D, double* theta) {
  const int n = D / 2;
  if ((n & (n - 1)) != 0 || !(base > 1e-100 && base < 1e100)) {
    for (int i = 0; i < n; ++i) theta[i] = pow(base, -2.0 * (double)i / (double)D);
    return;
  }
  AdsDd t[64], root;                                           // t[i] = base^(-i/n)
  root.hi = 1.0 / base;
  root.lo = fma(-root.hi, base, 1.0) / base;
  t[0] = AdsDd{1.0, 0.0};
  theta[0] = 1.0;
  for (int step = n / 2; step > 0; step /= 2) {                // root = base^(-step/n)
    const double s = sqrt(root.hi);
    root = ads_dd_sum(s, (fma(-s, s, root.hi) + root.lo) / (2.0 * s));
    for (int i = step; i < n; i += 2 * step) {                 // the indices whose lowest bit is `step`
      const AdsDd a = t[i - step];
      const double p = a.hi * root.hi;
      t[i] = ads_dd_sum(p, fma(a.hi, root.hi, -p) + (a.hi * root.lo + a.lo * root.hi));
      theta[i] = t[i].hi;
    }
  }
}
