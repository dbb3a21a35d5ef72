// The powers r^p and r^(p-1) of the SIMP interpolation.
//
// CUDA's pow executes about 105 FP64 operations (833 us for 4,915,200 moduli
// whose 79 MB move in 12 us).  The penalties of a continuation are multiples
// of 1/2, and for those the powers are products: r is multiplied up as an
// unevaluated sum hi + lo (the exact product error of each step by FMA), so the
// one rounding is that of the final sum, as good as pow's.  Outside
// [1e-30, 1e30] (where a product error could underflow; r = 0 apart) and for
// other p, pow itself.  Measured at p = 3: modulus of 4,915,200 elements 100
// against 833 us.
#pragma once

struct PowPlan {
  int k;      // floor(p), 0: use pow
  int half;   // p = k + 1/2
};

static inline PowPlan pow_plan(double p) {
  PowPlan q{0, 0};
  if (p >= 1.0 && p <= 8.0 && 2.0 * p == (double)(int)(2.0 * p)) {
    q.k = (int)p;
    q.half = (int)(2.0 * p) & 1;
  }
  return q;
}

// rp = r^p; rp1 = r^(p-1) if asked for
template <bool WITH_P1>
__device__ __forceinline__ void simp_powers(double r, double p, PowPlan q, double& rp,
                                            double& rp1) {
  if (q.k > 0 && r >= 1e-30 && r <= 1e30) {
    double h = 1.0, l = 0.0;
    if (q.half) {                        // sqrt(r) = s + (r - s^2) / (2 s)
      const double y = rsqrt(r);
      h = r * y;
      l = fma(-h, h, r) * (0.5 * y);
    } else if (q.k > 1) {
      h = r;
    }
    // h + l = r^(1/2), r (k > 1) or 1; multiplied up to r^(p-1)
    for (int i = q.half ? 1 : 2; i < q.k; ++i) {
      const double t = h * r;
      l = fma(l, r, fma(h, r, -t));
      h = t;
    }
    if (WITH_P1) rp1 = h + l;
    const double t = h * r;
    rp = t + fma(l, r, fma(h, r, -t));
  } else if (q.k > 0 && r == 0.0) {
    rp = 0.0;
    if (WITH_P1) rp1 = (q.k == 1 && !q.half) ? 1.0 : 0.0;
  } else {
    rp = pow(r, p);
    if (WITH_P1) rp1 = pow(r, p - 1.0);
  }
}
