// The powers r^p and r^(p-1) of the SIMP interpolation.
//
// CUDA's pow executes about 105 FP64 operations (833 us for 4,915,200 moduli
// whose 79 MB move in 12 us).  The penalties of a continuation are multiples
// of 1/2, and for those the powers are products: r is multiplied up as an
// unevaluated sum hi + lo (the exact product error of each step by FMA), so the
// one rounding is that of the final sum, as good as pow's.  Outside
// [2^-99, 2^99) (where a product error could underflow; r = 0 apart) and for
// other p, pow itself.  Measured at p = 3, 7 FP64 operations: modulus of
// 4,915,200 elements 66 against 833 us.
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
  // r in [2^-99, 2^99), by its exponent (a comparison takes the FP64 pipe)
  if (q.k > 0 && (unsigned)__double2hiint(r) - ((1023u - 99u) << 20) < (198u << 20)) {
    double h = 1.0, l = 0.0;
    if (q.half) {                        // sqrt(r) = s + (r - s^2) / (2 s)
      const double y = rsqrt(r);
      h = r * y;
      l = fma(-h, h, r) * (0.5 * y);
    } else if (q.k > 1) {
      h = r;
    }
    int i = q.half ? 1 : 2;
    if (!q.half && q.k > 2) {            // the first product has no l
      const double t = r * r;
      l = fma(r, r, -t);
      h = t;
      i = 3;
    }
    // h + l = r^(1/2), r (k > 1), r^2 or 1; multiplied up to r^(p-1)
    for (; i < q.k; ++i) {
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
