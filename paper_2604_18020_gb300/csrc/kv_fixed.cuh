// FP64 K.v (Eq. matfree) evaluated in 64-bit fixed point, z-columns of elements
// streamed as in kv_column64.cuh.
//
// The FP64 pipe runs 2 operations per clock and SM, the integer pipes 64; the
// 153 FP64 operations per element of kv_column64.cuh are additions and products
// by a few constants, so they are done on integers.  What floating point does
// by the operation is done once per node, face and element here: a block of
// values shares one exponent, and a block meets another at the larger of the two.
//   node      3 components, each with its own exponent: |S| < 2^(57-k), exact
//   face      4 nodes of a column; a component at the exponent of its largest
//   element   2 faces; all components at one exponent, directly where theirs lie
//             close, else as fix_modes says; mode operator, modulus (its
//             mantissa as a 62-bit fraction, its exponent added to the block's)
//   sum       with the element below, then over the 4 columns of a node;
//             converted back to FP64 by its owner
// Sums and differences are exact; alignments, products by constants and the
// modulus lose a few units of the last place.  So a share of an element carries
// an error of at most one FP64 rounding (2^-53) of each component's own largest
// value in the element, and a few 2^-56 of the largest mode difference of any
// component, times E.  A block without strain shifts nothing of its neighbours
// away, however stiff it is.
//
// FP64 sums in the mode basis carry 2^-53 E times the components' largest
// values, but where their sums happen to be exact: against extended precision
// (relative 2-norm; FP64 column kernel, then this) K u of a bending field over
// graded moduli 3.3e-15, 1.1e-16, of a solved cantilever's u 5.8e-14, 5.4e-15;
// the sensitivities 1.4e-15, 1.3e-16 and 2.3e-15, 1.5e-16.  What FP64 keeps and
// this does not: where one component's exact strain (a simple shear, a rigid
// rotation) exceeds another component's by more than 2^4, the smaller force keeps
// 57 bits of the larger, not of itself.  kv_column64.cuh serves callers for whom
// that matters (mfto_set_kv_variant).
//
// Measured on a GB300, y = K v, the FP64 column kernel, then this with components of one
// size and with components far apart: 1,971, 428 and 481 us at 256 x 128 x 150, 229, 52
// and 62 at 55 x 55 x 165, 114, 31 and 34 at 120 x 60 x 30, 18.5, 9.3 and 10.3 at 24 x 12
// x 12.  1,850 and 2,020 warp instructions per 32 elements, the tiles' halos included, issued
// on 54 % of the cycles; the rest waits for the layer's barrier and for dependent
// results.  (With one exponent for all components, 393 and 47 us at the first two.)
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define FIX_HD __host__ __device__ __forceinline__
#else
#define FIX_HD inline
#endif

// A constant 0 <= c < 1 as c 2^62 = hi 2^32 + lo (lo signed).
struct FixConst {
  int32_t hi, lo;
};
FIX_HD FixConst fix_const(int64_t c62) {
  return {(int32_t)((c62 + 0x80000000ll) >> 32), (int32_t)(uint32_t)(uint64_t)c62};
}

// x c / 4 for |x| < 2^63, to the nearest within a unit (errors of products do not
// lean one way)
FIX_HD int64_t fix_mul(int64_t x, FixConst c) {
  const uint32_t xl = (uint32_t)(uint64_t)x;
  const int32_t xh = (int32_t)(x >> 32);
  const int64_t low =
      (int64_t)((uint64_t)xl * (uint32_t)c.hi + 0x80000000ull) + (int64_t)xh * c.lo;
  return (int64_t)xh * c.hi + (low >> 32);
}
FIX_HD int64_t fix_shl(int64_t x, int s) { return (int64_t)((uint64_t)x << s); }

// The element operator in units of h mu / 2: with r = lam / mu every
// coefficient is an integer multiple of 1, 1/3, r, r/3 or (r + 4)/9.
struct FixOp {
  FixConst r;        // r / 2^(sr - 2)
  FixConst r3;       // (r / 3) / 2^(s3 - 2)
  FixConst third;    // 1 / 3
  FixConst q;        // ((r + 4) / 9) / 2^(s3 - 2)
  int sr, s3;
  int k;             // input bits given up for the range of the result
  double scale;      // h mu / 16: the unit, and the 8 of the mode transforms
};

// The operator for Poisson's ratio nu and element edge h; false where it does
// not fit.  The largest sum anywhere is 8 (3 r + 2) times the largest input
// (the row sum of the element matrix in these units), so k = 0 up to r = 1.97
// (nu = 0.33), and r < 10 (nu < 0.454) keeps 55 bits of the inputs.  Negative
// nu would need signed constants.
bool fixed_op(double nu, double h, FixOp* op);   // host.cu

FIX_HD int fix_min(int a, int b) { return a < b ? a : b; }
FIX_HD int fix_max(int a, int b) { return a > b ? a : b; }

// Exponents.  A component of a node value is S 2^(e - 1079 + k), e its own biased
// exponent (1 for subnormals).  A block's modes are X 2^(t - 1079 + k); a value after the modulus is
// Z 2^(e - 2099 + k).
constexpr int kFixNan = 1 << 14;          // a component that is an infinity or a NaN
constexpr int kFixEmpty = -(1 << 20);     // no contribution
constexpr int kFixNanOut = 1 << 20;

// x >> s for any s >= 0
FIX_HD int64_t fix_sar(int64_t x, int s) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(s));   // amounts above 63 count as 64
  return r;
#else
  return x >> (s < 63 ? s : 63);
#endif
}

// Exponents of three components in 16-bit lanes (0: the component is zero): the
// first two in xy, the third in the low lane of z.
struct FixExp {
  uint32_t xy, z;
  FIX_HD int at(int c) const { return (int)(c == 0 ? xy & 0xffffu : c == 1 ? xy >> 16 : z & 0xffffu); }
};
FIX_HD uint32_t fix_max_lanes(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __vmaxu2(a, b);
#else
  const uint32_t l = 0xffffu;
  return ((a & l) > (b & l) ? a & l : b & l) | ((a >> 16) > (b >> 16) ? a & ~l : b & ~l);
#endif
}

// four face modes (a + 2b) of three components and the components' exponents
struct FixFace {
  int64_t m[3][4];
  FixExp e;
};

// ... of a block of outputs, with one exponent
struct FixOut {
  int64_t m[3][4];
  int e;
};

// the value with these bits at its own exponent: its mantissa shifted left by
// `left` (4 - k), negated by the sign.  On the integer pipes: the conversion of
// the FP64 pipe, in front of the layer's barrier, made the warps wait.
FIX_HD int64_t fix_value(uint64_t bits, int left) {
  const uint64_t one = (bits << 1) >> 53 ? 0x10000000000000ull : 0ull;   // subnormals have none
  const int64_t m = (int64_t)(((bits & 0xfffffffffffffull) | one) << left);
  const int64_t sign = (int64_t)bits >> 63;
  return (m ^ sign) - sign;
}

// (sum, difference) modes of a face from its nodes' values v[node][component]
FIX_HD void fix_face(const int64_t (&v)[4][3], FixFace& F) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t s0 = v[0][c] + v[1][c], d0 = v[1][c] - v[0][c];
    const int64_t s1 = v[2][c] + v[3][c], d1 = v[3][c] - v[2][c];
    F.m[c][0] = s0 + s1;
    F.m[c][2] = s1 - s0;
    F.m[c][1] = d0 + d1;
    F.m[c][3] = d1 - d0;
  }
}

FIX_HD int fix_clz(uint32_t x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

FIX_HD bool fix_nan(const FixExp& e) {
  return fix_max(e.at(0), fix_max(e.at(1), e.at(2))) >= kFixNan;
}

// Whether the components' exponents lie so far apart that a common one would
// cost a component bits that FP64 holds (4 - k are spare), or so low that the
// values may be subnormals, which fill fewer bits.
FIX_HD bool fix_apart(const FixExp& e, int k) {
  const int a = e.at(0), b = e.at(1), c = e.at(2), top = fix_max(a, fix_max(b, c)), m = top - 4 + k;
  return (a != 0 && a < m) || (b != 0 && b < m) || (c != 0 && c < m) || (uint32_t)(top - 1) < 63u;
}

// z stage: modes f + 4 (z difference) of the element between two faces (e: their
// larger exponents); mode 0, a translation, is left out.  Returns the modes'
// common exponent (kFixEmpty: all zero).  each: form the modes of a component at
// its own exponent, where a common translation leaves exact zeros and what
// another component holds costs nothing, and then shift it to the exponent of
// the largest mode there is: what is lost lies 2^-57 or 2^-56 below that, not
// below the largest displacement.  |X| < 2^58 then (2^57 with k = 2): the modes' worst
// sum over a node of two elements, 9.3, 15.1 and 27.1 |X| for k = 0, 1 and 2
// after the quarter of fix_operator, stays below 2^62.
FIX_HD int fix_modes(const FixFace& lo, const FixFace& up, const FixExp& e, bool each, int k,
                     int64_t (&X)[3][8]) {
  const int common = fix_max(e.at(0), fix_max(e.at(1), e.at(2)));
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int at = each ? e.at(c) : common, dl = at - lo.e.at(c), du = at - up.e.at(c);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int64_t a = fix_sar(lo.m[c][f], dl), b = fix_sar(up.m[c][f], du);
      X[c][f] = f == 0 ? 0 : a + b;
      X[c][f | 4] = b - a;
    }
  }
  if (!each) return common;
  const int head = k > 1 ? 7 : 6;         // leading sign bits left
  int t = kFixEmpty;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    uint32_t big = 0;
#pragma unroll
    for (int m = 1; m < 8; ++m) {
      const int32_t hi = (int32_t)(X[c][m] >> 32);
      big |= (uint32_t)(hi ^ (hi >> 31));
    }
    int z = fix_clz(big);
    if (big == 0) {                       // below 2^32, or no modes at all
      uint32_t low = 0;
#pragma unroll
      for (int m = 1; m < 8; ++m) low |= (uint32_t)(X[c][m] ^ (X[c][m] >> 63));
      z = low != 0 ? 32 + fix_clz(low) : 1 << 16;
    }
    t = fix_max(t, e.at(c) + head - z);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    // (zero modes may be shifted by any amount)
    const int net = e.at(c) - t, l = fix_min(fix_max(net, 0), 63), r = fix_max(-net, 0);
#pragma unroll
    for (int m = 1; m < 8; ++m) X[c][m] = fix_sar(fix_shl(X[c][m], l), r);
  }
  return t;
}

// The modulus: fraction in [1/2, 1) (0: zero) and exponent e (0x7ff: no number).
struct FixModulus {
  FixConst f;
  int64_t f62;
  int e;
  bool negative;
};
FIX_HD FixModulus fix_modulus(uint64_t bits) {
  FixModulus E;
  E.negative = (bits >> 63) != 0;
  E.e = (int)((bits >> 52) & 0x7ff);
  uint64_t m = (bits & 0xfffffffffffffull) << 9;
  if (E.e != 0) {
    m |= 1ull << 61;
  } else if (m != 0) {                    // subnormal: its leading bit to where the others have it
    const uint32_t hi = (uint32_t)(m >> 32);
    const int up = (hi != 0 ? fix_clz(hi) : 32 + fix_clz((uint32_t)m)) - 2;
    m <<= up;
    E.e = 1 - up;
  }
  E.f62 = (int64_t)m;
  E.f = fix_const(E.f62);
  return E;
}

// Whether there is any strain: the modes but for the rotations in them.  (Asked of
// the modes: kept for the operator's results it would hold all of them at once.)
FIX_HD bool fix_strained(const int64_t (&X)[3][8]) {
  int64_t any = (X[0][2] + X[1][1]) | (X[0][4] + X[2][1]) | (X[1][4] + X[2][2]);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int m = 1; m < 8; ++m)
      if (m == 1 << c || (m & (m - 1)) != 0) any |= X[c][m];
  return any != 0;
}

// Z = E Kt X / 4 in the units above
FIX_HD void fix_operator(const int64_t (&X)[3][8], const FixOp& K, const FixModulus& E,
                         int64_t (&Z)[3][8]) {
  // constant strains: divergence and shears
  const int64_t T = fix_shl(fix_mul(X[0][1] + X[1][2] + X[2][4], K.r), K.sr);
  Z[0][1] = fix_mul(T + fix_shl(X[0][1], 1), E.f);
  Z[1][2] = fix_mul(T + fix_shl(X[1][2], 1), E.f);
  Z[2][4] = fix_mul(T + fix_shl(X[2][4], 1), E.f);
  Z[0][2] = Z[1][1] = fix_mul(X[0][2] + X[1][1], E.f);
  Z[0][4] = Z[2][1] = fix_mul(X[0][4] + X[2][1], E.f);
  Z[1][4] = Z[2][2] = fix_mul(X[1][4] + X[2][2], E.f);
  // strains linear in one axis
  const int64_t Tx = fix_shl(fix_mul(X[1][3] + X[2][5], K.r3), K.s3);
  Z[1][3] = fix_mul(Tx + X[1][3], E.f);
  Z[2][5] = fix_mul(Tx + X[2][5], E.f);
  const int64_t Ty = fix_shl(fix_mul(X[0][3] + X[2][6], K.r3), K.s3);
  Z[0][3] = fix_mul(Ty + X[0][3], E.f);
  Z[2][6] = fix_mul(Ty + X[2][6], E.f);
  const int64_t Tz = fix_shl(fix_mul(X[0][5] + X[1][6], K.r3), K.s3);
  Z[0][5] = fix_mul(Tz + X[0][5], E.f);
  Z[1][6] = fix_mul(Tz + X[1][6], E.f);
  const FixConst E3 = fix_const(fix_shl(fix_mul(E.f62, K.third), 2));
  const int64_t S = X[0][6] + X[1][5] + X[2][3];
  Z[0][6] = fix_mul(X[0][6] + S, E3);
  Z[1][5] = fix_mul(X[1][5] + S, E3);
  Z[2][3] = fix_mul(X[2][3] + S, E3);
  // and bilinear ones
  const FixConst Eq = fix_const(fix_shl(fix_mul(E.f62, K.q), 2));
#pragma unroll
  for (int c = 0; c < 3; ++c) Z[c][7] = fix_shl(fix_mul(X[c][7], Eq), K.s3 - 2);
}

// Undone z stage and the sum with the element below: Ms = upper outputs of the
// element below (U) + this one's lower ones; U becomes this one's upper ones.
FIX_HD void fix_join(const int64_t (&Z)[3][8], int e, FixOut& U, FixOut& Ms) {
  const int em = fix_max(U.e, e), du = em - U.e, dz = em - e;
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const int64_t s = f == 0 ? 0 : Z[c][f], d = Z[c][f | 4];
      Ms.m[c][f] = fix_sar(U.m[c][f], du) + fix_sar(s - d, dz);
      U.m[c][f] = s + d;
    }
  Ms.e = em;
  U.e = e;
}

// Shares of a column's four edges' nodes (a + 2b) from face modes.
FIX_HD void fix_corners(const FixOut& M, int64_t (&w)[4][3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const int64_t s0 = M.m[c][0] - M.m[c][2], d0 = M.m[c][1] - M.m[c][3];
    const int64_t s1 = M.m[c][0] + M.m[c][2], d1 = M.m[c][1] + M.m[c][3];
    w[0][c] = s0 - d0;
    w[1][c] = s0 + d0;
    w[2][c] = s1 - d1;
    w[3][c] = s1 + d1;
  }
}

// A sum of squares in units of 2^64 (exact but for the squares of the low
// words): 6 terms of |x| <= 2^61 or so fit.
struct FixSquares {
  int64_t h = 0, l = 0;
  FIX_HD void add(int64_t x) {
    const int32_t lo = (int32_t)(uint32_t)(uint64_t)x, hi = (int32_t)((x - lo) >> 32);
    h += (int64_t)hi * hi;
    l += (int64_t)hi * lo;
  }
  FIX_HD int64_t sum() const { return h + ((l + (1ll << 30)) >> 31); }
};

// X . Kt X in units of 2^(64 - 2 shift) (h mu / 2) of the modes' unit squared.
// With the sums of fix_operator the 45 terms are 23 squares in five classes.
// The sums are exact, and a rigid motion leaves none of them (a rotation
// cancels in the shears), so all are shifted left by `shift` before they are
// squared, the largest to about 2^60 (half of that with k > 0, where the
// coefficients are larger): the energy keeps its precision however far the
// strains lie below the displacements.
FIX_HD int64_t fix_energy(const int64_t (&X)[3][8], const FixOp& K, int& shift) {
  // normal strains, shears, those linear in one axis (two for each), twists
  // and bilinear ones
  int64_t v[18] = {X[0][1],           X[1][2],           X[2][4],
                   X[0][2] + X[1][1], X[0][4] + X[2][1], X[1][4] + X[2][2],
                   X[1][3],           X[2][5],           X[0][3],
                   X[2][6],           X[0][5],           X[1][6],
                   X[0][6],           X[1][5],           X[2][3],
                   X[0][7],           X[1][7],           X[2][7]};
  const int top = K.k > 0 ? 5 : 4;
  shift = 0;
  for (int pass = 0;; ++pass) {
    uint32_t big = 0;
#pragma unroll
    for (int n = 0; n < 18; ++n) {
      const int32_t hi = (int32_t)(v[n] >> 32);
      big |= (uint32_t)(hi ^ (hi >> 31));
    }
    // high words all zero: the values are below 2^32 (at most three passes,
    // the last for values of a few bits)
    const int s = big != 0 ? fix_max(fix_clz(big) - top, 0) : 32 - top;
#pragma unroll
    for (int n = 0; n < 18; ++n) v[n] = fix_shl(v[n], s);
    shift += s;
    if (big != 0 || pass == 2) break;
  }
  FixSquares div, lin, own, one, third, bil;
  div.add(v[0] + v[1] + v[2]);
  lin.add(v[6] + v[7]);
  lin.add(v[8] + v[9]);
  lin.add(v[10] + v[11]);
  third.add(v[12] + v[13] + v[14]);
#pragma unroll
  for (int n = 0; n < 3; ++n) {
    own.add(v[n]);
    third.add(v[12 + n]);
    bil.add(v[15 + n]);
  }
#pragma unroll
  for (int n = 3; n < 12; ++n) one.add(v[n]);
  // the classes at most 24, 9, 12, 12 and 3 times 2^56 (a quarter with k > 0)
  return one.sum() + 2 * own.sum() + fix_shl(fix_mul(div.sum(), K.r), K.sr) +
         fix_shl(fix_mul(lin.sum(), K.r3), K.s3) +
         fix_shl(fix_mul(third.sum(), K.third), 2) +
         fix_shl(fix_mul(bil.sum(), K.q), K.s3);
}
