// Compliance and sensitivities, the OC bisection update and one SIMP
// iteration (Sec. 3.1, Sec. 3.6 warm start).
#include <math.h>

#include "common.cuh"
#include "kv_column64.cuh"
#include "kv_column_fixed.cuh"
#include "simp_power.cuh"

namespace {

// u_e^T KE u_e of the element with modes X: KE = T^T Kt T / 8 (modes.cuh), so
// the energy is X . (Kt / 8) X.  By symmetry the 24 off-diagonal terms are 12
// products, and the 21 diagonal terms have 5 coefficients (the same for every
// component, by which of its axes a mode differences: its own, one other, its
// own and one other, both others, all three): 42 FP64 operations.
__device__ __forceinline__ double mode_energy(const double (&X)[3][8],
                                              const ModeCoef<double>& K) {
  double sq[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int m = 1; m < 8; ++m) {
      const int own = (m >> c) & 1;
      const int others = ((m & 1) + ((m >> 1) & 1) + ((m >> 2) & 1)) - own;
      const int cls = own ? (others == 0 ? 0 : (others == 1 ? 2 : 4)) : (others == 1 ? 1 : 3);
      sq[cls] = fma(X[c][m], X[c][m], sq[cls]);
    }
  double lam[2] = {0.0, 0.0}, mu[2] = {0.0, 0.0};
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a + 1; b < 3; ++b) {
      const int t = 3 - a - b;
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        const int tb = mt << t;
        lam[mt] = fma(X[a][(1 << a) | tb], X[b][(1 << b) | tb], lam[mt]);
        mu[mt] = fma(X[a][(1 << b) | tb], X[b][(1 << a) | tb], mu[mt]);
      }
    }
  double off = K.lamM[0] * lam[0];
  off = fma(K.lamM[1], lam[1], off);
  off = fma(K.muM[0], mu[0], off);
  off = fma(K.muM[1], mu[1], off);
  double ce = 2.0 * off;
  ce = fma(K.diag[0][1], sq[0], ce);
  ce = fma(K.diag[0][2], sq[1], ce);
  ce = fma(K.diag[0][3], sq[2], ce);
  ce = fma(K.diag[0][6], sq[3], ce);
  return fma(K.diag[0][7], sq[4], ce);
}

// What follows from an element's energy: its share of the compliance and of the
// grayness sum, and its sensitivity.
struct ElementEnergy {
  double E0, Emin, penal;
  const PowPlan& plan;
  double* dc;
  int e0, nexy;
  double (&acc)[2];
  __device__ __forceinline__ void operator()(double r, double ce, int ez) const {
    double rp, rp1;
    simp_powers<true>(r, penal, plan, rp, rp1);
    acc[0] = fma(fma(E0 - Emin, rp, Emin), ce, acc[0]);
    acc[1] += fma(-r, r, r);
    if (dc) dc[e0 + nexy * ez] = -penal * (E0 - Emin) * rp1 * ce;
  }
};

// ce_e = u_e^T KE u_e;  c = sum_e E_e ce_e;  dc_e = -p rho^(p-1) (E0-Emin) ce_e;
// grayness sum 4 rho (1 - rho).  Fixed-order sums.
//
// Bound by the FP64 pipe.  A tile of CX x CY element columns streams along z
// (Col64Stream): face modes are formed once per node layer and column and its
// edges once per row, 39 operations per element instead of 72, the energy 42
// instead of 72, the powers of rho 8 at p = 3 instead of two calls of pow (see
// simp_power.cuh): about 100 against 400 FP64 operations per element.
// Measured on a GB300: 945 against 3,125 us at 256 x 128 x 150, 55 against
// 157 us at 120 x 60 x 30 (p = 3; the operations take 780 and 34 us).
template <int CX, int CY>
__global__ void __launch_bounds__(CX * CY, kCol64Threads / (CX * CY))
compliance_kernel(const double* __restrict__ rho, const double* __restrict__ u,
                  double* __restrict__ dc, ModeCoef<double> K, Grid g, Col64Tiling tl, double E0,
                  double Emin, double penal, PowPlan plan, MiscScalars* s, double* partials) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sh[64];
  using S = Col64Shape<CX, CY>;
  const Col64LoadPlain ld{u};
  double acc[2] = {0.0, 0.0};
  for (int tile = blockIdx.x; tile < tl.count(); tile += gridDim.x) {
    const int bx = tile % tl.tx, by = (tile / tl.tx) % tl.ty, bz = tile / (tl.tx * tl.ty);
    const int kb = bz * tl.nzc, ke = min(kb + tl.nzc, g.nelz);   // element layers [kb, ke)
    Col64Stream<CX, CY, Col64LoadPlain> st(reinterpret_cast<double*>(smem_raw), ld, nullptr, g,
                                           bx * CX, by * CY, ke);
    const bool in = st.gi < g.nelx && st.gj < g.nely;
    const bool warp_in = __any_sync(0xffffffffu, in);
    const int e0 = st.gi + g.nelx * st.gj, nexy = g.nelx * g.nely;
    double own[3];
    st.issue(kb);
    st.issue(kb + 1);
    col64_wait<1>();
    st.stage(kb, 0u, own);
    st.issue(kb + 2);
    __syncthreads();
    Col64Face F0, F1;
    st.face(kb, F0);
    const ElementEnergy element{E0, Emin, penal, plan, dc, e0, nexy, acc};
    auto layer = [&](int ez, const Col64Face& lo, Col64Face& up) {
      double r = 0.0;
      if (in) r = rho[e0 + nexy * ez];
      col64_wait<1>();
      st.stage(ez + 1, 0u, own);
      st.issue(ez + 3);
      __syncthreads();
      if (!warp_in) return;
      st.face(ez + 1, up);
      double X[3][8];
      col64_modes(lo, up, X);
      const double ce = mode_energy(X, K);
      if (in) element(r, ce, ez);
    };
    for (int ez = kb; ez < ke; ez += 2) {
      layer(ez, F0, F1);
      if (ez + 1 < ke) layer(ez + 1, F1, F0);
    }
    col64_wait<0>();
    __syncthreads();   // the next tile's stages write what this one's faces read
  }
  double tot[2];
  if (last_block_reduce<2>(acc, partials, &s->ticket, tot, sh) && threadIdx.x == 0) {
    s->sum[0] = tot[0];
    s->sum[1] = 4.0 * tot[1];
  }
}

// The same on the fixed-point node stream (kv_column_fixed.cuh): the transforms
// and the energy's squares on the integer pipes, about 12 FP64 operations per
// element left (one conversion, powers and sums).  Measured on a GB300, p = 3,
// a displacement whose components lie far apart, against the kernel above, which
// serves the other Poisson's ratios and variant 2: 337 against 930 us at 256 x 128 x 150,
// 76 against 140 at 55 x 55 x 165, 43 against 67 at 120 x 60 x 30 (the call, with its host
// round trip of about 25 us).
template <int CX, int CY>
__global__ void __launch_bounds__(CX * CY, kCol64Threads / (CX * CY))
compliance_fixed_kernel(const double* __restrict__ rho, const double* __restrict__ u,
                        double* __restrict__ dc, FixOp K, Grid g, Col64Tiling tl, double E0,
                        double Emin, double penal, PowPlan plan, MiscScalars* s,
                        double* partials) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double sh[64];
  using St = FixStream<CX, CY, Col64LoadPlain, false>;
  const Col64LoadPlain ld{u};
  double* words = reinterpret_cast<double*>(smem_raw);
  double acc[2] = {0.0, 0.0};
  for (int tile = blockIdx.x; tile < tl.count(); tile += gridDim.x) {
    const int bx = tile % tl.tx, by = (tile / tl.tx) % tl.ty, bz = tile / (tl.tx * tl.ty);
    const int kb = bz * tl.nzc, ke = min(kb + tl.nzc, g.nelz);   // element layers [kb, ke)
    St st(words, reinterpret_cast<uint2*>(words + St::kWords), ld, nullptr, g, bx * CX, by * CY, ke,
          K.k);
    const int gi = bx * CX + threadIdx.x % CX, gj = by * CY + threadIdx.x / CX;
    const bool in = gi < g.nelx && gj < g.nely;
    const bool warp_in = __any_sync(0xffffffffu, in);
    const int e0 = gi + g.nelx * gj, nexy = g.nelx * g.nely;
    const ElementEnergy element{E0, Emin, penal, plan, dc, e0, nexy, acc};
    st.issue(kb);
    st.issue(kb + 1);
    col64_wait<1>();
    st.stage(kb, 0u);
    st.issue(kb + 2);
    double r_next = in ? rho[e0 + nexy * kb] : 0.0;
    __syncthreads();
    FixFace F0, F1;
    st.face(kb, F0);
    auto layer = [&](int ez, const FixFace& lo, FixFace& up) {
      const double r = r_next;
      if (in && ez + 1 < ke) r_next = rho[e0 + nexy * (ez + 1)];
      col64_wait<1>();
      st.stage(ez + 1, 0u);
      st.issue(ez + 3);
      __syncthreads();
      if (!warp_in) return;
      st.face(ez + 1, up);
      int64_t X[3][8];
      const FixExp both{fix_max_lanes(lo.e.xy, up.e.xy), fix_max_lanes(lo.e.z, up.e.z)};
      const int t = fix_modes(lo, up, both, __any_sync(0xffffffffu, fix_apart(both, K.k)), K.k, X);
      int shift;
      const double e = __ll2double_rn(fix_energy(X, K, shift));
      const double ce = fix_nan(both) ? __longlong_as_double(0x7ff8000000000000ll)
                                     : fix_scaled(e, 2 * (t - 1079 + K.k - shift) + 64, K);
      if (in) element(r, ce, ez);
    };
    for (int ez = kb; ez < ke; ez += 2) {
      layer(ez, F0, F1);
      if (ez + 1 < ke) layer(ez + 1, F1, F0);
    }
    col64_wait<0>();
    __syncthreads();
  }
  double tot[2];
  if (last_block_reduce<2>(acc, partials, &s->ticket, tot, sh) && threadIdx.x == 0) {
    s->sum[0] = tot[0];
    s->sum[1] = 4.0 * tot[1];
  }
}

template <typename S>
constexpr size_t energy_smem() {
  using St = FixStream<S::CX, S::CY, Col64LoadPlain, false>;
  return 8 * (size_t)(St::kWords + St::kExp);
}

// OC with bisection on lambda.  The candidate of a midpoint lambda is, per
// element, a_e s clipped to its move limits [lo_e, hi_e], with s = 1/sqrt(lambda)
// and a_e = rho_e sqrt(max(0, -dc_e) n) (the same value as rho_e sqrt(max(0,
// -dc_e) / (lambda / n)) up to rounding).  Its volume is a nondecreasing,
// piecewise linear function of s, which leaves little of the bisection's 60
// to 80 volume evaluations to be done:
//   1. a safeguarded Newton iteration in FP32 finds s* (where the volume is
//      the target) to about 1e-7, on FP32 copies of a and rho;
//   2. one FP64 pass classifies every element for all s within 1.5e-5 of that:
//      clipped (its bound goes into a constant C), linear (its a into a slope
//      A), or undecided (its breakpoint lies near; a few in 100,000);
//   3. every CTA then holds volume(s) = C + A s + sum over the undecided for
//      that window of s, in the same order of sums.  It confirms that the
//      volume crosses the target within the window, narrows the window by
//      Newton steps, and replays the bisection from [0, 1e9]: midpoints outside
//      the window are decided by monotonicity, those inside by evaluation.
// The replay takes the branches that the step by step bisection takes, but where
// a volume differs from the target by no more than the roundings of its sum, so
// its lambda and its last midpoint are the same to the bracket's 1e-10.  A target
// below the sum of the lower bounds, or above all that can be reached, decides
// every midpoint at once.  Where the crossing is not confirmed (a volume that is
// flat there, values beyond FP32's range, more undecided elements than the lists
// hold) the bisection evaluates every midpoint over all elements, after up to 24
// passes in FP32.
//
// One cooperative grid; a grid barrier counts arrivals (release-add of one per
// CTA, acquire-polls; bounded), and every CTA adds the per-CTA partials in the
// same order, so that all take the same branches.  Bound by the FP64 pipe in
// the first pass (a_e: 8 operations) and by about ten grid barriers of
// 2 to 3 us.  Measured on a GB300: 37 against 265 us at
// 216,000 elements (a bisection of about 37 full evaluations), 250 against
// 1,917 us at 4,915,200 (325 with the library's square root and FP64 comparisons).
constexpr int kOcThreads = 512;
constexpr int kOcSeg = 64;        // undecided elements a CTA may list
constexpr int kOcMine = 4;        // ... and a thread
constexpr int kOcList = 1024;     // ... and the grid
constexpr float kOcMargin = 3e-5f;
constexpr double kOcWindow = 1.5e-5;

struct OcElem {                   // an undecided element
  double a, lo, hi;
};

struct OcUp {                     // the bisection whose every midpoint exceeds the target
  double l1, l2, last;
  int step;
};

// The FP64 pipe bounds the passes over the elements, and comparisons, minima
// and conversions take it too: these go by the bits where the operands allow.

// a = r sqrt(max(0, -dc) n), neg_n = -n.  The square root by Goldschmidt's
// iteration with a final residual (P. Markstein, "Software division and square
// root using Goldschmidt's algorithms", 2004) from the hardware's
// approximation: 6 FP64 operations, the result within 0.51 ulp; sqrt where the
// argument lies near the ends of the exponent range.
__device__ __forceinline__ double oc_scale(double r, double dc, double neg_n) {
  const double x = dc * neg_n;
  const unsigned hi = (unsigned)__double2hiint(x);
  if (hi - 0x20000000u >= 0x40000000u) {
    // not positive (or NaN, as fmax(0, NaN) = 0)
    if (__double_as_longlong(x) <= 0 || hi >= 0x7ff80000u) return r * 0.0;
    return r * sqrt(x);
  }
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  double g = x * y;
  double h = __hiloint2double(__double2hiint(y) - 0x00100000, __double2loint(y));   // y / 2
  const double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  g = fma(fma(-g, g, x), h, g);
  return r * g;
}

// (float)x for x >= 0 in FP32's normal range (ties away from zero); the
// conversion elsewhere
__device__ __forceinline__ float oc_f32(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  if (hi - (897u << 20) >= (253u << 20)) return (hi | lo) == 0u ? 0.f : (float)x;
  return __uint_as_float(((hi - (896u << 20)) << 3 | lo >> 29) + (lo >> 28 & 1u));
}

// max(0, r - move) and min(1, r + move) (r no NaN)
__device__ __forceinline__ double oc_low(double r, double move) {
  const double v = r - move;
  return __double2hiint(v) < 0 ? 0.0 : v;
}
__device__ __forceinline__ double oc_high(double r, double move) {
  const double v = r + move;
  return __double_as_longlong(v) > 0x3ff0000000000000ll ? 1.0 : v;
}

template <int G>
__global__ void __launch_bounds__(kOcThreads, G > 0 ? 1 : 2)
oc_kernel(const double* __restrict__ rho, const double* __restrict__ dc,
          double* __restrict__ rho_new, double* __restrict__ a_s, float2* __restrict__ f_s, int n,
          double volfrac, double move, MiscScalars* s, double* partials, OcElem* list, int* counts,
          int k_end, OcUp up) {
  __shared__ double sh[64];
  __shared__ double s_tot[3];
  __shared__ float s_f[3];
  __shared__ int s_cnt, s_warp[32];
  __shared__ OcElem s_list[kOcList];
  const double target = volfrac * (double)n;
  const int first = blockIdx.x * blockDim.x + threadIdx.x;
  const int stride = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float movef = (float)move;
  const double neg_n = -(double)n;
  // per element a (FP64) and (a, rho) in FP32: in registers (G > 0: up to G
  // elements per thread) or in scratch arrays (G == 0, larger meshes)
  double ra[G > 0 ? G : 1];
  float2 rf[G > 0 ? G : 1];
  auto each = [&](auto&& f) {     // f(element, a, (a, rho) in FP32)
    if constexpr (G > 0) {
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (first + g * stride < n) f(first + g * stride, ra[g], rf[g]);
    } else {
      for (int e = first; e < n; e += stride) f(e, a_s[e], f_s[e]);
    }
  };
  auto each32 = [&](auto&& f) {   // f((a, rho) in FP32)
    if constexpr (G > 0) {
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (first + g * stride < n) f(rf[g]);
    } else {
      for (int e = first; e < n; e += stride) f(f_s[e]);
    }
  };
  unsigned int arrivals = 0;      // grid-barrier arrivals expected so far
  auto grid_sync = [&]() {
    arrivals += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) {
      red_release_add(&s->bar_count, 1u);
      volatile int32_t* verr = &s->error;
      unsigned int spins = 0;
      while (ld_acquire(&s->bar_count) < arrivals) {
        if (*verr) break;
        if (++spins > MFTO_SPIN_LIMIT) { atomicExch(&s->error, 1); break; }
      }
    }
    __syncthreads();
  };
  auto failed = [&]() { return *(volatile int32_t*)&s->error != 0; };
  // grid totals of three block sums (valid in thread 0), identical in every
  // thread: s_tot, and s_f in FP32 (s_f[0] less the target); partials
  // double-buffered by parity, one grid barrier
  int evals = 0;
  auto totals = [&](double b0, double b1, double b2) {
    double* buf = partials + (evals & 1) * 3 * MFTO_RED_SLOTS;
    ++evals;
    if (threadIdx.x == 0) {
      buf[blockIdx.x] = b0;
      buf[MFTO_RED_SLOTS + blockIdx.x] = b1;
      buf[2 * MFTO_RED_SLOTS + blockIdx.x] = b2;
    }
    grid_sync();
    if (warp < 3) {
      double t = 0.0;
      for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(&buf[warp * MFTO_RED_SLOTS + b]);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
      if (lane == 0) {
        s_tot[warp] = t;
        s_f[warp] = (float)(warp == 0 ? t - target : t);
      }
    }
    __syncthreads();
  };
  // block sums of FP32 thread sums: warps in FP32, then one conversion each
  auto block_f32 = [&](float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return block_sum_w0(lane == 0 ? (double)v : 0.0, sh);
  };

  // ---- a_e; sums of the lower bounds, of what each element can reach and of a
  float sum_lo = 0.f, sum_hi = 0.f, sum_a = 0.f;
  auto init = [&](int e, double& a, float2& f) {
    const double r = rho[e];
    a = oc_scale(r, dc[e], neg_n);
    f = make_float2(oc_f32(a), oc_f32(r));
    const float lo = fmaxf(0.f, f.y - movef);
    sum_lo += lo;
    // (a by its bits: its copy may be 0; a candidate that is no number counts as
    // the upper bound)
    sum_hi += __double_as_longlong(a) > 0 || f.x != f.x ? fmaxf(lo, fminf(1.f, f.y + movef)) : lo;
    sum_a += f.x;
  };
  if constexpr (G > 0) {
#pragma unroll
    for (int g = 0; g < G; ++g) {
      ra[g] = 0.0;
      rf[g] = make_float2(0.f, 0.f);
      if (first + g * stride < n) init(first + g * stride, ra[g], rf[g]);
    }
  } else {
    for (int e = first; e < n; e += stride) {
      double a;
      float2 f;
      init(e, a, f);
      a_s[e] = a;
      f_s[e] = f;
    }
  }
  {
    const double b0 = block_f32(sum_lo), b1 = block_f32(sum_hi);
    totals(b0, b1, block_f32(sum_a));
  }
  // the volume exceeds the target at every midpoint, or at none: the FP32 sums are off
  // by a rounding per element that a thread adds up, and by the roundings of rho
  // and move in each bound
  const double tol = 1e-5 + 6e-8 * (double)((n + stride - 1) / stride), off = 2.4e-7 * move * n;
  const bool always = s_tot[0] * (1.0 - tol) - off > target && move >= 0.0;
  const bool never = s_tot[1] * (1.0 + tol) + off < target && move >= 0.0;

  // ---- 1. Newton in FP32, kept between the scales known to give too little
  // (slo) and too much volume (shi); uniform over the grid
  float sf = (float)target / s_f[2], slo = 0.f, shi = INFINITY;
  bool found = false;
  if (!always && !never && s_f[2] < INFINITY && sf > 1e-30f && sf < 1e30f) {
    for (int it = 0; it < 24 && !failed(); ++it) {
      float vol = 0.f, slope = 0.f;
      each32([&](float2 f) {
        const float t = f.x * sf;
        const float lo = fmaxf(0.f, f.y - movef), hi = fminf(1.f, f.y + movef);
        vol += fmaxf(lo, fminf(hi, t));
        if (t > lo && t < hi) slope += f.x;
      });
      const double bv = block_f32(vol);
      totals(bv, block_f32(slope), 0.0);
      const float miss = s_f[0], A = s_f[1];
      if (miss > 0.f) shi = sf; else slo = sf;
      if (A > 0.f && fabsf(miss) <= 2e-6f * A * sf) { found = true; break; }
      float next = A > 0.f ? sf - miss / A : -1.f;
      if (!(next > slo && next < shi))    // outside what is known: halve in the logarithm
        next = shi == INFINITY ? 4.f * sf : (slo > 0.f ? sqrtf(slo) * sqrtf(shi) : 0.25f * sf);
      if (!(next > 1e-30f && next < 1e30f)) break;
      sf = next;
    }
  }

  // the bisection's state: bracket, last midpoint, its volume, steps
  double l1 = 0.0, l2 = 1e9, total = 0.0, last = -1.0;
  int step = 0;
  bool done = false;
  // the candidate volume at lambda over all elements
  auto eval_total = [&](double lam) {
    if (threadIdx.x == 0) sh[40] = 1.0 / sqrt(lam);
    __syncthreads();
    const double sc = sh[40];
    double acc = 0.0;
    each([&](int e, double a, float2) {
      const double r = rho[e];
      acc += fmax(fmax(0.0, r - move), fmin(fmin(1.0, r + move), a * sc));
    });
    __syncthreads();
    totals(block_sum(acc, sh), 0.0, 0.0);
    return s_tot[0];
  };
  // lambda_k = 1e9 halved k times (0 <= k <= k_end; exact for k <= 1083)
  auto lam_of = [](int k) {
    if (k <= 1083) return ldexp(1e9, -k);
    double x = ldexp(1e9, -1083);
    for (int i = 1083; i < k; ++i) x = 0.5 * x;
    return x;
  };

  if (always) {
    l1 = up.l1;
    l2 = up.l2;
    last = up.last;
    step = up.step;
    total = eval_total(last);
    done = true;
  } else if (never && k_end > 1) {
    // only the upper end ever moves, down to the last midpoint above 0
    l2 = lam_of(k_end - 1);
    last = l2;
    step = k_end - 1;
    total = eval_total(last);
    done = true;
  }

  if (found) {
    // ---- 2. classification for s in sf (1 -+ kOcWindow)
    double cacc = 0.0, aacc = 0.0;
    int mine = 0;
    OcElem und[kOcMine];
    each([&](int e, double a, float2 f) {
      // bounds that the FP64 ones are sure to lie between: rho, move and their sum
      // are rounded to FP32, which of a small lower bound leaves few bits
      const float off = 1.2e-7f * (fabsf(f.y) + movef), d = f.y - movef, u = f.y + movef;
      const float lo0 = fmaxf(0.f, d - off), lo1 = d > -off ? fmaxf(0.f, d) + off : 0.f;
      const float hi0 = u > 1.f + off ? 1.f : u - off, hi1 = fminf(1.f, u + off);
      // ... and candidates (a below FP32's normal range is 0 here)
      const float t0 = f.x * sf * (1.f - kOcMargin), t1 = (f.x + 1.2e-38f) * sf * (1.f + kOcMargin);
      if (t1 < lo0 || __double_as_longlong(a) == 0 || lo0 > hi1) {
        cacc += oc_low(rho[e], move);
      } else if (t0 > hi1 && hi0 > lo1) {
        cacc += oc_high(rho[e], move);
      } else if (t0 > lo1 && t1 < hi0 && t0 > 1e-30f) {
        aacc += a;
      } else {
        const double r = rho[e];
        const OcElem u{a, fmax(0.0, r - move), fmin(1.0, r + move)};
#pragma unroll
        for (int i = 0; i < kOcMine; ++i)
          if (i == mine) und[i] = u;
        ++mine;
      }
    });
    // the CTA's undecided elements, in thread order, into its list segment
    int before = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += v;
    }
    if (lane == 31) s_warp[warp] = before;
    before -= mine;
    int over = __syncthreads_or(mine > kOcMine);
    if (threadIdx.x == 0) {
      int t = 0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
        const int c = s_warp[w];
        s_warp[w] = t;
        t += c;
      }
      s_cnt = t;
    }
    __syncthreads();
    before += s_warp[warp];
    if (s_cnt > kOcSeg) over = 1;
    if (!over) {
#pragma unroll
      for (int i = 0; i < kOcMine; ++i)
        if (i < mine) list[(size_t)blockIdx.x * kOcSeg + before + i] = und[i];
    }
    if (threadIdx.x == 0) counts[blockIdx.x] = over ? -1 : s_cnt;
    const double bc = block_sum(cacc, sh);
    totals(bc, block_sum(aacc, sh), 0.0);
    const double C = s_tot[0], A = s_tot[1];
    // every CTA's undecided elements, in CTA order, into shared memory
    int have = 0, from = 0;
    if (threadIdx.x < gridDim.x) have = __ldcg(&counts[threadIdx.x]);
    over = __syncthreads_or(have < 0 || gridDim.x > blockDim.x);
    int upto = have;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, upto, o);
      if (lane >= o) upto += v;
    }
    if (lane == 31) s_warp[warp] = upto;
    __syncthreads();
    for (int w = 0; w < warp; ++w) from += s_warp[w];
    from += upto - have;
    over = __syncthreads_or(from + have > kOcList) || over;
    if (!over) {
      for (int i = 0; i < have; ++i) {
        const double* p = &list[(size_t)threadIdx.x * kOcSeg + i].a;
        s_list[from + i] = OcElem{__ldcg(p), __ldcg(p + 1), __ldcg(p + 2)};
      }
      if (threadIdx.x == blockDim.x - 1) s_cnt = from + have;
    }
    __syncthreads();

    // ---- 3. the window, by warp 0 of every CTA alike
    if (!over && warp == 0) {
      const int nu = s_cnt;
      double und_a = 0.0;   // slope of the undecided at the last evaluation
      auto volume = [&](double sc) {
        double v = 0.0, sl = 0.0;
        for (int i = lane; i < nu; i += 32) {
          const OcElem u = s_list[i];
          const double t = u.a * sc;
          v += fmax(u.lo, fmin(u.hi, t));
          if (t > u.lo && t < u.hi) sl += u.a;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          v += __shfl_xor_sync(0xffffffffu, v, o);
          sl += __shfl_xor_sync(0xffffffffu, sl, o);
        }
        und_a = sl;
        return fma(A, sc, C) + v;
      };
      double wl = (double)sf * (1.0 - kOcWindow), wh = (double)sf * (1.0 + kOcWindow);
      if (volume(wl) <= target && volume(wh) > target) {
        // Newton steps towards the crossing, then a window of 2e-12 around it
        double sc = (double)sf;
        for (int it = 0; it < 6; ++it) {
          const double v = volume(sc);
          if (v > target) wh = fmin(wh, sc); else wl = fmax(wl, sc);
          const double slope = A + und_a;
          const double next = slope > 0.0 ? sc + (target - v) / slope : sc;
          if (!(next > wl && next < wh) || fabs(next - sc) <= 1e-15 * sc) break;
          sc = next;
        }
        const double nl = sc * (1.0 - 1e-12), nh = sc * (1.0 + 1e-12);
        if (nl > wl && nl < wh && volume(nl) <= target) wl = nl;
        if (nh > wl && nh < wh && volume(nh) > target) wh = nh;
        // midpoints lambda below lam_h give too much volume, above lam_l not
        // (a margin of a few roundings: those between are evaluated)
        const double lam_l = 1.0 / (wl * wl) * (1.0 + 1e-15), lam_h = 1.0 / (wh * wh) * (1.0 - 1e-15);
        // (compared as integers where both are positive: the FP64 pipe is the
        // slow part of this serial chain)
        auto less = [](double a, double b) {
          return __double_as_longlong(a) < __double_as_longlong(b);
        };
        // while the lower end is 0 the midpoints are 1e9 halved k times: go
        // straight to the last but one before the first that may exceed
        const int k0 = ilogb(1e9 / lam_l) - 2;
        if (k0 >= 1 && k0 < 1000) {
          l2 = lam_of(k0);
          last = l2;
          step = k0;
        }
        bool known = false;
        int fine = 0;
        while (step < 4096) {
          const double sum = l1 + l2;
          // with the bracket at [l, 2 l] first, its relative width cannot have
          // fallen to 1e-10 before 29 more halvings
          if (!(sum > 0.0) || (l1 > 0.0 && ++fine > 29 && !((l2 - l1) / sum > 1e-10))) break;
          const double lmid = 0.5 * sum;
          if (!less(l1, lmid) || !less(lmid, l2)) break;
          last = lmid;
          known = !less(lmid, lam_h) && !less(lam_l, lmid);
          bool above = less(lmid, lam_h);
          if (known) {
            total = volume(1.0 / sqrt(lmid));
            above = total > target;
          }
          if (above) l1 = lmid; else l2 = lmid;
          ++step;
        }
        if (last > 0.0 && !known) total = volume(1.0 / sqrt(last));
        done = true;
      }
      if (lane == 0) {
        sh[0] = l1;
        sh[1] = l2;
        sh[2] = total;
        sh[3] = last;
        s_cnt = done ? step : -1;
      }
    }
    __syncthreads();
    done = !over && s_cnt >= 0;
    if (done) {
      l1 = sh[0];
      l2 = sh[1];
      total = sh[2];
      last = sh[3];
      step = s_cnt;
    }
    __syncthreads();
  }

  if (!done) {
    // every midpoint over all elements
    // the phase with lower end 0: midpoints lambda_k, up to the first k in
    // [1, k_end) whose volume exceeds the target, found by a binary search over
    // k (the volume is nondecreasing in k; k_end: the first k with lambda_k =
    // 0, where the step-by-step bisection stops); klo: volume known <= target
    // (0: none evaluated), khi: volume known > target (k_end: none found yet)
    if (k_end > 1) {
      int klo = 0, khi = k_end;
      double vlo = 0.0, vhi = 0.0;
      auto probe = [&](int k) {
        const double v = eval_total(lam_of(k));
        if (v > target) { khi = k; vhi = v; } else { klo = k; vlo = v; }
      };
      probe(k_end - 1);   // is there such a k at all?
      while (khi - klo > 1 && !failed()) probe((klo + khi) / 2);
      if (khi < k_end) {
        l1 = lam_of(khi);
        l2 = lam_of(khi - 1);
        last = l1;
        total = vhi;
        step = khi;
      } else {
        l2 = lam_of(k_end - 1);
        last = l2;
        total = vlo;
        step = k_end - 1;
      }
    }
    // Stops at the relative bracket width 1e-10, or when the midpoint no
    // longer lies strictly inside the bracket (lambda underflow when the target
    // is unreachable from above), and after at most 4096 steps in any case.
    while (l1 + l2 > 0.0 && (l2 - l1) / (l1 + l2) > 1e-10 && step < 4096) {
      const double lmid = 0.5 * (l1 + l2);
      if (!(l1 < lmid && lmid < l2)) break;   // uniform: every block holds the same l1, l2
      total = eval_total(lmid);
      last = lmid;
      if (total > target) l1 = lmid; else l2 = lmid;
      ++step;
      if (failed()) break;
    }
  }
  // the candidate of the last midpoint (rho itself if no step ran), and
  // change = max |rho_new - rho|
  if (threadIdx.x == 0) sh[40] = last > 0.0 ? 1.0 / sqrt(last) : 0.0;
  __syncthreads();
  const double sc = sh[40];
  double mx = 0.0;
  each([&](int e, double a, float2) {
    const double r = rho[e];
    double rn = r;
    if (last > 0.0) {
      if (__double2hiint(r) < 0x7ff00000) {
        // the candidate between its bounds; neither it nor the lower one is
        // negative, so the bits order as the values do
        const long long t = __double_as_longlong(a * sc);
        const long long lo = __double_as_longlong(oc_low(r, move));
        const long long hi = __double_as_longlong(oc_high(r, move));
        const long long m = t < hi ? t : hi;
        rn = __longlong_as_double(lo > m ? lo : m);
      } else {
        rn = fmax(fmax(0.0, r - move), fmin(fmin(1.0, r + move), a * sc));
      }
    }
    rho_new[e] = rn;
    const long long d = __double_as_longlong(rn - r) & 0x7fffffffffffffffll;
    mx = __double_as_longlong(mx) < d && d <= 0x7ff0000000000000ll ? __longlong_as_double(d) : mx;
  });
  double* buf = partials + 6 * MFTO_RED_SLOTS;
  const double bm = block_max(mx, sh);
  if (threadIdx.x == 0) buf[blockIdx.x] = bm;
  grid_sync();
  if (blockIdx.x == 0) {
    double m2 = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x) m2 = fmax(m2, __ldcg(&buf[b]));
    m2 = block_max(m2, sh);
    if (threadIdx.x == 0) {
      s->change = m2;
      s->volume = total / (double)n;
      s->lambda = 0.5 * (l1 + l2);
      s->oc_steps = step;
      s->oc_evals = evals;
    }
  }
}

constexpr int kOcRegs = 8;   // elements per thread held in registers

}  // namespace

mfto_status compliance_launch(mfto_handle* h, const double* rho, const double* u, double* dc,
                              double* c_out, double* gray_out) {
  const Grid g = make_grid(h->mesh);
  h->launches++;
  const mfto_status s = col64_dispatch(h->energy_shape, [&](auto shape) -> mfto_status {
    using S = decltype(shape);
    Col64Tiling tl;
    tl.tx = (g.nelx + S::CX - 1) / S::CX;
    tl.ty = (g.nely + S::CY - 1) / S::CY;
    tl.nzc = h->energy_nzc;
    tl.tz = (g.nelz + tl.nzc - 1) / tl.nzc;
    // one partial per CTA: on wider meshes a CTA takes several tiles
    const int grid = tl.count() < MFTO_RED_SLOTS ? tl.count() : MFTO_RED_SLOTS;
    if (fixed_route(h)) {
      compliance_fixed_kernel<S::CX, S::CY><<<grid, S::NT, energy_smem<S>(), h->stream>>>(
          rho, u, dc, h->fix, g, tl, h->p.E0, h->p.Emin, h->p.penal, pow_plan(h->p.penal),
          h->d_misc, h->d_partials);
      return MFTO_OK;
    }
    compliance_kernel<S::CX, S::CY>
        <<<grid, S::NT, S::template stream_bytes<1>(), h->stream>>>(
            rho, u, dc, h->mc64, g, tl, h->p.E0, h->p.Emin, h->p.penal, pow_plan(h->p.penal),
            h->d_misc, h->d_partials);
    return MFTO_OK;
  });
  if (s != MFTO_OK) return s;
  MFTO_LAUNCH_CHECK(h);
  MFTO_CUDA(h, cudaMemcpyAsync(h->h_misc, h->d_misc, sizeof(MiscScalars), cudaMemcpyDeviceToHost,
                               h->stream));
  MFTO_CUDA(h, cudaStreamSynchronize(h->stream));
  if (c_out) *c_out = h->h_misc->sum[0];
  if (gray_out) *gray_out = h->h_misc->sum[1] / (double)h->n_elem;
  return MFTO_OK;
}

mfto_status simp_init(mfto_handle* h) {
  const Grid g = make_grid(h->mesh);
  // (the FP64 pipe's rule for both energy kernels: the fixed-point one, bound by issue and
  // latency, has had none fitted to it)
  col64_choose(0, g.nelx, g.nely, g.nelz, 0.7, h->num_sms, &h->energy_shape, &h->energy_nzc);
  for (int i = 0; i < kCol64Shapes; ++i) {
    const mfto_status s = col64_dispatch(i, [&](auto shape) -> mfto_status {
      using S = decltype(shape);
      MFTO_CUDA(h, cudaFuncSetAttribute(compliance_kernel<S::CX, S::CY>,
                                        cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)S::template stream_bytes<1>()));
      static_assert(energy_smem<S>() <= 48 * 1024, "no attribute needed");
      return MFTO_OK;
    });
    if (s != MFTO_OK) return s;
  }
  return MFTO_OK;
}

mfto_status oc_launch(mfto_handle* h, const double* rho, const double* dc, double* rho_new,
                      mfto_iter_stats* st) {
  // one CTA per SM with its elements in registers where they fit, two (and
  // scratch arrays) on larger meshes; co-resident (cooperative launch)
  int blocks = h->num_sms;
  const int need = (int)((h->n_elem + kOcThreads - 1) / kOcThreads);
  const bool regs = h->n_elem <= (int64_t)blocks * kOcThreads * kOcRegs;
  if (!regs) {
    int per_sm = 0;
    MFTO_CUDA(h, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, oc_kernel<0>,
                                                               kOcThreads, 0));
    blocks = (per_sm < 2 ? (per_sm < 1 ? 1 : per_sm) : 2) * h->num_sms;
  }
  if (blocks > need) blocks = need;
  if (blocks < 1) blocks = 1;
  // partial rows 0 .. 6, the list segments and counts behind them
  static_assert(sizeof(OcElem) == 3 * sizeof(double), "list entries are three doubles");
  const int64_t list_doubles = (int64_t)blocks * (3 * kOcSeg + 1);
  if (list_doubles > (int64_t)(MFTO_RED_ROWS - 7) * MFTO_RED_SLOTS)
    return mfto_fail(h, MFTO_UNSUPPORTED, "OC: more CTAs than the list segments hold");
  MFTO_CUDA(h, cudaMemsetAsync(&h->d_misc->error, 0, sizeof(int32_t), h->stream));
  MFTO_CUDA(h, cudaMemsetAsync(&h->d_misc->bar_count, 0, sizeof(unsigned int), h->stream));
  int n = (int)h->n_elem;
  double volfrac = h->p.volfrac, move = h->p.move;
  MiscScalars* s = h->d_misc;
  double* partials = h->d_partials2;
  double* a_s = h->d_oc;
  float2* f_s = reinterpret_cast<float2*>(h->d_oc + h->n_elem);
  OcElem* list = reinterpret_cast<OcElem*>(partials + 7 * MFTO_RED_SLOTS);
  int* counts = reinterpret_cast<int*>(list + (size_t)blocks * kOcSeg);
  // k_end: the first k at which 1e9 halved k times is 0 (the bisection's
  // midpoint with lower end 0 no longer lies inside its bracket)
  static const int k_end = [] {
    double x = 1e9;
    int k = 0;
    while (x > 0.0) {
      x = 0.5 * x;
      ++k;
    }
    return k;
  }();
  static const OcUp up = [] {
    OcUp u{0.0, 1e9, -1.0, 0};
    while (u.l1 + u.l2 > 0.0 && (u.l2 - u.l1) / (u.l1 + u.l2) > 1e-10 && u.step < 4096) {
      const double lmid = 0.5 * (u.l1 + u.l2);
      if (!(u.l1 < lmid && lmid < u.l2)) break;
      u.last = u.l1 = lmid;
      ++u.step;
    }
    return u;
  }();
  void* args[] = {(void*)&rho, (void*)&dc, (void*)&rho_new, &a_s, &f_s, &n, &volfrac, &move, &s,
                  &partials, &list, &counts, (void*)&k_end, (void*)&up};
  h->launches++;
  const void* fn = regs ? (const void*)oc_kernel<kOcRegs> : (const void*)oc_kernel<0>;
  MFTO_CUDA(h, cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kOcThreads), args, 0, h->stream));
  MFTO_CUDA(h, cudaMemcpyAsync(h->h_misc, h->d_misc, sizeof(MiscScalars), cudaMemcpyDeviceToHost,
                               h->stream));
  MFTO_CUDA(h, cudaStreamSynchronize(h->stream));
  if (h->h_misc->error)
    return mfto_fail(h, MFTO_CUDA_ERROR, "OC: a grid barrier wait gave up (bounded spin)");
  if (st) {
    st->change = h->h_misc->change;
    st->volume = h->h_misc->volume;
    st->lambda = h->h_misc->lambda;
  }
  return MFTO_OK;
}

extern "C" mfto_status mfto_compliance_sens(mfto_handle* h, const double* rho_phys,
                                            const double* u, double* c_out, double* dc) {
  if (!h) return MFTO_INVALID_ARG;
  MFTO_REQUIRE(h, rho_phys && u && c_out, "mfto_compliance_sens: null pointer");
  return compliance_launch(h, rho_phys, u, dc, c_out, nullptr);
}

extern "C" mfto_status mfto_oc_update(mfto_handle* h, const double* rho, const double* dc,
                                      double* rho_new, mfto_iter_stats* st) {
  if (!h) return MFTO_INVALID_ARG;
  MFTO_REQUIRE(h, rho && dc && rho_new, "mfto_oc_update: null pointer");
  MFTO_REQUIRE(h, rho != rho_new, "mfto_oc_update: rho_new must not alias rho");
  return oc_launch(h, rho, dc, rho_new, st);
}

extern "C" mfto_status mfto_simp_step(mfto_handle* h, double* rho, double* u, const double* f,
                                      double* rho_phys_out, mfto_iter_stats* st) {
  if (!h) return MFTO_INVALID_ARG;
  MFTO_REQUIRE(h, rho && u && f, "mfto_simp_step: null pointer");
  double* rho_phys = rho_phys_out ? rho_phys_out : h->d_rho_phys;
  // filter, then (three-field form) project: rho -> rho_bar -> rho_phys
  const bool proj = projection_active(h);
  mfto_status s = filter_launch(h, rho, proj ? h->d_rho_bar : rho_phys, 0);
  if (s != MFTO_OK) return s;
  if (proj) {
    s = project_launch(h, h->d_rho_bar, rho_phys);
    if (s != MFTO_OK) return s;
  }
  s = modulus_launch(h, MFTO_FORM_F64, rho_phys, h->d_E);
  if (s != MFTO_OK) return s;
  mfto_solve_stats ss;
  if (learned_active(h)) {
    mfto_learned_stats ls;
    s = learned_run(h, h->d_E, rho_phys, f, u, &ls);
    if (s != MFTO_OK) return s;
    ss.iterations = ls.inner_iterations + ls.fp64_iterations;
    ss.status = ls.status;
    ss.rel_residual = ls.rel_residual;
    ss.fnorm = ls.fnorm;
  } else if (gmg_active(h)) {
    s = gmg_solve(h, h->d_E, f, u, &ss);
    if (s != MFTO_OK) return s;
} else if (h->solver_form == MFTO_FORM_F64) {
    s = pcg_run(h, h->d_E, f, u, &ss);
    if (s != MFTO_OK) return s;
  } else {
    mfto_ir_stats is;
    s = ir_run(h, (mfto_form)h->solver_form, h->inner_tol, h->d_E, f, u, &is);
    if (s != MFTO_OK) return s;
    ss.iterations = is.inner_iterations;
    ss.status = is.status;
    ss.rel_residual = is.rel_residual;
    ss.fnorm = is.fnorm;
  }
  double c = 0.0, gray = 0.0;
  s = compliance_launch(h, rho_phys, u, h->d_dc_phys, &c, &gray);
  if (s != MFTO_OK) return s;
  if (proj) {   // dc/drho_bar = dc/drho_phys * drho_phys/drho_bar
    s = project_chain_launch(h, h->d_rho_bar, h->d_dc_phys);
    if (s != MFTO_OK) return s;
  }
  s = filter_launch(h, h->d_dc_phys, h->d_dc, 1);
  if (s != MFTO_OK) return s;
  mfto_iter_stats local;
  mfto_iter_stats* out = st ? st : &local;
  // the OC candidate goes to scratch (the bisection re-reads rho every step)
  s = oc_launch(h, rho, h->d_dc, h->d_dc_phys, out);
  if (s != MFTO_OK) return s;
  MFTO_CUDA(h, cudaMemcpyAsync(rho, h->d_dc_phys, sizeof(double) * h->n_elem,
                               cudaMemcpyDeviceToDevice, h->stream));
  out->compliance = c;
  out->grayness = gray;
  out->cg_iterations = ss.iterations;
  out->cg_status = ss.status;
  out->rel_residual = ss.rel_residual;
  return MFTO_OK;
}
