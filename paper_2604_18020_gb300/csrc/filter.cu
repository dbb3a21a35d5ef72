// Cone density filter (Sec. 3.1) and its transpose.
//
//   forward:   y_e = sum_{i in N(e)} w_ei x_i / W_e
//   transpose: y_i = sum_{e in N(i)} w_ei x_e / W_e
// N(e): the stencil offsets of mfto_filter_stencil, truncated at the domain
// boundary; W_e = sum_{i in N(e)} w_ei.  Terms are added in stencil order with
// separate IEEE multiply and add (no fused multiply-add), so the result does
// not depend on the compiler's contraction choices.  The weight matrix is
// symmetric, so the transpose visits the same offsets and runs the forward sum
// on the quotients x / W, formed once per element (the same quotients the sum
// would form term by term).
//
// Radii in (sqrt 2, 2] (offsets of at most one element, 19 or 27 terms) take the
// streaming kernel below, which divides as it stages a layer; others the general
// one, after a pass that divides.
#include "common.cuh"

namespace {

__global__ void __launch_bounds__(MFTO_BLOCK)
filter_kernel(const double* __restrict__ x, double* __restrict__ y,
              const double* __restrict__ W, const int32_t* __restrict__ off,
              const double* __restrict__ w, int n_st, Grid g, int transpose,
              int rowsums_only) {
  extern __shared__ unsigned char smem_raw[];
  double* sw = reinterpret_cast<double*>(smem_raw);
  int* so = reinterpret_cast<int*>(sw + n_st);
  for (int t = threadIdx.x; t < n_st; t += blockDim.x) {
    sw[t] = w[t];
    so[3 * t + 0] = off[3 * t + 0];
    so[3 * t + 1] = off[3 * t + 1];
    so[3 * t + 2] = off[3 * t + 2];
  }
  __syncthreads();
  const int n = g.nelx * g.nely * g.nelz;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int i = e % g.nelx, j = (e / g.nelx) % g.nely, k = e / (g.nelx * g.nely);
    double acc = 0.0;
    for (int t = 0; t < n_st; ++t) {
      const int ii = i + so[3 * t], jj = j + so[3 * t + 1], kk = k + so[3 * t + 2];
      if (ii < 0 || jj < 0 || kk < 0 || ii >= g.nelx || jj >= g.nely || kk >= g.nelz) continue;
      const int nb = ii + g.nelx * (jj + g.nely * kk);
      double term;
      if (rowsums_only)
        term = sw[t];
      else
        term = __dmul_rn(sw[t], x[nb]);
      acc = __dadd_rn(acc, term);
    }
    y[e] = (rowsums_only || transpose) ? acc : __ddiv_rn(acc, W[e]);
  }
}

__global__ void __launch_bounds__(MFTO_BLOCK)
divide_kernel(const double* __restrict__ x, const double* __restrict__ W, double* __restrict__ q,
              int n) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x)
    q[e] = __ddiv_rn(x[e], W[e]);
}

// ---- one neighbour in each direction, 19 or 27 terms (sqrt 2 < rmin <= 2)
//
// The weights are then those of the distances 0, 1, sqrt 2 and sqrt 3 (classes
// 0 .. C of those below rmin, C = 2 or 3).  The FP64 pipe, two operations per clock and SM,
// is what bounds the sum, so an element's product with each weight is formed
// once, by the thread that stages it, and read by every neighbour: 18 additions
// and 3 products per element at 19 terms instead of 19 of each.  A CTA of TX x
// TY columns streams along z: a layer's products in shared memory (double
// buffered, one barrier per layer) feed the last nine terms of the layer below,
// the middle nine of its own and the first nine of the layer above, so each
// element's sum still runs in stencil order.  Products of elements outside the
// mesh are zero, and a first term of -0 counts as +0: the sum starts from +0,
// and neither changes a bit of it.
//
// Measured on a GB300, forward and transpose, against the general kernel (every
// product formed anew, a division per element): 19 terms at 256 x 128 x 150 289
// and 306 against 433 and 438 us, at 120 x 60 x 30 25 and 25 against 27 and 31;
// 27 terms 382 and 398 against 584 and 588 us.  At 7 terms (rmin <= sqrt 2) the
// products are few and the staging costs more: 33 against 27 us at 55 x 55 x
// 165, so these stay with the general kernel.
constexpr int kFilterThreads = 256;   // threads of a CTA
constexpr int kFilterResident = 1024; // ... and what an SM holds

struct FilterWeights {
  double w[4];
};

// A row sum w (between 1 and 54), its reciprocal r = RN(1 / w) and whether that
// is so close that a r is within an ulp of a / w (half an ulp of rounding and
// half of the reciprocal's error); renewed when the sum changes along z.
struct FilterRow {
  double w = 1.0, r = 1.0;
  bool close = true;
  __device__ __forceinline__ void set(double v) {
    if (__double_as_longlong(v) == __double_as_longlong(w)) return;
    w = v;
    r = __drcp_rn(v);
    close = fabs(__fma_rn(-v, r, 1.0)) <= 0.99 * 0x1p-54;
  }
};

// a / w in the IEEE rounding: Markstein's correction (P. Markstein, "Computation
// of elementary functions on the IBM RISC System/6000 processor", 1990) of a
// quotient good to an ulp; an r that is not close takes a first correction to
// get there.  Where a lies near the ends of the exponent range, or is no number,
// the division itself.
__device__ __forceinline__ double filter_divide(double a, const FilterRow& row) {
  const unsigned hi = (unsigned)__double2hiint(a) & 0x7fffffffu;
  if (hi - 0x10000000u >= 0x60000000u && (hi | (unsigned)__double2loint(a)) != 0u)
    return __ddiv_rn(a, row.w);
  double q = __dmul_rn(a, row.r);
  if (!row.close) q = __fma_rn(__fma_rn(-q, row.w, a), row.r, q);
  return __fma_rn(__fma_rn(-q, row.w, a), row.r, q);
}

// w x; x / 2 (half: w = 1/2, the neighbours' weight at rmin = 1.5) by the exponent
__device__ __forceinline__ double filter_product(double w, bool half, double x) {
  const int hi = __double2hiint(x);
  const unsigned e = (unsigned)hi & 0x7ff00000u;
  if (half && e - 0x00200000u < 0x7fd00000u)
    return __hiloint2double(hi - 0x00100000, __double2loint(x));
  return __dmul_rn(w, x);
}

// the first term of a sum that starts from +0
__device__ __forceinline__ double filter_first(double t) {
  const int hi = __double2hiint(t), lo = __double2loint(t);
  return __hiloint2double(hi == (int)0x80000000 && lo == 0 ? 0 : hi, lo);
}

template <int C, int TX, bool T>
__global__ void __launch_bounds__(kFilterThreads, kFilterResident / kFilterThreads)
filter_near_kernel(const double* __restrict__ x, double* __restrict__ y,
                   const double* __restrict__ W, FilterWeights fw, Grid g, int tiles_x,
                   int tiles_y, int nzc) {
  constexpr int TY = kFilterThreads / TX, PX = TX + 2, PY = TY + 2, P = PX * PY;
  constexpr int NH = P - TX * TY;                       // halo columns
  __shared__ double planes[2][C][P];
  const int tid = threadIdx.x;
  const int bx = blockIdx.x % tiles_x, by = (blockIdx.x / tiles_x) % tiles_y,
            bz = blockIdx.x / (tiles_x * tiles_y);
  const int i0 = bx * TX - 1, j0 = by * TY - 1;         // element of the plane's corner
  const int kb = bz * nzc, ke = min(kb + nzc, g.nelz);
  const int nxy = g.nelx * g.nely;
  const int tx = tid % TX, ty = tid / TX;
  const int q = (ty + 1) * PX + tx + 1;                 // this thread's place in a plane
  const int gi = i0 + 1 + tx, gj = j0 + 1 + ty;
  const bool in = gi < g.nelx && gj < g.nely;
  const int col = in ? gi + g.nelx * gj : 0;
  const bool warp_in = __any_sync(0xffffffffu, in);
  // the halo column it stages as well: top and bottom rows, then the sides
  static_assert(NH <= kFilterThreads, "one halo column per thread");
  int hx = 0, hy = 0;
  if (tid < 2 * PX) {
    hx = tid % PX;
    hy = tid < PX ? 0 : PY - 1;
  } else if (tid < NH) {
    hx = (tid - 2 * PX) & 1 ? PX - 1 : 0;
    hy = 1 + (tid - 2 * PX) / 2;
  }
  const int hi = i0 + hx, hj = j0 + hy, hq = hy * PX + hx;
  const bool halo = tid < NH;
  const bool hin = halo && hi >= 0 && hj >= 0 && hi < g.nelx && hj < g.nely;
  const int hcol = hin ? hi + g.nelx * hj : 0;
  const bool warp_halo = __any_sync(0xffffffffu, hin);
  const bool half = fw.w[1] == 0.5;
  // planes start as zeros: columns outside the mesh stay so
  for (int t = tid; t < 2 * C * P; t += kFilterThreads) (&planes[0][0][0])[t] = 0.0;
  __syncthreads();

  double xo = 0.0, xh = 0.0, wo = 1.0, wh = 1.0;        // the next layer's values
  FilterRow ro, rh, ry;
  auto load = [&](int L) {
    const bool lay = L >= 0 && L < g.nelz;
    xo = in && lay ? x[col + nxy * L] : 0.0;
    xh = hin && lay ? x[hcol + nxy * L] : 0.0;
    if constexpr (T) {
      wo = in && lay ? W[col + nxy * L] : wo;
      wh = hin && lay ? W[hcol + nxy * L] : wh;
    }
  };
  double lo = 0.0, mid = 0.0;                           // sums of layers L - 1 and L
  load(kb - 1);
  for (int L = kb - 1; L <= ke; ++L) {
    double p[2] = {0.0, 0.0};                           // own products of classes 0 and 1
    double(&pl)[C][P] = planes[L & 1];
    const bool lay = L >= 0 && L < g.nelz;
    if (lay) {
      if (warp_in) {
        double v = xo;
        if constexpr (T) {
          ro.set(wo);
          v = filter_divide(v, ro);
        }
        p[0] = __dmul_rn(fw.w[0], v);
        p[1] = filter_product(fw.w[1], half, v);
        pl[0][q] = p[1];
#pragma unroll
        for (int c = 2; c <= C; ++c) pl[c - 1][q] = __dmul_rn(fw.w[c], v);
      }
      if (warp_halo) {
        double v = xh;
        if constexpr (T) {
          rh.set(wh);
          v = filter_divide(v, rh);
        }
        if (halo) {
#pragma unroll
          for (int c = 1; c <= C; ++c)
            pl[c - 1][hq] = c == 1 ? filter_product(fw.w[1], half, v) : __dmul_rn(fw.w[c], v);
        }
      }
    }
    double wy = 1.0;
    if (!T && in && L > kb) wy = W[col + nxy * (L - 1)];
    if (L < ke) load(L + 1);
    __syncthreads();
    if (!warp_in) continue;
    double up = 0.0;                                    // sum of layer L + 1
    if (lay) {
      // terms of the plane at dz, in order; side: the class of a plane at
      // dz = +-1 is one more
      auto plane = [&](double s, int side, bool first) {
#pragma unroll
        for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
          for (int dx = -1; dx <= 1; ++dx) {
            const int c = side + dx * dx + dy * dy;
            if (c > C) continue;
            const double t = dx == 0 && dy == 0 ? p[side] : pl[c - 1][q + dy * PX + dx];
            s = first ? filter_first(t) : __dadd_rn(s, t);
            first = false;
          }
        return s;
      };
      if (L + 1 < ke) up = plane(0.0, 1, true);
      if (L >= kb && L < ke) mid = plane(mid, 0, false);
      if (L > kb) lo = plane(lo, 1, false);
    }
    if (L > kb && in) {
      double out = lo;
      if constexpr (!T) {
        ry.set(wy);
        out = filter_divide(out, ry);
      }
      y[col + nxy * (L - 1)] = out;
    }
    lo = mid;
    mid = up;
  }
}

template <typename F>
mfto_status filter_near_dispatch(int cls, int shape, int transpose, const F& f) {
#define MFTO_FN(C)                                                                            \
  switch (2 * shape + transpose) {                                                            \
    case 0: return f(filter_near_kernel<C, 32, false>, 32);                                   \
    case 1: return f(filter_near_kernel<C, 32, true>, 32);                                    \
    case 2: return f(filter_near_kernel<C, 16, false>, 16);                                   \
    case 3: return f(filter_near_kernel<C, 16, true>, 16);                                    \
    case 4: return f(filter_near_kernel<C, 8, false>, 8);                                     \
    default: return f(filter_near_kernel<C, 8, true>, 8);                                     \
  }
  if (cls == 2) MFTO_FN(2)
  MFTO_FN(3)
#undef MFTO_FN
}

// Tile width and z-chunk: the SM with the most work sets the time.  A CTA
// executes, per warp that holds elements, about 19 additions a layer it owns
// and 6 operations (products, quotient) a layer it stages, two more than it
// owns, and about four layers' worth of start and end; warps outside the mesh
// execute nothing.  Few resident warps leave gaps of the pipe (the factor of
// col64_choose).
static void filter_choose(mfto_handle* h, const Grid& g) {
  double best = 0.0;
  for (int shape = 0; shape < 3; ++shape) {
    const int tx = 32 >> shape, ty = kFilterThreads / tx, rows = 32 / tx;   // rows of a warp
    const int ntx = (g.nelx + tx - 1) / tx, nty = (g.nely + ty - 1) / ty;
    const double warps = (double)((g.nely + rows - 1) / rows) / nty;        // of a CTA
    for (int tz = 1; tz <= g.nelz; ++tz) {
      const int nzc = (g.nelz + tz - 1) / tz;
      if ((g.nelz + nzc - 1) / nzc != tz) continue;
      const int64_t n = (int64_t)ntx * nty * tz, per = (n + h->num_sms - 1) / h->num_sms;
      // CTAs of the busiest SM: full sets of the resident ones, then the rest
      constexpr int resident = kFilterResident / kFilterThreads;
      const int64_t full = per / resident * resident, rest = per - full;
      auto time = [&](int64_t ctas, int64_t at_once) {
        return ctas == 0 ? 0.0 : (double)ctas * (1.03 + 2.0 / (warps * (double)at_once));
      };
      const double cost = (time(full, resident) + time(rest, rest)) * warps *
                          (19.0 * nzc + 6.0 * (nzc + 2) + 24.0);
      if (best == 0.0 || cost < best) {
        best = cost;
        h->filter_shape = shape;
        h->filter_nzc = nzc;
      }
    }
  }
}

}  // namespace

static mfto_status launch_near(mfto_handle* h, const double* x, double* y, int transpose) {
  const Grid g = make_grid(h->mesh);
  FilterWeights fw;
  for (int c = 0; c < 4; ++c) fw.w[c] = h->p.rmin - sqrt((double)c);
  return filter_near_dispatch(
      fw.w[3] > 0.0 ? 3 : 2, h->filter_shape, transpose,
      [&](auto kernel, int tx) -> mfto_status {
        const int ty = kFilterThreads / tx;
        const int ntx = (g.nelx + tx - 1) / tx, nty = (g.nely + ty - 1) / ty;
        const int ntz = (g.nelz + h->filter_nzc - 1) / h->filter_nzc;
        h->launches++;
        kernel<<<ntx * nty * ntz, kFilterThreads, 0, h->stream>>>(x, y, h->d_filter_W, fw, g, ntx,
                                                                 nty, h->filter_nzc);
        MFTO_LAUNCH_CHECK(h);
        return MFTO_OK;
      });
}

static mfto_status launch_filter(mfto_handle* h, const double* x, double* y, int transpose,
                                 int rowsums) {
  const Grid g = make_grid(h->mesh);
  const size_t smem = (size_t)h->n_stencil * (sizeof(double) + 3 * sizeof(int));
  if (smem > 48 * 1024)
    MFTO_CUDA(h, cudaFuncSetAttribute(filter_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)smem));
  int blocks = (int)((h->n_elem + MFTO_BLOCK - 1) / MFTO_BLOCK);
  if (blocks > 16 * h->num_sms) blocks = 16 * h->num_sms;
  if (transpose) {   // quotients x / W into the OC scratch (free outside the OC update)
    h->launches++;
    divide_kernel<<<blocks, MFTO_BLOCK, 0, h->stream>>>(x, h->d_filter_W, h->d_oc,
                                                        (int)h->n_elem);
    x = h->d_oc;
  }
  h->launches++;
  filter_kernel<<<blocks, MFTO_BLOCK, smem, h->stream>>>(x, y, h->d_filter_W, h->d_stencil_off,
                                                         h->d_stencil_w, h->n_stencil, g,
                                                         transpose, rowsums);
  MFTO_LAUNCH_CHECK(h);
  return MFTO_OK;
}

mfto_status filter_rowsums(mfto_handle* h) {
  filter_choose(h, make_grid(h->mesh));
  return launch_filter(h, nullptr, h->d_filter_W, 0, 1);
}

mfto_status filter_launch(mfto_handle* h, const double* x, double* y, int transpose) {
  // n_stencil tells sqrt 2 < rmin <= 2 from smaller radii (1 or 7 terms) and
  // larger ones (33 and more)
  if (h->n_stencil == 19 || h->n_stencil == 27) return launch_near(h, x, y, transpose);
  return launch_filter(h, x, y, transpose, 0);
}

extern "C" mfto_status mfto_filter(mfto_handle* h, const double* x, double* y,
                                   int32_t transpose) {
  if (!h) return MFTO_INVALID_ARG;
  MFTO_REQUIRE(h, x && y, "mfto_filter: null pointer");
  MFTO_REQUIRE(h, x != y, "mfto_filter: y must not alias x");
  return filter_launch(h, x, y, transpose ? 1 : 0);
}
