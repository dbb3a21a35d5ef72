// Column-streaming FP64 K.v (Eq. matfree): the element operator of modes.cuh
// applied along z-columns of elements, one column per thread, with every
// partial transform formed once and shared.
//
// The FP64 pipe runs 2 operations per clock and SM (1/64 of the FP32 rate),
// so this kernel is bound by the number of FP64 operations it executes, not by
// memory, shared memory or latency: one warp instruction keeps its quarter of
// the pipe busy for 64 clocks, and two warps per quarter hide everything else.
// The layout is therefore chosen to execute as few of them as possible.  A CTA
// covers CX x CY element columns and owns the (CX-1) x (CY-1) interior nodes of
// every node layer of a z-chunk.  Per element layer and column it executes
//    6  x stage of the column's lower-y edge (s, d) of the new node layer (the
//       neighbouring column's edge comes from shared memory)
//   12  y stage: face modes of the new node layer; those of the old one are
//       kept in registers
//   21  z stage (the sum of sums is a translation, which the element maps to
//       zero: neither formed nor multiplied)
//   45  mode operator
//   42  modulus, undone z stage and the sum with the element below
//   12  undone y stage: the column's share of its two edges
//    6  sum of the two columns that share an edge
//    6  undone x stage, and 3 for the sum of the two columns along x
// = 153, against 220 (and a 1.3 times larger halo) when every element
// transforms its 8 corners by itself.  The stages are pipelined over the
// layers so that one barrier per layer is enough.
//
// The operators that kv_fixed.cuh holds (Poisson's ratios of 0 to 0.454) run
// there; this kernel serves the others.
//
// Measured on a GB300, y = K v, against the kernel that transformed each
// element's corners by itself in 16 x 12 node tiles: 229 against 394 us at
// 55 x 55 x 165, 18.4 against 79.9 us at 24 x 12 x 12 (the operations above on
// the padded tiles take 192 and 12 us at the FP64 pipe's rate).
#pragma once
#include "common.cuh"

template <int CX_, int CY_>
struct Col64Shape {
  static constexpr int CX = CX_, CY = CY_, NT = CX * CY;   // element columns = threads
  static constexpr int NX = CX + 1, NY = CY + 1, NV = NX * NY;
  static constexpr int OX = CX - 1, OY = CY - 1;           // owned nodes per layer
  static constexpr int ROW = 6 * CX;                       // one edge row: s, d x 3 components
  static_assert(NT % 32 == 0 && CX <= 32, "whole warps, x neighbours within a warp");
  // shared memory of the node stream (ring, node edges) and, for the K.v, of
  // the back edges [2][CY][ROW] and own values [3][3][NT]
  template <int KSRC>
  static constexpr size_t stream_bytes() {
    return sizeof(double) * (size_t)(2 * 3 * KSRC * NV + 2 * (CY + 1) * ROW);
  }
  template <int KSRC>
  static constexpr size_t smem_bytes() {
    return stream_bytes<KSRC>() + sizeof(double) * (size_t)(2 * CY * ROW + 9 * NT);
  }
};

// Tile t owns nodes [tx OX, +OX) x [ty OY, +OY) x [tz nzc, +nzc).
struct Col64Tiling {
  int tx, ty, tz, nzc;
  __host__ __device__ int count() const { return tx * ty * tz; }
};

__device__ __forceinline__ void col64_cp8(void* sdst, const void* gsrc, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(sdst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(d), "l"(gsrc),
               "r"(valid ? 8 : 0)
               : "memory");
}
__device__ __forceinline__ void col64_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void col64_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// Loaders: the staged source arrays and how they combine into the vector.
struct Col64LoadPlain {
  static constexpr int kSrc = 1;
  const double* v;
  __device__ __forceinline__ const double* src(int) const { return v; }
  __device__ __forceinline__ double combine(const double (&r)[1]) const { return r[0]; }
};
struct Col64LoadDirection {           // z + beta p
  static constexpr int kSrc = 2;
  const double* z;
  const double* p;
  double beta;
  __device__ __forceinline__ const double* src(int i) const { return i == 0 ? z : p; }
  __device__ __forceinline__ double combine(const double (&r)[2]) const { return fma(beta, r[1], r[0]); }
};

// face modes (a + 2b) of one node layer for the three components
struct Col64Face {
  double m[3][4];
};

// z stage: modes m = f + 4 (z difference) of the element between face modes lo
// (below) and up (above).  Mode 0, a translation, is left 0.
__device__ __forceinline__ void col64_modes(const Col64Face& lo, const Col64Face& up,
                                            double (&X)[3][8]) {
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      X[c][f] = f == 0 ? 0.0 : lo.m[c][f] + up.m[c][f];
      X[c][f | 4] = up.m[c][f] - lo.m[c][f];
    }
}

// Element layer between face modes lo_f (below) and up_f (above), unit mode
// operator, modulus and undone z stage: up (in: the upper-face outputs of the
// element below, out: this one's) and Ms = up_in + this element's lower-face
// outputs, both in face modes.
__device__ __forceinline__ void col64_element(const Col64Face& lo_f, const Col64Face& up_f,
                                              double E, const ModeCoef<double>& K, Col64Face& up,
                                              Col64Face& Ms) {
  double X[3][8], Y[3][8];
  col64_modes(lo_f, up_f, X);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int m = 1; m < 8; ++m) Y[c][m] = K.diag[c][m] * X[c][m];
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      if (i == j) continue;
      const int t = 3 - i - j;
#pragma unroll
      for (int mt = 0; mt < 2; ++mt) {
        const int tb = mt << t;
        Y[i][(1 << i) | tb] = fma(K.lamM[mt], X[j][(1 << j) | tb], Y[i][(1 << i) | tb]);
        Y[i][(1 << j) | tb] = fma(K.muM[mt], X[j][(1 << i) | tb], Y[i][(1 << j) | tb]);
      }
    }
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const double ed = E * Y[c][f | 4];
      if (f == 0) {                       // no sum-of-sums output
        Ms.m[c][0] = up.m[c][0] - ed;
        up.m[c][0] = ed;
      } else {
        Ms.m[c][f] = fma(E, Y[c][f], up.m[c][f] - ed);
        up.m[c][f] = fma(E, Y[c][f], ed);
      }
    }
}

// Epilogues: what the owner of a node does with its 3 sums.
struct Col64Store {                   // plain K.v: y = sum, y_fixed = v
  static constexpr bool kOwn = false;   // pn unused
  const double* v;
  double* y;
  __device__ __forceinline__ void operator()(int node, const double (&acc)[3],
                                             const double (&pn)[3], uint8_t fm,
                                             double& red) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) y[3 * node + c] = ((fm >> c) & 1) ? v[3 * node + c] : acc[c];
  }
};
struct Col64Pcg {                     // CG: p_new stored, q = K p_new, p_new.q accumulated
  static constexpr bool kOwn = true;
  double* p_new;
  double* q;
  __device__ __forceinline__ void operator()(int node, const double (&acc)[3],
                                             const double (&pn)[3], uint8_t fm,
                                             double& red) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double qc = ((fm >> c) & 1) ? pn[c] : acc[c];
      p_new[3 * node + c] = pn[c];
      q[3 * node + c] = qc;
      red = fma(pn[c], qc, red);
    }
  }
};

// The node layers of a tile of CX x CY element columns, streamed along z: raw
// values copied asynchronously two layers ahead into a ring (each thread reads
// only its own copies, so the ring needs no barrier), the x stage of every
// edge row into shared memory, the y stage into registers.  fixed NULL: no
// masks.
template <int CX, int CY, typename Load>
struct Col64Stream {
  using S = Col64Shape<CX, CY>;
  static constexpr int KS = Load::kSrc;
  // ring [2][3 KS][NV], node edges [2][CY + 1][6][CX]; slot of layer k: k & 1
  static constexpr int kRing = 2 * 3 * KS * S::NV, kEdges = 2 * (CY + 1) * S::ROW;
  static constexpr int kDoubles = kRing + kEdges;
  double *ring, *edges;
  const Load& ld;
  const uint8_t* fixed;
  const Grid& g;
  int ex, ey, gi, gj, nb0, nxy, last;   // last: the topmost node layer to copy
  bool re, te, in0, in1, in2, in3;
  double eo[6];   // this column's lower-y edge of the node layer staged last

  // (i0, j0): element column and node of thread 0
  __device__ __forceinline__ Col64Stream(double* smem, const Load& load, const uint8_t* fix,
                                         const Grid& grid, int i0, int j0, int last_layer)
      : ring(smem), edges(smem + kRing), ld(load), fixed(fix), g(grid) {
    ex = threadIdx.x % CX;
    ey = threadIdx.x / CX;
    gi = i0 + ex;
    gj = j0 + ey;
    last = min(last_layer, g.nz - 1);
    nxy = g.nx * g.ny;
    nb0 = gi + g.nx * gj;
    // the thread's nodes of a layer: its own, the tile's last column for the
    // last thread of a row, the tile's last row for the threads of the last row
    re = ex == CX - 1;
    te = ey == CY - 1;
    const bool in_x0 = gi >= 0 && gi < g.nx, in_x1 = gi + 1 < g.nx;
    const bool in_y0 = gj >= 0 && gj < g.ny, in_y1 = gj + 1 < g.ny;
    in0 = in_x0 && in_y0;
    in1 = re && in_x1 && in_y0;
    in2 = te && in_x0 && in_y1;
    in3 = re && te && in_x1 && in_y1;
  }

  // copies node layer L into its ring slot; returns the masks of the thread's
  // nodes (own | right << 8 | top << 16 | corner << 24)
  __device__ __forceinline__ uint32_t issue(int L) {
    double* R = ring + (L & 1) * 3 * KS * S::NV;
    const bool lay = L >= 0 && L <= last;
    uint32_t fm = 0;
    auto one = [&](bool in, int node, int q, int shift) {
      in = in && lay;
      const int n = in ? node : 0;
#pragma unroll
      for (int s = 0; s < KS; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c)
          col64_cp8(R + (3 * s + c) * S::NV + q, ld.src(s) + 3 * n + c, in);
      if (in && fixed != nullptr) fm |= (uint32_t)fixed[node] << shift;
    };
    const int base = nb0 + nxy * L, q = ey * S::NX + ex;
    one(in0, base, q, 0);
    if (re) one(in1, base + 1, q + 1, 8);
    if (te) one(in2, base + g.nx, q + S::NX, 16);
    if (re && te) one(in3, base + g.nx + 1, q + S::NX + 1, 24);
    col64_commit();
    return fm;
  }

  __device__ __forceinline__ void take(int L, int q, uint32_t fm, double (&v)[3]) const {
    const double* R = ring + (L & 1) * 3 * KS * S::NV + q;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double r[KS];
#pragma unroll
      for (int s = 0; s < KS; ++s) r[s] = R[(3 * s + c) * S::NV];
      v[c] = ((fm >> c) & 1) ? 0.0 : ld.combine(r);
    }
  }

  // x stage of one edge row: the edge from this thread's node to the next
  __device__ __forceinline__ void edge(const double (&a)[3], const double (&right)[3],
                                       double (&e)[6]) const {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      double b = __shfl_down_sync(0xffffffffu, a[c], 1);
      if (re) b = right[c];
      e[c] = a[c] + b;
      e[3 + c] = b - a[c];
    }
  }

  // x stage of node layer L (its copies have landed); own: the thread's node
  __device__ __forceinline__ void stage(int L, uint32_t fm, double (&own)[3]) {
    const int q = ey * S::NX + ex;
    double right[3] = {0.0, 0.0, 0.0};
    take(L, q, fm, own);
    if (re) take(L, q + 1, fm >> 8, right);
    edge(own, right, eo);
    double* Eb = edges + (L & 1) * (CY + 1) * S::ROW + ey * S::ROW + ex;
#pragma unroll
    for (int i = 0; i < 6; ++i) Eb[i * CX] = eo[i];
    if (__any_sync(0xffffffffu, te)) {   // the tile's last edge row
      double top[3] = {0.0, 0.0, 0.0}, corner[3] = {0.0, 0.0, 0.0}, et[6];
      if (te) take(L, q + S::NX, fm >> 16, top);
      if (re && te) take(L, q + S::NX + 1, fm >> 24, corner);
      edge(top, corner, et);
      if (te) {
#pragma unroll
        for (int i = 0; i < 6; ++i) Eb[S::ROW + i * CX] = et[i];
      }
    }
  }

  // y stage of node layer L, staged last, a barrier after its stage()
  __device__ __forceinline__ void face(int L, Col64Face& F) const {
    const double* Eb = edges + (L & 1) * (CY + 1) * S::ROW + (ey + 1) * S::ROW + ex;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double s1 = Eb[c * CX], d1 = Eb[(3 + c) * CX];
      F.m[c][0] = eo[c] + s1;
      F.m[c][2] = s1 - eo[c];
      F.m[c][1] = eo[3 + c] + d1;
      F.m[c][3] = d1 - eo[3 + c];
    }
  }
};

// Tile `tile` of `tl`; returns this thread's share of the epilogue reduction.
// Iteration ez (element layer ez, between node layers ez and ez + 1) stages
// node layer ez + 1, crosses the layer's barrier, finishes node layer ez - 1
// and computes element layer ez.
template <int CX, int CY, typename Load, typename Epi>
__device__ __forceinline__ double kv_column64_body(const double* __restrict__ E,
                                                   const uint8_t* __restrict__ fixed,
                                                   const ModeCoef<double>& K, const Grid& g,
                                                   const Col64Tiling& tl, int tile,
                                                   const Load& ld, const Epi& epi, double* smem) {
  using S = Col64Shape<CX, CY>;
  using Stream = Col64Stream<CX, CY, Load>;
  double* back = smem + Stream::kDoubles;              // [2][CY][6][CX], slot of layer k: k & 1
  double* ownv = back + 2 * CY * S::ROW;               // [3][3][NT], slot of layer k: (k + 3) % 3
  const int tid = threadIdx.x;
  const int bx = tile % tl.tx, by = (tile / tl.tx) % tl.ty, bz = tile / (tl.tx * tl.ty);
  const int kb = bz * tl.nzc, ke = min(kb + tl.nzc, g.nz);        // owned node layers [kb, ke)
  Stream st(smem, ld, fixed, g, bx * S::OX - 1, by * S::OY - 1, ke);
  const int ex = st.ex, ey = st.ey, gi = st.gi, gj = st.gj;
  const int nexy = g.nelx * g.nely;
  const bool elem_in = gi >= 0 && gj >= 0 && gi < g.nelx && gj < g.nely;
  const bool own_node = ex >= 1 && ey >= 1 && st.in0;
  const bool warp_elem = __any_sync(0xffffffffu, elem_in);
  const bool warp_own = __any_sync(0xffffffffu, own_node);
  double red = 0.0;

  auto stage = [&](int L, uint32_t fm) {
    double own[3];
    st.stage(L, fm, own);
    double* O = ownv + ((L + 3) % 3) * 3 * S::NT + tid;
#pragma unroll
    for (int c = 0; c < 3; ++c) O[c * S::NT] = own[c];
  };
  double front[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // this column's share of its lower-y edge
  // owner's sum of node layer k: the shares of the columns at y - 1 (back
  // edge) and y (front edge), then of the columns at x - 1 and x
  auto finish = [&](int k, uint32_t fm) {
    if (!warp_own) return;
    const double* Bb = back + (k & 1) * CY * S::ROW + (ey > 0 ? ey - 1 : 0) * S::ROW + ex;
    double acc[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double s = Bb[c * CX] + front[c], d = Bb[(3 + c) * CX] + front[3 + c];
      const double up = __shfl_up_sync(0xffffffffu, s + d, 1);
      acc[c] = up + (s - d);
    }
    if (own_node) {
      const double* O = ownv + ((k + 3) % 3) * 3 * S::NT + tid;
      const double pn[3] = {O[0], O[S::NT], O[2 * S::NT]};
      epi(st.nb0 + st.nxy * k, acc, pn, (uint8_t)fm, red);
    }
  };

  // a warp without elements contributes nothing: its back edges stay zero
  if (!warp_elem) {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int i = 0; i < 6; ++i) back[s * CY * S::ROW + ey * S::ROW + i * CX + ex] = 0.0;
  }
  uint32_t fm_prev = 0, fm_cur = st.issue(kb - 1), fm_next = st.issue(kb);
  col64_wait<1>();
  stage(kb - 1, fm_cur);
  uint32_t fm_load = st.issue(kb + 1);
  __syncthreads();
  Col64Face F0, F1, U, Ms;
  if (warp_elem) st.face(kb - 1, F0);
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int f = 0; f < 4; ++f) U.m[c][f] = 0.0;
  // one element layer: Flo the face modes of node layer ez (in), Fup those of
  // ez + 1 (out)
  auto layer = [&](int ez, const Col64Face& Flo, Col64Face& Fup) {
    double Ee = 0.0;
    if (elem_in && ez >= 0 && ez < g.nelz) Ee = E[gi + g.nelx * gj + nexy * ez];
    // node layer ez + 1 has landed: its x stage, then the copies of ez + 3
    // into the slot it leaves
    col64_wait<1>();
    stage(ez + 1, fm_next);
    const uint32_t fm_new = st.issue(ez + 3);
    __syncthreads();
    if (ez - 1 >= kb) finish(ez - 1, fm_prev);
    if (warp_elem) {
      st.face(ez + 1, Fup);
      if (ez >= 0 && ez < g.nelz) {
        col64_element(Flo, Fup, Ee, K, U, Ms);
      } else {   // below or above the mesh: no element layer
        Ms = U;
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
          for (int f = 0; f < 4; ++f) U.m[c][f] = 0.0;
      }
      double* Bb = back + (ez & 1) * CY * S::ROW + ey * S::ROW + ex;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        front[c] = Ms.m[c][0] - Ms.m[c][2];
        front[3 + c] = Ms.m[c][1] - Ms.m[c][3];
        Bb[c * CX] = Ms.m[c][0] + Ms.m[c][2];
        Bb[(3 + c) * CX] = Ms.m[c][1] + Ms.m[c][3];
      }
    }
    fm_prev = fm_cur;
    fm_cur = fm_next;
    fm_next = fm_load;
    fm_load = fm_new;
  };
  fm_prev = fm_cur;
  for (int ez = kb - 1; ez < ke; ez += 2) {
    layer(ez, F0, F1);
    if (ez + 1 < ke) layer(ez + 1, F1, F0);
  }
  __syncthreads();
  finish(ke - 1, fm_prev);
  col64_wait<0>();
  return red;
}

// Threads an SM holds at the kernels' launch bounds: registers for a whole
// element in each (at most 168).
constexpr int kCol64Threads = 384;

// The tile shapes, by index, and the one (with its z-chunk) that a mesh gets.
constexpr int kCol64Shapes = 5;
template <typename F>
mfto_status col64_dispatch(int i, const F& f) {
  switch (i) {
    case 0: return f(Col64Shape<32, 8>{});
    case 1: return f(Col64Shape<16, 16>{});
    case 2: return f(Col64Shape<32, 4>{});
    case 3: return f(Col64Shape<16, 8>{});
    default: return f(Col64Shape<8, 16>{});
  }
}

// A CTA of NT threads over nzc layers executes (nzc + extra) layers of NT / 32
// warps, and an SM's FP64 pipe takes its CTAs one after another, so the time is
// that of the SM with the most CTAs: ceil(tiles / SMs) x NT x (nzc + extra), or
// about half a CTA beyond the mean where there are more than are resident.
// Few resident warps leave gaps: sweeps of shapes and chunks on seven meshes
// (3,456 to 1,000,000 elements) gave 1.5 times the pipe's time with 4 warps on
// an SM, 1.25 with 8 and 1.18 with 12, hence the factor 1.03 + 2 / warps.  Every
// shape and every balanced chunk length is tried (host arithmetic, once per
// handle).  halo: columns (in x and y) of a tile that it does not own; nx, ny,
// nz: what the tiles own together; extra: the recomputed layer and about half a
// layer of prologue and tail; copies: launches' worth of tiles in one grid.
static inline void col64_choose(int halo, int nx, int ny, int nz, double extra, int num_sms,
                                int* shape_out, int* nzc_out, int copies = 1) {
  double best = 0.0;
  bool best_fits = false;
  for (int i = 0; i < kCol64Shapes; ++i)
    col64_dispatch(i, [&](auto shape) -> mfto_status {
      using S = decltype(shape);
      const int ox = S::CX - halo, oy = S::CY - halo;
      const int64_t txy = (int64_t)((nx + ox - 1) / ox) * ((ny + oy - 1) / oy);
      for (int tz = 1; tz <= nz; ++tz) {
        const int nzc = (nz + tz - 1) / tz;
        if ((nz + nzc - 1) / nzc != tz) continue;          // not a balanced count
        const bool fits = txy * tz <= MFTO_RED_SLOTS;       // one partial per CTA
        if (!fits && tz > 1) break;
        constexpr int resident = kCol64Threads / S::NT;
        const double mean = (double)(txy * tz * copies) / num_sms;
        const int64_t ctas = (txy * tz * copies + num_sms - 1) / num_sms;
        const double busy = ctas > resident ? mean + 0.5 : (double)ctas;
        const double warps = (double)(ctas > resident ? resident : ctas) * S::NT / 32;
        const double cost = busy * S::NT * (nzc + extra) * (1.03 + 2.0 / warps);
        if (best == 0.0 || (fits == best_fits ? cost < best : fits)) {
          best = cost;
          best_fits = fits;
          *shape_out = i;
          *nzc_out = nzc;
        }
      }
      return MFTO_OK;
    });
}
