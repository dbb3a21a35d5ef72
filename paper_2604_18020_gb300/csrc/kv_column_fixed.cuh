// Column-streaming kernel body of the fixed-point FP64 K.v (kv_fixed.cuh): one
// z-column of elements per thread, tiles, loaders and epilogues as in
// kv_column64.cuh.
//
// Per node layer the tile's nodes are copied asynchronously into a ring two
// layers ahead; the thread that copied a node converts it (masked, combined)
// to fixed point with its components' exponents in shared memory.  A barrier later
// every column forms its face modes from four nodes, its element from two
// faces, and leaves three of its four node shares in shared memory, where the
// nodes' owners add them a layer later.  One barrier per layer.
#pragma once
#include "kv_column64.cuh"
#include "kv_fixed.cuh"

// The node layers of a tile of CX x CY element columns in fixed point, streamed
// along z.  OWN: the FP64 values are kept as well, for the node's owner.  fixed
// NULL: no masks.
template <int CX, int CY, typename Load, bool OWN>
struct FixStream {
  using S = Col64Shape<CX, CY>;
  static constexpr int NT = S::NT, NX = S::NX, NV = S::NV, KS = Load::kSrc;
  static constexpr int kRing = 2 * 3 * KS * NV;              // doubles, slot of layer k: k & 1
  static constexpr int kNodes = 2 * 3 * NV;                  // int64, slot k & 1
  static constexpr int kOwn = OWN ? 4 * 3 * NV : 0;          // doubles, slot k & 3
  static constexpr int kExp = 4 * NV;                        // uint2, slot k & 3
  static constexpr int kWords = kRing + kNodes + kOwn;       // 8-byte words
  static_assert(NV > NT && NV <= 2 * NT, "two nodes at most per thread and layer");

  double* ring;
  int64_t* nodes;
  double* ownv;
  uint2* nexp;              // exponents (x | y << 16, z) and the mask (<< 16)
  const Load& ld;
  const uint8_t* fixed;
  int last, nxy, q, left;
  bool in[2], second;
  int node0[2];             // the nodes this thread stages: tid and tid + NT of the tile's

  // words, exps: shared memory; (i0, j0): node of the tile's corner; last
  // layer: the topmost to copy; k: the operator's FixOp::k
  __device__ __forceinline__ FixStream(double* words, uint2* exps, const Load& load,
                                       const uint8_t* fix, const Grid& g, int i0, int j0,
                                       int last_layer, int k)
      : ring(words), nodes(reinterpret_cast<int64_t*>(words + kRing)),
        ownv(words + kRing + kNodes), nexp(exps), ld(load), fixed(fix) {
    const int tid = threadIdx.x;
    last = min(last_layer, g.nz - 1);
    nxy = g.nx * g.ny;
    q = tid / CX * NX + tid % CX;       // the column's first node
    left = 4 - k;
    second = tid + NT < NV;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int t = tid + p * NT, ni = i0 + t % NX, nj = j0 + t / NX;
      in[p] = t < NV && ni >= 0 && nj >= 0 && ni < g.nx && nj < g.ny;
      node0[p] = in[p] ? ni + g.nx * nj : 0;
    }
  }

  // copies node layer L into its ring slot; the masks of the thread's nodes
  __device__ __forceinline__ uint32_t issue(int L) {
    const bool lay = L >= 0 && L <= last;
    uint32_t fm = 0;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (p == 1 && !second) break;
      const bool ok = in[p] && lay;
      const int n = ok ? node0[p] + nxy * L : 0;
      double* R = ring + (L & 1) * 3 * KS * NV + threadIdx.x + p * NT;
#pragma unroll
      for (int s = 0; s < KS; ++s)
#pragma unroll
        for (int c = 0; c < 3; ++c) col64_cp8(R + (3 * s + c) * NV, ld.src(s) + 3 * n + c, ok);
      if (ok && fixed != nullptr) fm |= (uint32_t)fixed[n] << (8 * p);
    }
    col64_commit();
    return fm;
  }

  // node layer L (its copies have landed) in fixed point
  __device__ __forceinline__ void stage(int L, uint32_t masks) {
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      if (p == 1 && !second) break;
      const int t = threadIdx.x + p * NT;
      const uint32_t fm = (masks >> (8 * p)) & 0xffu;
      const double* R = ring + (L & 1) * 3 * KS * NV + t;
      double v[3];
      uint32_t e[3];
      int64_t* N = nodes + (L & 1) * 3 * NV + t;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        double r[KS];
#pragma unroll
        for (int s = 0; s < KS; ++s) r[s] = R[(3 * s + c) * NV];
        v[c] = ((fm >> c) & 1) ? 0.0 : ld.combine(r);
        const int hi = __double2hiint(v[c]) & 0x7fffffff;
        const bool finite = hi < 0x7ff00000, zero = (hi | __double2loint(v[c])) == 0;
        e[c] = zero ? 0u : finite ? (uint32_t)max(hi >> 20, 1) : (uint32_t)kFixNan;
        N[c * NV] = finite ? fix_value((uint64_t)__double_as_longlong(v[c]), left) : 0ll;
      }
      const int slot = L & 3;
      nexp[slot * NV + t] = make_uint2(e[0] | e[1] << 16, e[2] | fm << 16);
      if constexpr (OWN) {
#pragma unroll
        for (int c = 0; c < 3; ++c) ownv[(slot * 3 + c) * NV + t] = v[c];
      }
    }
  }

  // face modes of node layer L, a barrier after its stage()
  __device__ __forceinline__ void face(int L, FixFace& F) const {
    const int64_t* N = nodes + (L & 1) * 3 * NV + q;
    const uint2* X = nexp + (L & 3) * NV + q;
    constexpr int at[4] = {0, 1, NX, NX + 1};
    uint2 e[4];
#pragma unroll
    for (int n = 0; n < 4; ++n) e[n] = X[at[n]];
    // 16-bit lanes: none borrows below, as none exceeds its maximum
    F.e.xy = fix_max_lanes(fix_max_lanes(e[0].x, e[1].x), fix_max_lanes(e[2].x, e[3].x));
    F.e.z = fix_max_lanes(fix_max_lanes(e[0].y, e[1].y), fix_max_lanes(e[2].y, e[3].y));
    int64_t v[4][3];
#pragma unroll
    for (int n = 0; n < 4; ++n) {
      const uint32_t dx = F.e.xy - e[n].x, dy = F.e.z - e[n].y;
      v[n][0] = fix_sar(N[at[n]], (int)(dx & 0xffffu));
      v[n][1] = fix_sar(N[NV + at[n]], (int)(dx >> 16));
      v[n][2] = fix_sar(N[2 * NV + at[n]], (int)(dy & 0xffffu));
    }
    fix_face(v, F);
  }
};

// Threads an SM holds at the K.v's launch bounds (at most 128 registers).  The
// upper outputs of the element below wait in shared memory, each thread's own
// (24 registers): 31 us at 120 x 60 x 30, against 33 with 12 warps of 168 (52 both
// at 55 x 55 x 165).
constexpr int kFixThreads = 512;

// Shared memory of the K.v: the stream, the shares of the other columns' nodes
// and their exponents (slot of layer k: k & 1).
template <int CX, int CY, typename Load, typename Epi>
struct FixShape {
  using St = FixStream<CX, CY, Load, Epi::kOwn>;
  static constexpr int kUp = 12 * St::NT;   // int64, upper outputs of the element below
  static constexpr int kBack = 2 * 9 * St::NT, kBackExp = 2 * St::NT;
  static constexpr size_t kBytes =
      8 * (size_t)(St::kWords + kBack + kUp + St::kExp) + 4 * (size_t)kBackExp;
};

// d 2^t times the operator's unit.
__device__ __forceinline__ double fix_scaled(double d, int t, const FixOp& K) {
  const int hi = __double2hiint(K.scale), lo = __double2loint(K.scale);
  const int eb = (hi >> 20) + t;
  if (eb >= 1 && eb <= 2046) return d * __hiloint2double(hi + t * (1 << 20), lo);
  const int t1 = fix_max(-2040, fix_min(2040, t)), half = t1 / 2;   // near FP64's ends
  return d * K.scale * __hiloint2double((1023 + half) << 20, 0) *
         __hiloint2double((1023 + t1 - half) << 20, 0);
}

// Tile `tile` of `tl`; returns this thread's share of the epilogue reduction.
// Iteration ez (element layer ez, between node layers ez and ez + 1) stages
// node layer ez + 1, crosses the layer's barrier, finishes node layer ez - 1
// and computes element layer ez.
template <int CX, int CY, typename Load, typename Epi>
__device__ __forceinline__ double kv_column_fixed_body(const double* __restrict__ E,
                                                       const uint8_t* __restrict__ fixed,
                                                       const FixOp& K, const Grid& g,
                                                       const Col64Tiling& tl, int tile,
                                                       const Load& ld, const Epi& epi,
                                                       double* smem) {
  using S = Col64Shape<CX, CY>;
  using L = FixShape<CX, CY, Load, Epi>;
  using St = typename L::St;
  constexpr int NT = St::NT;
  int64_t* back = reinterpret_cast<int64_t*>(smem + St::kWords);
  int64_t* ups = back + L::kBack + threadIdx.x;
  uint2* nexp = reinterpret_cast<uint2*>(back + L::kBack + L::kUp);
  int* bexp = reinterpret_cast<int*>(nexp + St::kExp);

  const int tid = threadIdx.x;
  const int bx = tile % tl.tx, by = (tile / tl.tx) % tl.ty, bz = tile / (tl.tx * tl.ty);
  const int kb = bz * tl.nzc, ke = min(kb + tl.nzc, g.nz);        // owned node layers [kb, ke)
  const int i0 = bx * S::OX - 1, j0 = by * S::OY - 1;             // node of the tile's corner
  const int nxy = g.nx * g.ny, nexy = g.nelx * g.nely;
  const int ex = tid % CX, ey = tid / CX, gi = i0 + ex, gj = j0 + ey;
  const bool elem_in = gi >= 0 && gj >= 0 && gi < g.nelx && gj < g.nely;
  const bool own_node = ex >= 1 && ey >= 1 && gi < g.nx && gj < g.ny;
  const bool warp_elem = __any_sync(0xffffffffu, elem_in);
  double red = 0.0;
  St st(smem, nexp, ld, fixed, g, i0, j0, ke, K.k);

  int64_t front[3] = {0, 0, 0};         // this column's share of its own node
  int front_e = kFixEmpty;
  // owner's sum of node layer k: the shares of the columns at (x - 1, y),
  // (x, y - 1), (x - 1, y - 1) and its own
  auto finish = [&](int k) {
    if (!own_node) return;
    const int64_t* Bk = back + (k & 1) * 9 * NT + tid;
    const int* Be = bexp + (k & 1) * NT + tid;
    const int e0 = Be[-1], e1 = Be[-CX], e2 = Be[-CX - 1];
    const int em = max(max(front_e, e0), max(e1, e2));
    // one bit of headroom for the sum of four
    const int df = min(em - front_e, 62) + 1, d0 = min(em - e0, 62) + 1,
              d1 = min(em - e1, 62) + 1, d2 = min(em - e2, 62) + 1;
    double acc[3], pn[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int64_t s = (front[c] >> df) + (Bk[c * NT - 1] >> d0) +
                        (Bk[(3 + c) * NT - CX] >> d1) + (Bk[(6 + c) * NT - CX - 1] >> d2);
      acc[c] = em >= kFixNanOut ? __longlong_as_double(0x7ff8000000000000ll)
                               : fix_scaled(__ll2double_rn(s), em - 2098 + K.k, K);
    }
    const int slot = k & 3;
    const uint32_t fm = nexp[slot * St::NV + st.q].y >> 16;
    if constexpr (Epi::kOwn) {
#pragma unroll
      for (int c = 0; c < 3; ++c) pn[c] = st.ownv[(slot * 3 + c) * St::NV + st.q];
    }
    epi(gi + g.nx * gj + nxy * k, acc, pn, (uint8_t)fm, red);
  };

  // a warp without elements contributes nothing
  if (!warp_elem) {
#pragma unroll
    for (int s = 0; s < 2; ++s) {
#pragma unroll
      for (int i = 0; i < 9; ++i) back[(s * 9 + i) * NT + tid] = 0;
      bexp[s * NT + tid] = kFixEmpty;
    }
  }
  uint32_t fm_cur = st.issue(kb - 1), fm_next = st.issue(kb);
  col64_wait<1>();
  st.stage(kb - 1, fm_cur);
  uint32_t fm_load = st.issue(kb + 1);
  auto load_modulus = [&](int ez) -> uint64_t {
    return elem_in && ez >= 0 && ez < g.nelz && ez < ke
               ? (uint64_t)__double_as_longlong(E[gi + g.nelx * gj + nexy * ez])
               : 0ull;
  };
  uint64_t Ebits = load_modulus(kb - 1);
  __syncthreads();
  FixFace F0, F1;
  FixOut U;
  if (warp_elem) st.face(kb - 1, F0);
  auto clear = [&]() {
    U.e = kFixEmpty;
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
      for (int f = 0; f < 4; ++f) U.m[c][f] = 0;
#pragma unroll
    for (int i = 0; i < 12; ++i) ups[i * NT] = 0;
  };
  clear();
  // one element layer: Flo the face modes of node layer ez (in), Fup those of
  // ez + 1 (out)
  auto layer = [&](int ez, const FixFace& Flo, FixFace& Fup) {
    const uint64_t Enext = load_modulus(ez + 1);
    // node layer ez + 1 has landed: its conversion, then the copies of ez + 3
    // into the ring slot it leaves
    col64_wait<1>();
    st.stage(ez + 1, fm_next);
    const uint32_t fm_new = st.issue(ez + 3);
    __syncthreads();
    if (ez - 1 >= kb) finish(ez - 1);
    if (warp_elem) {
      st.face(ez + 1, Fup);
      FixOut Ms;
      if (ez >= 0 && ez < g.nelz) {
        int64_t X[3][8], Z[3][8];
        const FixExp e{fix_max_lanes(Flo.e.xy, Fup.e.xy), fix_max_lanes(Flo.e.z, Fup.e.z)};
        const bool nan = fix_nan(e);
        const int t = fix_modes(Flo, Fup, e, __any_sync(0xffffffffu, fix_apart(e, K.k)), K.k, X);
        // (by a vote: the answer is then formed here, before the operator needs the
        // modes' registers)
        const unsigned strained = __ballot_sync(0xffffffffu, fix_strained(X));
        const FixModulus Em = fix_modulus(Ebits);
        fix_operator(X, K, Em, Z);
        if (__any_sync(0xffffffffu, Em.negative)) {
#pragma unroll
          for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int m = 1; m < 8; ++m) Z[c][m] = Em.negative ? -Z[c][m] : Z[c][m];
        }
        // a block that holds nothing shifts no neighbour's bits away
        const bool any = (strained >> (tid & 31)) & 1u;
        const int eo = nan || Em.e == 0x7ff ? (elem_in ? kFixNanOut : kFixEmpty)
                       : Em.f62 == 0 || !any         ? kFixEmpty
                                                     : t + Em.e;
#pragma unroll
        for (int i = 0; i < 12; ++i) U.m[i / 4][i % 4] = ups[i * NT];
        fix_join(Z, eo, U, Ms);
#pragma unroll
        for (int i = 0; i < 12; ++i) ups[i * NT] = U.m[i / 4][i % 4];
      } else {   // below or above the mesh: no element layer
#pragma unroll
        for (int i = 0; i < 12; ++i) U.m[i / 4][i % 4] = ups[i * NT];
        Ms = U;
        clear();
      }
      int64_t w[4][3];
      fix_corners(Ms, w);
      int64_t* Bk = back + (ez & 1) * 9 * NT + tid;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        front[c] = w[0][c];
        Bk[c * NT] = w[1][c];
        Bk[(3 + c) * NT] = w[2][c];
        Bk[(6 + c) * NT] = w[3][c];
      }
      front_e = Ms.e;
      bexp[(ez & 1) * NT + tid] = Ms.e;
    }
    fm_next = fm_load;
    fm_load = fm_new;
    Ebits = Enext;
  };
  for (int ez = kb - 1; ez < ke; ez += 2) {
    layer(ez, F0, F1);
    if (ez + 1 < ke) layer(ez + 1, F1, F0);
  }
  __syncthreads();
  finish(ke - 1);
  col64_wait<0>();
  return red;
}

// Tile shape and z-chunk: an SM's resident CTAs advance a layer in about 1.28 +
// 0.00625 us per thread (measured, with one exponent for all components; now a
// tenth more of both: the integer pipes are half busy at 16
// warps, so a layer's latency counts as much as its work), a CTA takes its
// layers and about 1.3 more, and the SM with the most CTAs sets the time.
// copies: launches' worth of tiles in one grid.
static inline void fixed_choose(int nx, int ny, int nz, int num_sms, int* shape_out, int* nzc_out,
                                int copies = 1) {
  double best = 0.0;
  bool best_fits = false;
  for (int i = 0; i < kCol64Shapes; ++i)
    col64_dispatch(i, [&](auto shape) -> mfto_status {
      using S = decltype(shape);
      const int64_t txy = (int64_t)((nx + S::OX - 1) / S::OX) * ((ny + S::OY - 1) / S::OY);
      for (int tz = 1; tz <= nz; ++tz) {
        const int nzc = (nz + tz - 1) / tz;
        if ((nz + nzc - 1) / nzc != tz) continue;          // not a balanced count
        const bool fits = txy * tz <= MFTO_RED_SLOTS;       // one partial per CTA, first choice
        if (!fits && tz > 1) break;
        constexpr int resident = kFixThreads / S::NT;
        const int64_t ctas = (txy * tz * copies + num_sms - 1) / num_sms;
        const int64_t sets = ctas / resident, rest = ctas % resident;
        auto layer = [](int64_t n) { return n == 0 ? 0.0 : 1.28 + 0.00625 * (double)(n * S::NT); };
        // larger CTAs wait longer at their barriers
        const double cost = ((double)sets * layer(resident) + layer(rest)) * (nzc + 1.3) *
                            (S::NT > 128 ? 1.05 : 1.0);
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
