// Inner FP32 CG of a batch: two kernels per iteration over all instances, and
// no grid-wide step.
//
//   A(k)  K.v: a CTA sums its instance's shares of r.z and r.r left by B(k-1),
//         decides convergence, forms beta, then p = z + beta p_old, q = K p and
//         its share of p.q;
//   B(k)  update: a CTA sums its instance's shares of p.q, forms alpha,
//         updates u, r, z and leaves its shares of r.z and r.r.
// Every CTA of an instance sums the same shares in the same order and takes the
// same decisions; the instance's first one records them.  Scalars are double
// buffered by the iteration's parity.  CTAs of finished instances end at once.
//
// A streams z-columns of elements like kv_column.cuh, on tiles that fit small
// meshes: a CTA of 256 threads covers whole rows of nodes (pitch w, all of x
// where the mesh is at most 64 nodes wide), so there is no halo along x, one
// halo row along y, and few idle lanes; the last node of a row has no element
// and contributes nothing, so that the columns left of a row's first node need
// no test.
//
// Bound by the FP32 work and shared-memory traffic of A (its element layers
// stream as in kv_column.cuh) and by L2 bandwidth in B.  Measured on a GB300, 64
// instances of 16 x 8 x 8 to 48 x 24 x 24: A 24 and B 9.5 us per iteration, against
// 45 us of 8 x 8 x 4 element blocks that recompute 1.7 times their nodes'
// elements and end in a grid-wide ticket, and 36 us of an update that did so
// too, one CTA summing every instance's shares while the others idled.
#pragma once
#include "common.cuh"
#include "kv_column.cuh"

constexpr int kBatchRow = 64;                           // widest row of nodes
constexpr int kBatchNodes = MFTO_BLOCK + kBatchRow + 2; // staged nodes of a layer, at most
constexpr int kBatchSums = MFTO_BLOCK + 1;              // column sums, one (zero) in front
constexpr int kBatchUpdate = 1024;                      // DOFs of an update CTA
constexpr int kBatchLayer = 3 * kBatchNodes;            // floats of a staged layer
constexpr int kBatchPerSm = 2;                          // CTAs of A (three: registers spill)

// The tiles of an instance (bx + ntx (by + nty bz), from tile0): rows of
// pitch w, `rows` of them (the first a halo), ow owned nodes along x from
// column c0 on.
struct BatchTiles {
  int tile0, ntile, ntx, nty, nzc;
  int w, c0, ow, rows;
  int up0, nup;              // update CTAs
};

struct BatchScal {
  double rz, pq, alpha, beta, rr, ff, rtol2ff;
  int32_t it, done, status, pad;
};

// The dot products: a warp's sums as FP32 pairs (DotAcc<float>), from there on in
// FP64, where the chains of dependent operations are what they cost (an FP64
// instruction takes a warp 64 clocks): a lane per row and warp, short trees.
//
// Sums of an instance's n shares in K (1 or 2) rows `stride` apart, fixed order,
// by 32 / K lanes of the calling warp each; all its lanes get them.
template <int K>
__device__ __forceinline__ void batch_sum(const double* part, int stride, int n,
                                          double (&out)[K]) {
  constexpr int W = 32 / K;
  const int lane = threadIdx.x & 31;
  const double* row = part + lane / W * stride;
  double t = 0.0;
  for (int b = lane % W; b < n; b += W) t += row[b];
#pragma unroll
  for (int o = W / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
#pragma unroll
  for (int c = 0; c < K; ++c) out[c] = __shfl_sync(0xffffffffu, t, c * W);
}

// The block's sums of K double-float values held by lane 0 of each warp, in FP64,
// as share `at` of its rows.
template <int K>
__device__ __forceinline__ void batch_publish(const DFloat (&v)[K], double* part, int stride,
                                              int at) {
  constexpr int W = MFTO_BLOCK / 32;
  __shared__ float2 sh[K * W];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
#pragma unroll
    for (int c = 0; c < K; ++c) sh[c * W + warp] = make_float2(v[c].hi, v[c].lo);
  }
  __syncthreads();
  if (warp == 0) {
    const float2 x = sh[lane % (K * W)];
    double t = (double)x.x + (double)x.y;
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane < K * W && lane % W == 0) part[lane / W * stride + at] = t;
  }
}

// face modes of one layer from its staged nodes, pitch w
__device__ __forceinline__ void batch_face(const float* layer, int at, int w, ColFace& F) {
  const float2* Lxy = reinterpret_cast<const float2*>(layer) + at;
  const float* Lz = layer + 2 * kBatchNodes + at;
  const float2 c0 = Lxy[0], c1 = Lxy[1], c2 = Lxy[w], c3 = Lxy[w + 1];
  const float2 m0 = add2(c0, c1), m1 = sub2(c1, c0), m2 = add2(c2, c3), m3 = sub2(c3, c2);
  F.xy[0] = add2(m0, m2);
  F.xy[2] = sub2(m2, m0);
  F.xy[1] = add2(m1, m3);
  F.xy[3] = sub2(m3, m1);
  const float z0 = Lz[0], z1 = Lz[1], z2 = Lz[w], z3 = Lz[w + 1];
  const float n0 = z0 + z1, n1 = z1 - z0, n2 = z2 + z3, n3 = z3 - z2;
  F.z[0] = n0 + n2;
  F.z[2] = n2 - n0;
  F.z[1] = n1 + n3;
  F.z[3] = n3 - n1;
}

struct BatchCgArgs {
  const float* E;
  const float* z;
  const float* p_old;
  float* p_new;
  float* q;
  const uint8_t* fixed;
  const BatchInst* inst;
  const BatchTiles* tiles;
  const int* tile_inst;       // instance of a tile
  const BatchScal* prev;      // scalars of iteration k - 1
  BatchScal* cur;             // ... and k
  const double* part_b;       // r.z and r.r of the update CTAs, rows n_update apart
  double* part_a;             // p.q of the tiles
  int n_update, maxit;
  double rtol2;
};

// shared memory of A: three staged layers, the ring of source values, sums
constexpr int kBatchRingFloats = 3 * 6 * kBatchNodes;
constexpr int kBatchSumFloats = 2 * 12 * kBatchSums;
constexpr size_t kBatchCgSmem =
    sizeof(float) * (size_t)(3 * kBatchLayer + kBatchRingFloats + kBatchSumFloats);
static_assert(kBatchLayer % 2 == 0 && kBatchNodes % 2 == 0 && kBatchRingFloats % 2 == 0,
              "pairs are 8-byte aligned");

__global__ void __launch_bounds__(MFTO_BLOCK, kBatchPerSm)
batch_cg_kv(BatchCgArgs a, ModeCoef<float> K) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ float s_beta;
  __shared__ int s_skip;
  float* nodes = reinterpret_cast<float*>(smem_raw);   // slot of layer k: (k + 3) % 3
  float* ring = nodes + 3 * kBatchLayer;                // [3][6][kBatchNodes], slot (k + 3) % 3
  float* sums = ring + kBatchRingFloats;                // slot k & 1: 4 pairs, then 4 z
  const int tid = threadIdx.x;
  pdl_wait();
  const int i = a.tile_inst[blockIdx.x];
  const BatchTiles t = a.tiles[i];
  const BatchInst in = a.inst[i];
  const BatchScal scal = a.prev[i];
  const int lb = blockIdx.x - t.tile0;
  if (scal.done) {
    if (lb == 0 && tid == 0) a.cur[i] = scal;
    return;
  }
  const int bx = lb % t.ntx, by = (lb / t.ntx) % t.nty, bz = lb / (t.ntx * t.nty);
  const int w = t.w, nslot = t.rows * w;
  const int kb = bz * t.nzc, ke = min(kb + t.nzc, in.nz);   // owned node layers [kb, ke)
  const int x0 = bx * t.ow - t.c0, y0 = by * (t.rows - 1) - 1;
  const int ex = tid % w, ey = tid / w, gi = x0 + ex, gj = y0 + ey;
  const int nxy = in.nx * in.ny, nexy = in.nelx * in.nely;
  const bool own_in = tid < nslot && gi >= 0 && gi < in.nx && gj >= 0 && gj < in.ny;
  const bool elem_in = tid < nslot && ex + 1 < w && gi >= 0 && gi < in.nelx && gj >= 0 &&
                       gj < in.nely;
  const bool own_node = own_in && ey >= 1 && ex >= t.c0 && ex < t.c0 + t.ow;
  const bool warp_elem = __any_sync(0xffffffffu, elem_in);
  // the node row above the tile, staged by the first w threads
  const int hx = x0 + tid, hy = y0 + t.rows;
  const bool top = tid < w;
  const bool top_in = top && hx >= 0 && hx < in.nx && hy < in.ny;
  const int own_base = own_in ? gi + in.nx * gj : 0, top_base = top_in ? hx + in.nx * hy : 0;
  const int elem_base = elem_in ? gi + in.nelx * gj : 0;
  const float* zs = a.z + 3 * in.node_off;
  const float* ps = a.p_old + 3 * in.node_off;
  const float* Es = a.E + in.elem_off;
  const uint8_t* fx = a.fixed + in.node_off;
  const int last = min(ke, in.nz - 1);

  // copies of node layer L into ring slot rs; the masks of the own and the
  // top node (<< 8)
  auto issue = [&](int L, int rs) {
    const bool lay = L >= 0 && L <= last;
    uint32_t fm = 0;
    if (tid < nslot) {
      const bool ok = lay && own_in;
      const int n = ok ? own_base + nxy * L : 0;
      float* R = ring + rs * 6 * kBatchNodes + tid;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        col_cp4(R + c * kBatchNodes, zs + 3 * n + c, ok);
        col_cp4(R + (3 + c) * kBatchNodes, ps + 3 * n + c, ok);
      }
      if (ok) fm = fx[n];
    }
    if (top) {
      const bool ok = lay && top_in;
      const int n = ok ? top_base + nxy * L : 0;
      float* R = ring + rs * 6 * kBatchNodes + nslot + tid;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        col_cp4(R + c * kBatchNodes, zs + 3 * n + c, ok);
        col_cp4(R + (3 + c) * kBatchNodes, ps + 3 * n + c, ok);
      }
      if (ok) fm |= (uint32_t)fx[n] << 8;
    }
    col_cp_commit();
    return fm;
  };
  auto load_E = [&](int el) {
    return elem_in && el >= 0 && el < in.nelz && el < ke ? Es[elem_base + nexy * el] : 0.f;
  };
  const int first_slot = (kb + 2) % 3;                  // of node layer kb - 1
  auto next = [](int s) { return s == 2 ? 0 : s + 1; };
  uint32_t fm_prev = 0, fm_cur = issue(kb - 1, first_slot),
           fm_next = issue(kb, next(first_slot));
  uint32_t fm_load = issue(kb + 1, next(next(first_slot)));
  float Ecur = load_E(kb - 1);

  // beta, and whether the instance is done, by the first warp
  if (tid < 32) {
    double tot[2];
    batch_sum<2>(a.part_b + t.up0, a.n_update, t.nup, tot);
    if (tid == 0) {
      BatchScal o = scal;
      const int k = scal.it + 1;                        // iterations completed
      o.it = k;
      o.rz = tot[0];
      o.rr = tot[1];
      o.beta = tot[0] / scal.rz;
      if (k == 0) {
        o.ff = tot[1];
        o.rtol2ff = a.rtol2 * tot[1];
      }
      if (!isfinite(tot[0]) || !isfinite(tot[1])) {
        o.done = 1;
        o.status = MFTO_BREAKDOWN;
      } else if (tot[1] <= o.rtol2ff) {
        o.done = 1;
        o.status = MFTO_OK;
      } else if (k >= a.maxit) {
        o.done = 1;
        o.status = MFTO_NOT_CONVERGED;
      }
      if (lb == 0) a.cur[i] = o;
      s_skip = o.done;
      s_beta = (float)o.beta;
    }
  }
  // nothing may be read that no thread stages; the sums in front of column 0
  // and those of warps without elements stay zero
  for (int k = tid; k < 3 * kBatchLayer; k += MFTO_BLOCK) nodes[k] = 0.f;
  for (int k = tid; k < kBatchSumFloats; k += MFTO_BLOCK) sums[k] = 0.f;
  __syncthreads();
  if (s_skip) {
    col_cp_wait<0>();
    return;
  }
  const float beta = s_beta;
  auto put = [&](int slot, int at, uint32_t fm) {
    const float* R = ring + slot * 6 * kBatchNodes + at;
    float v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c)
      v[c] = ((fm >> c) & 1) ? 0.f : R[c * kBatchNodes] + beta * R[(3 + c) * kBatchNodes];
    float* N = nodes + slot * kBatchLayer;
    reinterpret_cast<float2*>(N)[at] = make_float2(v[0], v[1]);
    N[2 * kBatchNodes + at] = v[2];
  };
  auto stage = [&](int slot, uint32_t fm) {
    if (tid < nslot) put(slot, tid, fm & 0xffu);
    if (top) put(slot, nslot + tid, fm >> 8);
  };
  float* pn_out = a.p_new + 3 * in.node_off;
  float* q_out = a.q + 3 * in.node_off;
  DotAcc<float> acc;
  // owner's sum of node layer k (staged in `slot`): the columns at
  // (x - 1, y - 1), (x, y - 1), (x - 1, y), (x, y)
  auto finish = [&](int k, int slot, uint32_t fm) {
    if (!own_node) return;
    const float* S = sums + (k & 1) * 12 * kBatchSums;
    const float2* S2 = reinterpret_cast<const float2*>(S) + 1 + tid;
    const float* Sz = S + 8 * kBatchSums + 1 + tid;
    float2 s = S2[3 * kBatchSums - w - 1];
    s = add2(s, S2[2 * kBatchSums - w]);
    s = add2(s, S2[kBatchSums - 1]);
    s = add2(s, S2[0]);
    float sz = Sz[3 * kBatchSums - w - 1];
    sz += Sz[2 * kBatchSums - w];
    sz += Sz[kBatchSums - 1];
    sz += Sz[0];
    const float* N = nodes + slot * kBatchLayer;
    const float2 pxy = reinterpret_cast<const float2*>(N)[tid];
    const float pz = N[2 * kBatchNodes + tid];
    const int at = 3 * (own_base + nxy * k);
    const float q0 = (fm & 1) ? pxy.x : s.x, q1 = (fm & 2) ? pxy.y : s.y,
                q2 = (fm & 4) ? pz : sz;
    pn_out[at] = pxy.x;
    pn_out[at + 1] = pxy.y;
    pn_out[at + 2] = pz;
    q_out[at] = q0;
    q_out[at + 1] = q1;
    q_out[at + 2] = q2;
    acc.add(fmaf(pz, q2, fmaf(pxy.y, q1, pxy.x * q0)));
  };

  int sp = first_slot, sc = next(sp);                   // slots of layers ez and ez + 1
  col_cp_wait<2>();
  stage(sp, fm_cur);
  __syncthreads();
  ColFace F0, F1, U0, U1;
  face_zero(U0);
  face_zero(U1);
  if (warp_elem) batch_face(nodes + sp * kBatchLayer, tid, w, F0);
  fm_prev = fm_cur;
  // element layer ez: Flo the face modes of node layer ez (in), Fup of ez + 1
  // (out), upp the upper outputs of the element below (in), up this one's
  auto layer = [&](int ez, const ColFace& Flo, ColFace& Fup, const ColFace& upp, ColFace& up) {
    const float Ee = Ecur;
    Ecur = load_E(ez + 1);
    col_cp_wait<1>();
    stage(sc, fm_next);
    // layer ez + 3 into the ring slot of layer ez
    const uint32_t fm_new = issue(ez + 3, sp);
    __syncthreads();
    // slot of layer ez - 1: its nodes stay until layer ez + 2 is staged there
    if (ez - 1 >= kb) finish(ez - 1, next(sc), fm_prev & 0xffu);
    if (warp_elem) {
      batch_face(nodes + sc * kBatchLayer, tid, w, Fup);
      ColFace lo;
      col_element(Flo, Fup, Ee, K, lo, up);
      if (ez >= kb && tid < nslot) {
        ColFace Ms, Sc;
        face_add(upp, lo, Ms);
        face_inverse(Ms, Sc);
        float* S = sums + (ez & 1) * 12 * kBatchSums;
        float2* S2 = reinterpret_cast<float2*>(S) + 1 + tid;
        float* Sz = S + 8 * kBatchSums + 1 + tid;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          S2[c * kBatchSums] = Sc.xy[c];
          Sz[c * kBatchSums] = Sc.z[c];
        }
      }
    }
    fm_prev = fm_cur;
    fm_cur = fm_next;
    fm_next = fm_load;
    fm_load = fm_new;
    sp = sc;
    sc = next(sc);
  };
  for (int ez = kb - 1; ez < ke; ez += 2) {
    layer(ez, F0, F1, U0, U1);
    if (ez + 1 < ke) layer(ez + 1, F1, F0, U1, U0);
  }
  __syncthreads();
  finish(ke - 1, next(sc), fm_prev & 0xffu);
  col_cp_wait<0>();
  const DFloat v[1] = {acc.finish_df()};
  batch_publish<1>(v, a.part_a, 0, blockIdx.x);
}

// B: u += alpha p, r -= alpha q, z = r / d and the shares of r.z and r.r.
__global__ void __launch_bounds__(MFTO_BLOCK)
batch_cg_update(float* __restrict__ u, const float* __restrict__ p, const float* __restrict__ q,
                float* __restrict__ r, float* __restrict__ z, const float* __restrict__ dinv,
                const BatchInst* __restrict__ inst, const BatchTiles* __restrict__ tiles,
                const int* __restrict__ up_inst, BatchScal* sc, const double* part_a,
                double* part_b, int n_update) {
  constexpr int N = kBatchUpdate / MFTO_BLOCK;
  __shared__ float s_alpha;
  __shared__ int s_skip;
  pdl_wait();
  const int i = up_inst[blockIdx.x];
  const int up0 = tiles[i].up0;
  const int n = 3 * inst[i].nx * inst[i].ny * inst[i].nz;
  const long long o = 3 * inst[i].node_off;
  if (sc[i].done) return;
  const int k0 = (blockIdx.x - up0) * kBatchUpdate + threadIdx.x;
  float uu[N], pp[N], qq[N], rr[N], dd[N];
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int k = k0 + j * MFTO_BLOCK;
    const bool in = k < n;
    uu[j] = in ? u[o + k] : 0.f;
    pp[j] = in ? p[o + k] : 0.f;
    qq[j] = in ? q[o + k] : 0.f;
    rr[j] = in ? r[o + k] : 0.f;
    dd[j] = in ? dinv[o + k] : 0.f;
  }
  if (threadIdx.x < 32) {
    const double rz = sc[i].rz;
    double pq[1];
    batch_sum<1>(part_a + tiles[i].tile0, 0, tiles[i].ntile, pq);
    if (threadIdx.x == 0) {
      const bool broken = !(pq[0] > 0.0) || !isfinite(pq[0]);
      const double alpha = broken ? 0.0 : rz / pq[0];
      s_skip = broken;
      s_alpha = (float)alpha;
      if ((int)blockIdx.x == up0) {
        sc[i].pq = pq[0];
        sc[i].alpha = alpha;
        if (broken) {   // the instance's other CTAs come to the same end
          sc[i].status = MFTO_BREAKDOWN;
          sc[i].done = 1;
        }
      }
    }
  }
  __syncthreads();
  if (s_skip) return;
  const float alpha = s_alpha;
  DotAcc<float> d0, d1;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int k = k0 + j * MFTO_BLOCK;
    if (k >= n) continue;
    const float ri = rr[j] - alpha * qq[j];
    const float zi = ri * dd[j];
    u[o + k] = uu[j] + alpha * pp[j];
    r[o + k] = ri;
    z[o + k] = zi;
    d0.add_prod(ri, zi);
    d1.add_prod(ri, ri);
  }
  const DFloat v[2] = {d0.finish_df(), d1.finish_df()};
  batch_publish<2>(v, part_b, n_update, blockIdx.x);
}

// Inner solve start: z = r / d, the shares of r.z and r.r, and the scalars
// before iteration 0 (rz_prev > 0: the direction in p is continued).
__global__ void __launch_bounds__(MFTO_BLOCK)
batch_cg_start(const float* __restrict__ r, float* __restrict__ z, const float* __restrict__ dinv,
               const BatchInst* __restrict__ inst, const BatchTiles* __restrict__ tiles,
               const int* __restrict__ up_inst, BatchScal* sc, const double* __restrict__ rz_prev,
               double* part_b, int n_update) {
  const int i = up_inst[blockIdx.x];
  const int up0 = tiles[i].up0;
  const int n = 3 * inst[i].nx * inst[i].ny * inst[i].nz;
  const long long o = 3 * inst[i].node_off;
  DotAcc<float> d0, d1;
  for (int j = 0; j < kBatchUpdate / MFTO_BLOCK; ++j) {
    const int k = (blockIdx.x - up0) * kBatchUpdate + j * MFTO_BLOCK + threadIdx.x;
    if (k >= n) break;
    const float ri = r[o + k], zi = ri * dinv[o + k];
    z[o + k] = zi;
    d0.add_prod(ri, zi);
    d1.add_prod(ri, ri);
  }
  if (threadIdx.x == 0 && (int)blockIdx.x == up0) {
    BatchScal s{};
    s.rz = rz_prev[i] > 0.0 ? rz_prev[i] : INFINITY;   // beta = 0: p = z
    s.it = -1;
    sc[i] = s;
  }
  const DFloat v[2] = {d0.finish_df(), d1.finish_df()};
  batch_publish<2>(v, part_b, n_update, blockIdx.x);
}

// whether every instance is done, after a chunk of iterations
__global__ void __launch_bounds__(MFTO_BLOCK)
batch_cg_done(const BatchScal* sc, int count, int* all_done) {
  pdl_wait();
  int live = 0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) live |= !sc[i].done;
  live = __syncthreads_or(live);
  if (threadIdx.x == 0) *all_done = !live;
}
