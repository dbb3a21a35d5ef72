// Weight and bias gradients of a 3x3x3 convolution on the FP32 FMA pipe:
//   dW[co][ci][k] = sum_v g[co][v] x[ci][v + d_k],   db[co] = sum_v g[co][v].
//
// A contraction over voxels with 27 shifted copies of x.  A thread owns one
// (ci, dz, dy) and CO output channels: walking along x it reads one x value per
// step (the three dx are a sliding window in registers) and CO gradient values
// that the whole warp shares (vector loads, broadcast), for 3 CO multiply-adds
// as packed pairs.  With CO = 14 that is 42 per 5 shared-memory reads, so the
// kernel is bound by the FMA pipe, where one block per (co, ci) re-read both
// operands from L1 for every product.  One extra "pair" with x = 1 gives the
// bias gradient.
//
// A block covers 128 (ci, dz, dy) pairs, CO output channels and one task: a
// range of units, each a segment of at most kWgX voxels of kWgRows consecutive
// y rows of one z plane.  The x rows of y - 1 .. y + 2 sit in a
// ring of four slots filled by asynchronous copies one row ahead.  Sums run in
// a fixed order: along a row into one set of accumulators, rows into a second
// set, tasks by wgrad_sum -- short chains, so that the rounding stays below
// that of the products' inputs.  Measured on a GB300, 72 x 40 x 40 voxels, 14 to 14
// channels: 48 against 389 us; all 14 layers of a gradient 0.58 against 3.9 ms (0.60 with
// three CTAs per SM).
#pragma once

constexpr int kWgX = 62;           // voxels of a row segment (with its halo: two warp passes)
constexpr int kWgCi = 16;          // input channels that 128 pairs can touch
constexpr int kWgRows = 8;         // y rows of a unit
constexpr int kWgG = 16;           // staged gradient values per voxel

struct WgradPlan {
  int pairs, pblocks, cblocks;     // 9 Cin + 1 pairs; blocks of 128 pairs and CO channels
  int xtiles, xt, yblocks, units;  // row segments and their length; row blocks per z; units
  int per_task, tasks;             // units per task; tasks
  int pitch;                       // floats of a staged x row: odd, lanes read different rows
};

// shared memory of segments of xt voxels, and the CTAs an SM holds with it (four
// by the registers; segments of 39 voxels and more: three)
__host__ __device__ constexpr int wg_pitch(int xt) { return (xt + 2) | 1; }
constexpr size_t wg_smem_bytes(int xt) {
  return sizeof(float) * (size_t)(kWgCi * 3 * 4 * wg_pitch(xt) + 2 * xt * kWgG);
}
constexpr int wg_per_sm(int xt) {
  const int fit = (int)(227 * 1024 / (wg_smem_bytes(xt) + 1024));
  return fit < 4 ? fit : 4;
}

__device__ __forceinline__ void wg_cp4(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src),
               "r"(valid ? 4 : 0)
               : "memory");
}

template <int CO>
__global__ void __launch_bounds__(128, 4)
wgrad3(const float* __restrict__ in, int Cin, const float* __restrict__ dout, int Cout, Dims d,
       WgradPlan pl, float* __restrict__ partial) {
  static_assert(CO % 2 == 0 && CO <= kWgG, "pairs of output channels");
  extern __shared__ __align__(16) float wg_smem[];
  const int pitch = pl.pitch, gstep = pl.xt * kWgG;
  float* gs = wg_smem;                              // [2][xt][kWgG]
  float* xs = wg_smem + 2 * gstep;                  // [kWgCi][3][4 slots][pitch]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int pb = blockIdx.x % pl.pblocks, cb = blockIdx.x / pl.pblocks;
  const int co0 = cb * CO, c0 = pb * 128 / 9;
  int x0 = 0, xn = 0;                               // the current row segment
  const size_t V = (size_t)d.V();
  // this thread's pair
  const int p = pb * 128 + tid;
  const bool is_bias = p == 9 * Cin, live = p < 9 * Cin;
  const int ci = live ? p / 9 - c0 : 0, k9 = live ? p % 9 : 0;
  const int dz = k9 / 3, dy = k9 % 3;
  const float* xrow = xs + (ci * 3 + dz) * 4 * pitch;

  // copies of x row y (planes z - 1 .. z + 1, this block's channels) into slot
  // y & 3, and of gradient row yg into buffer yg & 1 (zero outside the grid)
  auto load_x = [&](int z, int y) {
    const int nrow = 3 * kWgCi;
    for (int r = warp; r < nrow; r += 4) {
      const int c = r / 3, zz = z - 1 + (r - 3 * c);
      const bool row_in = c0 + c < Cin && zz >= 0 && zz < d.D && y >= 0 && y < d.H;
      const float* src = in + (size_t)(row_in ? c0 + c : 0) * V +
                         (row_in ? ((size_t)zz * d.H + y) * d.W : 0);
      float* dst = xs + (r * 4 + (y & 3)) * pitch;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h, x = x0 - 1 + i;
        if (i < pl.xt + 2) {
          const bool ok = row_in && x >= 0 && x < d.W;
          wg_cp4(dst + i, src + (ok ? x : 0), ok);
        }
      }
    }
  };
  auto load_g = [&](int z, int y) {
    float* dst = gs + (y & 1) * gstep;
    for (int j = warp; j < CO; j += 4) {
      const bool row_in = co0 + j < Cout && y < d.H;
      const float* src = dout + (size_t)(row_in ? co0 + j : 0) * V +
                         (row_in ? ((size_t)z * d.H + y) * d.W : 0);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = lane + 32 * h;
        if (i < pl.xt) {
          const bool ok = row_in && i < xn;
          wg_cp4(dst + i * kWgG + j, src + (ok ? x0 + i : 0), ok);
        }
      }
    }
  };
  auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };

  float2 tot[CO / 2][3];
#pragma unroll
  for (int j = 0; j < CO / 2; ++j)
#pragma unroll
    for (int q = 0; q < 3; ++q) tot[j][q] = make_float2(0.f, 0.f);

  const int u1 = min(pl.units, ((int)blockIdx.y + 1) * pl.per_task);
  for (int u = blockIdx.y * pl.per_task; u < u1; ++u) {
    const int zy = u / pl.xtiles, z = zy / pl.yblocks;
    const int ya = (zy % pl.yblocks) * kWgRows, yb = min(ya + kWgRows, d.H);
    x0 = (u % pl.xtiles) * pl.xt;
    xn = min(pl.xt, d.W - x0);
    __syncthreads();              // the previous row block's reads are done
    load_x(z, ya - 1);
    load_x(z, ya);
    load_x(z, ya + 1);
    load_g(z, ya);
    commit();
    for (int y = ya; y < yb; ++y) {
      if (y + 1 < yb) {
        load_x(z, y + 2);
        load_g(z, y + 1);
      }
      commit();
      asm volatile("cp.async.wait_group 1;\n" ::: "memory");
      __syncthreads();
      const float* xr = xrow + ((y - 1 + dy) & 3) * pitch;
      const float* gr = gs + (y & 1) * gstep;
      float2 acc[CO / 2][3];
#pragma unroll
      for (int j = 0; j < CO / 2; ++j)
#pragma unroll
        for (int q = 0; q < 3; ++q) acc[j][q] = make_float2(0.f, 0.f);
      float xm = is_bias ? 1.f : xr[0], xc = is_bias ? 1.f : xr[1];
#pragma unroll 2
      for (int x = 0; x < xn; ++x) {
        const float xp = is_bias ? 1.f : xr[x + 2];
        float g[kWgG];
#pragma unroll
        for (int j = 0; j < (CO + 3) / 4; ++j)
          *reinterpret_cast<float4*>(g + 4 * j) =
              *reinterpret_cast<const float4*>(gr + x * kWgG + 4 * j);
        const float2 m2 = make_float2(xm, xm), c2 = make_float2(xc, xc), p2 = make_float2(xp, xp);
#pragma unroll
        for (int j = 0; j < CO / 2; ++j) {
          const float2 gj = make_float2(g[2 * j], g[2 * j + 1]);
          acc[j][0] = __ffma2_rn(gj, m2, acc[j][0]);
          acc[j][1] = __ffma2_rn(gj, c2, acc[j][1]);
          acc[j][2] = __ffma2_rn(gj, p2, acc[j][2]);
        }
        xm = xc;
        xc = xp;
      }
#pragma unroll
      for (int j = 0; j < CO / 2; ++j)
#pragma unroll
        for (int q = 0; q < 3; ++q) tot[j][q] = __fadd2_rn(tot[j][q], acc[j][q]);
      __syncthreads();            // row y - 1's slot and this gradient row are free
    }
  }
  if (!live && !is_bias) return;
  // partial[task][co][3 p + dx]
  float* out = partial + (size_t)blockIdx.y * Cout * pl.pairs * 3 + 3 * p;
#pragma unroll
  for (int j = 0; j < CO; ++j)
    if (co0 + j < Cout) {
      float* o = out + (size_t)(co0 + j) * pl.pairs * 3;
#pragma unroll
      for (int q = 0; q < 3; ++q) o[q] = (j & 1) ? tot[j / 2][q].y : tot[j / 2][q].x;
    }
}

// gw, gb = sums of the tasks' partials, by threads (i, s): thread s of 8 adds
// every eighth task, then the 8 in a tree
__global__ void __launch_bounds__(256)
wgrad_sum(const float* __restrict__ partial, int Cin, int Cout, WgradPlan pl,
          float* __restrict__ gw, float* __restrict__ gb) {
  __shared__ float sh[8][33];
  const int i = blockIdx.x * 32 + (threadIdx.x & 31), s = threadIdx.x >> 5;
  const int row = pl.pairs * 3, n = Cout * row, tasks = pl.tasks;
  float v = 0.f;
  if (i < n)
    for (int t = s; t < tasks; t += 8) v += partial[(size_t)t * n + i];
  sh[s][threadIdx.x & 31] = v;
  __syncthreads();
  if (s != 0 || i >= n) return;
  const int l = threadIdx.x;
  const float a = (sh[0][l] + sh[1][l]) + (sh[2][l] + sh[3][l]);
  const float b = (sh[4][l] + sh[5][l]) + (sh[6][l] + sh[7][l]);
  const int co = i / row, q = i % row;
  if (q < 27 * Cin) gw[(size_t)co * 27 * Cin + q] = a + b;
  else if (q == 27 * Cin + 1) gb[co] = a + b;   // the x = 1 pair, dx = 0
}

// Tasks of a layer: units grouped into one wave of blocks, as far as the
// partials (max_partial floats) allow.
static inline WgradPlan wgrad_plan(int Cin, int Cout, const Dims& d, int co, int num_sms,
                                   size_t max_partial) {
  WgradPlan p;
  p.pairs = 9 * Cin + 1;
  p.pblocks = (p.pairs + 127) / 128;
  p.cblocks = (Cout + co - 1) / co;
  p.xtiles = (d.W + kWgX - 1) / kWgX;
  p.xt = (d.W + p.xtiles - 1) / p.xtiles;
  p.pitch = wg_pitch(p.xt);
  p.yblocks = (d.H + kWgRows - 1) / kWgRows;
  p.units = d.D * p.yblocks * p.xtiles;
  const size_t one = (size_t)Cout * p.pairs * 3;   // partials of one task
  long long tasks = (long long)wg_per_sm(p.xt) * num_sms / ((long long)p.pblocks * p.cblocks);
  if (tasks > (long long)(max_partial / one)) tasks = (long long)(max_partial / one);
  if (tasks < 1) tasks = 1;
  if (tasks > p.units) tasks = p.units;
  p.per_task = (int)((p.units + tasks - 1) / tasks);
  p.tasks = (p.units + p.per_task - 1) / p.per_task;
  return p;
}
