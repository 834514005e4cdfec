// factrow.cuh -- the 2-D operator of eq. (Brinkman-weak) in FP64, applied with its
// tensor structure.
//
// The FP64 units (two FMAs per clock and SM) bound the operator in FP64, so what
// counts is the number of products per row.  Row by row the interior-penalty term
// multiplies every pair of a mass entry M along the component's direction and an
// entry of the penalty operator across it: 36 FP64 instructions per row for RT_1
// (320^2: 87 us, the units 89 % busy).  Here a thread takes one cell along the
// component's direction at one node across it: it applies the penalty operator to
// the cell's nodes first, Z = F u, and then
//   y_a = sum_b M_ab (c_K u_b + Z_b) + K_ab u_b + G_ba p_b,
// the cell's share of its K + 2 nodes; a face node adds the share of the cell before.
// Z of the first node and that share come from the neighbouring cell: of the next
// lane (component x, lanes = cells along x) or warp (component y, lanes = cells along
// x at the same position inside them, warps = cells along y).  The first two cells of
// a warp (of a block) only supply them: 24 instructions per row for RT_1, 59 us (the
// units 88 % busy).
#pragma once

#include "device.cuh"

namespace mgd {

constexpr int FR_WARPS = 16, FR_LANES = 30, FR_CELLS = FR_WARPS - 2;

// Blocks of the three parts (components x and y, pressure).
struct FactRowGrid {
  int bx[3];     // blocks along x (lanes)
  int64_t first[4];
};
template <int K>
inline FactRowGrid fact_row_grid(int n) {
  FactRowGrid g;
  const int64_t N = (int64_t)n * (K + 1);
  auto cd = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
  g.bx[0] = (int)cd(n + 1, FR_LANES);
  g.bx[1] = g.bx[2] = (int)cd(n, 32);
  g.first[0] = 0;
  g.first[1] = g.bx[0] * cd(N, FR_WARPS);
  g.first[2] = g.first[1] + (int64_t)g.bx[1] * (K + 1) * cd(n + 1, FR_CELLS);
  g.first[3] = g.first[2] + (int64_t)g.bx[2] * (K + 1) * cd(N, FR_WARPS);
  return g;
}

// Scaled 1-D operators of the level.
template <int K>
struct FactRowTab {
  static constexpr int K1 = K + 1, NG = K + 2;
  double m[NG][NG];            // M
  double k[K1][NG][NG];        // mu w_b K
  double g[K1][K1][NG];        // -w_b G
  double f[4][K1][3][K1];      // penalty rows [first | last << 1][b][cell before, own, behind]
};

// sink(flat index, value of A x, constrained): called once for every row.
template <int D, int K, class Sink>
__device__ __forceinline__ void fact_rows(const Lvl<D, K, double>& L, const Tab<K, double>& tb, const FactRowGrid& fg,
                                          const double* __restrict__ x, Sink sink) {
  static_assert(D == 2, "a node across a cell has one coordinate");
  constexpr int K1 = K + 1, NG = K + 2;
  __shared__ FactRowTab<K> S;
  __shared__ double ex[2][FR_WARPS][32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = L.n, N = L.N, N1 = N + 1;
  for (int q = tid; q < NG * NG; q += 32 * FR_WARPS) S.m[q / NG][q % NG] = tb.Mcg[q / NG][q % NG];
  for (int q = tid; q < K1 * NG * NG; q += 32 * FR_WARPS) {
    const int b = q / (NG * NG), a = q / NG % NG, c = q % NG;
    S.k[b][a][c] = L.s_mu * tb.wg[b] * tb.Kcg[a][c];
  }
  for (int q = tid; q < K1 * K1 * NG; q += 32 * FR_WARPS) {
    const int b = q / (K1 * NG), c = q / NG % K1, a = q % NG;
    S.g[b][c][a] = -L.s_b * tb.wg[b] * tb.G[c][a];
  }
  for (int q = tid; q < 4 * K1 * K1; q += 32 * FR_WARPS) {
    const int var = q / (K1 * K1), b = q / K1 % K1, c = q % K1;
    const bool lo = !(var & 1), hi = !(var & 2);
    S.f[var][b][0][c] = lo ? L.s_mu * tb.F21[b][c] : 0.0;
    S.f[var][b][1][c] = L.s_mu * (tb.Kdg[b][c] + (lo ? tb.F22[b][c] : tb.Blo[b][c]) + (hi ? tb.F11[b][c] : tb.Bhi[b][c]));
    S.f[var][b][2][c] = hi ? L.s_mu * tb.F12[b][c] : 0.0;
  }
  __syncthreads();
  const int64_t blk = blockIdx.x;
  if (blk >= fg.first[2]) {   // pressure: lanes = cells along x at one position, warps = nodes along y
    const int64_t q = blk - fg.first[2];
    const int lx = (int)(q % fg.bx[2]), bx = (int)(q / fg.bx[2] % K1);
    const int64_t row = q / fg.bx[2] / K1 * FR_WARPS + warp;
    const int cx = lx * 32 + lane;
    if (row >= N || cx >= n) return;
    const int sy = (int)row, cy = sy / K1, by = sy - cy * K1, sx = cx * K1 + bx;
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < NG; ++a) {
      const int t = cx * K1 + a;
      if (t > 0 && t < N) acc += S.g[by][bx][a] * x[L.off[0] + t + (int64_t)sy * N1];
    }
#pragma unroll
    for (int a = 0; a < NG; ++a) {
      const int t = cy * K1 + a;
      if (t > 0 && t < N) acc += S.g[bx][by][a] * x[L.off[1] + sx + (int64_t)t * N];
    }
    sink(L.off[2] + sx + (int64_t)sy * N, acc, false);
    return;
  }
  const bool cy_comp = blk >= fg.first[1];   // component y
  int ct, s;                                 // cell along the component's direction, node across
  bool out;                                  // this cell's rows are written by this thread
  if (!cy_comp) {
    const int64_t row = blk / fg.bx[0] * FR_WARPS + warp;
    ct = (int)(blk % fg.bx[0]) * FR_LANES + lane - 2;
    s = (int)row;
    out = row < N && lane >= 2 && ct <= n;
    if (row >= N) ct = -1;
  } else {
    const int64_t q = blk - fg.first[1];
    const int cx = (int)(q % fg.bx[1]) * 32 + lane, b = (int)(q / fg.bx[1] % K1);
    ct = (int)(q / fg.bx[1] / K1) * FR_CELLS + warp - 2;
    s = cx * K1 + b;
    out = cx < n && warp >= 2 && ct <= n;
    if (cx >= n) ct = -1;
  }
  const bool live = ct >= 0 && ct < n;
  const int cs = s / K1, b = s - cs * K1;
  const int64_t st = cy_comp ? N : 1, ss = cy_comp ? 1 : N1, off = cy_comp ? L.off[1] : L.off[0];
  const double(&f)[3][K1] = S.f[(cs == 0 ? 1 : 0) | (cs == n - 1 ? 2 : 0)][b];
  double u[NG], z[NG], y[NG];
#pragma unroll
  for (int a = 0; a < NG; ++a) u[a] = z[a] = y[a] = 0.0;
  if (live) {
    const double* xu = x + off + (int64_t)ct * K1 * st;
#pragma unroll
    for (int a = 0; a < NG; ++a) {
      const int t = ct * K1 + a;
      if (t == 0 || t == N) continue;   // constrained column
      u[a] = xu[a * st + (int64_t)s * ss];
      if (a == 0) continue;
      const double* xs = xu + a * st + (int64_t)cs * K1 * ss;
#pragma unroll
      for (int c = 0; c < K1; ++c) {
        z[a] += f[1][c] * xs[c * ss];
        if (cs > 0) z[a] += f[0][c] * xs[(c - K1) * ss];
        if (cs < n - 1) z[a] += f[2][c] * xs[(c + K1) * ss];
      }
    }
  }
  // Z of the first node: the last one of the cell before
  if (!cy_comp) {
    z[0] = __shfl_up_sync(0xffffffffu, z[K1], 1);
  } else {
    ex[0][warp][lane] = z[K1];
    __syncthreads();
    if (warp > 0) z[0] = ex[0][warp - 1][lane];
  }
  if (live) {
    const double cw = L.s_c * tb.wg[b] * L.c[cy_comp ? (int64_t)ct * n + cs : (int64_t)cs * n + ct];
#pragma unroll
    for (int a = 0; a < NG; ++a) z[a] += cw * u[a];
    const double* xp = x + L.off[2] + (int64_t)ct * K1 * (cy_comp ? N : 1) + (int64_t)s * (cy_comp ? 1 : N);
    double p[K1];
#pragma unroll
    for (int c = 0; c < K1; ++c) p[c] = xp[(int64_t)c * (cy_comp ? N : 1)];
#pragma unroll
    for (int a = 0; a < NG; ++a) {
#pragma unroll
      for (int c = 0; c < NG; ++c) y[a] += S.m[a][c] * z[c];
#pragma unroll
      for (int c = 0; c < NG; ++c) y[a] += S.k[b][a][c] * u[c];
#pragma unroll
      for (int c = 0; c < K1; ++c) y[a] += S.g[b][c][a] * p[c];
    }
  }
  // the share of the cell before in the first node's row
  double y0 = 0.0;
  if (!cy_comp) {
    y0 = __shfl_up_sync(0xffffffffu, y[K1], 1);
  } else {
    ex[1][warp][lane] = y[K1];
    __syncthreads();
    if (warp > 0) y0 = ex[1][warp - 1][lane];
  }
  if (!out) return;
  const int64_t g0 = off + (int64_t)ct * K1 * st + (int64_t)s * ss;
  sink(g0, y0 + y[0], ct == 0 || ct == n);
  if (ct < n)
#pragma unroll
    for (int a = 1; a < K1; ++a) sink(g0 + a * st, y[a], false);
}

// y = A x (b null; the identity on constrained rows), or r = b - A x on free rows and
// on constrained rows 0 (zero_c) or b - x, for the vector blockIdx.y.
template <int D, int K>
__global__ void __launch_bounds__(32 * FR_WARPS) k_fact_apply(const Lvl<D, K, double> L0, const __grid_constant__ Tab<K, double> tb,
                                                             const FactRowGrid fg, const double* __restrict__ x,
                                                             const double* b, double* y, int zero_c, int64_t vs,
                                                             const ProbStride ps) {
  Lvl<D, K, double> L = L0;
  L.c += ps.of(blockIdx.y) * ps.c;
  x += blockIdx.y * vs;
  y += blockIdx.y * vs;
  if (b) b += blockIdx.y * vs;
  fact_rows(L, tb, fg, x, [&](int64_t g, double v, bool con) {
    if (con) v = x[g];
    y[g] = b ? (con && zero_c ? 0.0 : b[g] - v) : v;
  });
}

// r = b - A x (stored if r is given) and a partial sum of its squares per block.
template <int D, int K>
__global__ void __launch_bounds__(32 * FR_WARPS) k_fact_residual_norm(const Lvl<D, K, double> L,
                                                                     const __grid_constant__ Tab<K, double> tb,
                                                                     const FactRowGrid fg, const double* __restrict__ x,
                                                                     const double* b, double* r, double* __restrict__ partial) {
  __shared__ double red[FR_WARPS];
  double sq = 0.0;
  fact_rows(L, tb, fg, x, [&](int64_t g, double v, bool con) {
    const double rv = b[g] - (con ? x[g] : v);
    if (r) r[g] = rv;
    sq += rv * rv;
  });
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < FR_WARPS; ++w) s += red[w];
    partial[blockIdx.x] = s;
  }
}

}  // namespace mgd
