// xg_dynamics.cu -- hyper-diffusion, sponge and the RI-velocity diagnostic
// (include/xg_dynamics.h).
//
// The weak Laplacian on the box is, per direction, a 1-D operator along grid
// lines: with the collocated LGL quadrature the transverse weights cancel
// against the diagonal mass (as for the right-hand side), leaving
//   (L_d q)_I = -nu_d (2/h_d)^2 / W_d(g) sum_{segments s of I} sum_l K[a_s][l] q_{s,l},
// K[a][l] = sum_k w_k D[k][a] D[k][l] the 1-D stiffness and W_d the assembled
// 1-D weight (w_a inside an element, 2 w_0 on a shared face, w_0 on a wall).
// The rows are pre-scaled by -nu_d (2/h_d)^2 / w_a, rows 0 and N by half of
// that over 2 w_0; a face node adds its two segments' rows and a wall node
// doubles its one row -- the same structure as the derivative rows of the
// right-hand side.  Hyper-diffusion applies it twice (FP64, one thread per
// node, loads along the three lines through the node) and the second pass
// adds the sponge, into the extra tendency E that the FP64 stage adds
// before the wall condition.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include <cuda_runtime.h>

#include "../../include/xg_dynamics.h"
#include "xg_ctx.h"
#include "xg_fixed.cuh"
#include "xg_setup.h"

namespace xg {

struct LapParams {
  int n[3], nseg[3], per[3];
  long long np;
  double Km[3][kMaxOrder + 1][kMaxOrder + 1];
  FixRows Kf[3];   // Km in fixed point
};

template <int N>
__device__ __forceinline__ double line_apply(const LapParams& P, int d, const double* __restrict__ f,
                                             long long base, long long sd, int g) {
  const int nd = P.n[d], nseg = P.nseg[d];
  int s = g / N;
  if (s >= nseg) s = nseg - 1;
  const int a = g - s * N;
  double acc = 0.0;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    int k = s * N + l;
    if (k >= nd) k -= nd;
    acc = fma(P.Km[d][a][l], f[base + sd * k], acc);
  }
  if (a == 0) {
    if (s > 0 || P.per[d]) {
      const int s2 = s > 0 ? s - 1 : nseg - 1;
#pragma unroll
      for (int l = 0; l <= N; ++l) {
        int k = s2 * N + l;
        if (k >= nd) k -= nd;
        acc = fma(P.Km[d][N][l], f[base + sd * k], acc);
      }
    } else {
      acc = acc + acc;
    }
  } else if (a == N) {
    acc = acc + acc;
  }
  return acc;
}

// The Laplacian runs in two passes, the x and y parts over plane tiles and the
// z part along columns, with the contractions in 64-bit fixed point
// (xg_fixed.cuh): one thread per node with FP64 FMAs spent 3 (N + 1) (1 + 1/N)
// of them a value, at the FP64 pipe's rate.  Grid of the plane pass: tiles, n_z,
// 5 variables; out gets the x and y parts.  One Laplacian of the 64 x 64 x 16
// order-4 box: 0.93-1.02 -> 0.25 + 0.13-0.17 ms; the plane pass is bound by
// instruction issue (2.9 a clock of 4, 340 instructions a value), the z pass by the
// FP64 pipe (79 % busy, 3 to 4 instructions a value: conversion, scale-and-add, face
// sum).
template <int N, int W>
__global__ void __launch_bounds__(32 * W) k_lap_plane(const LapParams P, const double* __restrict__ in,
                                                          double* __restrict__ out) {
  using L = FixPlane<N>;
  __shared__ double V[L::V];
  __shared__ FixPlaneRows<N> R;
  stage_kernel_begin();
  const int z = blockIdx.y, var = blockIdx.z;
  const int tilesx = (P.nseg[0] + L::E - 1) / L::E;
  const int nx = P.n[0], ny = P.n[1];
  const long long off = var * P.np + (long long)nx * ny * z;
  FixTile T;
  T.init<N>(P, blockIdx.x % tilesx, blockIdx.x / tilesx);
  fix_plane_load<N, W, true, true>(in + off, T, nx, ny, V);
  __syncthreads();
  fix_plane_rows<N, W>(P.Kf[0], P.Kf[1], T, V, V, R);
  __syncthreads();
  fix_plane_nodes<N, W>(T, [&](int i, int j) {
    const long long I = T.x0 + i + (long long)nx * (T.y0 + j);
    const FixSum r = fix_add(fix_plane_x<N>(R, i, j), fix_plane_y<N>(T, R, i, j));
    if (r.u < kFixBad) {
      out[off + I] = fix_double(r);
    } else {   // an infinity or NaN in a segment of the node: FP64
      double s = line_apply<N>(P, 0, in + off, (long long)nx * (T.y0 + j), 1, T.x0 + i);
      s += line_apply<N>(P, 1, in + off, T.x0 + i, nx, T.y0 + j);
      out[off + I] = s;
    }
  });
}

// The same x and y parts with a thread a node, for levels that fill no tile.
template <int N>
__global__ void __launch_bounds__(128) k_lap_nodes(const LapParams P, const double* __restrict__ in,
                                                  double* __restrict__ out) {
  __shared__ FixTable<N> R[2];
  stage_kernel_begin();
  fix_stage_rows<N>(P.Kf[0], R[0]);
  fix_stage_rows<N>(P.Kf[1], R[1]);
  __syncthreads();
  const long long I = blockIdx.x * 128ll + threadIdx.x;
  if (I >= P.np) return;
  const int nx = P.n[0], ny = P.n[1];
  const long long line = I / nx;
  const int gx = (int)(I - line * nx), gy = (int)(line % ny);
  const double* __restrict__ f = in + blockIdx.y * P.np;
  const long long x0 = I - gx, y0 = I - (long long)nx * gy;
  const FixSum r = fix_add(fix_line_node<N>(R[0], f, x0, 1, gx, nx, P.nseg[0], P.per[0]),
                           fix_line_node<N>(R[1], f, y0, nx, gy, ny, P.nseg[1], P.per[1]));
  double s;
  if (r.u < kFixBad) {
    s = fix_double(r);
  } else {
    s = line_apply<N>(P, 0, f, x0, 1, gx);
    s += line_apply<N>(P, 1, f, y0, nx, gy);
  }
  out[blockIdx.y * P.np + I] = s;
}

// out += the z part (FIRST: the x and y parts are in out), or out = -(out + z
// part) - gamma(z) rho w.  One thread per column of one variable (blockIdx.z),
// marching the segments of its chunk (blockIdx.y).
template <int N, bool SECOND>
__global__ void __launch_bounds__(128) k_lap_z(const LapParams P, const double* __restrict__ in, double* out,
                                               const double* __restrict__ q, const double* __restrict__ gamma,
                                               int chunk) {
  stage_kernel_begin();
  const long long nxy = (long long)P.n[0] * P.n[1];
  const long long col = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int var = blockIdx.z, nz = P.n[2], nseg = P.nseg[2];
  const int s0 = (blockIdx.y * blockDim.y + threadIdx.y) * chunk, s1 = min(nseg, s0 + chunk);
  if (col >= nxy || s0 >= nseg) return;
  const double* __restrict__ f = in + var * P.np + col;
  double* o = out + var * P.np + col;
  const FixRows& K = P.Kf[2];
  auto at = [&](int g) -> double { return f[nxy * (g == nz ? 0 : g)]; };
  auto put = [&](int g, double s) {   // the FP64 pipe bounds this pass: signs ride in the operands
    if (SECOND && var == 3 && gamma) s = fma(-gamma[g], q[3 * P.np + col + nxy * g], s);
    o[nxy * g] = s;
  };
  double v[N + 1], next[N], carry = 0.0;
  fix2 w[N + 1];
  bool left = s0 > 0 || P.per[2];
  if (left) {
    const int sp = s0 > 0 ? s0 - 1 : nseg - 1;
#pragma unroll
    for (int l = 0; l <= N; ++l) v[l] = at(sp * N + l);
    const int E = fix_segment<N>(v, K.sc, w);
    carry = (double)fix_row<N>(K, N, w) * (SECOND ? -fix_unit<N>(E, K.sc) : fix_unit<N>(E, K.sc));
  }
  v[0] = at(s0 * N);
#pragma unroll
  for (int l = 0; l < N; ++l) next[l] = at(s0 * N + l + 1);
  for (int s = s0; s < s1; ++s) {
    double part[N];
#pragma unroll
    for (int a = 0; a < N; ++a) {
      part[a] = o[nxy * (s * N + a)];
      v[a + 1] = next[a];
    }
    if (s + 1 < s1) {   // the next segment's values while this one is computed
#pragma unroll
      for (int l = 0; l < N; ++l) next[l] = at((s + 1) * N + l + 1);
    }
    const int E = fix_segment<N>(v, K.sc, w);
    const double unit = SECOND ? -fix_unit<N>(E, K.sc) : fix_unit<N>(E, K.sc);
#pragma unroll
    for (int a = 0; a < N; ++a) {
      long long r = fix_row<N>(K, a, w);
      if (a == 0 && !left) r += r;          // a wall's first node: its row twice
      double x = fma((double)r, unit, SECOND ? -part[a] : part[a]);
      if (a == 0 && left) x += carry;
      put(s * N + a, x);
    }
    carry = (double)fix_row<N>(K, N, w) * unit;
    v[0] = v[N];
    left = true;
  }
  if (!P.per[2] && s1 == nseg) {
    const double part = o[nxy * (nseg * N)];
    put(nseg * N, fma(2.0, carry, SECOND ? -part : part));
  }
}

// Order 1, where a row is a difference and a factor, on levels that leave tiles
// empty: a thread a node takes all three directions in FP64 (two Laplacians of 1 M
// nodes 0.32 ms at any shape; the tiles 0.29 where full, 0.41 where half full).
template <bool SECOND>
__global__ void __launch_bounds__(128) k_lap_linear(const LapParams P, const double* __restrict__ in,
                                                   double* __restrict__ out, const double* __restrict__ q,
                                                   const double* __restrict__ gamma) {
  stage_kernel_begin();
  const long long I = blockIdx.x * 128ll + threadIdx.x;
  if (I >= P.np) return;
  const int nx = P.n[0], ny = P.n[1], var = blockIdx.y;
  const long long line = I / nx;
  const int z = (int)(line / ny);
  const int at[3] = {(int)(I - line * nx), (int)(line - (long long)z * ny), z};
  const double* __restrict__ f = in + var * P.np + I;
  const double c = *f;
  double s = 0.0;
  long long sd = 1;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const int n = P.n[d], g = at[d];
    const bool right = g < n - 1 || P.per[d], left = g > 0 || P.per[d];
    double r = c, l = c;
    if (right) r = f[sd * (g < n - 1 ? 1 : 1 - n)];
    if (left) l = f[sd * (g > 0 ? -1 : n - 1)];
    const double k = P.Km[d][0][1];                  // = Km[1][0]; a wall's node: its row twice
    s = fma(right && left ? k : k + k, (r - c) + (l - c), s);
    sd *= n;
  }
  if (SECOND) {
    s = -s;
    if (var == 3 && gamma) s = fma(-gamma[z], q[3 * P.np + I], s);
  }
  out[var * P.np + I] = s;
}

// E = sponge only (no hyper-diffusion)
__global__ void k_sponge_only(long long np, int nxy, const double* __restrict__ q,
                              const double* __restrict__ gamma, double* __restrict__ out) {
  stage_kernel_begin();
  for (long long I = blockIdx.x * (long long)blockDim.x + threadIdx.x; I < 5 * np;
       I += (long long)gridDim.x * blockDim.x) {
    const long long v = I / np, J = I - v * np;
    out[I] = v == 3 ? -gamma[J / nxy] * q[I] : 0.0;
  }
}

// ------------------------------------------------------------------ RI velocity
//
// Two passes over the state, then one small one.  Both are bound by the FP64
// pipe (17 FP64 instructions a node for the centroid, 25 for the strips), not
// by HBM, so neither divides nor takes an IEEE square root: a speed is
// |m|^2 rsqrt(|m|^2 rho^2) and a tangential speed |cross| rsqrt(rho^2 r^2),
// the hardware estimate refined by two Newton steps, and a node's strip comes
// from an FP32 square root wherever that is far enough from a boundary.  Each
// node is visited once (a block per strip would visit it nstrips times):
// a warp takes 32 neighbours of a row, whose strips come in runs, sums each
// run by a segmented scan and adds it to the warp's own bins, so that no
// atomic is needed and the order of every sum is fixed.  128 x 128 x 16
// order-4 box, 50 strips: centroid 3.77 -> 0.70 ms, strips 39.8 -> 0.99 ms.

constexpr int kRiThreads = 256, kRiWarps = kRiThreads / 32;

__device__ __forceinline__ double rsqrt_newton(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double e = fma(-(x * y), y, 1.0);
    y = fma(0.5 * y, e, y);
  }
  return y;
}

// far from under- and overflow, where rsqrt_newton is good to an ulp or two
__device__ __forceinline__ bool rsqrt_range(double x) { return x > 1.0e-280 && x < 1.0e280; }

// A sum with what its roundings left out (Knuth's TwoSum): the last steps of a
// centroid's sums, over warps and chunks, where positions of both signs cancel.
// In FP64 alone they put it off by up to eight times as much as the lanes' own
// sums do.
struct Sum2 {
  double h, l;
};

__device__ __forceinline__ Sum2 sum2(Sum2 a, Sum2 b) {
  const double s = a.h + b.h, t = s - a.h;
  return {s, (a.l + b.l) + ((a.h - (s - t)) + (b.h - t))};
}

// (an infinity leaves no remainder)
__device__ __forceinline__ double value_of(Sum2 a) { return a.l == a.l ? a.h + a.l : a.h; }

// grid (chunks, n_z): |u|, |u| x and |u| y over a chunk of a level's rows
template <typename R>
__global__ void __launch_bounds__(kRiThreads) k_ri_centroid(const R* __restrict__ q,
                                                           const double* __restrict__ rho0,
                                                           const double* __restrict__ px,
                                                           const double* __restrict__ py, int nx,
                                                           int ny, long long np,
                                                           Sum2* __restrict__ part) {
  __shared__ double red[3][kRiWarps];
  const int gz = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y0 = (int)((long long)ny * blockIdx.x / gridDim.x), y1 = (int)((long long)ny * (blockIdx.x + 1) / gridDim.x);
  const double r0 = rho0[gz];
  double s = 0.0, sx = 0.0, sy = 0.0;
  for (int y = y0 + warp; y < y1; y += kRiWarps) {
    const R* row = q + (long long)nx * (y + (long long)ny * gz);
    double sr = 0.0;
    for (int x = lane; x < nx; x += 32) {
      const double rho = r0 + (double)row[x];
      const double mu = row[np + x], mv = row[2 * np + x], mw = row[3 * np + x];
      const double m2 = fma(mu, mu, fma(mv, mv, mw * mw)), t = m2 * (rho * rho);
      double sp;
      if (rsqrt_range(t)) {
        sp = m2 * rsqrt_newton(t);
      } else {
        const double u = mu / rho, v = mv / rho, w = mw / rho;
        sp = sqrt(u * u + v * v + w * w);
      }
      sr += sp;
      sx = fma(sp, px[x], sx);
    }
    s += sr;
    sy = fma(sr, py[y], sy);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_down_sync(0xffffffffu, s, o);
    sx += __shfl_down_sync(0xffffffffu, sx, o);
    sy += __shfl_down_sync(0xffffffffu, sy, o);
  }
  if (lane == 0) {
    red[0][warp] = s;
    red[1][warp] = sx;
    red[2][warp] = sy;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    Sum2 t = {red[threadIdx.x][0], 0.0};
#pragma unroll
    for (int k = 1; k < kRiWarps; ++k) t = sum2(t, {red[threadIdx.x][k], 0.0});
    part[3 * (blockIdx.x + (long long)gridDim.x * gz) + threadIdx.x] = t;
  }
}

// The centroid of level gz from its chunks' sums, in chunk order, to c2; called by
// a whole block.
__device__ __forceinline__ void level_centroid(const Sum2* __restrict__ part, int chunks, int gz, double cx0,
                                               double cy0, double (&c2)[2]) {
  __shared__ double sums[3];
  if (threadIdx.x < 3) {
    Sum2 t = {0.0, 0.0};
    for (int k = 0; k < chunks; ++k) t = sum2(t, part[3 * (k + (long long)chunks * gz) + threadIdx.x]);
    sums[threadIdx.x] = value_of(t);
  }
  __syncthreads();
  if (threadIdx.x < 2) c2[threadIdx.x] = sums[0] > 0.0 ? sums[1 + threadIdx.x] / sums[0] : (threadIdx.x == 0 ? cx0 : cy0);
  __syncthreads();
}

// grid (chunks, n_z): tangential-speed sums and node counts per strip over a
// chunk of a level's rows.  Dynamic shared memory: per warp nstrips sums and
// counts.
template <typename R>
__global__ void __launch_bounds__(kRiThreads) k_ri_strip(const R* __restrict__ q,
                                                        const double* __restrict__ rho0,
                                                        const double* __restrict__ px,
                                                        const double* __restrict__ py, int nx, int ny,
                                                        long long np, const Sum2* __restrict__ cpart,
                                                        double cx0, double cy0, int nstrips, double eps,
                                                        double* __restrict__ cent,
                                                        double* __restrict__ part, int* __restrict__ cntp) {
  extern __shared__ double bins[];
  int* cnts = reinterpret_cast<int*>(bins + kRiWarps * nstrips);
  __shared__ double c2[2];
  const int gz = blockIdx.y, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int y0 = (int)((long long)ny * blockIdx.x / gridDim.x), y1 = (int)((long long)ny * (blockIdx.x + 1) / gridDim.x);
  for (int k = threadIdx.x; k < kRiWarps * nstrips; k += kRiThreads) {
    bins[k] = 0.0;
    cnts[k] = 0;
  }
  level_centroid(cpart, gridDim.x, gz, cx0, cy0, c2);
  if (threadIdx.x < 2 && blockIdx.x == 0) cent[2 * gz + threadIdx.x] = c2[threadIdx.x];
  const double cx = c2[0], cy = c2[1], r0 = rho0[gz];
  const float ieps = (float)(1.0 / eps);
  double* wb = bins + warp * nstrips;
  int* wc = cnts + warp * nstrips;
  for (int y = y0 + warp; y < y1; y += kRiWarps) {
    const R* row = q + (long long)nx * (y + (long long)ny * gz);
    const double ry = py[y] - cy;
    for (int xb = 0; xb < nx; xb += 32) {
      const int x = xb + lane;
      const double rx = x < nx ? px[x] - cx : 0.0;
      const double r2 = fma(rx, rx, ry * ry);
      int j = nstrips;
      if (x < nx) {
        // the strip floor(r / eps): FP32's rounding (below 4e-7 of t) decides
        // it except near a boundary
        const float t = sqrtf((float)r2) * ieps, f = floorf(t), tol = 1.0e-6f + 1.0e-6f * t;
        if (t - f > tol && t - f < 1.0f - tol && t < 4096.0f && r2 > 1.0e-30 && r2 < 1.0e30)
          j = min((int)f, nstrips);
        else
          j = (int)fmin(floor(sqrt(rx * rx + ry * ry) / eps), (double)nstrips);
      }
      const bool in = j < nstrips;
      if (!__any_sync(0xffffffffu, in)) continue;
      double ut = 0.0;
      if (in) {
        const double rho = r0 + (double)row[x], mu = row[np + x], mv = row[2 * np + x];
        const double d = (rho * rho) * r2;
        if (rsqrt_range(d)) {
          ut = fabs(fma(mv, rx, -(mu * ry))) * rsqrt_newton(d);
        } else {
          const double r = sqrt(rx * rx + ry * ry), u = mu / rho, v = mv / rho;
          const double erx = r > 0.0 ? rx / r : 0.0, ery = r > 0.0 ? ry / r : 0.0;
          const double ur = u * erx + v * ery;
          const double tx = u - ur * erx, ty = v - ur * ery;
          ut = sqrt(tx * tx + ty * ty);
        }
      }
      // runs of equal strips: each run's sum at its first lane
      const int jl = __shfl_up_sync(0xffffffffu, j, 1);
      const bool head = lane == 0 || jl != j;
      const unsigned heads = __ballot_sync(0xffffffffu, head);
      const unsigned after = lane == 31 ? 0u : heads & (0xffffffffu << (lane + 1));
      const int end = after ? __ffs(after) - 1 : 32;   // the run's end (exclusive)
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double v = __shfl_down_sync(0xffffffffu, ut, o);
        if (lane + o < end) ut += v;
      }
      // a strip may come twice in a row of 32 (left and right of the centre):
      // its runs are added one after the other, in lane order
      unsigned todo = __ballot_sync(0xffffffffu, head && in);
      while (todo) {
        const bool mine = (todo >> lane) & 1u;
        const unsigned same = __match_any_sync(0xffffffffu, mine ? j : nstrips + 1 + lane) & todo;
        const bool go = mine && (__ffs(same) - 1) == lane;
        if (go) {
          wb[j] += ut;
          wc[j] += end - lane;
        }
        __syncwarp();
        todo &= ~__ballot_sync(0xffffffffu, go);
      }
    }
  }
  __syncthreads();
  const long long o = ((long long)gz * gridDim.x + blockIdx.x) * nstrips;
  for (int k = threadIdx.x; k < nstrips; k += kRiThreads) {
    double s = 0.0;
    int n = 0;
    for (int w = 0; w < kRiWarps; ++w) {
      s += bins[w * nstrips + k];
      n += cnts[w * nstrips + k];
    }
    part[o + k] = s;
    cntp[o + k] = n;
  }
}

// strip means per level, the chunks' sums in chunk order
__global__ void k_ri_means(const double* __restrict__ part, const int* __restrict__ cntp, int chunks, int nz,
                           int nstrips, double* __restrict__ means) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nz * nstrips) return;
  const int gz = t / nstrips, k = t - gz * nstrips;
  double s = 0.0;
  long long n = 0;
  for (int c = 0; c < chunks; ++c) {
    const long long o = ((long long)gz * chunks + c) * nstrips + k;
    s += part[o];
    n += cntp[o];
  }
  means[t] = n > 0 ? s / (double)n : 0.0;
}

}  // namespace xg

using xg::LapParams;

namespace {

xg_status status_of(xg_ctx* c, cudaError_t e, const char* where) {
  if (e == cudaSuccess) return XG_OK;
  fprintf(stderr, "xg_dynamics: %s: %s\n", where, cudaGetErrorString(e));
  cudaGetLastError();
  if (e == cudaErrorMemoryAllocation) return XG_ERR_OOM;
  c->failed = true;
  return XG_ERR_CUDA;
}

// Global node positions along direction d (the mesh's own formula).
std::vector<double> axis_positions(const xg_ctx* c, int d) {
  const int N = c->d.order;
  long double xi[xg::kMaxOrder + 1];
  xg::lgl_nodes(N, xi);
  const double h = (c->d.hi[d] - c->d.lo[d]) / c->d.nel[d];
  std::vector<double> p(c->n[d]);
  for (int g = 0; g < c->n[d]; ++g) {
    const int e = std::min(g / N, c->d.nel[d] - 1);
    const int a = g - N * e;
    p[g] = c->d.lo[d] + ((double)e + (double)((xi[a] + 1.0L) / 2.0L)) * h;
  }
  return p;
}

template <int N>
void launch_lap(const LapParams& P, const double* q, double* L1, const double* gamma, double* E,
                bool hyper, int sms, cudaStream_t st) {
  const long long nxy = (long long)P.n[0] * P.n[1];
  if (!hyper) {
    xg::launch_stage_kernel(xg::k_sponge_only, (unsigned)std::min<long long>((5 * P.np + 255) / 256, 65535), 256, 0, st, P.np, (int)nxy, q, gamma, E);
    return;
  }
  constexpr int TE = xg::fix_plane_elems(N);
  const dim3 gp(((P.nseg[0] + TE - 1) / TE) * ((P.nseg[1] + TE - 1) / TE), P.n[2], 5);
  const dim3 gn((unsigned)((P.np + 127) / 128), 5);
  const int chunk = xg::fix_z_chunk(P.nseg[2], 5 * nxy, sms);
  const int cols = xg::fix_z_columns(nxy), par = xg::kFixZThreads / cols;
  const dim3 bz(cols, par), gz((unsigned)((nxy + cols - 1) / cols), ((P.nseg[2] + chunk - 1) / chunk + par - 1) / par, 5);
  const bool tiles = xg::fix_plane_pays(N, P.n[0], P.n[1], P.nseg[0], P.nseg[1]);
  const bool wide = xg::fix_plane_wide((long long)gp.x * gp.y * gp.z, sms);
  if (N == 1 && !tiles) {
    xg::launch_stage_kernel(xg::k_lap_linear<false>, gn, 128, 0, st, P, q, L1, nullptr, nullptr);
    xg::launch_stage_kernel(xg::k_lap_linear<true>, gn, 128, 0, st, P, L1, E, q, gamma);
    return;
  }
  auto plane = [&](const double* in, double* out) {
    constexpr int W = xg::fix_plane_warps(N), WW = xg::kFixWideWarps;
    if (tiles && wide) {
      xg::launch_stage_kernel(xg::k_lap_plane<N, WW>, gp, 32 * WW, 0, st, P, in, out);
    } else if (tiles) {
      xg::launch_stage_kernel(xg::k_lap_plane<N, W>, gp, 32 * W, 0, st, P, in, out);
    } else {
      if constexpr (N > 1) xg::launch_stage_kernel(xg::k_lap_nodes<N>, gn, 128, 0, st, P, in, out);
    }
  };
  plane(q, L1);
  xg::launch_stage_kernel(xg::k_lap_z<N, false>, gz, bz, 0, st, P, q, L1, nullptr, nullptr, chunk);
  plane(L1, E);
  xg::launch_stage_kernel(xg::k_lap_z<N, true>, gz, bz, 0, st, P, L1, E, q, gamma, chunk);
}

}  // namespace

// Called by the FP64 stage before its line kernels: E = H(q) + sponge(q).
cudaError_t dynamics_launch(xg_ctx* c, const double* q, cudaStream_t st) {
  const LapParams& P = *static_cast<const LapParams*>(c->dyn_params);
  const bool hyper = c->dyn_hyper;
  switch (c->d.order) {
    case 1: launch_lap<1>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 2: launch_lap<2>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 3: launch_lap<3>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 4: launch_lap<4>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 5: launch_lap<5>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 6: launch_lap<6>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 7: launch_lap<7>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    case 8: launch_lap<8>(P, q, c->dyn_L1, c->dyn_gamma, c->dyn_E, hyper, c->sms, st); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

void dynamics_free(xg_ctx* c) {
  cudaFree(c->dyn_L1);
  cudaFree(c->dyn_E);
  cudaFree(c->dyn_gamma);
  cudaFree(c->ri_buf);
  c->ri_buf = nullptr;
  c->ri_bytes = 0;
  delete static_cast<LapParams*>(c->dyn_params);
  c->dyn_L1 = c->dyn_E = c->dyn_gamma = nullptr;
  c->dyn_params = nullptr;
  c->dyn = c->dyn_hyper = false;
}

extern "C" {

xg_status xg_set_dynamics(xg_ctx* c, const xg_dynamics* dyn) {
  if (!c) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (!dyn) {
    c->dyn = false;
    return XG_OK;
  }
  if (c->dfm || c->f32) return XG_ERR_UNSUPPORTED;
  if (c->part_open[0] || c->part_open[1]) return XG_ERR_UNSUPPORTED;   // partitioned contexts
  const double H = c->d.hi[2] - c->d.lo[2];
  bool hyper = false;
  for (int k = 0; k < 3; ++k) {
    if (!(dyn->hyper_c[k] >= 0.0) || !std::isfinite(dyn->hyper_c[k])) return XG_ERR_ARG;
    hyper |= dyn->hyper_c[k] > 0.0;
  }
  if (hyper && !(dyn->hyper_dt > 0.0 && std::isfinite(dyn->hyper_dt))) return XG_ERR_ARG;
  if (!(dyn->sponge_depth >= 0.0 && dyn->sponge_depth <= H)) return XG_ERR_ARG;
  if (!(dyn->sponge_gamma >= 0.0 && std::isfinite(dyn->sponge_gamma))) return XG_ERR_ARG;
  const bool sponge = dyn->sponge_depth > 0.0 && dyn->sponge_gamma > 0.0;

  const int N = c->d.order;
  LapParams* P = static_cast<LapParams*>(c->dyn_params);
  if (!P) {
    P = new (std::nothrow) LapParams();
    if (!P) return XG_ERR_OOM;
    c->dyn_params = P;
  }
  memset(P, 0, sizeof(*P));
  for (int k = 0; k < 3; ++k) {
    P->n[k] = c->n[k];
    P->nseg[k] = c->d.nel[k];
    P->per[k] = c->d.periodic[k] ? 1 : 0;
  }
  P->np = c->np;
  // principal axes: descending element size, x, y, z on ties
  double h[3];
  int order[3] = {0, 1, 2};
  for (int k = 0; k < 3; ++k) h[k] = (c->d.hi[k] - c->d.lo[k]) / c->d.nel[k];
  std::stable_sort(order, order + 3, [&](int a, int b) { return h[a] > h[b]; });
  double nu[3];
  for (int i = 0; i < 3; ++i) {
    const int d = order[i];
    const double dx = h[d] / N;
    nu[d] = hyper ? std::sqrt(dyn->hyper_c[i]) * dx * dx / std::sqrt(dyn->hyper_dt) : 0.0;
  }
  long double D[xg::kMaxOrder + 1][xg::kMaxOrder + 1], w[xg::kMaxOrder + 1];
  xg::lgl_derivative(N, D);
  xg::lgl_weights(N, w);
  for (int d = 0; d < 3; ++d) {
    xg::FixMatrix Kl;
    const long double s = -(long double)nu[d] * (2.0L / h[d]) * (2.0L / h[d]);
    for (int a = 0; a <= N; ++a) {
      const long double wa = (a == 0 || a == N) ? 2.0L * w[0] : w[a];
      for (int l = 0; l <= N; ++l) {
        long double K = 0.0L;
        for (int k = 0; k <= N; ++k) K += w[k] * D[k][a] * D[k][l];
        Kl[a][l] = s * K / wa;
        P->Km[d][a][l] = (double)Kl[a][l];
      }
    }
    xg::fix_rows(N, Kl, &P->Kf[d]);
  }
  cudaError_t e = cudaSuccess;
  const size_t vec = sizeof(double) * 5 * (size_t)c->np;
  if (!c->dyn_L1) e = cudaMalloc((void**)&c->dyn_L1, vec);
  if (e == cudaSuccess && !c->dyn_E) e = cudaMalloc((void**)&c->dyn_E, vec);
  if (e == cudaSuccess && !c->dyn_gamma) e = cudaMalloc((void**)&c->dyn_gamma, sizeof(double) * c->n[2]);
  if (e == cudaSuccess) {
    const std::vector<double> z = axis_positions(c, 2);
    std::vector<double> g(c->n[2], 0.0);
    if (sponge) {
      const double zs = c->d.hi[2] - dyn->sponge_depth;
      const double pi = 3.14159265358979323846;
      for (int k = 0; k < c->n[2]; ++k) {
        if (z[k] > zs) {
          const double sn = std::sin(0.5 * pi * std::min(1.0, (z[k] - zs) / dyn->sponge_depth));
          g[k] = dyn->sponge_gamma * sn * sn;
        }
      }
    }
    e = cudaMemcpy(c->dyn_gamma, g.data(), sizeof(double) * c->n[2], cudaMemcpyHostToDevice);
  }
  if (e != cudaSuccess) {
    dynamics_free(c);
    return status_of(c, e, "xg_set_dynamics");
  }
  c->dyn_hyper = hyper;
  c->dyn = hyper || sponge;
  return XG_OK;
}

xg_status xg_dynamics_tendency(xg_ctx* c, double* out, int where, void* stream) {
  if (!c || !out) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (c->dfm || c->f32) return XG_ERR_UNSUPPORTED;
  if (!c->has_state || (where != XG_HOST && where != XG_DEVICE)) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const size_t bytes = sizeof(double) * 5 * (size_t)c->np;
  cudaError_t e;
  if (!c->dyn) {
    e = where == XG_DEVICE ? cudaMemsetAsync(out, 0, bytes, st) : cudaSuccess;
    if (where == XG_HOST) memset(out, 0, bytes);
    return status_of(c, e, "xg_dynamics_tendency");
  }
  e = dynamics_launch(c, c->A, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out, c->dyn_E, bytes, where == XG_DEVICE ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                        st);
  if (e == cudaSuccess && where == XG_HOST) e = cudaStreamSynchronize(st);
  return status_of(c, e, "xg_dynamics_tendency");
}

xg_status xg_ri_velocity(xg_ctx* c, int nstrips, double* u_ri, double* centroid, double* means,
                         void* stream) {
  if (!c || !u_ri || nstrips < 1 || nstrips > 1024) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (!c->has_state) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int nx = c->n[0], ny = c->n[1], nz = c->n[2];
  const long long np = c->np;
  // chunks of a level's rows: eight blocks per SM over all levels
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev);
  const int chunks = std::max(1, std::min((ny + xg::kRiWarps - 1) / xg::kRiWarps, (8 * std::max(1, sms) + nz - 1) / nz));
  // one buffer: positions, results (centroids, then means), chunk sums and
  // counts
  const size_t nres = 2 * (size_t)nz + (size_t)nz * nstrips;
  const size_t nd = (size_t)nx + ny + nres + (size_t)nz * chunks * (6 + nstrips);
  const size_t bytes = sizeof(double) * nd + sizeof(int) * (size_t)nz * chunks * nstrips;
  cudaError_t e = cudaSuccess;
  if (c->ri_bytes < bytes) {   // kept by the context: every call waits for its own work
    cudaFree(c->ri_buf);
    c->ri_buf = nullptr;
    c->ri_bytes = 0;
    e = cudaMalloc((void**)&c->ri_buf, bytes);
    if (e == cudaSuccess) c->ri_bytes = bytes;
  }
  double* buf = c->ri_buf;
  std::vector<double> pos, res(nres);
  if (e == cudaSuccess) {
    pos = axis_positions(c, 0);
    const std::vector<double> ay = axis_positions(c, 1);
    pos.insert(pos.end(), ay.begin(), ay.end());
    double *px = buf, *py = px + nx, *cent = py + ny, *mn = cent + 2 * nz, *part = cent + nres + 6 * (size_t)nz * chunks;
    xg::Sum2* cpart = reinterpret_cast<xg::Sum2*>(cent + nres);
    int* cntp = reinterpret_cast<int*>(buf + nd);
    const double cx0 = 0.5 * (c->d.lo[0] + c->d.hi[0]), cy0 = 0.5 * (c->d.lo[1] + c->d.hi[1]);
    const double R = 0.5 * std::min(c->d.hi[0] - c->d.lo[0], c->d.hi[1] - c->d.lo[1]);
    const dim3 g(chunks, nz);
    const size_t smem = (sizeof(double) + sizeof(int)) * xg::kRiWarps * (size_t)nstrips;
    e = cudaMemcpyAsync(px, pos.data(), sizeof(double) * pos.size(), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = c->f32 ? xg::raise_dynamic_smem(xg::k_ri_strip<float>, smem)
                                     : xg::raise_dynamic_smem(xg::k_ri_strip<double>, smem);
    if (e == cudaSuccess) {
      if (c->f32) {
        const float* q = (const float*)c->A;
        xg::k_ri_centroid<float><<<g, xg::kRiThreads, 0, st>>>(q, c->base64, px, py, nx, ny, np, cpart);
        xg::k_ri_strip<float><<<g, xg::kRiThreads, smem, st>>>(q, c->base64, px, py, nx, ny, np, cpart, cx0, cy0,
                                                             nstrips, R / nstrips, cent, part, cntp);
      } else {
        xg::k_ri_centroid<double><<<g, xg::kRiThreads, 0, st>>>(c->A, c->base64, px, py, nx, ny, np, cpart);
        xg::k_ri_strip<double><<<g, xg::kRiThreads, smem, st>>>(c->A, c->base64, px, py, nx, ny, np, cpart, cx0, cy0,
                                                              nstrips, R / nstrips, cent, part, cntp);
      }
      xg::k_ri_means<<<(nz * nstrips + 127) / 128, 128, 0, st>>>(part, cntp, chunks, nz, nstrips, mn);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(res.data(), cent, sizeof(double) * nres, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) return status_of(c, e, "xg_ri_velocity");
  const double* hmean = res.data() + 2 * (size_t)nz;
  double best = 0.0;
  for (size_t k = 0; k < (size_t)nz * nstrips; ++k) best = std::max(best, hmean[k]);
  *u_ri = best;
  if (centroid) memcpy(centroid, res.data(), sizeof(double) * 2 * (size_t)nz);
  if (means) memcpy(means, hmean, sizeof(double) * (size_t)nz * nstrips);
  return XG_OK;
}

}  // extern "C"
