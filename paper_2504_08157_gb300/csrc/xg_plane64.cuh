// xg_plane64.cuh -- the x and y passes of the FP64-accurate paths (XG_FP64 and
// XG_DF64) as one kernel over plane tiles.
//
// A CTA takes E_x x E_y elements of one level: the pointwise primitives of the
// tile's nodes (FP64, or the mixed arithmetic of xg_kernels_df.cuh), the x and
// y fluxes of the five equations, and the x + y part of each node's tendency
// by 1-D contractions in 64-bit fixed point (xg_fixed.cuh): GB300 issues 1.9
// FP64 FMAs a clock and SM against 60 IMAD.WIDE, and an order-4 row is 15 of
// those.  The kernel writes T (the x + y part) and W (w, p', theta), which the
// z pass reads; v and the x part never leave the chip.
//
// Every element segment of a line has an exponent of its own, so its rows carry
// the bits of its own values whatever the tile holds elsewhere, and no result
// depends on the tiles: a domain cut into y-slabs gets the same bits as the
// whole.  x and y rows of a node are integers, added in the larger one's unit
// (fix_add); a shared y face adds the row N of the segment before it in the
// format of T (t0 + row N, the order in which a partition face is completed).
// The Theta' flux theta (rho u_d) is formed as an integer product of 62 bits, so
// only theta's own rounding is in it; the difference form of the FP64 chains is
// not needed.  (One exponent for an x tile and y segment, found by a reduction
// over the block, took the same time, 0.413 against 0.404 ms for 4.3 M nodes, but
// left values below 2^-8 of the tile's largest fewer bits than FP64 has.)
//
// XG_FP64, a stage on the 128 x 128 x 16 order-4 box (17.0 M nodes): three line
// kernels with FP64 chains 1.87 + 1.44 + 2.02 ms; tiles 1.57 + 1.39 ms (FP64
// pipe 63 and 73 % busy with 37 and 38 instructions a node; 2,180 and 1,220
// instructions a node in all).  33^3 nodes: 66 -> 21 us.  At the full-size vortex,
// where the parts of rho' cancel to 1e-3 and less, its tendency's error is 6e-14
// (FP64 chains 7e-14).
#pragma once

#include <type_traits>

#include <cuda_runtime.h>

#include "xg_fixed.cuh"
#include "xg_kernels.cuh"
#include "xg_kernels_df.cuh"

namespace xg {

// FP64 launch constants with the fixed-point matrices of the three directions.
struct F64Params {
  LineParams P64;
  FixRows F[3];
};

// Launch constants of the mixed x-y tiles.
struct DfTileParams {
  DfParams D;
  FixRows F[2];
};

// Segments of a z tile and its launch bounds: two segments (of order 4) at 4
// CTAs per SM (56 registers).
__host__ __device__ constexpr int z_tile_segments(int N) { return N >= 8 ? 1 : 8 / N; }
__host__ __device__ constexpr int z_tile_threads(int N) { return kTileCols * (z_tile_segments(N) * N + 1); }
__host__ __device__ constexpr int z_tile_min_blocks(int N) { return 1152 / z_tile_threads(N); }

// Elements of a tile along x; element rows: about 8 nodes, so that the N + 1
// columns before and after a tile and its closing line are a quarter of its nodes.
__host__ __device__ constexpr int xy_elems_x(int N) { return fix_plane_elems(N); }
__host__ __device__ constexpr int xy_elems_y(int N) { return N == 1 ? 9 : (N == 3 ? 3 : (N >= 5 ? 1 : 8 / N)); }

template <int N>
struct XYTile {
  static constexpr int EX = xy_elems_x(N), EY = xy_elems_y(N);
  static constexpr int TX = EX * N, TY = EY * N;
  static constexpr int CX = TX == 32 ? N + 1 : N;       // columns beside the 32 that a warp's lanes take
  static constexpr int PX = (N + TX + 1) | 1;           // V: columns -N .. TX
  static constexpr int LY = TY + 1, LX = TX + 1;
  static constexpr int PR = LX | 1;                     // x rows, a wall's last node included
  static constexpr int V = LY * PX;                     // one value
  static constexpr int RX = LY * PR, UX = LY * (2 * EX + 1);
  static constexpr int RY = TY * LX, RNY = EY * LX;
  static constexpr size_t bytes = 8 * (size_t)(8 * V + 5 * (RX + RY + RNY)) + 4 * 5 * (size_t)(UX + RNY);
  static constexpr int side_warps(int ey) { return ((ey * N + 1) * CX + 31) / 32; }
  static constexpr int threads(int ey) { return 32 * (ey * N + 1 + side_warps(ey)); }
};

#ifdef __CUDACC__

// x and y fluxes of one node (M: the momentum's type)
template <typename M>
struct XYFlux {
  double mu, mv, th;     // rho u, rho v, theta: the rho' fluxes and the factors of the Theta' ones
  M xx, xy, xz, yy, yz;  // rho u u + p', rho u v, rho u w, rho v v + p', rho v w
};

// FP64: primitives and fluxes of the node I of level z; w, p', theta to W
// where the tile owns the node.
__device__ __forceinline__ void xy_point(const F64Params& Q, const StageBufs& B, long long I, int z, bool own,
                                         XYFlux<double>& f) {
  const LineParams& P = Q.P64;
  const long long np = P.np;
  const int nz = P.n[2];
  const double* __restrict__ q = B.q;
  const double rp = q[I], mu = q[np + I], mv = q[2 * np + I], mw = q[3 * np + I], tp = q[4 * np + I];
  const double ir = rcp_newton(__ldg(B.base + z) + rp);
  const double u = mu * ir, v = mv * ir;
  const double pp = __ldg(B.base + 2 * nz + z) * eos_phi(P, tp * __ldg(B.base + 3 * nz + z));
  f.mu = mu;
  f.mv = mv;
  f.th = (__ldg(B.base + nz + z) + tp) * ir;
  f.xx = fma(mu, u, pp);
  f.xy = mv * u;
  f.xz = mw * u;
  f.yy = fma(mv, v, pp);
  f.yz = mw * v;
  if (own) {
    B.W[np + I] = mw * ir;
    B.W[2 * np + I] = pp;
    B.W[3 * np + I] = f.th;
  }
}

// Mixed: theta in FP64 from a double-float estimate and one Newton correction
// (t1 = t0 + (Theta - t0 rho) / rho: the estimate's 2^-47 error squares away),
// two FP64 additions and two FMAs; everything else in double-float.
__device__ __forceinline__ void xy_point(const DfTileParams& Q, const DfBufs& B, long long I, int z, bool own,
                                         XYFlux<df>& f) {
  const DfParams& P = Q.D;
  const long long np = P.np;
  const int nz = P.n[2];
  const double* __restrict__ q = B.q;
  const double rp = q[I], mu = q[np + I], mv = q[2 * np + I], mw = q[3 * np + I], tp = q[4 * np + I];
  const double rho = B.base64[z] + rp, Th = B.base64[nz + z] + tp;
  const df ir = df_rcp(df_of_double(rho));
  const double t0 = dbl_of_df(df_mul(df_of_double(Th), ir));
  f.th = fma(fma(-t0, rho, Th), dbl_of_df(ir), t0);
  f.mu = mu;
  f.mv = mv;
  const df muD = df_of_double(mu), mvD = df_of_double(mv), mwD = df_of_double(mw);
  const df u = df_mul(muD, ir), v = df_mul(mvD, ir);
  const df pp = df_mul(B.base[2 * nz + z], df_eos_phi(P, df_mul(df_of_double(tp), B.base[3 * nz + z])));
  f.xx = df_add(df_mul(muD, u), pp);
  f.xy = df_mul(mvD, u);
  f.xz = df_mul(mwD, u);
  f.yy = df_add(df_mul(mvD, v), pp);
  f.yz = df_mul(mwD, v);
  if (own) {
    B.W[np + I] = df_mul(mwD, ir);
    B.W[2 * np + I] = pp;
    B.W64[I] = f.th;
  }
}

template <typename Params>
struct XYTypes;
template <>
struct XYTypes<F64Params> {
  using Bufs = StageBufs;
  using M = double;
  static constexpr bool mixed = false;
  static __device__ __forceinline__ const LineParams& line(const F64Params& P) { return P.P64; }
};
template <>
struct XYTypes<DfTileParams> {
  using Bufs = DfBufs;
  using M = df;
  static constexpr bool mixed = true;
  static __device__ __forceinline__ const LineParams& line(const DfTileParams& P) { return P.D.P64; }
};

// grid (x tiles, y tiles, n_z), block XYTile<N>::threads(ey), dynamic shared
// memory XYTile<N>::bytes; ey <= EY element rows a tile.  Fy [5][y tiles][n_z]
// [n_x] gets row N of the segment that ends at each tile's first line, which
// the z pass adds.
template <int N, typename Params>
__global__ void __launch_bounds__(XYTile<N>::threads(XYTile<N>::EY), 1088 / XYTile<N>::threads(XYTile<N>::EY))
    k_plane_xy(const __grid_constant__ Params P, const __grid_constant__ typename XYTypes<Params>::Bufs B, int ey) {
  using L = XYTile<N>;
  using M = typename XYTypes<Params>::M;
  constexpr bool MIXED = XYTypes<Params>::mixed;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  double* V = reinterpret_cast<double*>(smem_raw);    // rho u, rho v, theta, then the momentum's fluxes
  long long* RX = reinterpret_cast<long long*>(V + 8 * L::V);
  long long* RY = RX + 5 * L::RX;
  long long* RNY = RY + 5 * L::RY;
  int* UX = reinterpret_cast<int*>(RNY + 5 * L::RNY);   // units of the x rows and the y segments
  int* UY = UX + 5 * L::UX;

  const LineParams& G = XYTypes<Params>::line(P);
  const int nx = G.n[0], ny = G.n[1];
  const long long np = G.np;
  const int z = blockIdx.z;
  const int ekx = min(L::EX, G.nseg[0] - (int)blockIdx.x * L::EX), eky = min(ey, G.nseg[1] - (int)blockIdx.y * ey);
  const int x0 = blockIdx.x * L::TX, y0 = blockIdx.y * ey * N;
  const bool endx = !G.per[0] && (int)blockIdx.x * L::EX + ekx == G.nseg[0];
  const bool endy = !G.per[1] && (int)blockIdx.y * ey + eky == G.nseg[1];
  const bool open_lo = G.open_y[0] && blockIdx.y == 0, open_hi = endy && G.open_y[1];
  const int fx = ekx * N, fy = eky * N;                    // the closing column and line
  const int ox = fx + (endx ? 1 : 0), oy = fy + (endy ? 1 : 0);   // owned columns and lines
  const int oyx = fy + (endy && !open_hi ? 1 : 0);         // lines with x rows
  const bool hxl = blockIdx.x > 0 || G.per[0], hyl = blockIdx.y > 0 || G.per[1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int warps = blockDim.x >> 5;
  const int lines = ey * N + 1;                            // warps that take a line each

  stage_kernel_begin();

  // this thread's node (i, j) of the tile: a warp takes a line, the warps
  // after them the N columns before the tile and its 33rd
  int i, j;
  if (warp < lines) {
    j = warp;
    i = lane;
  } else {
    const int t = (int)threadIdx.x - 32 * lines;
    j = t / L::CX;
    const int k = t - j * L::CX;
    i = k == N ? 32 : k - N;
  }
  const bool inside = i >= 0 && i < ox && j <= fy;         // takes part in y rows
  const bool need = inside || (j < oyx && i <= fx && (i >= 0 || hxl));
  // the y segment of the node (its own), and the one it closes
  const int sj = j < fy ? j / N : eky - 1, aj = j - sj * N;
  const bool closes = aj == 0 && sj > 0 && inside;

  if (need) {
    XYFlux<M> f;
    int gx = x0 + i, gy = y0 + j;
    if (gx < 0) gx += nx;
    if (gx >= nx) gx -= nx;
    if (gy >= ny) gy -= ny;
    xy_point(P, B, gx + (long long)nx * (gy + (long long)ny * z), z, i >= 0 && i < ox && j < oy, f);
    double* v = V + j * L::PX + i + N;
    v[0] = f.mu;
    v[L::V] = f.mv;
    v[2 * L::V] = f.th;
    M* p = reinterpret_cast<M*>(v);
    p[3 * L::V] = f.xx;
    p[4 * L::V] = f.xy;
    p[5 * L::V] = f.xz;
    p[6 * L::V] = f.yy;
    p[7 * L::V] = f.yz;
  }
  __syncthreads();

  // one thread per segment, variable and direction; a warp's tasks are of one
  // kind.  Values of variable c along x: rho u, xx, xy, xz, rho u (and theta);
  // along y: rho v, xy, yy, yz, rho v.  Mixed momentum in double-float, the rest
  // in fixed point.
  constexpr unsigned kFx = 0x05430u, kFy = 0x17641u;
  auto limbs = [&](int c, const double* p, int at, int sp, int sc, fix2 (&v)[N + 1]) -> int {
    if (c == 4) return fix_products<N>(p, V + 2 * L::V + at, sp, sc, v);
    double a[N + 1];
#pragma unroll
    for (int l = 0; l <= N; ++l) a[l] = p[l * sp];
    return fix_values<N>(a, sc, v);
  };
  const int cy = ox > L::TX ? L::LX : L::TX;              // columns of the y tasks
  const bool low = L::EY > 1 && ey < L::EY;               // a small launch: a tile's time counts
  const int div = low ? fix_x_div(ekx) : 0;
  const int wx = fix_x_tasks(oyx, low ? ekx : L::EX), wy = (eky * cy + 31) / 32;
  for (int w = warp; w < 5 * (wx + wy); w += warps) {
    if (w < 5 * wx) {
      const int c = w / wx;
      int o, s;
      if (low) fix_x_slot(w - c * wx, lane, ekx, div, o, s);
      else fix_x_slot<L::EX>(w - c * wx, lane, o, s);
      const bool act = o >= 0 && o < oyx && s < ekx && (s >= 0 || hxl), own = act && s >= 0 && lane > 0;
      const bool left = s > 0 || hxl, end = endx && s == ekx - 1;
      const int at = o * L::PX + (s + 1) * N;
      const double* p = V + ((kFx >> (4 * c)) & 15u) * L::V + at;
      long long* r = RX + c * L::RX + o * L::PR + s * N;
      if (MIXED && c != 0 && c != 4) {
        if constexpr (MIXED) {
          df v[N + 1], last = {0.0f, 0.0f}, before;
          if (act) {
#pragma unroll
            for (int l = 0; l <= N; ++l) v[l] = reinterpret_cast<const df*>(p)[l];
            last = df_row<N, 0>(P.D, N, v);
          }
          before.h = __shfl_up_sync(0xffffffffu, last.h, 1);
          before.l = __shfl_up_sync(0xffffffffu, last.l, 1);
          if (own) {
            df* q = reinterpret_cast<df*>(r);
            const df first = df_row<N, 0>(P.D, 0, v);
            q[0] = left ? df_add(first, before) : df_scale2(first, 2.0f);
#pragma unroll
            for (int a = 1; a < N; ++a) q[a] = df_row<N, 0>(P.D, a, v);
            if (end) q[N] = df_scale2(last, 2.0f);
          }
        }
      } else {
        fix2 v[N + 1];
        int u = 0;
        if (act) u = limbs(c, p, at, 1, P.F[0].sc, v);
        int* ur = UX + c * L::UX + o * (2 * L::EX + 1) + 2 * s;
        fix_x_rows<N>(P.F[0], v, u, act, own, left, end, [&](int a, FixSum x) {
          r[a] = x.r;
          if (a < 2 || a == N) ur[a == N ? 2 : a] = x.u;
        });
      }
    } else {
      const int c = (w - 5 * wx) / wy, t = (w - 5 * wx - c * wy) * 32 + lane;
      const int s = ox > L::TX ? t / L::LX : t / L::TX, k = t - s * cy;
      if (s >= eky || k >= ox) continue;
      const int at = s * N * L::PX + N + k;
      const double* p = V + ((kFy >> (4 * c)) & 15u) * L::V + at;
      long long *r = RY + c * L::RY + s * N * L::LX + k, *rn = RNY + c * L::RNY + s * L::LX + k;
      if (MIXED && c != 0 && c != 4) {
        if constexpr (MIXED) {
          df v[N + 1];
#pragma unroll
          for (int l = 0; l <= N; ++l) v[l] = reinterpret_cast<const df*>(p)[l * L::PX];
#pragma unroll
          for (int a = 0; a < N; ++a) reinterpret_cast<df*>(r)[a * L::LX] = df_row<N, 1>(P.D, a, v);
          *reinterpret_cast<df*>(rn) = df_row<N, 1>(P.D, N, v);
        }
      } else {
        fix2 v[N + 1];
        UY[c * L::RNY + s * L::LX + k] = limbs(c, p, at, L::PX, P.F[1].sc, v);
#pragma unroll
        for (int a = 0; a < N; ++a) r[a * L::LX] = fix_row<N>(P.F[1], a, v);
        *rn = fix_row<N>(P.F[1], N, v);
      }
    }
  }
  __syncthreads();

  if (i < 0 || i >= ox || j > fy) return;
  const bool closing = j == fy && (!endy || open_hi);     // row N alone: the next tile's, or the neighbour's
  if (closing && !open_hi && gridDim.y == 1) return;
  double* faces = nullptr;
  long long fstride = 0, fat = 0;
  if (closing) {
    if (open_hi) {
      faces = B.face_hi;
      fstride = (long long)nx * G.n[2];
      fat = (long long)nx * z + x0 + i;
    } else {
      const int next = (int)blockIdx.y + 1 < (int)gridDim.y ? blockIdx.y + 1 : 0;
      faces = B.Fy;
      fstride = (long long)gridDim.y * G.n[2] * nx;
      fat = ((long long)next * G.n[2] + z) * nx + x0 + i;
    }
  }
  const bool wraps = j == 0 && hyl && gridDim.y == 1;     // one tile around: its own closing row
  const int sl = wraps ? eky - 1 : sj - 1;                // the y segment that ends at this line
  const long long I = x0 + i + (long long)nx * (y0 + j + (long long)ny * z);
  // a variable in fixed point
  auto node = [&](int c) {
    auto end_row = [&](int s) -> FixSum {
      return {RNY[c * L::RNY + s * L::LX + i], UY[c * L::RNY + s * L::LX + i]};
    };
    if (closing) {
      faces[c * fstride + fat] = fix_sum_out<MIXED>(end_row(eky - 1));
      return;
    }
    const FixSum rx = {RX[c * L::RX + j * L::PR + i], UX[c * L::UX + j * (2 * L::EX + 1) + fix_unit_slot<N>(i)]};
    FixSum ry;
    if (j == fy) {
      ry = fix_twice(end_row(eky - 1));                   // a wall's last node: its row twice
    } else {
      ry = {RY[c * L::RY + j * L::LX + i], UY[c * L::RNY + sj * L::LX + i]};
      if (j == 0 && !hyl && !open_lo) ry = fix_twice(ry);
    }
    double v = fix_sum_out<MIXED>(fix_add(rx, ry));
    if (closes || wraps) v = v + fix_sum_out<MIXED>(end_row(sl));
    B.T[c * np + I] = v;
  };
  node(0);
  node(4);
  if constexpr (!MIXED) {
    node(1);
    node(2);
    node(3);
  } else {
    const df* RXm = reinterpret_cast<const df*>(RX);
    const df* RYm = reinterpret_cast<const df*>(RY);
    const df* RNYm = reinterpret_cast<const df*>(RNY);
#pragma unroll
    for (int c = 1; c < 4; ++c) {
      if (closing) {
        reinterpret_cast<df*>(faces)[c * fstride + fat] = RNYm[c * L::RNY + (eky - 1) * L::LX + i];
        continue;
      }
      df r = RXm[c * L::RX + j * L::PR + i];
      if (j == fy) {
        r = df_add(r, df_scale2(RNYm[c * L::RNY + (eky - 1) * L::LX + i], 2.0f));
      } else {
        df t = RYm[c * L::RY + j * L::LX + i];
        if (j == 0 && !hyl && !open_lo) t = df_scale2(t, 2.0f);
        r = df_add(r, t);
      }
      if (closes || wraps) r = df_add(r, RNYm[c * L::RNY + sl * L::LX + i]);
      B.Tm[c * np + I] = r;
    }
  }
}

// ---------------------------------------------------------------- z lines + sources + stage, FP64
// One CTA per (32 x-columns) x (K element segments along z) x y, one thread per
// node: block (32, K N + 1), a warp a level.  The loads of the fluxes come
// first; fluxes go to shared memory with those of the N levels of the segment
// before the tile (Theta' as rho w and theta); then one thread per (column,
// segment) and variable takes its rows in fixed point, with an exponent of its
// own; after a barrier each thread assembles its node: sources, walls, stage.
template <int N>
__global__ void __launch_bounds__(z_tile_threads(N), z_tile_min_blocks(N))
    k_tile_z(const __grid_constant__ F64Params P, const __grid_constant__ StageBufs B) {
  constexpr int K = z_tile_segments(N);
  constexpr int NS = K * N + N + 1;            // flux slots: N halo levels + K N + 1
  __shared__ double Fm[3][NS][kTileCols];           // momentum fluxes
  __shared__ double Fs[2][NS][kTileCols];      // rho w and theta
  __shared__ double Rz[5][K * N][kTileCols];  // rows 0..N-1 of every segment, in the order 0, 4, 1, 2, 3
  __shared__ double RN[5][K + 1][kTileCols];  // row N, from the segment before the tile on
  const LineParams& G = P.P64;
  const int nx = G.n[0], ny = G.n[1], nz = G.n[2];
  const int nseg = G.nseg[2];
  const bool per = G.per[2] != 0;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = blockIdx.x * kTileCols + tx;
  const bool xin = x < nx;
  const int s0 = blockIdx.y * K;
  const int kc = min(K, nseg - s0);             // segments in this tile
  const int y = blockIdx.z;
  const long long np = G.np;
  const long long sd = (long long)nx * ny;
  const long long base = x + (long long)nx * y;
  const bool has_left = s0 > 0 || per;
  auto level = [&](int g) -> int { return g >= nz ? g - nz : (g < 0 ? g + nz : g); };

  const int own = s0 * N + ty;
  const bool owns = xin && (ty < kc * N || (ty == kc * N && s0 + kc == nseg && !per));
  const bool main_level = xin && ty <= kc * N;   // the extra row fills the end face
  const bool halo = xin && has_left && ty < N;   // the N levels before the tile
  const int g = level(own);
  const int gh = level((s0 - 1) * N + ty);
  const long long I = base + sd * (main_level ? g : 0);
  const long long Ih = base + sd * (halo ? gh : 0);
  const double* __restrict__ W = B.W;

  stage_kernel_begin();
  // the global loads the fluxes and rows need first (one memory round trip);
  // q^n and S, needed only by the stage at the end, are loaded there
  double qv[5], hq[3], th = 0.0, hth = 0.0, vel, pp, hvel, hpp;
  if (main_level) {
#pragma unroll
    for (int c = 0; c < 5; ++c) qv[c] = B.q[c * np + I];
    vel = W[np + I];
    pp = W[2 * np + I];
    th = W[3 * np + I];
  }
  if (halo) {
#pragma unroll
    for (int c = 0; c < 3; ++c) hq[c] = B.q[(c + 1) * np + Ih];
    hvel = W[np + Ih];
    hpp = W[2 * np + Ih];
    hth = W[3 * np + Ih];
  }
  if (main_level) {
    Fm[0][N + ty][tx] = qv[1] * vel;
    Fm[1][N + ty][tx] = qv[2] * vel;
    Fm[2][N + ty][tx] = fma(qv[3], vel, pp);
    Fs[0][N + ty][tx] = qv[3];
    Fs[1][N + ty][tx] = th;
  }
  if (halo) {
    Fm[0][ty][tx] = hq[0] * hvel;
    Fm[1][ty][tx] = hq[1] * hvel;
    Fm[2][ty][tx] = fma(hq[2], hvel, hpp);
    Fs[0][ty][tx] = hq[2];
    Fs[1][ty][tx] = hth;
  }
  __syncthreads();

  // a warp takes one variable of one segment (the segment before the tile, of
  // which only row N is needed, last)
  if (xin) {
    const int sc = P.F[2].sc;
    for (int w = ty; w < 5 * (kc + (has_left ? 1 : 0)); w += K * N + 1) {
      const int k = w < 5 * kc ? w / 5 + 1 : 0, e = w % 5;      // segment k - 1 of the tile
      const double* src = e < 2 ? &Fs[0][k * N][tx] : &Fm[e >= 2 ? e - 2 : 0][k * N][tx];
      bool b = false;
      int E = 0, u;
      fix2 v[N + 1];
      double a[N + 1];
#pragma unroll
      for (int l = 0; l <= N; ++l) a[l] = src[l * kTileCols];
      if (e == 1) {
        double t[N + 1];
#pragma unroll
        for (int l = 0; l <= N; ++l) {
          t[l] = src[(NS + l) * kTileCols];
          E = max(E, fix_prod_top(a[l], fix_exp_finite(a[l], b), t[l], fix_exp_finite(t[l], b)));
        }
        E = fix_prod_exp<N>(E, sc);
#pragma unroll
        for (int l = 0; l <= N; ++l) v[l] = fix_prod<N>(t[l], a[l], E);
        u = fix_prod_field<N>(E, sc);
      } else {
#pragma unroll
        for (int l = 0; l <= N; ++l) E = max(E, fix_exp_finite(a[l], b));
        E = fix_block_exp(E, sc);
#pragma unroll
        for (int l = 0; l <= N; ++l) v[l] = fix_of<N>(a[l], E);
        u = fix_field<N>(E, sc);
      }
      if (k > 0) {
#pragma unroll
        for (int r = 0; r < N; ++r)
          Rz[e][(k - 1) * N + r][tx] = b ? xg_nan(0.0) : fix_out<false>(fix_row<N>(P.F[2], r, v), u);
      }
      RN[e][k][tx] = b ? xg_nan(0.0) : fix_out<false>(fix_row<N>(P.F[2], N, v), u);
    }
  }

  __syncthreads();
  if (!owns) return;

  // the node's segment k and local index a; the wall node is row N of the last
  const int k = ty < kc * N ? ty / N : kc - 1;
  const int a = ty < kc * N ? ty - k * N : N;
  const long long fat = xy_face_at(G, B.fy, B.nty, x, y, g), nf = (long long)B.nty * nz * nx;
  double L[5];
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    const int e = c == 0 ? 0 : (c == 4 ? 1 : c + 1);
    double t = B.T[c * np + I];
    if (fat >= 0) t = t + B.Fy[c * nf + fat];           // the y face's row N: t0 + row N
    if (a == N) {                                       // wall node: its one-sided row counts twice
      const double r = RN[e][kc][tx];
      L[c] = t + (r + r);
    } else {
      const double r = Rz[e][ty][tx];
      t = t + r;
      L[c] = a == 0 ? t + (k > 0 || has_left ? RN[e][k][tx] : r) : t;
    }
  }
  bool bad = false;
  finish_node(G, B, qv, I, x, y, g, L, bad);
  if (bad) *B.flag = 1;
}

#endif  // __CUDACC__

// Element rows of the x-y tiles of a mesh: the most, EY, unless fewer give the
// chip blocks that it would lack.
inline int xy_tile_rows(int N, const int (&nseg)[3], int levels, int sms) {
  const int most = xy_elems_y(N), ex = xy_elems_x(N);
  const long long columns = (long long)((nseg[0] + ex - 1) / ex) * levels;
  int ey = most;
  while (ey > 1 && columns * ((nseg[1] + ey - 1) / ey) < 3ll * sms) --ey;
  return ey;
}

// Whether the mixed form takes the x-y tiles instead of the x and y line
// kernels.  The tiles do the pointwise work 1.4 times and the rho' and Theta'
// rows without the FP64 pipe; a short x line fills only part of its CTA, and a tile
// that is not full costs almost as much as one that is.  So the line lies at a number of
// elements for each order, two tiles' (three at orders 4 and 5).  A right-hand side of
// 3 M nodes, tiles over lines, is 0.75 / 0.97 / 1.05 at 32, 64 and 80 nodes (order 2),
// 0.91 / 0.90 / 1.15 at 33, 48 and 63 (order 3), 0.63 / 0.89 / 1.03 / 1.11 at 32, 64, 96
// and 128 (order 4), 0.45 / 0.90 / 1.12 / 1.22 at 30, 80, 95 and 125 (order 5), and
// 1.0 or more at order 1.  Boxes of few nodes would gain from the tiles beyond it
// (order 4, 128 nodes: 0.83 at 30,000 nodes, equal at 300,000), but the rule leaves
// n_y out, so that a y-slab of a domain takes the path of the whole.
inline bool df_uses_plane(int N, int nelx) {
  constexpr int kMost[kDfLineOrder + 1] = {0, 0, 32, 20, 24, 18};
  return N > kDfLineOrder || nelx <= kMost[N];
}

}  // namespace xg
