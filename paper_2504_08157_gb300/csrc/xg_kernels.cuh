// xg_kernels.cuh -- what the FP64-state kernels of the explicit CG Euler path share
// (sm_103a): launch constants, the equation of state, the FP64 contractions, and
// the completion of a node.
//
// The right-hand side of Sec. 2.1 (Eq. 1 restated for q = (rho', rho u,
// rho v, rho w, Theta'), pressure from Eq. 3) is evaluated by the collocated
// strong form of Sec. 2.2 (Eqs. 7-8) with DSS (Eqs. 9-11, Alg. 3) and the
// inverse diagonal mass (Eq. 12).  On an axis-aligned box of equal elements
// the metric is the same constant diagonal in every element, and the mass
// is the tensor product M_I = J W_x(gx) W_y(gy) W_z(gz) of assembled 1-D LGL
// weights.  The assembled divergence then splits into three 1-D operators:
// along each grid line, a node interior to an element takes that element's
// derivative (D F)_a, and a node on a shared face takes
// (w_N (D F^left)_N + w_0 (D F^right)_0) / (w_N + w_0) =
// ((D F^left)_N + (D F^right)_0) / 2 (w_0 = w_N); the transverse weights
// cancel against M.  This is the paper's gather/assembly/scatter of
// Alg. 1-3, reached without element-local storage and without atomics.
//
// A stage of an XG_FP64 context is two kernels over the SoA state
// (xg_plane64.cuh), with the contractions in 64-bit fixed point:
//   k_plane_xy  tiles of a level: pointwise primitives (w, p', theta =
//               Theta/rho to W), x and y fluxes, the x + y part of the tendency
//               to T;
//   k_tile_z    32 columns by a few element segments: z fluxes, the z part,
//               the sources (-rho' g k, -f k x rho u, rho S_theta), no-flux
//               walls, and either dq/dt or the fused SSP-RK stage combination
//               out = alpha q^n + beta (q + dt L(q)) into a buffer distinct from
//               every input.
// XG_DF64 contexts have kernels of their own (xg_kernels_df.cuh) or the first
// of these in mixed arithmetic.
//
// The derivative matrices come pre-scaled by -2/h_d (chain rule of the affine
// map, sign of the divergence) with rows 0 and N halved for the face average;
// wall nodes undo the halving.  The FP64 pipe (2 DFMA/clk/SM on GB300) bounds
// what runs on it, so the arithmetic is arranged to spend few FP64 instructions:
// 1/rho is one hardware reciprocal estimate refined by two Newton steps and the
// equation of state is a short binomial series.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace xg {

constexpr int kMaxOrder = 8;
constexpr int kXThreads = 128;
constexpr int kEosTerms = 8;

// Launch-time constants of one mesh (passed by value as a kernel parameter).
struct LineParams {
  int n[3];       // global nodes per direction
  int nseg[3];    // elements per direction
  int per[3];     // 1 = periodic
  // y ends that are faces of an element partition (a domain split into
  // y-slabs, Sec. 3.1): the face node's y part is completed by the
  // neighbouring partition's one-sided row (xg_partition_*) instead of the
  // wall's doubled row, and no wall condition applies there
  int open_y[2];
  long long np;   // n[0] n[1] n[2]
  // Dm[d][a][l] = -(2/h_d) D[a][l] (x 1/2 for a = 0 and a = N)
  double Dm[3][kMaxOrder + 1][kMaxOrder + 1];
  // (1 + x)^gamma - 1 = sum_{k=1..8} eos_c[k-1] x^k for |x| < eos_xmax
  double eos_c[kEosTerms];
  double eos_xmax;
  double gamma;
  double f, g;    // Coriolis parameter, gravity
};

// Buffers and stage coefficients of one launch.
struct StageBufs {
  const double* q;      // [5][np] state the tendency is taken of
  const double* qn;     // [5][np] q^n of the RK combination (alpha != 0)
  double* out;          // [5][np] new state, or dq/dt when rhs_only
  double* W;            // [4][np]: w, p', theta = Theta/rho in rows 1..3 (written by k_plane_xy)
  double* T;            // [5][np] x + y parts of the tendency
  const double* S;      // [np] heating S_theta (K/s)
  const double* base;   // [4][nz]: rho0, Theta0, p0, 1/Theta0 per level
  int* flag;            // set to 1 when a non-finite value is stored
  double dt, alpha, beta;
  int rhs_only;
  const double* E = nullptr;  // [5][np] extra tendency (hyper-diffusion, sponge) or null
  // open_y[1]: the one-sided row N of the slab's last y segment at every
  // (x, z) of the end face, [5][n_z][n_x] (written by k_plane_xy instead of the
  // wall's doubled row)
  double* face_hi = nullptr;
  // row N of the y segment that ends at each y tile's first line, written by
  // the x-y pass and added by the z pass: [5][nty][n_z][n_x], fy lines a tile
  double* Fy = nullptr;
  int fy = 1, nty = 1;
};

// Start of a stage kernel (launched by launch_stage_kernel): waits for the end of
// the kernel before it on the stream, all its writes included.
__device__ __forceinline__ void stage_kernel_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// (1 + x)^gamma - 1: the binomial series (Horner) for small |x|, where the
// truncation error after 8 terms is below 2^-56 relative (bound checked on
// the host), else expm1(gamma log1p(x)).
__device__ __forceinline__ double eos_phi(const LineParams& P, double x) {
  if (fabs(x) < P.eos_xmax) {
    double acc = P.eos_c[kEosTerms - 1];
#pragma unroll
    for (int k = kEosTerms - 2; k >= 0; --k) acc = fma(acc, x, P.eos_c[k]);
    return acc * x;
  }
  return expm1(P.gamma * log1p(x));
}

// 1/a for positive normal a: the hardware reciprocal estimate refined by two
// Newton-Raphson steps r <- r + r (1 - a r) (quadratic convergence; the
// estimate's error squared twice is far below the FP64 rounding, and the
// last FMA step leaves the result within an ulp).
__device__ __forceinline__ double rcp_newton(double a) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  double e = fma(-a, r, 1.0);
  r = fma(r, e, r);
  e = fma(-a, r, 1.0);
  return fma(r, e, r);
}

__device__ __forceinline__ bool is_nonfinite(double v) {
  return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
}

// ---------------------------------------------------------------- difference form
// (the y and z passes of the mixed lines; contractions in fixed point depend on
// differences by themselves, xg_fixed.cuh)
// The rho' and Theta' tendencies are residuals of cancelling flux
// derivatives where the flow is nearly non-divergent (in a vortex the x and
// y parts nearly cancel), so their rounding must stay far below the size of
// each part.  Every row of the LGL derivative matrix sums to zero (D 1 = 0,
// the derivative of a constant), so a row may be applied to the flux minus
// its value at the segment's first node:
//     sum_l Dm[a][l] f_l = sum_{l>=1} Dm[a][l] (f_l - f_0);
// the roundings then scale with the flux's variation across the segment
// instead of the flux.  The Theta' flux Theta u_d is written theta (rho u_d)
// with theta = Theta / rho (W[3]), and its differences as
//     F_l - F_0 = theta_l (m_l - m_0) + (theta_l - theta_0) m_0,
// so the product's rounding scales with the variation as well.  The exact
// value is unchanged.

// start + sum_{l>=1} Dm[d][a][l] d[l] (d[0] = 0 is not used)
template <int N, int D>
__device__ __forceinline__ double drow_from(const LineParams& P, int a, const double (&d)[N + 1],
                                            double start) {
  double acc = start;
#pragma unroll
  for (int l = 1; l <= N; ++l) acc = fma(P.Dm[D][a][l], d[l], acc);
  return acc;
}

// (the first product rounded by itself: at order 1, where it is the whole row,
// the compiler would fuse it with the sum it is added to, and a face between two
// tiles or slabs, which hand the row on, would differ from one inside a tile)
template <int N, int D>
__device__ __forceinline__ double drow_N(const LineParams& P, const double (&d)[N + 1]) {
  double acc = __dmul_rn(P.Dm[D][N][1], d[1]);
#pragma unroll
  for (int l = 2; l <= N; ++l) acc = fma(P.Dm[D][N][l], d[l], acc);
  return acc;
}

// Row N of the y segment before a y tile, for the tile's first line (written by
// the y or x-y pass): its offset in one variable of Fy, or -1 where the node at line
// y has none.  fy: lines of a tile, nty: tiles.
__device__ __forceinline__ long long xy_face_at(const LineParams& P, int fy, int nty, int x, int y, int z) {
  if (nty == 1 || !(P.per[1] || (y > 0 && y < P.n[1] - 1))) return -1;
  // y / fy without an integer division (exact: y < 2^16, so the float quotient
  // of y + 1/2 is nearer to it than 1 / (2 fy))
  const int t = (int)__fdividef((float)y + 0.5f, (float)fy);
  if (y != t * fy) return -1;
  return ((long long)t * P.n[2] + z) * P.n[0] + x;
}

// ---------------------------------------------------------------- z lines + sources + stage
// Completes node I at level gz given its state qv and L[5] = T + z part (the
// assembled flux divergence): sources, no-flux walls, then the stage store.
// Every array of a launch is distinct (the stage output never overwrites an
// input).
__device__ __forceinline__ void finish_node(const LineParams& P, const StageBufs& B, const double (&qv)[5],
                                            long long I, int x, int y, int gz, double (&L)[5], bool& bad) {
  const long long np = P.np;
  if (B.E) {
#pragma unroll
    for (int c = 0; c < 5; ++c) L[c] += B.E[c * np + I];
  }
  L[1] = fma(P.f, qv[2], L[1]);                  // -f k x (rho u): +f rho v
  L[2] = fma(-P.f, qv[1], L[2]);                 //                 -f rho u
  L[3] = fma(-P.g, qv[0], L[3]);                 // -rho' g
  if (B.S) L[4] = fma(__ldg(B.base + gz) + qv[0], __ldg(B.S + I), L[4]);  // rho S_theta
  if (!P.per[0] && (x == 0 || x == P.n[0] - 1)) L[1] = 0.0;
  if (!P.per[1] && ((y == 0 && !P.open_y[0]) || (y == P.n[1] - 1 && !P.open_y[1]))) L[2] = 0.0;
  if (!P.per[2] && (gz == 0 || gz == P.n[2] - 1)) L[3] = 0.0;
#pragma unroll
  for (int c = 0; c < 5; ++c) {
    double o = L[c];
    if (!B.rhs_only) {
      o = fma(B.dt, L[c], qv[c]);
      if (B.alpha != 0.0) o = fma(B.alpha, B.qn[c * np + I], B.beta * o);
    }
    B.out[c * np + I] = o;
    bad |= is_nonfinite(o);
  }
}

}  // namespace xg
