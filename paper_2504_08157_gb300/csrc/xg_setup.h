// xg_setup.h -- host-side mesh checks and launch constants shared by the
// entry points: the LGL derivative matrix (Sec. 2.2, Eq. 5), the binomial
// series of the equation of state (Eq. 3), the pre-scaled per-direction
// derivative matrices.
#pragma once

#include <cmath>
#include <cstring>
#include <mutex>

#include <cuda_runtime.h>

#include "../../include/xg.h"
#include "xg_kernels.cuh"
#include "xg_kernels_df.cuh"
#include "xg_kernels_f32.cuh"
#include "xg_plane64.cuh"
#include "xg_plane_f32.cuh"

namespace xg {

inline bool finite_pos(double v) { return std::isfinite(v) && v > 0.0; }

// Legendre P_N and P_{N-1} at x by the three-term recurrence.
inline void legendre2(int N, long double x, long double* pN, long double* pN1) {
  long double p0 = 1.0L, p1 = x;
  if (N == 0) { *pN = 1.0L; *pN1 = 0.0L; return; }
  for (int k = 1; k < N; ++k) {
    long double p2 = ((2 * k + 1) * x * p1 - k * p0) / (k + 1);
    p0 = p1;
    p1 = p2;
  }
  *pN = p1;
  *pN1 = p0;
}

// LGL points: the zeros of x P_N - P_{N-1} = -(1 - x^2) P_N' / N, found by
// Newton's method (its derivative is (N+1) P_N) from the Chebyshev-Lobatto
// points; then the derivative matrix of the Lagrange basis,
// D[i][j] = P_N(x_i) / (P_N(x_j) (x_i - x_j)) for i != j,
// D[0][0] = -N(N+1)/4, D[N][N] = N(N+1)/4, else 0 on the diagonal.
inline void lgl_nodes(int N, long double* x) {
  const long double pi = 3.14159265358979323846264338327950288L;
  for (int j = 0; j <= N; ++j) {
    long double xj = -cosl(pi * j / N);
    for (int it = 0; it < 100; ++it) {
      long double pn, pn1;
      legendre2(N, xj, &pn, &pn1);
      long double dx = (xj * pn - pn1) / ((N + 1) * pn);
      xj -= dx;
      if (fabsl(dx) < 1e-30L) break;
    }
    x[j] = xj;
  }
  x[0] = -1.0L;
  x[N] = 1.0L;
}

template <typename T>
inline void lgl_derivative(int N, T D[kMaxOrder + 1][kMaxOrder + 1]) {
  long double x[kMaxOrder + 1], PN[kMaxOrder + 1];
  lgl_nodes(N, x);
  for (int j = 0; j <= N; ++j) {
    long double pn1;
    legendre2(N, x[j], &PN[j], &pn1);
  }
  for (int i = 0; i <= N; ++i)
    for (int j = 0; j <= N; ++j) {
      long double v;
      if (i != j) v = PN[i] / (PN[j] * (x[i] - x[j]));
      else if (i == 0) v = -(long double)N * (N + 1) / 4.0L;
      else if (i == N) v = (long double)N * (N + 1) / 4.0L;
      else v = 0.0L;
      D[i][j] = (T)v;
    }
}

// LGL weights w_j = 2 / (N (N+1) P_N(x_j)^2) at the points of lgl_derivative.
template <typename T>
inline void lgl_weights(int N, T* w) {
  const long double pi = 3.14159265358979323846264338327950288L;
  for (int j = 0; j <= N; ++j) {
    long double xj = -cosl(pi * j / N);
    for (int it = 0; it < 100; ++it) {
      long double pn, pn1;
      legendre2(N, xj, &pn, &pn1);
      long double dx = (xj * pn - pn1) / ((N + 1) * pn);
      xj -= dx;
      if (fabsl(dx) < 1e-30L) break;
    }
    if (j == 0) xj = -1.0L;
    if (j == N) xj = 1.0L;
    long double pn, pn1;
    legendre2(N, xj, &pn, &pn1);
    w[j] = (T)(2.0L / ((long double)N * (N + 1) * pn * pn));
  }
}

// Binomial coefficients C(gamma, k), k = 1..K (K = kEosTerms), of
// (1+x)^gamma - 1 and the largest |x| (<= 0.1) for which the truncation
// error after K terms stays below 2^-56 of the sum:
// |R| <= |C(gamma,K+1)| |x|^(K+1) / (1 - |x|) (the coefficients decrease in
// magnitude for 1 < gamma < 2) against a sum of at least 0.9 gamma |x|.
inline void eos_series(double gamma, double* c, double* xmax) {
  long double ck = 1.0L;
  for (int k = 1; k <= kEosTerms; ++k) {
    ck = ck * ((long double)gamma - (k - 1)) / k;
    c[k - 1] = (double)ck;
  }
  long double cK1 = fabsl(ck * ((long double)gamma - kEosTerms) / (kEosTerms + 1));
  long double bound = ldexpl(1.0L, -56) * 0.9L * gamma * 0.9L / (cK1 > 0 ? cK1 : 1e-300L);
  long double xm = powl(bound, 1.0L / kEosTerms);
  *xmax = (double)(xm < 0.1L ? xm : 0.1L);
}

// Sizes a mesh description implies.
struct MeshGeom {
  int n[3];        // global nodes per direction
  long long np;    // n[0] n[1] n[2]
};

// Host-side checks of a mesh description (no GPU work).  XG_ERR_ARG for
// invalid values, XG_ERR_UNSUPPORTED for valid ones this build cannot run.
inline xg_status check_desc(const xg_mesh_desc* d, MeshGeom* g) {
  if (!d) return XG_ERR_ARG;
  for (int k = 0; k < 3; ++k) {
    if (d->nel[k] < 1) return XG_ERR_ARG;
    if (!(std::isfinite(d->lo[k]) && std::isfinite(d->hi[k]) && d->hi[k] > d->lo[k])) return XG_ERR_ARG;
    if (d->periodic[k] != 0 && d->periodic[k] != 1) return XG_ERR_ARG;
  }
  if (d->order < 1 || d->order > kMaxOrder) return XG_ERR_ARG;
  if (!(finite_pos(d->R) && finite_pos(d->cp) && finite_pos(d->cv) && finite_pos(d->p_a))) return XG_ERR_ARG;
  if (!(std::isfinite(d->g) && d->g >= 0.0 && std::isfinite(d->f_coriolis))) return XG_ERR_ARG;
  const double gamma = d->cp / d->cv;
  if (!(gamma > 1.0 && gamma < 2.0)) return XG_ERR_ARG;
  if (d->precision != XG_FP64 && d->precision != XG_DF64 && d->precision != XG_FP32)
    return XG_ERR_UNSUPPORTED;
  const int N = d->order;
  for (int k = 0; k < 3; ++k) {
    long long nk = (long long)N * d->nel[k] + (d->periodic[k] ? 0 : 1);
    if (nk > (1 << 24)) return XG_ERR_UNSUPPORTED;
    g->n[k] = (int)nk;
  }
  g->np = (long long)g->n[0] * g->n[1] * g->n[2];
  // one x line per CTA of the mixed form's x pass
  if (sizeof(double) * (5 * (size_t)(g->n[0] + 1) + 5 * (size_t)d->nel[0]) > 220 * 1024) return XG_ERR_UNSUPPORTED;
  if (g->n[1] > 65535 || g->n[2] > 65535) return XG_ERR_UNSUPPORTED;  // grid y/z limits
  return XG_OK;
}

// Launch constants of the line kernels for a checked description.
inline void fill_line_params(const xg_mesh_desc* d, const MeshGeom& g, LineParams* P) {
  memset(P, 0, sizeof(*P));
  const int N = d->order;
  double D[kMaxOrder + 1][kMaxOrder + 1];
  lgl_derivative(N, D);
  for (int k = 0; k < 3; ++k) {
    P->n[k] = g.n[k];
    P->nseg[k] = d->nel[k];
    P->per[k] = d->periodic[k];
    const double h = (d->hi[k] - d->lo[k]) / d->nel[k];
    for (int a = 0; a <= N; ++a) {
      const double face = (a == 0 || a == N) ? 0.5 : 1.0;
      for (int l = 0; l <= N; ++l) P->Dm[k][a][l] = -(2.0 / h) * face * D[a][l];
    }
  }
  P->np = g.np;
  const double gamma = d->cp / d->cv;
  eos_series(gamma, P->eos_c, &P->eos_xmax);
  P->gamma = gamma;
  P->f = d->f_coriolis;
  P->g = d->g;
}

// The same matrices -(2/h_d) D (rows 0 and N halved) in fixed point.
inline void fill_fix_params(const xg_mesh_desc* d, FixRows (&F)[3]) {
  const int N = d->order;
  long double D[kMaxOrder + 1][kMaxOrder + 1];
  lgl_derivative(N, D);
  FixMatrix M;
  for (int k = 0; k < 3; ++k) {
    const long double h = ((long double)d->hi[k] - d->lo[k]) / d->nel[k];
    for (int a = 0; a <= N; ++a)
      for (int l = 0; l <= N; ++l) M[a][l] = -(2.0L / h) * ((a == 0 || a == N) ? 0.5L : 1.0L) * D[a][l];
    fix_rows(N, M, &F[k]);
  }
}

// A double split into a double-float pair (host).
inline df split_df(double v) {
  const float h = (float)v;
  return {h, (float)(v - (double)h)};
}

// Launch constants of the double-float line kernels, from the FP64 ones.
inline void fill_df_params(const LineParams& P, DfParams* Q) {
  memset(Q, 0, sizeof(*Q));
  for (int k = 0; k < 3; ++k) {
    Q->n[k] = P.n[k];
    Q->nseg[k] = P.nseg[k];
    Q->per[k] = P.per[k];
    for (int a = 0; a <= kMaxOrder; ++a)
      for (int l = 0; l <= kMaxOrder; ++l) Q->Dm[k][a][l] = split_df(P.Dm[k][a][l]);
  }
  Q->np = P.np;
  for (int k = 0; k < 3; ++k) Q->eos_c[k] = split_df(P.eos_c[k]);
  for (int k = 3; k < kEosTerms; ++k) Q->eos_g[k - 3] = (float)P.eos_c[k];
  Q->eos_xmax = (float)P.eos_xmax;
  Q->gamma = P.gamma;
  Q->f = split_df(P.f);
  Q->g = split_df(P.g);
  Q->P64 = P;
}

// Launch constants of the FP32 line kernels, from the FP64 ones.
inline void fill_f32_params(const LineParams& P, FParams* Q) {
  memset(Q, 0, sizeof(*Q));
  for (int k = 0; k < 3; ++k) {
    Q->n[k] = P.n[k];
    Q->nseg[k] = P.nseg[k];
    Q->per[k] = P.per[k];
    for (int a = 0; a <= kMaxOrder; ++a)
      for (int l = 0; l <= kMaxOrder; ++l) Q->Dm[k][a][l] = (float)P.Dm[k][a][l];
  }
  Q->np = P.np;
  for (int k = 0; k < 3; ++k) Q->eos_c[k] = split_df(P.eos_c[k]);
  for (int k = 3; k < kEosTerms; ++k) Q->eos_g[k - 3] = (float)P.eos_c[k];
  Q->eos_xmax = (float)P.eos_xmax;
  Q->gamma = P.gamma;
  Q->f = (float)P.f;
  Q->g = (float)P.g;
}

// Raise a kernel's dynamic shared-memory limit to at least `bytes`.  The
// limit is an attribute of the kernel function on the device, shared by
// every context (and every translation unit that launches the kernel), so
// it is only ever raised: lowering it for one mesh would break the launches
// of a larger mesh that is still alive.
template <typename F>
inline cudaError_t raise_dynamic_smem(F* func, size_t bytes) {
  static std::mutex m;
  std::lock_guard<std::mutex> lock(m);
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, (const void*)func);
  if (e != cudaSuccess) return e;
  if ((size_t)a.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
  return cudaFuncSetAttribute((const void*)func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Launch of a kernel that begins with stage_kernel_begin: where the stream's last
// work is a kernel, the launch is paid while that one runs, and the wait at the
// kernel's start keeps the order (no kernel lets its successor in before its own
// end: blocks that wait took room and issue slots from blocks that work, 24.1
// against 16.4 us below).  A mixed stage on 33^3 nodes 20.9 -> 16.4 us, FP32 18.6
// -> 13.3, FP64 26.5 -> 20.5.
template <typename... P, typename... A>
inline cudaError_t launch_stage_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                       const A&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

}  // namespace xg
