// xg_closure.cu -- learned subgrid closure (include/xg_closure.h).
//
// Kernels:
//   * features of a state: q, assembled gradients, heating (k_features);
//   * restriction of fine fields to coarse nodes, one axis at a time
//     (k_interp_z, k_interp_y, k_interp_x);
//   * training in FP32 on the CUDA cores: forward and back-propagation over
//     chunks of samples with the weights and activations in shared memory
//     and the block's gradient sums in registers (k_mlp_grad, each gradient
//     entry owned by one thread so the sums are deterministic), the
//     fixed-order reduction of the block partials (k_mlp_reduce), Adam
//     (k_adam), column statistics (k_col_stats);
//   * inference on the fifth-generation tensor cores (tcgen05.mma, bfloat16
//     operands in shared memory, FP32 accumulators in TMEM): persistent CTAs
//     of 128 threads take 128 samples per tile, one row of every product per
//     thread; bias, SiLU and the bfloat16 rounding of the hidden activations
//     run on the CUDA cores between the layers.  k_closure computes the
//     features of each tile's nodes straight from the state and runs the
//     network on them; k_mlp_bf16 runs it on given features.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include "../../include/xg_closure.h"
#include "xg_ctx.h"
#include "xg_setup.h"
#include "xg_tc.cuh"

namespace xg {

constexpr int kIn = XG_CLOSURE_IN, kHid = XG_CLOSURE_HIDDEN, kOut = XG_CLOSURE_OUT;
constexpr int kParams = XG_CLOSURE_PARAMS;
// Normalised inputs are clamped to [-kClampIn, kClampIn]: a state outside
// the training distribution cannot drive the network's output without bound.
constexpr float kClampIn = 8.0f;
__device__ __forceinline__ float norm_in(float x, float mean, float scale) {
  return fminf(fmaxf((x - mean) * scale, -kClampIn), kClampIn);
}
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid,
              kOffB2 = kOffW2 + kHid * kHid, kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kOut * kHid;
static_assert(kOffB3 + kOut == kParams, "parameter layout");

// ------------------------------------------------------------------ features

// The stencil of the assembled derivative along direction d at global
// index g of a line starting at offset base (stride sd): the node's segment
// (row a of the scaled matrix Dm = -(2/h) D, rows 0 and N halved), at a
// shared face also the segment before (its row N), at a wall the one
// segment's row doubled.  Built once per direction and applied to all five
// variables.
template <int N>
struct LineStencil {
  int off[2 * (N + 1)];   // within one variable's array (np < 2^31)
  float r0[N + 1], r1[N + 1];
  bool two;
  float scale;
};

template <int N>
__device__ __forceinline__ void line_stencil(const FParams& P, int d, long long base, long long sd, int g,
                                             LineStencil<N>& L) {
  const int nd = P.n[d], nseg = P.nseg[d];
  int s = g / N;
  if (s >= nseg) s = nseg - 1;
  const int a = g - s * N;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    int k = s * N + l;
    if (k >= nd) k -= nd;
    L.off[l] = (int)(base + sd * k);
    L.r0[l] = P.Dm[d][a][l];
  }
  L.two = a == 0 && (s > 0 || P.per[d]);
  L.scale = (a == N || (a == 0 && !L.two)) ? -2.0f : -1.0f;   // the sign undoes Dm's minus
  const int s2 = s > 0 ? s - 1 : nseg - 1;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    int k = s2 * N + l;
    if (k >= nd) k -= nd;
    L.off[N + 1 + l] = L.two ? (int)(base + sd * k) : L.off[l];
    L.r1[l] = L.two ? P.Dm[d][N][l] : 0.0f;
  }
}

template <int N>
__device__ __forceinline__ float line_apply(const LineStencil<N>& L, const float* __restrict__ f) {
  float acc = 0.0f;
#pragma unroll
  for (int l = 0; l <= N; ++l) acc = fmaf(L.r0[l], f[L.off[l]], acc);
  if (L.two) {
#pragma unroll
    for (int l = 0; l <= N; ++l) acc = fmaf(L.r1[l], f[L.off[N + 1 + l]], acc);
  }
  return L.scale * acc;
}

// The 21 features of node I, handed to emit(f, value): per direction the
// stencil once, then that direction's derivative of all five variables.
template <int N, typename Emit>
__device__ __forceinline__ void node_features(const FParams& P, const float* __restrict__ q,
                                              const float* __restrict__ S, long long I, Emit emit) {
  const long long np = P.np;
  const int nx = P.n[0], ny = P.n[1];
  const int gx = (int)(I % nx);
  const long long r = I / nx;
  const int gy = (int)(r % ny), gz = (int)(r / ny);
#pragma unroll
  for (int v = 0; v < 5; ++v) emit(v, q[v * np + I]);
#pragma unroll 1
  for (int d = 0; d < 3; ++d) {
    LineStencil<N> L;
    if (d == 0) line_stencil<N>(P, 0, I - gx, 1, gx, L);
    else if (d == 1) line_stencil<N>(P, 1, I - (long long)gy * nx, nx, gy, L);
    else line_stencil<N>(P, 2, I - (long long)gz * nx * ny, (long long)nx * ny, gz, L);
#pragma unroll
    for (int v = 0; v < 5; ++v) emit(5 + 3 * v + d, line_apply<N>(L, q + v * np));
  }
  emit(20, S ? S[I] : 0.0f);
}

template <int N>
__global__ void __launch_bounds__(128) k_features(const FParams P, const float* __restrict__ q,
                                                  const float* __restrict__ S, float* __restrict__ X) {
  const long long I = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (I >= P.np) return;
  const long long np = P.np;
  node_features<N>(P, q, S, I, [&](int f, float v) { X[f * np + I] = v; });
}

// ------------------------------------------------------------------ restriction

// One axis of the restriction: coarse node c takes the np_f = N_f + 1 values of
// its fine element from fine node start[c] on, with weights w[c][.].  one[c]:
// the point that the coarse node falls on (its weight is 1 and the others are
// below 2^-60), or -1: half of the coarse nodes of a mesh refined by two, which
// then cost no FP64 operation.
struct InterpAxis {
  const int* start;
  const int* one;
  const double* w;
  int n_in, n_out, npts;
};

// One coarse node's weights and points, in registers.
template <int NP>
struct InterpNode {
  int k[NP], one;   // one: the fine node it falls on, or -1
  double w[NP];
  __device__ __forceinline__ void load(const InterpAxis& A, int c) {
    const int s = A.start[c], o = A.one[c];
    one = o < 0 ? -1 : (s + o >= A.n_in ? s + o - A.n_in : s + o);
#pragma unroll
    for (int a = 0; a < NP; ++a) {
      k[a] = s + a >= A.n_in ? s + a - A.n_in : s + a;
      w[a] = A.w[c * NP + a];
    }
  }
  // at(k): the value of fine node k.  A value that is not finite counts with
  // every weight, a zero among them.
  template <typename At>
  __device__ __forceinline__ double value(At at) const {
    if (one >= 0) {
      unsigned e = 0;
#pragma unroll
      for (int a = 0; a < NP; ++a)
        if (k[a] != one) e = max(e, (unsigned)__double2hiint(at(k[a])) & 0x7ff00000u);
      const double v = at(one);
      return e == 0x7ff00000u ? __hiloint2double(0x7ff80000, 0) : v;
    }
    double r = 0.0;
#pragma unroll
    for (int a = 0; a < NP; ++a) r = fma(w[a], at(k[a]), r);
    return r;
  }
};

// The three passes, z, y, x, over the n planes from p0 on (of nvar n_zc
// [variable][coarse level]) of one chunk: z reads src and writes out [plane]
// [y_f][x_f], y writes [plane][y_c][x_f], x the result.  With z first every
// pass runs along contiguous lines, no index is divided, and a chunk's
// intermediates stay in L2.  A thread of the z and y passes walks along the
// interpolated axis, so that the fine values that consecutive coarse nodes share
// come from L1: one coarse node a thread read five values from L2 for each.
// Blocks are as wide as the lines are (interp_width), with several planes or lines
// where these are short, and a small plane's walk along z is cut into slices
// (blockIdx.y): one element of 5 x 5 fine columns by 2,000 along z, five variables,
// 13.7 -> 0.18 ms a call.
template <int NP>
__global__ void __launch_bounds__(256) k_interp_z(const double* __restrict__ in, double* __restrict__ out,
                                                  const InterpAxis A, long long plane, int p0, int np) {
  const int lo = (int)((long long)np * blockIdx.y / gridDim.y), hi = (int)((long long)np * (blockIdx.y + 1) / gridDim.y);
  for (long long i = blockIdx.x * 256ll + threadIdx.x; i < plane; i += gridDim.x * 256ll) {
    int v = (p0 + lo) / A.n_out, c = p0 + lo - v * A.n_out;
    const double* f = in + (long long)v * A.n_in * plane + i;
    double* o = out + lo * plane + i;
    for (int p = lo; p < hi; ++p) {
      InterpNode<NP> n;
      n.load(A, c);
      *o = n.value([&](int k) { return f[k * plane]; });
      o += plane;
      if (++c == A.n_out) {
        c = 0;
        f += A.n_in * plane;
      }
    }
  }
}

constexpr int kInterpRows = 16;   // coarse lines a thread of the y pass walks
template <int NP>
__global__ void __launch_bounds__(128) k_interp_y(const double* __restrict__ in, double* __restrict__ out,
                                                  const InterpAxis A, int nx, int np) {
  const int p = blockIdx.z * blockDim.y + threadIdx.y;
  if (p >= np) return;
  const double* f = in + (long long)p * A.n_in * nx;
  double* o = out + (long long)p * A.n_out * nx;
  for (int c0 = blockIdx.y * kInterpRows; c0 < A.n_out; c0 += gridDim.y * kInterpRows)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nx; i += gridDim.x * blockDim.x)
      for (int c = c0; c < min(c0 + kInterpRows, A.n_out); ++c) {
        InterpNode<NP> n;
        n.load(A, c);
        o[(long long)c * nx + i] = n.value([&](int k) { return f[(long long)k * nx + i]; });
      }
}

// A thread keeps its coarse node and walks down the lines.
template <int NP>
__global__ void __launch_bounds__(128) k_interp_x(const double* __restrict__ in, double* __restrict__ out,
                                                  const InterpAxis A, long long lines) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= A.n_out) return;
  InterpNode<NP> n;
  n.load(A, c);
  for (long long j = (long long)blockIdx.y * blockDim.y + threadIdx.y; j < lines; j += (long long)gridDim.y * blockDim.y)
    out[j * A.n_out + c] = n.value([&](int k) { return in[j * A.n_in + k]; });
}

// Threads along a line of n nodes in a block of 128.
inline int interp_width(int n) {
  int w = 128;
  while (w > 1 && w / 2 >= n) w /= 2;
  return w;
}

// The passes of one chunk of n planes.
template <int NP>
cudaError_t interp_chunk(const double* src, double* t1, double* t2, double* dst, const InterpAxis (&A)[3], int p0,
                         unsigned n, cudaStream_t st) {
  const int nx = A[0].n_in, nyf = A[1].n_in, nyc = A[1].n_out;
  const long long plane = (long long)nx * nyf;
  const unsigned bz = (unsigned)std::min<long long>((plane + 255) / 256, 1 << 20);
  const unsigned slices = std::min(n, (1024u + bz - 1) / bz);   // about 2^18 threads
  k_interp_z<NP><<<dim3(bz, slices), 256, 0, st>>>(src, t1, A[2], plane, p0, (int)n);
  const int wy = interp_width(nx), ry = 128 / wy;
  const unsigned by = (unsigned)std::min((nyc + kInterpRows - 1) / kInterpRows, 65535);
  k_interp_y<NP><<<dim3((unsigned)((nx + wy - 1) / wy), by, (n + ry - 1) / ry), dim3(wy, ry), 0, st>>>(t1, t2, A[1], nx, (int)n);
  const int wx = interp_width(A[0].n_out), rx = 128 / wx;
  const long long lines = (long long)nyc * n;
  k_interp_x<NP><<<dim3((unsigned)((A[0].n_out + wx - 1) / wx), (unsigned)std::min<long long>((lines + 4 * rx - 1) / (4 * rx), 65535)),
                   dim3(wx, rx), 0, st>>>(t2, dst, A[0], lines);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ training (FP32)

__device__ __forceinline__ float silu_f(float z) { return z / (1.0f + expf(-z)); }

// Sums of products over shared memory are bound by its reads (an output per
// thread reads two floats per FMA), so every product below gives a thread a
// tile of outputs and reads four floats at a time: 4 x 4 for the layers and the
// back-propagated delta, 8 x 4 for the second layer's gradient.  Rows of
// samples are kPitch = 36 floats apart, so lanes on consecutive rows read
// distinct banks.  The gradients stay in registers over the block's chunks,
// each entry owned by one thread (the sums are deterministic); SiLU and its
// derivative come from one exponential.  4,096 samples: 57 -> 23 us a launch
// (four warps an SM, latency); a whole call with 200,000: 2.0 -> 0.42 ms.
constexpr int kTrainThreads = 128;
constexpr int kChunk = 32;   // samples per pass through the network
constexpr int kPitch = kChunk + 4;
constexpr int kWPitch = kHid + 4;
constexpr int kTrainX = (kIn * kChunk + kTrainThreads - 1) / kTrainThreads;    // input values per thread
constexpr int kTrainT = (kOut * kChunk + kTrainThreads - 1) / kTrainThreads;

struct TrainSmem {
  float W1t[kIn][kHid];       // [input][output]
  float W2t[kHid][kWPitch];   // [input][output]
  float W2[kHid][kHid];       // [output][input]
  float W3[kOut][kHid];
  float b1[kHid], b2[kHid], b3[8];
  float stat[48];             // input mean and scale, 1 / output scale
  float x[kIn][kPitch];
  float h1[kHid][kPitch], g1[kHid][kPitch];   // SiLU and its derivative; g1 later the first layer's delta
  float h2[kHid][kPitch], g2[kHid][kPitch];   // g2 later the second layer's delta
  float t[kOut][kPitch];                      // targets, then the output delta
  float ypart[4][kOut][kChunk];
};

__device__ __forceinline__ void silu_both(float z, float& h, float& d) {
  const float s = 1.0f / (1.0f + expf(-z));
  h = z * s;
  d = s * (1.0f + z * (1.0f - s));
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

// a[k][l] += sum_i W[i][o0 + k] v[i][s0 + l], i < K
template <int K, int WP>
__device__ __forceinline__ void train_product(const float* W, const float* v, int o0, int s0, float (&a)[4][4]) {
#pragma unroll 4
  for (int i = 0; i < K; ++i) {
    const float4 w = ld4(W + i * WP + o0), x = ld4(v + i * kPitch + s0);
    const float wk[4] = {w.x, w.y, w.z, w.w}, xl[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int l = 0; l < 4; ++l) a[k][l] = fmaf(wk[k], xl[l], a[k][l]);
  }
}

// a hidden layer: rows o0.. of SiLU(W v + b) and its derivative
template <int K, int WP>
__device__ __forceinline__ void train_layer(const float* W, const float* b, const float* v, float (*h)[kPitch],
                                            float (*g)[kPitch], int o0, int s0) {
  float a[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int l = 0; l < 4; ++l) a[k][l] = b[o0 + k];
  train_product<K, WP>(W, v, o0, s0, a);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float hv[4], gv[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) silu_both(a[k][l], hv[l], gv[l]);
    *reinterpret_cast<float4*>(&h[o0 + k][s0]) = make_float4(hv[0], hv[1], hv[2], hv[3]);
    *reinterpret_cast<float4*>(&g[o0 + k][s0]) = make_float4(gv[0], gv[1], gv[2], gv[3]);
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float c) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, c))));
}

// Samples [begin, end) of this block; writes the block's gradient sums and
// loss partial.  scale = 2 / (5 n) (the derivative of the mean square).
__global__ void __launch_bounds__(kTrainThreads, 2)
    k_mlp_grad(const float* __restrict__ params, const float* __restrict__ X, const float* __restrict__ T,
               long long ld, long long n, const float* __restrict__ in_mean, const float* __restrict__ in_scale,
               const float* __restrict__ out_scale, float* __restrict__ partial, double* __restrict__ lossp,
               float scale) {
  extern __shared__ __align__(16) unsigned char smraw[];
  TrainSmem& S = *reinterpret_cast<TrainSmem*>(smraw);
  __shared__ double red[kTrainThreads / 32];
  const int tid = threadIdx.x;
  for (int k = tid; k < kHid * kIn; k += kTrainThreads) S.W1t[k % kIn][k / kIn] = params[kOffW1 + k];
  for (int k = tid; k < kHid * kHid; k += kTrainThreads) {
    const float w = params[kOffW2 + k];
    S.W2[k / kHid][k % kHid] = w;
    S.W2t[k % kHid][k / kHid] = w;
  }
  for (int k = tid; k < kOut * kHid; k += kTrainThreads) S.W3[k / kHid][k % kHid] = params[kOffW3 + k];
  if (tid < kHid) {
    S.b1[tid] = params[kOffB1 + tid];
    S.b2[tid] = params[kOffB2 + tid];
  }
  if (tid < kIn) {
    S.stat[tid] = in_mean[tid];
    S.stat[kIn + tid] = in_scale[tid];
  }
  if (tid < kOut) {
    S.stat[2 * kIn + tid] = 1.0f / out_scale[tid];
    S.b3[tid] = params[kOffB3 + tid];
  }
  const long long begin = n * blockIdx.x / gridDim.x, end = n * (blockIdx.x + 1) / gridDim.x;
  double lacc = 0.0;
  const int lane = tid & 31, warp = tid >> 5;
  const int o0 = 4 * (tid & 15), s0 = 4 * (tid >> 4);   // this thread's 4 x 4 tile
  const int wi = tid & 15, wo = tid >> 4;               // W2 gradient: rows wo + 8 k, columns wi + 16 l
  const int ro = tid & 63, half = tid >> 6;             // W1 and W3 gradients, biases
  float G2[8][4] = {}, G1[11] = {}, G3[3] = {}, gb = 0.0f, gb3 = 0.0f;
  float xin[kTrainX], tin[kTrainT];
  auto fetch = [&](long long c0) {
    const int cn = (int)min((long long)kChunk, end - c0);
#pragma unroll
    for (int k = 0; k < kTrainX; ++k) {
      const int j = tid + k * kTrainThreads, f = j / kChunk, s = j % kChunk;
      xin[k] = j < kIn * kChunk && s < cn ? X[f * ld + c0 + s] : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kTrainT; ++k) {
      const int j = tid + k * kTrainThreads, o = j / kChunk, s = j % kChunk;
      tin[k] = j < kOut * kChunk && s < cn ? T[o * ld + c0 + s] : 0.0f;
    }
  };
  fetch(begin);
  __syncthreads();
  for (long long c0 = begin; c0 < end; c0 += kChunk) {
    const int cn = (int)min((long long)kChunk, end - c0);
#pragma unroll
    for (int k = 0; k < kTrainX; ++k) {
      const int j = tid + k * kTrainThreads, f = j / kChunk, s = j % kChunk;
      if (j < kIn * kChunk) S.x[f][s] = s < cn ? norm_in(xin[k], S.stat[f], S.stat[kIn + f]) : 0.0f;
    }
#pragma unroll
    for (int k = 0; k < kTrainT; ++k) {
      const int j = tid + k * kTrainThreads, o = j / kChunk, s = j % kChunk;
      if (j < kOut * kChunk) S.t[o][s] = tin[k] * S.stat[2 * kIn + o];
    }
    if (c0 + kChunk < end) fetch(c0 + kChunk);   // the next chunk's samples while this one is computed
    __syncthreads();
    train_layer<kIn, kHid>(&S.W1t[0][0], S.b1, &S.x[0][0], S.h1, S.g1, o0, s0);
    __syncthreads();
    train_layer<kHid, kWPitch>(&S.W2t[0][0], S.b2, &S.h1[0][0], S.h2, S.g2, o0, s0);
    __syncthreads();
    {   // outputs: a quarter of the hidden units per warp, one sample per lane
      float y[kOut] = {};
#pragma unroll 4
      for (int i = warp * (kHid / 4); i < (warp + 1) * (kHid / 4); ++i) {
        const float h = S.h2[i][lane];
#pragma unroll
        for (int o = 0; o < kOut; ++o) y[o] = fmaf(S.W3[o][i], h, y[o]);
      }
#pragma unroll
      for (int o = 0; o < kOut; ++o) S.ypart[warp][o][lane] = y[o];
    }
    __syncthreads();
    for (int k = tid; k < kOut * kChunk; k += kTrainThreads) {   // residual and output delta
      const int o = k / kChunk, s = k % kChunk;
      const float y = S.b3[o] + ((S.ypart[0][o][s] + S.ypart[1][o][s]) + (S.ypart[2][o][s] + S.ypart[3][o][s]));
      const float r = s < cn ? y - S.t[o][s] : 0.0f;
      lacc += (double)r * r;
      S.t[o][s] = scale * r;
    }
    __syncthreads();
    {   // second hidden layer's delta, in place of its derivative
      float d3[kOut];
#pragma unroll
      for (int o = 0; o < kOut; ++o) d3[o] = S.t[o][lane];
#pragma unroll 4
      for (int i = warp; i < kHid; i += kTrainThreads / 32) {
        float a = 0.0f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) a = fmaf(S.W3[o][i], d3[o], a);
        S.g2[i][lane] *= a;
      }
    }
    // W3 and b3 gradients (h2 and the output delta)
#pragma unroll 2
    for (int s = 0; s < kChunk; s += 4) {
      const float4 h = ld4(&S.h2[ro][s]);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int o = 3 * half + k;
        if (o < kOut) G3[k] = dot4(h, ld4(&S.t[o][s]), G3[k]);
      }
    }
    if (warp < kOut) {
      float a = S.t[warp][lane];
      if (warp == 0) {   // four warps, five outputs
        float a4 = S.t[4][lane];
#pragma unroll
        for (int q = 16; q > 0; q >>= 1) a4 += __shfl_xor_sync(0xffffffffu, a4, q);
        if (lane == 4) gb3 += a4;
      }
#pragma unroll
      for (int q = 16; q > 0; q >>= 1) a += __shfl_xor_sync(0xffffffffu, a, q);
      if (lane == warp) gb3 += a;
    }
    __syncthreads();
    // W2 gradient (the second delta and h1)
#pragma unroll 2
    for (int s = 0; s < kChunk; s += 4) {
      float4 h[4];
#pragma unroll
      for (int l = 0; l < 4; ++l) h[l] = ld4(&S.h1[wi + 16 * l][s]);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 d = ld4(&S.g2[wo + 8 * k][s]);
#pragma unroll
        for (int l = 0; l < 4; ++l) G2[k][l] = dot4(d, h[l], G2[k][l]);
      }
    }
    {   // first hidden layer's delta, in place of its derivative
      float a[4][4] = {};
      train_product<kHid, kHid>(&S.W2[0][0], &S.g2[0][0], o0, s0, a);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float4 g = ld4(&S.g1[o0 + k][s0]);
        *reinterpret_cast<float4*>(&S.g1[o0 + k][s0]) =
            make_float4(a[k][0] * g.x, a[k][1] * g.y, a[k][2] * g.z, a[k][3] * g.w);
      }
    }
    __syncthreads();
    // W1 gradient (the first delta and x), and a hidden bias: b1 by the first
    // half of the threads, b2 by the second
#pragma unroll 2
    for (int s = 0; s < kChunk; s += 4) {
      const float4 d = ld4(&S.g1[ro][s]);
      const float4 e = half == 0 ? d : ld4(&S.g2[ro][s]);
      gb += (e.x + e.y) + (e.z + e.w);
#pragma unroll
      for (int k = 0; k < 11; ++k) {
        const int f = 11 * half + k;
        if (f < kIn) G1[k] = dot4(d, ld4(&S.x[f][s]), G1[k]);
      }
    }
    __syncthreads();
  }
  float* out = partial + (long long)blockIdx.x * kParams;
#pragma unroll
  for (int k = 0; k < 11; ++k)
    if (11 * half + k < kIn) out[kOffW1 + ro * kIn + 11 * half + k] = G1[k];
#pragma unroll
  for (int k = 0; k < 8; ++k)
#pragma unroll
    for (int l = 0; l < 4; ++l) out[kOffW2 + (wo + 8 * k) * kHid + wi + 16 * l] = G2[k][l];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (3 * half + k < kOut) out[kOffW3 + (3 * half + k) * kHid + ro] = G3[k];
  out[(half == 0 ? kOffB1 : kOffB2) + ro] = gb;
  if (lane == warp) out[kOffB3 + warp] = gb3;
  if (warp == 0 && lane == 4) out[kOffB3 + 4] = gb3;
#pragma unroll
  for (int q = 16; q > 0; q >>= 1) lacc += __shfl_down_sync(0xffffffffu, lacc, q);
  if (lane == 0) red[warp] = lacc;
  __syncthreads();
  if (tid == 0) lossp[blockIdx.x] = (red[0] + red[1]) + (red[2] + red[3]);
}

// The blocks' gradient sums (32 entries a block, 8 threads over the partials of
// each) and, in the last block, the loss, all in a fixed order.
constexpr int kReduceWays = 8;
__global__ void __launch_bounds__(32 * kReduceWays)
    k_mlp_reduce(const float* __restrict__ partial, const double* __restrict__ lossp, int nblocks, double norm,
                 float* __restrict__ grad, double* __restrict__ loss) {
  __shared__ float sum[kReduceWays][32];
  const int k = blockIdx.x * 32 + threadIdx.x, w = threadIdx.y;
  float a = 0.0f;
  if (k < kParams)
    for (int b = w; b < nblocks; b += kReduceWays) a += partial[(long long)b * kParams + k];
  sum[w][threadIdx.x] = a;
  __syncthreads();
  if (w == 0 && k < kParams) {
#pragma unroll
    for (int j = 1; j < kReduceWays; ++j) a += sum[j][threadIdx.x];
    grad[k] = a;
  }
  if (blockIdx.x == gridDim.x - 1 && w == 1) {
    double s = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += 32) s += lossp[b];
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) s += __shfl_down_sync(0xffffffffu, s, q);
    if (threadIdx.x == 0) *loss = s * norm;
  }
}

// Adam; 1 - beta1 and 1 - beta2 come from the host in double precision
// (1.0f - 0.999f would carry a 5e-5 relative error into v).
__global__ void k_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                       const float* __restrict__ g, int n, float lr, float b1, float b2, float omb1,
                       float omb2, float eps, float c1, float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + omb1 * gk;
  const float vk = b2 * v[k] + omb2 * gk * gk;
  m[k] = mk;
  v[k] = vk;
  p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

__global__ void k_col_stats(const float* __restrict__ X, long long ld, long long n, double* __restrict__ out) {
  __shared__ double red[256];
  const int c = blockIdx.x, tid = threadIdx.x;
  const float* x = X + c * ld;
  double s = 0.0;
  for (long long i = tid; i < n; i += blockDim.x) s += x[i];
  red[tid] = s;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (tid < h) red[tid] += red[tid + h];
    __syncthreads();
  }
  const double mean = red[0] / (double)n;
  __syncthreads();
  double q = 0.0;
  for (long long i = tid; i < n; i += blockDim.x) {
    const double d = x[i] - mean;
    q += d * d;
  }
  red[tid] = q;
  __syncthreads();
  for (int h = blockDim.x / 2; h > 0; h >>= 1) {
    if (tid < h) red[tid] += red[tid + h];
    __syncthreads();
  }
  if (tid == 0) {
    out[2 * c] = mean;
    out[2 * c + 1] = sqrt(red[0] / (double)n);
  }
}

__global__ void k_mlp_fp32(const float* __restrict__ params, const float* __restrict__ X, long long ld,
                           long long n, const float* __restrict__ in_mean, const float* __restrict__ in_scale,
                           const float* __restrict__ out_scale, float* __restrict__ Y, long long ldy) {
  const long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (s >= n) return;
  float x[kIn], h1[kHid], h2[kHid];
  for (int f = 0; f < kIn; ++f) x[f] = norm_in(X[f * ld + s], in_mean[f], in_scale[f]);
  for (int o = 0; o < kHid; ++o) {
    float a = params[kOffB1 + o];
    for (int i = 0; i < kIn; ++i) a = fmaf(params[kOffW1 + o * kIn + i], x[i], a);
    h1[o] = silu_f(a);
  }
  for (int o = 0; o < kHid; ++o) {
    float a = params[kOffB2 + o];
    for (int i = 0; i < kHid; ++i) a = fmaf(params[kOffW2 + o * kHid + i], h1[i], a);
    h2[o] = silu_f(a);
  }
  for (int o = 0; o < kOut; ++o) {
    float a = params[kOffB3 + o];
    for (int i = 0; i < kHid; ++i) a = fmaf(params[kOffW3 + o * kHid + i], h2[i], a);
    Y[o * ldy + s] = a * out_scale[o];
  }
}

// ------------------------------------------------------------------ inference (tcgen05)
//
// Inference runs on the fifth-generation tensor cores.  A persistent CTA of
// 128 threads takes 128 samples at a time: they are the M = 128 rows of every
// product, one row per thread and per TMEM lane.  Per tile:
//   features -> A (bfloat16, shared memory)              all threads
//   D = A W1h^T   (K 32, N 64)                           one thread issues tcgen05.mma
//   A <- bf16(SiLU(2 (D + b1/2)))                        all threads: tcgen05.ld, FP32
//   D = A W2h^T   (K 64, N 64)
//   A <- bf16(SiLU(2 (D + b2/2)))
//   D = A W3^T    (K 64, N 16; outputs 5..15 are zero rows of W3)
//   y = (D + b3) * out_scale                             all threads, coalesced stores
// W1h and W2h are the bfloat16 weights halved (exact), so the accumulator
// holds h = z / 2 and SiLU(z) = h + h tanh(h) needs no further scaling.  The
// accumulator takes 64 TMEM columns; shared memory (31.5 KB per CTA) lets at
// most 7 CTAs share an SM (448 of its 512 columns), the launch bound 4.
constexpr int kTcRows = 128;             // samples per tile, the MMA's M
constexpr int kK1 = 32;                  // layer-1 K: 21 features, zero padded
constexpr int kN3 = 16;                  // layer-3 N: 5 outputs, zero padded
constexpr int kTcCols = 64;              // TMEM columns per CTA

// Packed inference constants (one device blob, copied to shared memory):
// the bfloat16 weights in the canonical K-major layout (tc::kmajor), then
// FP32 b1/2, b2/2, b3, in_mean, in_scale, out_scale.
struct InferPack {
  __nv_bfloat16 W1[kHid * kK1];
  __nv_bfloat16 W2[kHid * kHid];
  __nv_bfloat16 W3[kN3 * kHid];
  float hb1[kHid], hb2[kHid], b3[8];
  float mean[24], scale[24], oscale[8];
};
static_assert(sizeof(InferPack) % 16 == 0, "InferPack is copied as int4");

__global__ void k_pack(const float* __restrict__ p, const float* __restrict__ mean,
                       const float* __restrict__ scale, const float* __restrict__ oscale,
                       InferPack* __restrict__ out) {
  for (int k = threadIdx.x; k < kHid * kK1; k += blockDim.x) {
    const int o = k / kK1, i = k % kK1;
    out->W1[tc::kmajor(kHid, o, i)] = __float2bfloat16_rn(i < kIn ? 0.5f * p[kOffW1 + o * kIn + i] : 0.0f);
  }
  for (int k = threadIdx.x; k < kHid * kHid; k += blockDim.x) {
    const int o = k / kHid, i = k % kHid;
    out->W2[tc::kmajor(kHid, o, i)] = __float2bfloat16_rn(0.5f * p[kOffW2 + o * kHid + i]);
  }
  for (int k = threadIdx.x; k < kN3 * kHid; k += blockDim.x) {
    const int o = k / kHid, i = k % kHid;
    out->W3[tc::kmajor(kN3, o, i)] = __float2bfloat16_rn(o < kOut ? p[kOffW3 + o * kHid + i] : 0.0f);
  }
  for (int k = threadIdx.x; k < kHid; k += blockDim.x) {
    out->hb1[k] = 0.5f * p[kOffB1 + k];
    out->hb2[k] = 0.5f * p[kOffB2 + k];
  }
  for (int k = threadIdx.x; k < 24; k += blockDim.x) {
    out->mean[k] = k < kIn ? mean[k] : 0.0f;
    out->scale[k] = k < kIn ? scale[k] : 0.0f;
  }
  for (int k = threadIdx.x; k < 8; k += blockDim.x) {
    out->b3[k] = k < kOut ? p[kOffB3 + k] : 0.0f;
    out->oscale[k] = k < kOut ? oscale[k] : 0.0f;
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// SiLU(2h) = h (1 + tanh h) with the hardware tanh approximation (relative
// error ~2^-11), below the bfloat16 rounding that follows it.
__device__ __forceinline__ float silu_of_half(float h) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(h));
  return fmaf(h, t, h);
}

struct TcSmem {
  InferPack K;
  __nv_bfloat16 A[kTcRows * kHid];   // features (first 4 K-chunks) or hidden activations
  unsigned long long bar;            // mbarrier: MMA completion
  uint32_t tmem;                     // TMEM base address
};

__device__ __forceinline__ void load_pack(InferPack& dst, const InferPack* src) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(&dst);
  for (int k = threadIdx.x; k < (int)(sizeof(InferPack) / 16); k += blockDim.x) d[k] = s[k];
}

// One layer's products: makes this thread's writes of A visible to the
// tensor cores, synchronises the CTA, issues the K/16 MMAs from thread 0 and
// waits for them.  False (on every thread) when a wait ran out; the kernel
// then reports XG_ERR_TIMEOUT through the flag and stops.
__device__ __forceinline__ bool tc_layer(TcSmem& S, uint32_t w_addr, uint32_t w_lbo, int ksteps,
                                         uint32_t idesc, uint32_t& phase) {
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t bar = tc::smem_addr(&S.bar);
  if (threadIdx.x == 0) {
    const uint32_t a_addr = tc::smem_addr(S.A);
    constexpr uint32_t a_lbo = kTcRows * 16;
    for (int k = 0; k < ksteps; ++k) {
      tc::mma_bf16(S.tmem, tc::smem_desc(a_addr + 2 * k * a_lbo, a_lbo, 128),
                   tc::smem_desc(w_addr + 2 * k * w_lbo, w_lbo, 128), idesc, k > 0);
    }
    tc::commit(bar);
  }
  const bool ok = tc::mbar_wait(bar, phase, tc::kWaitNs);
  phase ^= 1u;
  const int bad = __syncthreads_or(!ok);
  tc::fence_after_sync();
  return !bad;
}

// The hidden layer's epilogue: this thread's row of D (64 columns) plus the
// halved bias, SiLU, bfloat16 into its row of A.
__device__ __forceinline__ void tc_hidden(TcSmem& S, uint32_t lane_addr, const float* hb) {
  char* A = reinterpret_cast<char*>(S.A);
#pragma unroll
  for (int c0 = 0; c0 < kHid; c0 += 16) {
    uint32_t r[16];
    tc::tmem_ld16(lane_addr + c0, r);
    tc::tmem_wait_ld();
    uint32_t pk[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      pk[j] = pack_bf16(silu_of_half(__uint_as_float(r[2 * j]) + hb[c0 + 2 * j]),
                        silu_of_half(__uint_as_float(r[2 * j + 1]) + hb[c0 + 2 * j + 1]));
    const int off = (c0 >> 3) * (kTcRows * 16) + threadIdx.x * 16;
    *reinterpret_cast<uint4*>(A + off) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
    *reinterpret_cast<uint4*>(A + off + kTcRows * 16) = make_uint4(pk[4], pk[5], pk[6], pk[7]);
  }
}

// The persistent inference loop over the tiles of n samples: feat(s, emit)
// hands the raw features f = 0..20 of sample s < n to emit(f, value);
// Y[o * ldy + s] = out_scale_o * y_o.  On a wait that runs out, sets bit 1
// (value 2) of *flag and returns after freeing its TMEM.  blockDim.x = kTcRows.
template <typename Feat>
__device__ __forceinline__ void tc_infer(TcSmem& S, const InferPack* __restrict__ pack, long long n,
                                         float* __restrict__ Y, long long ldy, int* flag, Feat feat) {
  const int tid = threadIdx.x, warp = tid >> 5;
  load_pack(S.K, pack);
#pragma unroll
  for (int k = kIn; k < kK1; ++k) S.A[tc::kmajor(kTcRows, tid, k)] = __float2bfloat16_rn(0.0f);
  if (tid == 0) tc::mbar_init(tc::smem_addr(&S.bar), 1);
  if (warp == 0) tc::tmem_alloc(tc::smem_addr(&S.tmem), kTcCols);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t lane_addr = S.tmem + ((uint32_t)(32 * warp) << 16);
  const uint32_t w1 = tc::smem_addr(S.K.W1), w2 = tc::smem_addr(S.K.W2), w3 = tc::smem_addr(S.K.W3);
  uint32_t phase = 0;
  bool ok = true;
  const long long ntiles = (n + kTcRows - 1) / kTcRows;
  for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
    const long long s = t * kTcRows + tid;
    if (s < n) {
      feat(s, [&](int f, float v) {
        S.A[tc::kmajor(kTcRows, tid, f)] = __float2bfloat16_rn(norm_in(v, S.K.mean[f], S.K.scale[f]));
      });
    } else {
#pragma unroll
      for (int f = 0; f < kIn; ++f) S.A[tc::kmajor(kTcRows, tid, f)] = __float2bfloat16_rn(0.0f);
    }
    ok = tc_layer(S, w1, kHid * 16, kK1 / 16, tc::idesc_bf16(kTcRows, kHid), phase);
    if (!ok) break;
    tc_hidden(S, lane_addr, S.K.hb1);
    ok = tc_layer(S, w2, kHid * 16, kHid / 16, tc::idesc_bf16(kTcRows, kHid), phase);
    if (!ok) break;
    tc_hidden(S, lane_addr, S.K.hb2);
    ok = tc_layer(S, w3, kN3 * 16, kHid / 16, tc::idesc_bf16(kTcRows, kN3), phase);
    if (!ok) break;
    uint32_t r[8];
    tc::tmem_ld8(lane_addr, r);
    tc::tmem_wait_ld();
    if (s < n) {
#pragma unroll
      for (int o = 0; o < kOut; ++o) Y[o * ldy + s] = (__uint_as_float(r[o]) + S.K.b3[o]) * S.K.oscale[o];
    }
  }
  if (!ok && tid == 0) {
    // the products whose completion was not seen may still write tensor
    // memory: wait (bounded) once more for their commit before freeing it
    atomicOr(flag, 2);
    tc::mbar_wait(tc::smem_addr(&S.bar), phase ^ 1u, tc::kWaitNs);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(S.tmem, kTcCols);
  }
}

constexpr int kTcCtasPerSm = 4;

__global__ void __launch_bounds__(kTcRows, kTcCtasPerSm)
    k_mlp_bf16(const InferPack* __restrict__ pack, const float* __restrict__ X, long long ld, long long n,
               float* __restrict__ Y, long long ldy, int* flag) {
  __shared__ __align__(128) TcSmem S;
  tc_infer(S, pack, n, Y, ldy, flag, [&](long long s, auto&& emit) {
#pragma unroll
    for (int f = 0; f < kIn; ++f) emit(f, X[f * ld + s]);
  });
}

// The closure correction C [5][np]: the features of each tile's 128 nodes
// straight from the state, then the network.
template <int N>
__global__ void __launch_bounds__(kTcRows, kTcCtasPerSm)
    k_closure(const FParams P, const InferPack* __restrict__ pack, const float* __restrict__ q,
              const float* __restrict__ Sth, float* __restrict__ C, int* flag) {
  __shared__ __align__(128) TcSmem S;
  stage_kernel_begin();
  tc_infer(S, pack, P.np, C, P.np, flag,
           [&](long long I, auto&& emit) { node_features<N>(P, q, Sth, I, emit); });
}

// The bounded wait of the tensor-core kernels, made to run out: one CTA
// allocates TMEM, initialises an mbarrier that nothing will complete, waits
// for it with the limit, records the timeout in *status and frees its TMEM
// (the path every tcgen05 kernel here takes when a wait gives up).
__global__ void k_tc_wait_selftest(unsigned long long limit_ns, int* status) {
  __shared__ unsigned long long bar;
  __shared__ uint32_t tmem;
  const int warp = threadIdx.x >> 5;
  if (warp == 0) tc::tmem_alloc(tc::smem_addr(&tmem), 32);
  if (threadIdx.x == 0) tc::mbar_init(tc::smem_addr(&bar), 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const bool ok = tc::mbar_wait(tc::smem_addr(&bar), 0, limit_ns);
  const int bad = __syncthreads_or(!ok);
  if (threadIdx.x == 0) *status = bad ? 2 : 0;
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, 32);
  }
}

// Persistent grid: kTcCtasPerSm CTAs per SM, at most one per tile.  (The
// occupancy calculator reports one CTA per SM for these kernels, although
// their registers and shared memory admit kTcCtasPerSm, and the hardware
// does co-schedule them; the grid is therefore sized from the launch bound.)
inline int tc_grid(long long n) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long tiles = (n + kTcRows - 1) / kTcRows;
  return (int)std::max(1LL, std::min(tiles, (long long)kTcCtasPerSm * std::max(sms, 1)));
}

}  // namespace xg

using xg::InferPack;

// ------------------------------------------------------------------ stage hook

// Called by the FP32 stage before its passes when the closure is on:
// C = correction of the stage's input state.
cudaError_t closure_launch(xg_ctx* c, const float* q, cudaStream_t st) {
  const float* S = c->has_forcing ? (const float*)c->S : nullptr;
  const InferPack* K = (const InferPack*)c->cl_pack;
  const long long np = c->np;
  switch (c->d.order) {
#define XG_CLOSURE_CASE(n)                                                                              \
  case n: {                                                                                             \
    if (!c->cl_grid) c->cl_grid = xg::tc_grid(np);                                                      \
    const unsigned g = (unsigned)c->cl_grid;                                                            \
    xg::launch_stage_kernel(xg::k_closure<n>, g, xg::kTcRows, 0, st, c->Pf, K, q, S, c->cl_C, c->flag);   \
    break;                                                                                              \
  }
    XG_CLOSURE_CASE(1) XG_CLOSURE_CASE(2) XG_CLOSURE_CASE(3) XG_CLOSURE_CASE(4)
    XG_CLOSURE_CASE(5) XG_CLOSURE_CASE(6) XG_CLOSURE_CASE(7) XG_CLOSURE_CASE(8)
#undef XG_CLOSURE_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

void closure_free(xg_ctx* c) {
  cudaFree(c->cl_pack);
  cudaFree(c->cl_C);
  c->cl_pack = nullptr;
  c->cl_C = nullptr;
  c->closure = false;
  c->cl_fixed = false;
}

namespace xg {

// out = s (a - b), FP64 (out may alias a or b: each element is read before it is written)
__global__ void k_scaled_difference(const double* a, const double* b, double s, long long n, double* out) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    out[i] = s * (a[i] - b[i]);
}

// dst = (float) src, rounded to nearest
__global__ void k_round_to_f32(const double* __restrict__ src, long long n, float* __restrict__ dst) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    dst[i] = __double2float_rn(src[i]);
}

inline unsigned stream_grid(long long n) {
  return (unsigned)std::max(1LL, std::min((n + 255) / 256, 152LL * 16));
}

}  // namespace xg

namespace {

xg_status cuda_status(cudaError_t e, const char* where) {
  if (e == cudaSuccess) return XG_OK;
  fprintf(stderr, "xg_closure: %s: %s\n", where, cudaGetErrorString(e));
  cudaGetLastError();
  return e == cudaErrorMemoryAllocation ? XG_ERR_OOM : XG_ERR_CUDA;
}

// Scratch of the entry points that have no context, from a memory pool of the
// library's own per device: stream-ordered, so calls on several streams and
// threads each get memory of their own, and freed by each call.  The pool keeps
// up to kScratchKept bytes for the next call (cudaMalloc and cudaFree took most
// of a training step) and gives what is beyond that back at the next
// synchronisation.  The driver grows a pool by 32 MB at a time, so a smaller
// limit would keep nothing: 218 us a call with 16 MB, 61 us with 64.
constexpr unsigned long long kScratchKept = 64ull << 20;
constexpr int kScratchDevices = 64;
cudaError_t scratch_alloc(void** p, size_t bytes, int dev, cudaStream_t st) {
  static std::mutex m;
  static cudaMemPool_t pools[kScratchDevices] = {};
  if (dev < 0 || dev >= kScratchDevices) return cudaMallocAsync(p, bytes, st);
  {
    std::lock_guard<std::mutex> lock(m);
    if (!pools[dev]) {
      cudaMemPoolProps props;
      memset(&props, 0, sizeof(props));
      props.allocType = cudaMemAllocationTypePinned;
      props.location.type = cudaMemLocationTypeDevice;
      props.location.id = dev;
      cudaMemPool_t pool;
      cudaError_t e = cudaMemPoolCreate(&pool, &props);
      unsigned long long keep = kScratchKept;
      if (e == cudaSuccess) e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
      if (e != cudaSuccess) return e;
      pools[dev] = pool;
    }
  }
  return cudaMallocFromPoolAsync(p, bytes, pools[dev], st);
}

// 1-D restriction table: for each coarse node its fine element's first
// global node, the N_f + 1 Lagrange weights of the fine element's LGL points at
// the coarse node's position, and the point it falls on (InterpAxis::one).
// Coarse element e starts at fine element e nel_f / nel_c, in whole numbers and
// a remainder, and elements of one remainder share their weights (a mesh
// refined by a whole factor has one): long double is software arithmetic on
// Arm, where weights for every node took more than a millisecond an axis.
void axis_table(const xg_ctx* f, const xg_ctx* c, int d, std::vector<int>& start, std::vector<int>& one,
                std::vector<double>& w) {
  const int Nf = f->d.order, Nc = c->d.order;
  long double xf[xg::kMaxOrder + 1], xc[xg::kMaxOrder + 1];
  xg::lgl_nodes(Nf, xf);
  xg::lgl_nodes(Nc, xc);
  const int nelf = f->d.nel[d], nelc = c->d.nel[d];
  const int nf = f->n[d], ncn = c->n[d];
  start.assign(ncn, 0);
  one.assign(ncn, -1);
  w.assign((size_t)ncn * (Nf + 1), 0.0);
  struct Entry { int ef = -1, one = -1; double w[xg::kMaxOrder + 1]; };
  std::map<std::pair<int, int>, Entry> seen;   // (remainder, local node)
  for (int g = 0; g < ncn; ++g) {
    const int e = std::min(g / Nc, nelc - 1);
    const int a = g - Nc * e;
    const int whole = (int)((long long)e * nelf / nelc), rem = (int)((long long)e * nelf % nelc);
    Entry& t = seen[{rem, a}];
    if (t.ef < 0) {   // fine elements past `whole`, and the weights there
      const long double sf = ((long double)rem + (xc[a] + 1.0L) / 2.0L * nelf) / nelc;
      t.ef = std::max(0, (int)floorl(sf));
      if (whole + t.ef >= nelf) t.ef = nelf - 1 - whole;   // the last node of the box
      const long double loc = 2.0L * (sf - t.ef) - 1.0L;
      int big = 0, small = 0;
      for (int l = 0; l <= Nf; ++l) {
        long double L = 1.0L;
        for (int k = 0; k <= Nf; ++k)
          if (k != l) L *= (loc - xf[k]) / (xf[l] - xf[k]);
        t.w[l] = (double)L;
        if (std::fabs(t.w[l]) > std::fabs(t.w[big])) big = l;
      }
      for (int l = 0; l <= Nf; ++l) small += l != big && std::fabs(t.w[l]) < 0x1p-60;
      if (small == Nf && t.w[big] == 1.0) t.one = big;
    }
    start[g] = (int)((long long)Nf * (whole + t.ef) % nf);
    one[g] = t.one;
    for (int l = 0; l <= Nf; ++l) w[(size_t)g * (Nf + 1) + l] = t.w[l];
    if (whole + t.ef == nelf - 1) seen.erase({rem, a});    // (an entry made at the box's end is its own)
  }
}

}  // namespace

extern "C" {

xg_status xg_features(xg_ctx* c, float* X, void* stream) {
  if (!c || !X) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (!c->f32) return XG_ERR_UNSUPPORTED;
  if (!c->has_state) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const unsigned blocks = (unsigned)((c->np + 127) / 128);
  const float* q = (const float*)c->A;
  const float* S = c->has_forcing ? (const float*)c->S : nullptr;
  switch (c->d.order) {
    case 1: xg::k_features<1><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 2: xg::k_features<2><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 3: xg::k_features<3><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 4: xg::k_features<4><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 5: xg::k_features<5><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 6: xg::k_features<6><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 7: xg::k_features<7><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    case 8: xg::k_features<8><<<blocks, 128, 0, st>>>(c->Pf, q, S, X); break;
    default: return XG_ERR_ARG;
  }
  return cuda_status(cudaGetLastError(), "xg_features");
}

xg_status xg_restrict(const xg_ctx* f, const xg_ctx* c, const double* src, int nvar, double* dst,
                      void* stream) {
  if (!f || !c || !src || !dst || nvar < 1) return XG_ERR_ARG;
  for (int d = 0; d < 3; ++d) {
    if (f->d.lo[d] != c->d.lo[d] || f->d.hi[d] != c->d.hi[d]) return XG_ERR_ARG;
    if ((f->d.periodic[d] != 0) != (c->d.periodic[d] != 0)) return XG_ERR_ARG;
  }
  cudaStream_t st = (cudaStream_t)stream;
  const int* nf = f->n;
  const int* nc = c->n;
  // the tables of the three axes in one buffer: weights, starts, points
  const int npts = f->d.order + 1;
  const size_t nodes = (size_t)nc[0] + nc[1] + nc[2];
  std::vector<double> table(nodes * (npts + 1));
  double* hw = table.data();
  int* hs = reinterpret_cast<int*>(hw + nodes * npts);
  int* ho = hs + nodes;
  size_t off[3], at = 0;
  for (int d = 0; d < 3; ++d) {
    std::vector<int> start, one;
    std::vector<double> w;
    axis_table(f, c, d, start, one, w);
    std::copy(w.begin(), w.end(), hw + at * npts);
    std::copy(start.begin(), start.end(), hs + at);
    std::copy(one.begin(), one.end(), ho + at);
    off[d] = at;
    at += (size_t)nc[d];
  }
  // chunks of planes whose intermediates fit half the scratch that the pool keeps
  const long long plane = (long long)nf[0] * nf[1], mid = (long long)nf[0] * nc[1];
  const long long planes = (long long)nvar * nc[2];
  const long long per = 8 * (plane + mid);
  int chunk = (int)std::max<long long>(1, std::min<long long>(planes, (long long)(kScratchKept / 2) / per));
  chunk = std::min(chunk, 65535);
  // a result over the source is written only once all of it is read
  const size_t out_bytes = 8 * (size_t)planes * nc[0] * nc[1];
  const uintptr_t s0 = (uintptr_t)src, d0 = (uintptr_t)dst;
  const bool over = s0 < d0 + out_bytes && d0 < s0 + 8 * (size_t)nvar * f->np;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  const size_t tbytes = (8 * table.size() + 255) / 256 * 256;
  double* scratch = nullptr;
  if (e == cudaSuccess) e = scratch_alloc((void**)&scratch, tbytes + (size_t)per * chunk + (over ? out_bytes : 0), dev, st);
  if (e != cudaSuccess) return cuda_status(e, "xg_restrict");
  e = cudaMemcpyAsync(scratch, hw, 8 * table.size(), cudaMemcpyHostToDevice, st);
  const int* ds = reinterpret_cast<const int*>(scratch + nodes * npts);
  xg::InterpAxis A[3];
  for (int d = 0; d < 3; ++d)
    A[d] = {ds + off[d], ds + nodes + off[d], scratch + off[d] * npts, nf[d], nc[d], npts};
  double* t1 = scratch + tbytes / 8;
  double* t2 = t1 + plane * chunk;
  double* res = over ? t2 + mid * chunk : dst;
  for (long long p = 0; p < planes && e == cudaSuccess; p += chunk) {
    const unsigned n = (unsigned)std::min<long long>(chunk, planes - p);
    double* out = res + p * (long long)nc[0] * nc[1];
    switch (npts) {
      case 2: e = xg::interp_chunk<2>(src, t1, t2, out, A, (int)p, n, st); break;
      case 3: e = xg::interp_chunk<3>(src, t1, t2, out, A, (int)p, n, st); break;
      case 4: e = xg::interp_chunk<4>(src, t1, t2, out, A, (int)p, n, st); break;
      case 5: e = xg::interp_chunk<5>(src, t1, t2, out, A, (int)p, n, st); break;
      case 6: e = xg::interp_chunk<6>(src, t1, t2, out, A, (int)p, n, st); break;
      case 7: e = xg::interp_chunk<7>(src, t1, t2, out, A, (int)p, n, st); break;
      case 8: e = xg::interp_chunk<8>(src, t1, t2, out, A, (int)p, n, st); break;
      case 9: e = xg::interp_chunk<9>(src, t1, t2, out, A, (int)p, n, st); break;
      default: e = cudaErrorInvalidValue;
    }
  }
  if (e == cudaSuccess && over) e = cudaMemcpyAsync(dst, res, out_bytes, cudaMemcpyDeviceToDevice, st);
  const cudaError_t ef = cudaFreeAsync(scratch, st);
  if (e == cudaSuccess) e = ef;
  const cudaError_t es = cudaStreamSynchronize(st);
  if (e == cudaSuccess) e = es;
  return cuda_status(e, "xg_restrict");
}

xg_status xg_column_stats(const float* X, int ncol, long long ld, long long n, double* mean,
                          double* stdev, void* stream) {
  if (!X || ncol < 1 || n < 1 || ld < n || !mean || !stdev) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  double* d = nullptr;
  cudaError_t e = cudaMalloc((void**)&d, sizeof(double) * 2 * ncol);
  if (e == cudaSuccess) {
    xg::k_col_stats<<<ncol, 256, 0, st>>>(X, ld, n, d);
    e = cudaGetLastError();
  }
  std::vector<double> h(2 * (size_t)ncol);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), d, sizeof(double) * 2 * ncol, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(d);
  if (e != cudaSuccess) return cuda_status(e, "xg_column_stats");
  for (int k = 0; k < ncol; ++k) {
    mean[k] = h[2 * k];
    stdev[k] = h[2 * k + 1];
  }
  return XG_OK;
}

xg_status xg_mlp_loss_grad(const float* params, const float* X, const float* T, long long ld,
                           long long n, const float* in_mean, const float* in_scale,
                           const float* out_scale, float* grad, double* loss, void* stream) {
  if (!params || !X || !T || !in_mean || !in_scale || !out_scale || !grad || !loss) return XG_ERR_ARG;
  if (n < 1 || ld < n) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = (int)std::min<long long>((n + xg::kChunk - 1) / xg::kChunk, 2LL * sms);
  const size_t smem = sizeof(xg::TrainSmem);
  // the loss, the blocks' losses, their gradient sums
  double* buf = nullptr;
  cudaError_t e = xg::raise_dynamic_smem(xg::k_mlp_grad, smem);
  if (e == cudaSuccess)
    e = scratch_alloc((void**)&buf, sizeof(double) * (1 + (size_t)blocks) + sizeof(float) * (size_t)blocks * xg::kParams,
                      dev, st);
  double h = 0.0;
  if (e == cudaSuccess) {
    double* lossp = buf + 1;
    float* partial = (float*)(lossp + blocks);
    xg::k_mlp_grad<<<blocks, xg::kTrainThreads, smem, st>>>(params, X, T, ld, n, in_mean, in_scale, out_scale,
                                                           partial, lossp, (float)(2.0 / (5.0 * (double)n)));
    xg::k_mlp_reduce<<<(xg::kParams + 31) / 32, dim3(32, xg::kReduceWays), 0, st>>>(
        partial, lossp, blocks, 1.0 / (5.0 * (double)n), grad, buf);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, buf, sizeof(double), cudaMemcpyDeviceToHost, st);
    const cudaError_t ef = cudaFreeAsync(buf, st);
    if (e == cudaSuccess) e = ef;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e != cudaSuccess) return cuda_status(e, "xg_mlp_loss_grad");
  *loss = h;
  return XG_OK;
}

xg_status xg_mlp_adam(float* params, float* m, float* v, const float* grad, int nparams, int t,
                      double lr, double beta1, double beta2, double eps, void* stream) {
  if (!params || !m || !v || !grad || nparams < 1 || t < 1) return XG_ERR_ARG;
  if (!(lr > 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps >= 0.0))
    return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const double c1 = 1.0 - pow(beta1, t), c2 = 1.0 - pow(beta2, t);
  xg::k_adam<<<(nparams + 255) / 256, 256, 0, st>>>(params, m, v, grad, nparams, (float)lr, (float)beta1,
                                                    (float)beta2, (float)(1.0 - beta1), (float)(1.0 - beta2),
                                                    (float)eps, (float)c1, (float)c2);
  return cuda_status(cudaGetLastError(), "xg_mlp_adam");
}

xg_status xg_mlp_forward(const float* params, const float* X, long long ld, long long n,
                         const float* in_mean, const float* in_scale, const float* out_scale, float* Y,
                         long long ldy, int precision, void* stream) {
  if (!params || !X || !in_mean || !in_scale || !out_scale || !Y) return XG_ERR_ARG;
  if (n < 1 || ld < n || ldy < n) return XG_ERR_ARG;
  if (precision != XG_MLP_FP32 && precision != XG_MLP_BF16) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (precision == XG_MLP_FP32) {
    xg::k_mlp_fp32<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(params, X, ld, n, in_mean, in_scale,
                                                                 out_scale, Y, ldy);
    return cuda_status(cudaGetLastError(), "xg_mlp_forward");
  }
  // the packed network, then the timeout flag
  int dev = 0;
  cudaGetDevice(&dev);
  char* blob = nullptr;
  cudaError_t e = scratch_alloc((void**)&blob, sizeof(InferPack) + 16, dev, st);
  int hflag = 0;
  if (e == cudaSuccess) {
    InferPack* K = (InferPack*)blob;
    int* flag = (int*)(blob + sizeof(InferPack));
    e = cudaMemsetAsync(flag, 0, sizeof(int), st);
    if (e == cudaSuccess) {
      xg::k_pack<<<1, 256, 0, st>>>(params, in_mean, in_scale, out_scale, K);
      xg::k_mlp_bf16<<<xg::tc_grid(n), xg::kTcRows, 0, st>>>(K, X, ld, n, Y, ldy, flag);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hflag, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
    const cudaError_t ef = cudaFreeAsync(blob, st);
    if (e == cudaSuccess) e = ef;
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  if (e == cudaSuccess && hflag) return XG_ERR_TIMEOUT;
  return cuda_status(e, "xg_mlp_forward");
}

xg_status xg_tc_wait_selftest(long long limit_ns, void* stream) {
  if (limit_ns < 1 || limit_ns > 1000000000LL) return XG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int* d = nullptr;
  int h = -1;
  cudaError_t e = cudaMalloc((void**)&d, sizeof(int));
  if (e == cudaSuccess) {
    xg::k_tc_wait_selftest<<<1, 128, 0, st>>>((unsigned long long)limit_ns, d);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  }
  cudaFree(d);
  if (e != cudaSuccess) return cuda_status(e, "xg_tc_wait_selftest");
  return h == 2 ? XG_ERR_TIMEOUT : XG_OK;
}

xg_status xg_closure_set(xg_ctx* c, const float* params, const float* in_mean, const float* in_scale,
                         const float* out_scale, void* stream) {
  if (!c) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (!params) {
    c->closure = false;
    return XG_OK;
  }
  if (!in_mean || !in_scale || !out_scale) return XG_ERR_ARG;
  if (!c->f32) return XG_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  if (!c->cl_pack) e = cudaMalloc(&c->cl_pack, sizeof(InferPack));
  if (e == cudaSuccess && !c->cl_C) e = cudaMalloc((void**)&c->cl_C, sizeof(float) * 5 * (size_t)c->np);
  if (e == cudaSuccess) {
    xg::k_pack<<<1, 256, 0, st>>>(params, in_mean, in_scale, out_scale, (InferPack*)c->cl_pack);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    closure_free(c);
    return cuda_status(e, "xg_closure_set");
  }
  c->closure = true;
  c->cl_fixed = false;
  return XG_OK;
}

xg_status xg_correction_set(xg_ctx* c, const double* C, void* stream) {
  if (!c) return XG_ERR_ARG;
  if (c->failed) return XG_ERR_CUDA;
  if (!C) {
    if (c->cl_fixed) c->closure = c->cl_fixed = false;
    return XG_OK;
  }
  if (!c->f32) return XG_ERR_UNSUPPORTED;
  cudaStream_t st = (cudaStream_t)stream;
  const long long n = 5 * c->np;
  cudaError_t e = cudaSuccess;
  if (!c->cl_C) e = cudaMalloc((void**)&c->cl_C, sizeof(float) * (size_t)n);
  if (e == cudaSuccess) {
    xg::k_round_to_f32<<<xg::stream_grid(n), 256, 0, st>>>(C, n, c->cl_C);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    closure_free(c);
    return cuda_status(e, "xg_correction_set");
  }
  c->closure = true;
  c->cl_fixed = true;
  return XG_OK;
}

xg_status xg_closure_target(const double* a, const double* b, double s, long long n, double* out,
                            void* stream) {
  if (!a || !b || !out || n < 0) return XG_ERR_ARG;
  if (n == 0) return XG_OK;
  xg::k_scaled_difference<<<xg::stream_grid(n), 256, 0, (cudaStream_t)stream>>>(a, b, s, n, out);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? XG_OK : cuda_status(e, "xg_closure_target");
}

}  // extern "C"
