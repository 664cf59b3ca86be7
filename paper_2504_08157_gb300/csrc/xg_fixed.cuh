// xg_fixed.cuh -- FP64 line contractions in 64-bit fixed point on the integer
// pipe.
//
// GB300 issues 1.9 FP64 FMAs per clock and SM but 60 IMAD.WIDE (32 x 32 -> 64
// bits with a 64-bit addend; both measured), so a contraction of FP64 data
// with a constant matrix is cheaper in exact integer arithmetic:
//   * the values of a block (an element segment, or a plane tile) are written
//     as V = v 2^sv, |V| < 2^B, with one exponent for the block, B = 61 for
//     orders up to 4 and 60 above: the largest value keeps B bits and
//     every value down to 2^-8 (2^-7) of it all of its 53;
//   * the matrix is written once per mesh as C = c 2^sc, from its long double
//     entries, with sum_l |C_l| <= 2^60 over every assembled row (59 bits
//     against FP64's 53);
//   * both are split into limbs, X = h 2^30 + l with |l| <= 2^29 (so that what
//     is left out has no bias), and a product takes three IMAD.WIDE, hi += ch h
//     and mid += ch l + cl h; the low product (below 2^-60 of sum |c| max |v|) is
//     left out;
//   * a row that sums to zero up to its entries' rounding is made to sum to
//     zero in both limbs, which takes a few |cl| up to 2^30: then a constant
//     has no derivative at all, as in the difference form (with the low limbs'
//     sum left over it had one unit of r at some spacings).  Nothing overflows:
//     |hi| <= 2^61 and, with sum |cl| <= 4/3 (N + 1) 2^29 where sum cl = 0,
//     |mid| <= 2^60 + 4/3 (N + 1) 2^(B - 1) < 2^63;
//   * r = hi + mid 2^-30, rounded, is one FP64 value again by one conversion, times
//     2^(60 - sc - sv).
// The sums of a block are exact up to those cuts, about 2^-59 of
// sum |c| max |v|, where an FP64 FMA chain rounds at 2^-53 of its partial
// sums.  A block with an infinity or NaN has no exponent; its callers take
// the FP64 path or return NaN for the segment, as an FP64 chain would.
#pragma once

#include <cmath>

#include <cuda_runtime.h>

#include "xg_kernels.cuh"

namespace xg {

// c[a][l] = (ch[a][l] 2^30 + cl[a][l]) 2^-sc, rows a = 0..N
struct FixRows {
  int ch[kMaxOrder + 1][kMaxOrder + 1], cl[kMaxOrder + 1][kMaxOrder + 1];
  int sc;
};

// The largest absolute row sum that a node of the assembled operator sees: an
// interior row, or rows 0 and N together at a shared face.
using FixMatrix = long double[kMaxOrder + 1][kMaxOrder + 1];

inline double fix_row_sum(int N, const FixMatrix& c) {
  double most = 0.0, face = 0.0;
  for (int a = 0; a <= N; ++a) {
    double s = 0.0;
    for (int l = 0; l <= N; ++l) s += (double)fabsl(c[a][l]);
    if (a == 0 || a == N) face += s;
    most = std::fmax(most, s);
  }
  return std::fmax(most, face);
}

// sc for matrices whose largest row sum is `most` (directions that are summed
// as integers share it); ldexp of zero rows is harmless.
inline int fix_scale_of(double most) {
  int e = 0;
  if (most > 0.0 && std::isfinite(most)) std::frexp(most, &e);
  return 60 - e;
}

inline void fix_rows(int N, const FixMatrix& c, int sc, FixRows* F) {
  F->sc = sc;
  for (int a = 0; a <= kMaxOrder; ++a)
    for (int l = 0; l <= kMaxOrder; ++l) F->ch[a][l] = F->cl[a][l] = 0;
  for (int a = 0; a <= N; ++a) {
    long long C[kMaxOrder + 1], sum = 0;
    int big = 0;
    for (int l = 0; l <= N; ++l) {
      C[l] = llrintl(ldexpl(c[a][l], sc));
      sum += C[l];
      if (std::llabs(C[l]) > std::llabs(C[big])) big = l;
    }
    const bool zero = std::llabs(sum) <= 8 * (N + 1);   // up to the entries' rounding
    if (zero) C[big] -= sum;
    long long high[kMaxOrder + 1], low[kMaxOrder + 1], over = 0;
    for (int l = 0; l <= N; ++l) {
      low[l] = (long long)((unsigned long long)C[l] << 34) >> 34;   // signed 30 bits
      high[l] = (C[l] - low[l]) >> 30;
      over += high[l];
    }
    // the high limbs to a sum of zero as well (|over| <= (N + 1) / 2: the low
    // ones sum to -over 2^30), at the entries with the farthest low limbs
    while (zero && over != 0) {
      const int sg = over > 0 ? 1 : -1;
      int far = 0;
      for (int l = 1; l <= N; ++l)
        if (sg * low[l] < sg * low[far]) far = l;
      high[far] -= sg;
      low[far] += (long long)sg << 30;
      over -= sg;
    }
    for (int l = 0; l <= N; ++l) {
      F->ch[a][l] = (int)high[l];
      F->cl[a][l] = (int)low[l];
    }
  }
}

#ifdef __CUDACC__

struct fix2 {
  int h, l;
};

// biased exponent field of v
__device__ __forceinline__ int fix_exp(double v) { return (int)(((unsigned)__double2hiint(v) >> 20) & 0x7ffu); }

constexpr int kFixNonfinite = 0x7ff;

// The exponent used for a block whose largest field is e, against rows of
// scale sc: tiny blocks are cut at 2^-900 or so.
__device__ __forceinline__ int fix_block_exp(int e, int sc) { return max(e, max(128, sc + 2)); }

// Bits of a block's values for order N (see the overflow bound above).
__host__ __device__ constexpr int fix_bits(int N) { return N <= 4 ? 61 : 60; }

// sg V in limbs, V < 2^61: the high one rounded to nearest, but kept below 2^31
// (the low one is then up to 2^30).
__device__ __forceinline__ fix2 fix_limbs(unsigned long long V, int sg) {
  const unsigned h = min((unsigned)((V + (1ull << 29)) >> 30), 0x7fffffffu);
  return {(int)h * sg, (int)((unsigned)V - (h << 30)) * sg};
}

// v in the limbs of a block of exponent E >= fix_exp(v): |v| 2^(B - 1 - (E -
// 1023)) cut to an integer, both limbs with v's sign.
template <int N>
__device__ __forceinline__ fix2 fix_of(double v, int E) {
  constexpr int up = fix_bits(N) - 53;
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned long long M = ((unsigned long long)__funnelshift_l(lo, mh, up) << 32) | (unsigned long long)(lo << up);
  const unsigned s = (unsigned)E - ((hi >> 20) & 0x7ffu);
  unsigned long long V;
  asm("shr.u64 %0, %1, %2;" : "=l"(V) : "l"(M), "r"(s));   // clamps: 0 for s >= 64
  return fix_limbs(V, ((int)hi >> 31) | 1);
}

// 2^(60 - sc - sv) of a block of exponent E (NaN for a block that has none)
template <int N>
__device__ __forceinline__ double fix_unit(int E, int sc) {
  if (E == kFixNonfinite) return __hiloint2double(0x7ff80000, 0);
  return __hiloint2double(min(E + 61 - fix_bits(N) - sc, 2046) << 20, 0);
}

// hi + mid 2^-30 of row a, rounded
template <int N>
__device__ __forceinline__ long long fix_row(const FixRows& F, int a, const fix2 (&v)[N + 1]) {
  long long hi = 0, mid = 1ll << 29;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    hi += (long long)F.ch[a][l] * v[l].h;
    mid += (long long)F.ch[a][l] * v[l].l;
    mid += (long long)F.cl[a][l] * v[l].h;
  }
  return hi + (mid >> 30);
}

// ---------------------------------------------------------------- plane tiles
// A CTA takes E x E elements of one level.  Its nodes' x and y rows need the
// tile extended by the segment before it and its end face along each
// direction (a cross); the extended tile is converted once, with one exponent,
// into shared memory (two limbs a node), one thread takes a whole element
// segment of a line -- the matrix then comes from the constant bank at fixed
// offsets, and a segment's N + 1 values are read once for its N + 1 rows --
// and leaves its rows as 64-bit integers, which the nodes add up exactly: rows
// 0..N-1 in RA, row N, which belongs to the next segment's first node, in RB.
__host__ __device__ constexpr int fix_plane_elems(int N) { return 32 / N; }
constexpr int kFixThreads = 256;

template <int N>
struct FixPlane {
  static constexpr int E = fix_plane_elems(N);
  static constexpr int TS = E * N;            // <= 32: a warp takes a row of the tile, a lane a column
  static constexpr int LO = TS + 1;           // owned extent (a wall's last node included)
  static constexpr int LX = TS + N + 1;       // extended extent
  static constexpr int PV = LX | 1;           // odd pitches: lanes along either axis hit distinct banks
  static constexpr int PR = LO | 1;
  static constexpr int V = LX * PV;           // 8-byte slots
  static constexpr int RA = LO * PR;
  static constexpr int RB = (E + 1) * LO;
  static constexpr int kWarps = kFixThreads / 32;
  static constexpr int kRows = (LX + kWarps - 1) / kWarps;                   // rows per warp
  static constexpr int kSide = (LO * N + LX + kFixThreads - 1) / kFixThreads;    // the columns beside the tile's
  static constexpr int kLoads = kRows + kSide;
};

// Extent of tile (bx, by) as PlaneTile (xg_plane_f32.cuh) for any line
// parameters.
struct FixTile {
  int ekx, eky, x0, y0, ox, oy;
  bool hxl, hyl;
  template <int N, typename P>
  __device__ __forceinline__ void init(const P& p, int bx, int by) {
    constexpr int E = fix_plane_elems(N);
    ekx = min(E, p.nseg[0] - bx * E);
    eky = min(E, p.nseg[1] - by * E);
    x0 = bx * E * N;
    y0 = by * E * N;
    ox = ekx * N + (!p.per[0] && bx * E + ekx == p.nseg[0] ? 1 : 0);
    oy = eky * N + (!p.per[1] && by * E + eky == p.nseg[1] ? 1 : 0);
    hxl = bx > 0 || p.per[0];
    hyl = by > 0 || p.per[1];
  }
};

// Slot k of this thread in the extended tile: row jj and column ii (both
// offset by N); false where the thread has none.  The first kRows slots are
// rows of the tile's own TS columns, one warp a row; the rest are the N columns
// before them, of the owned rows, and the one after them, of every row (a
// wall's last column has y segments of its own).
template <int N>
__device__ __forceinline__ bool fix_plane_slot(int k, int& jj, int& ii) {
  using L = FixPlane<N>;
  if (k < L::kRows) {
    jj = (int)(threadIdx.x >> 5) + k * L::kWarps;
    ii = N + (int)(threadIdx.x & 31);
    return jj < L::LX && ii < N + L::TS;
  }
  const int t = (int)threadIdx.x + (k - L::kRows) * kFixThreads;
  if (t < L::LO * N) {
    const int r = t / N;
    jj = N + r;
    ii = t - r * N;
    return true;
  }
  jj = t - L::LO * N;
  ii = N + L::TS;
  return jj < L::LX;
}

// Loads the cross of one variable f (a level's first node) into registers and
// raises *emax to its largest exponent field.  X, Y: which directions' segments
// are needed.
template <int N, bool X, bool Y>
__device__ __forceinline__ void fix_plane_load(const double* __restrict__ f, const FixTile& T, int nx, int ny,
                                               double (&v)[FixPlane<N>::kLoads], int* emax) {
  using L = FixPlane<N>;
  int e = 0;
#pragma unroll
  for (int k = 0; k < L::kLoads; ++k) {
    int jj, ii;
    const bool has = fix_plane_slot<N>(k, jj, ii);
    const int i = ii - N, j = jj - N;
    // owned rows extended along x, owned columns extended along y
    const bool inx = j >= 0 && j < T.oy && (i >= 0 || T.hxl) && i <= T.ekx * N;
    const bool iny = i >= 0 && i < T.ox && (j >= 0 || T.hyl) && j <= T.eky * N;
    v[k] = 0.0;
    if (has && ((X && inx) || (Y && iny))) {
      int gx = T.x0 + i, gy = T.y0 + j;
      if (gx < 0) gx += nx;
      if (gy < 0) gy += ny;
      if (gx >= nx) gx -= nx;
      if (gy >= ny) gy -= ny;
      v[k] = f[gx + (long long)nx * gy];
    }
  }
#pragma unroll
  for (int k = 0; k < L::kLoads; ++k) e = max(e, fix_exp(v[k]));
  e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if ((threadIdx.x & 31) == 0) atomicMax(emax, e);
}

// The loaded values in limbs of a block of exponent E.
template <int N>
__device__ __forceinline__ void fix_plane_convert(const double (&v)[FixPlane<N>::kLoads], int E, fix2* V) {
  using L = FixPlane<N>;
#pragma unroll
  for (int k = 0; k < L::kLoads; ++k) {
    int jj, ii;
    if (fix_plane_slot<N>(k, jj, ii)) V[jj * L::PV + ii] = fix_of<N>(v[k], E);
  }
}

// Rows of every x segment (DIR 0) or y segment (DIR 1) of the tile: RA[j][i]
// the row of node (i, j) in the segment that starts at or before it, RB[s][.]
// row N of segment s - 1 (s = 0: the segment before the tile).
template <int N, int DIR>
__device__ __forceinline__ void fix_plane_rows(const FixRows& F, const FixTile& T, const fix2* V, long long* RA,
                                               long long* RB) {
  using L = FixPlane<N>;
  const int ns = (DIR == 0 ? T.ekx : T.eky) + 1, no = DIR == 0 ? T.oy : T.ox;
  const bool left = DIR == 0 ? T.hxl : T.hyl;
  for (int t = threadIdx.x; t < ns * L::LO; t += kFixThreads) {
    const int s = t / L::LO, o = t - s * L::LO;   // s - 1: the segment; o: the line
    if (o >= no || (s == 0 && !left)) continue;
    const fix2* p = DIR == 0 ? V + (o + N) * L::PV + s * N : V + s * N * L::PV + o + N;
    fix2 v[N + 1];
#pragma unroll
    for (int l = 0; l <= N; ++l) v[l] = p[DIR == 0 ? l : l * L::PV];
    RB[s * L::LO + o] = fix_row<N>(F, N, v);
    if (s > 0) {
#pragma unroll
      for (int a = 0; a < N; ++a) {
        const int g = (s - 1) * N + a;
        RA[DIR == 0 ? o * L::PR + g : g * L::PR + o] = fix_row<N>(F, a, v);
      }
    }
  }
}

// The assembled row of node g (0-based in the tile) on line o along DIR.
template <int N, int DIR>
__device__ __forceinline__ long long fix_plane_node(const FixTile& T, const long long* RA, const long long* RB,
                                                    int g, int o) {
  using L = FixPlane<N>;
  const int s = g / N, ek = DIR == 0 ? T.ekx : T.eky;
  if (s == ek) return 2 * RB[ek * L::LO + o];            // a wall's last node: its row twice
  const long long r = RA[DIR == 0 ? o * L::PR + g : g * L::PR + o];
  if (g != s * N) return r;
  if (s > 0 || (DIR == 0 ? T.hxl : T.hyl)) return r + RB[s * L::LO + o];
  return 2 * r;
}

// node(i, j) for every owned node of the tile: a warp takes a row, a lane a
// column; a wall's last column (i = TS) goes to the threads of its own.
template <int N, typename F>
__device__ __forceinline__ void fix_plane_nodes(const FixTile& T, F node) {
  using L = FixPlane<N>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane < min(T.ox, L::TS)) {
    for (int j = warp; j < T.oy; j += L::kWarps) node(lane, j);
  }
  if (T.ox > L::TS && (int)threadIdx.x < T.oy) node(L::TS, (int)threadIdx.x);
}

// One z segment's values (FP64, in registers) in limbs, with its own exponent.
template <int N>
__device__ __forceinline__ int fix_segment(const double (&v)[N + 1], int sc, fix2 (&f)[N + 1]) {
  int e = fix_exp(v[0]);
#pragma unroll
  for (int l = 1; l <= N; ++l) e = max(e, fix_exp(v[l]));
  const int E = e == kFixNonfinite ? e : fix_block_exp(e, sc);
#pragma unroll
  for (int l = 0; l <= N; ++l) f[l] = fix_of<N>(v[l], E);
  return E;
}

// Segments per thread of a marching z pass: enough chunks to give every SM
// 1,024 threads (a chunk start recomputes one segment's last row).
inline int fix_z_chunk(int nseg, long long columns, int sms) {
  long long chunks = (1024ll * sms + columns - 1) / columns;
  if (chunks < 1) chunks = 1;
  if (chunks > nseg) chunks = nseg;
  return (int)((nseg + chunks - 1) / chunks);
}

// ---------------------------------------------------------------- fluxes
// exponent field of v, 0 for an infinity or NaN
__device__ __forceinline__ int fix_exp_finite(double v, bool& bad) {
  const int e = fix_exp(v);
  const bool b = e == kFixNonfinite;
  bad |= b;
  return b ? 0 : e;
}

__device__ __forceinline__ bool fix_bad(double v) { return fix_exp(v) == kFixNonfinite; }

constexpr int kFixMark = (int)0x80000000;   // high limb of a value without an exponent: |h| < 2^31 for all others

__device__ __forceinline__ unsigned long long fix_shr(unsigned long long m, unsigned s) {
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(s));   // clamps: 0 for s >= 64
  return v;
}

// Exponent field of a b on a scale of its own: the fields' sum, and one where the
// significands' product reaches 2 (from their leading 32 bits; fix_limbs takes a
// product that reaches it in the bits below).  ea, eb: the fields.
__device__ __forceinline__ int fix_prod_top(double a, int ea, double b, int eb) {
  const unsigned ah = (unsigned)__double2hiint(a), bh = (unsigned)__double2hiint(b);
  const unsigned A1 = __funnelshift_l((unsigned)__double2loint(a), (ah & 0xfffffu) | 0x100000u, 11);
  const unsigned B1 = __funnelshift_l((unsigned)__double2loint(b), (bh & 0xfffffu) | 0x100000u, 11);
  return ea + eb + (int)(__umulhi(A1, B1) >> 31);
}

// a b in limbs of a block whose largest fix_prod_top is G: |a b| 2^(B - 1 - (G -
// 2046)) cut to an integer (values below 2^-1022 count as zero).
template <int N>
__device__ __forceinline__ fix2 fix_prod(double a, double b, int G) {
  const unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
  const unsigned bh = (unsigned)__double2hiint(b), bl = (unsigned)__double2loint(b);
  const unsigned ea = (ah >> 20) & 0x7ffu, eb = (bh >> 20) & 0x7ffu;
  // mantissas with their leading bit at 2^63
  const unsigned A1 = __funnelshift_l(al, (ah & 0xfffffu) | 0x100000u, 11), A0 = al << 11;
  const unsigned B1 = __funnelshift_l(bl, (bh & 0xfffffu) | 0x100000u, 11), B0 = bl << 11;
  unsigned long long P = (unsigned long long)A1 * B1 + __umulhi(A1, B0) + __umulhi(A0, B1);
  if (ea == 0 || eb == 0) P = 0;
  return fix_limbs(fix_shr(P, (unsigned)(63 - fix_bits(N) + G) - (ea + eb)), ((int)(ah ^ bh) >> 31) | 1);
}

// Block exponents usable with rows of scale sc (for fix_prod's largest
// fix_prod_top), and the exponent field of the unit 2^(60 - sc - sv) of its rows.
template <int N>
__device__ __forceinline__ int fix_prod_exp(int G, int sc) { return max(G, 963 + fix_bits(N) + sc); }
template <int N>
__device__ __forceinline__ int fix_field(int E, int sc) { return E + 61 - fix_bits(N) - sc; }
template <int N>
__device__ __forceinline__ int fix_prod_field(int G, int sc) { return G - 962 - fix_bits(N) - sc; }

// r 2^(u - 1023) as an FP64 value, rounded to nearest, in integer operations
// (I2F.F64 and the scaling product would cost two at the FP64 rate); u >= 1,
// |r| < 2^63.
__device__ __forceinline__ void fix_value(long long r, int u, double& out) {
  const int sg = (int)(r >> 63);
  const unsigned long long m = (unsigned long long)((r ^ sg) - sg);
  const int n = __clzll((long long)m);
  const unsigned long long a = m << (n & 63);
  const unsigned long long b = (a >> 11) + ((a >> 10) & 1ull);      // 2^52 .. 2^53
  const int e = u + 62 - n;
  unsigned long long bits = ((unsigned long long)(unsigned)e << 52) + b;
  if (e >= 2046) bits = 0x7ff0000000000000ull;
  if (m == 0) bits = 0;
  out = __hiloint2double((int)((unsigned)(bits >> 32) | ((unsigned)sg & 0x80000000u)), (int)(unsigned)bits);
}

__device__ __forceinline__ double xg_nan(double) { return __hiloint2double(0x7ff80000, 0); }

// r 2^(u - 1023) for the form at hand: the FP64 form, bound by the FP64 pipe,
// converts in integer operations; the mixed one, bound by issue slots, spends
// two FP64 operations.
template <bool MIXED>
__device__ __forceinline__ double fix_out(long long r, int u) {
  double v;
  if (MIXED) v = (double)r * __hiloint2double(min(u, 2046) << 20, 0);
  else fix_value(r, u, v);
  return v;
}

// Rows of the rho' and Theta' fluxes m and theta m of one segment, with an
// exponent each, handed to put0(a, row) and put4 (a value that is not finite
// makes its rows NaN); MIXED as fix_out.
template <int N, typename Put0, typename Put4>
__device__ __forceinline__ void fix_flux_rows(const FixRows& F, const double (&m)[N + 1], const double (&th)[N + 1],
                                              Put0 put0, Put4 put4) {
  bool b0 = false, b4 = false;
  int e0 = 0, e4 = 0;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    const int em = fix_exp_finite(m[l], b0);
    e0 = max(e0, em);
    e4 = max(e4, fix_prod_top(m[l], em, th[l], fix_exp_finite(th[l], b4)));
  }
  b4 |= b0;
  fix2 v[N + 1];
  const int E0 = fix_block_exp(e0, F.sc), E4 = fix_prod_exp<N>(e4, F.sc);
#pragma unroll
  for (int l = 0; l <= N; ++l) v[l] = fix_of<N>(m[l], E0);
#pragma unroll
  for (int a = 0; a <= N; ++a) put0(a, b0 ? xg_nan(0.0) : fix_out<true>(fix_row<N>(F, a, v), fix_field<N>(E0, F.sc)));
#pragma unroll
  for (int l = 0; l <= N; ++l) v[l] = fix_prod<N>(th[l], m[l], E4);
#pragma unroll
  for (int a = 0; a <= N; ++a)
    put4(a, b4 ? xg_nan(0.0) : fix_out<true>(fix_row<N>(F, a, v), fix_prod_field<N>(E4, F.sc)));
}

#endif  // __CUDACC__

}  // namespace xg
