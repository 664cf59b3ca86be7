// xg_fixed.cuh -- FP64 line contractions in 64-bit fixed point on the integer
// pipe.
//
// GB300 issues 1.9 FP64 FMAs per clock and SM but 60 IMAD.WIDE (32 x 32 -> 64
// bits with a 64-bit addend; both measured), so a contraction of FP64 data
// with a constant matrix is cheaper in exact integer arithmetic:
//   * the N + 1 values of an element segment are written as V = v 2^sv, |V| <
//     2^B, B = 61 for orders up to 4 and 60 above, with one exponent for the
//     segment: the largest value keeps B bits and every value down to 2^-8 (2^-7)
//     of it all of its 53;
//   * the matrix is written once per mesh as C = c 2^sc, from its long double
//     entries, with sum_l |C_l| <= 2^60 over every assembled row (59 bits
//     against FP64's 53);
//   * both are split into limbs, X = h 2^30 + l, and a product takes three
//     IMAD.WIDE, hi += ch h and mid += ch l + cl h; the low product (below 2^-58
//     of sum |c| max |v|) is left out;
//   * a row that sums to zero up to its entries' rounding is made to sum to
//     zero in both limbs, so that rows depend on the values' differences only:
//     a constant has no derivative at all, as in the difference form, and what is
//     left out has no bias.  That takes a few |cl| up to 2^30, with sum |cl| <=
//     4/3 (N + 1) 2^29; nothing overflows: |hi| <= 2^61 and |mid| <= 2^60 +
//     4/3 (N + 1) 2^(B - 1) < 2^63;
//   * r = hi + mid 2^-30, rounded, is one FP64 value again by one conversion, times
//     2^(60 - sc - sv).
// A segment's sums are exact up to those cuts, a few 2^-59 of its
// sum |c| max |v|, where an FP64 FMA chain rounds at 2^-53 of its partial
// sums.  Sums over segments and directions are taken in the larger one's unit
// (fix_add), so a node's error is one of the values in its own segments.  A
// segment with an infinity or NaN has no exponent; its callers take the FP64
// path or return NaN, as an FP64 chain would.
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

// c in fixed point, on a scale of its own: sums of rows of two matrices are taken
// in the larger one's unit (fix_add), and a direction of wide spacing, whose
// matrix is small, keeps its bits beside one of narrow spacing.
inline void fix_rows(int N, const FixMatrix& c, FixRows* F) {
  const double most = fix_row_sum(N, c);
  int e = 0;
  if (most > 0.0 && std::isfinite(most)) std::frexp(most, &e);
  // (a matrix of zeros: a unit so small that its rows never set that of a sum)
  const int sc = F->sc = most == 0.0 ? 1000 : 60 - e;
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

// The exponent used for a segment whose largest field is e, against rows of
// scale sc: tiny ones are cut at 2^-900 or so.
__device__ __forceinline__ int fix_block_exp(int e, int sc) { return max(e, max(128, sc + 2)); }

// Bits B of a segment's values (see the overflow bound above).
__host__ __device__ constexpr int fix_bits(int N) { return N <= 4 ? 61 : 60; }

// sg V in limbs, V < 2^61: the low one cut, 0 .. 2^30 with v's sign.  (Rows
// depend on differences, so the low limbs' mean does not bias them.)
__device__ __forceinline__ fix2 fix_limbs(unsigned long long V, int sg) {
  return {(int)(V >> 30) * sg, (int)((unsigned)V & 0x3fffffffu) * sg};
}

// v in the limbs of a segment of exponent E >= fix_exp(v): |v| 2^(B - 1 - (E -
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

// 2^(60 - sc - sv) of a segment of exponent E (NaN for one that has none)
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

// ---------------------------------------------------------------- fluxes
// exponent field of v, 0 for an infinity or NaN
__device__ __forceinline__ int fix_exp_finite(double v, bool& bad) {
  const int e = fix_exp(v);
  const bool b = e == kFixNonfinite;
  bad |= b;
  return b ? 0 : e;
}

__device__ __forceinline__ unsigned long long fix_shr(unsigned long long m, unsigned s) {
  unsigned long long v;
  asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(m), "r"(s));   // clamps: 0 for s >= 64
  return v;
}

// Exponent field of a b on a scale of its own: the fields' sum, and one where the
// significands' product reaches 2 (from their leading 32 bits; fix_prod takes a
// product that reaches it in the bits below).  ea, eb: the fields.
__device__ __forceinline__ int fix_prod_top(double a, int ea, double b, int eb) {
  const unsigned ah = (unsigned)__double2hiint(a), bh = (unsigned)__double2hiint(b);
  const unsigned A1 = __funnelshift_l((unsigned)__double2loint(a), (ah & 0xfffffu) | 0x100000u, 11);
  const unsigned B1 = __funnelshift_l((unsigned)__double2loint(b), (bh & 0xfffffu) | 0x100000u, 11);
  return ea + eb + (int)(__umulhi(A1, B1) >> 31);
}

// a b in limbs of a segment whose largest fix_prod_top is G: |a b| 2^(B - 1 - (G -
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
  const int sg = ((int)(ah ^ bh) >> 31) | 1;
  unsigned long long V = fix_shr(P, (unsigned)(63 - fix_bits(N) + G) - (ea + eb));
  if (fix_bits(N) == 61) V = min(V, (1ull << 61) - 1);   // (see fix_prod_top; h stays below 2^31)
  return fix_limbs(V, sg);
}

// Exponents usable with rows of scale sc (for fix_prod's largest
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

// ---------------------------------------------------------------- sums of rows
// r 2^(u - 1023), |r| < 2^62: the rows of one segment share u, an exponent field.
struct FixSum {
  long long r;
  int u;
};

constexpr int kFixBad = 0x4000;   // u of a segment that holds an infinity or NaN

// a + b in the larger of the two units, the other rounded to it: the segments
// keep the bits of their own values, whatever a neighbour or the other direction
// holds.
__device__ __forceinline__ FixSum fix_add(FixSum a, FixSum b) {
  const bool swap = a.u < b.u;
  const long long big = swap ? b.r : a.r, low = swap ? a.r : b.r;
  const int d = min(abs(a.u - b.u), 62);
  return {big + ((((low + low) >> d) + 1) >> 1), max(a.u, b.u)};
}

__device__ __forceinline__ FixSum fix_twice(FixSum a) { return {a.r + a.r, a.u}; }

// Its FP64 value (u < kFixBad), in two FP64 operations.
__device__ __forceinline__ double fix_double(FixSum a) {
  return (double)a.r * __hiloint2double(min(a.u, 2046) << 20, 0);
}

// Its value for the form at hand (fix_out), NaN for a bad one.
template <bool MIXED>
__device__ __forceinline__ double fix_sum_out(FixSum a) {
  return a.u >= kFixBad ? xg_nan(0.0) : fix_out<MIXED>(a.r, a.u);
}

// u, or 0 where all values are equal: the rows are zero, which is exact in any
// unit, and must not cost the sums that they are added to any bits.
template <int N>
__device__ __forceinline__ int fix_unit_of(const fix2 (&v)[N + 1], int u) {
  int differ = 0;
#pragma unroll
  for (int l = 1; l <= N; ++l) {
    differ |= v[l].h ^ v[0].h;
    differ |= v[l].l ^ v[0].l;
  }
  return differ != 0 ? u : 0;
}

// The values a of one segment, or the products t m, in limbs of an exponent of
// their own; returns the u of their rows against a matrix of scale sc.
template <int N>
__device__ __forceinline__ int fix_values(const double (&a)[N + 1], int sc, fix2 (&v)[N + 1]) {
  int e = fix_exp(a[0]);
#pragma unroll
  for (int l = 1; l <= N; ++l) e = max(e, fix_exp(a[l]));
  const int E = fix_block_exp(e, sc);
#pragma unroll
  for (int l = 0; l <= N; ++l) v[l] = fix_of<N>(a[l], E);
  return e == kFixNonfinite ? kFixBad : fix_unit_of<N>(v, fix_field<N>(E, sc));
}

template <int N>
__device__ __forceinline__ int fix_products(const double* m, const double* t, int stride, int sc,
                                            fix2 (&v)[N + 1]) {
  bool bad = false;
  int G = 0;
#pragma unroll
  for (int l = 0; l <= N; ++l) {
    const double x = m[l * stride], y = t[l * stride];
    G = max(G, fix_prod_top(x, fix_exp_finite(x, bad), y, fix_exp_finite(y, bad)));
  }
  G = fix_prod_exp<N>(G, sc);
#pragma unroll
  for (int l = 0; l <= N; ++l) v[l] = fix_prod<N>(t[l * stride], m[l * stride], G);
  return bad ? kFixBad : fix_unit_of<N>(v, fix_prod_field<N>(G, sc));
}

// x segments of a tile's lines, n of each line and the one before the tile, go to
// lanes in line order, 31 to a warp: a warp's lane 0 repeats the last one of the warp
// before.  Each lane so finds the segment before its own on the lane before it.  n is a
// full tile's number, a constant; small launches, where a tile's time counts, take the
// tile's own (dynamics on 20 x 40 x 45 nodes 193 -> 180 us; on full tiles it costs 1 %).
constexpr int kFixLanes = 31;
__host__ __device__ constexpr int fix_x_tasks(int lines, int n) { return (lines * (n + 1) + kFixLanes - 1) / kFixLanes; }
// 2^16 / (n + 1) rounded up: f fix_x_div(n) >> 16 = floor(f / (n + 1)) for -1 <= f < 1300
__device__ __forceinline__ int fix_x_div(int n) { return (int)__fdividef(65536.0f, (float)(n + 1)) + 1; }
__device__ __forceinline__ void fix_x_slot(int task, int lane, int n, int div, int& line, int& s) {
  const int f = task * kFixLanes + lane - 1;   // -1: none (line -1)
  line = (f * div) >> 16;
  s = f - line * (n + 1) - 1;                  // -1: the segment before the tile
}
template <int E>
__device__ __forceinline__ void fix_x_slot(int task, int lane, int& line, int& s) {
  const int f = task * kFixLanes + lane - 1;
  line = f < 0 ? 1 << 30 : f / (E + 1);
  s = f - (f < 0 ? 0 : line * (E + 1)) - 1;
}

// Rows of x segments on the lanes of fix_x_slot, so that a first node's row is
// joined with row N of the segment before (left; a wall's first and, where end,
// last node take theirs twice) without a barrier.  Called by all lanes of a warp:
// act the lanes that have a segment, own those whose rows are wanted; put(a, row)
// gets the nodes' rows.
template <int N, typename Put>
__device__ __forceinline__ void fix_x_rows(const FixRows& F, const fix2 (&v)[N + 1], int u, bool act, bool own,
                                           bool left, bool end, Put put) {
  FixSum last = {0, u}, before;
  if (act) last.r = fix_row<N>(F, N, v);
  before.r = __shfl_up_sync(0xffffffffu, last.r, 1);
  before.u = __shfl_up_sync(0xffffffffu, last.u, 1);
  if (!own) return;
  const FixSum first = {fix_row<N>(F, 0, v), u};
  put(0, left ? fix_add(first, before) : fix_twice(first));
#pragma unroll
  for (int a = 1; a < N; ++a) put(a, FixSum{fix_row<N>(F, a, v), u});
  if (end) put(N, fix_twice(last));
}

// Slot of node i's unit among the 2 E + 1 of a line of E segments: a segment's
// first node, which two segments meet in, has one of its own.
template <int N>
__device__ __forceinline__ int fix_unit_slot(int i) {
  const int s = i / N;
  return 2 * s + (i != s * N);
}

// ---------------------------------------------------------------- plane tiles
// A CTA takes E x E elements of one level.  Its nodes' x and y rows need the
// tile extended by the segment before it and its end face along each
// direction (a cross), which is put into shared memory once; one thread takes a
// whole element segment of a line -- the matrix then comes from the constant
// bank at fixed offsets, and a segment's N + 1 values are read once for its
// N + 1 rows -- converts its values with an exponent of their own and leaves its
// rows as 64-bit integers, which the nodes add up (fix_add).  A warp takes 31 x
// segments or a y segment of every column.
// (One exponent and one conversion a value for the whole tile, 0.234 against
// 0.253 ms a Laplacian's pass over 5 x 4.3 M nodes, left a quiet segment the bits
// that the loudest one of the tile had to spare.)
__host__ __device__ constexpr int fix_plane_elems(int N) { return 32 / N; }
// Warps of a tile's block: seven, six at order 8, whose tiles have few and long
// tasks (two Laplacians over 4.3 M nodes at order 4 0.841 ms with seven, 0.854 with
// eight, 0.879 with ten; over 5.7 M at order 8 0.915 with six, 0.983 with seven).
// Twelve where a launch has fewer blocks than fit the chip at once, and a tile's
// own time counts.
__host__ __device__ constexpr int fix_plane_warps(int N) { return N == 8 ? 6 : 7; }
constexpr int kFixWideWarps = 12;
inline bool fix_plane_wide(long long blocks, int sms) { return blocks <= 3ll * sms; }

template <int N>
struct FixPlane {
  static constexpr int E = fix_plane_elems(N);
  static constexpr int TS = E * N;            // <= 32: a warp takes a row of the tile, a lane a column
  static constexpr int LO = TS + 1;           // owned extent (a wall's last node included)
  static constexpr int LX = TS + N + 1;       // extended extent
  static constexpr int PV = LX | 1;           // odd pitches: lanes along either axis hit distinct banks
  static constexpr int PR = LO | 1;
  static constexpr int V = LX * PV;           // 8-byte slots
  static constexpr int RX = LO * PR, UX = LO * (2 * E + 1);   // x rows (wall ends included) and units
  static constexpr int RY = TS * PR, RB = (E + 1) * LO;       // y rows; rows N, and units, of segments -1..E-1
};

// Rows of a tile's segments.
template <int N>
struct FixPlaneRows {
  using L = FixPlane<N>;
  long long x[L::RX], y[L::RY], yn[L::RB];
  int ux[L::UX], uy[L::RB];
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

// Loads the cross of one variable f (a level's first node) into V[j + N][i + N]:
// a warp takes a row of the tile's own columns; the rest are the N columns before
// them, of the owned rows, and the one after them, of every row (a wall's last
// column has y segments of its own).  X, Y: which directions' segments are needed
// (owned rows extended along x, owned columns along y).
template <int N, int W, bool X, bool Y>
__device__ __forceinline__ void fix_plane_load(const double* __restrict__ f, const FixTile& T, int nx, int ny,
                                               double* V) {
  using L = FixPlane<N>;
  constexpr int kRows = (L::LX + W - 1) / W;                           // rows of a warp
  constexpr int kSide = (L::LO * N + L::LX + 32 * W - 1) / (32 * W);   // columns beside the tile's of a thread
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int fx = T.ekx * N, fy = T.eky * N;
  auto value = [&](int i, int j) -> double {
    const bool inx = X && j >= 0 && j < T.oy && (i >= 0 || T.hxl) && i <= fx;
    const bool iny = Y && i >= 0 && i < T.ox && (j >= 0 || T.hyl) && j <= fy;
    if (!inx && !iny) return 0.0;
    int gx = T.x0 + i, gy = T.y0 + j;
    if (gx < 0) gx += nx;
    if (gy < 0) gy += ny;
    if (gx >= nx) gx -= nx;
    if (gy >= ny) gy -= ny;
    return f[gx + (long long)nx * gy];
  };
  double v[kRows], w[kSide];
  const int gx = T.x0 + lane - (T.x0 + lane >= nx ? nx : 0);
  const bool colx = X && lane < L::TS && lane <= fx, coly = Y && lane < L::TS && lane < T.ox;
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int j = warp + k * W - N;
    int gy = T.y0 + j;
    if (j < 0) gy += gy < 0 ? ny : 0;
    else gy -= gy >= ny ? ny : 0;
    v[k] = 0.0;
    if ((colx && j >= 0 && j < T.oy) || (coly && (j >= 0 || T.hyl) && j <= fy)) v[k] = f[gx + (long long)nx * gy];
  }
#pragma unroll
  for (int k = 0; k < kSide; ++k) {
    const int t = (int)threadIdx.x + k * 32 * W, r = t / N;
    if (t < L::LO * N) w[k] = value(t - r * N - N, r);
    else w[k] = value(L::TS, t - L::LO * N - N);
  }
#pragma unroll
  for (int k = 0; k < kRows; ++k) {
    const int jj = warp + k * W;
    if (lane < L::TS && jj < L::LX) V[jj * L::PV + N + lane] = v[k];
  }
#pragma unroll
  for (int k = 0; k < kSide; ++k) {
    const int t = (int)threadIdx.x + k * 32 * W, r = t / N;
    if (t < L::LO * N) V[(N + r) * L::PV + t - r * N] = w[k];
    else if (t < L::LO * N + L::LX) V[(t - L::LO * N) * L::PV + N + L::TS] = w[k];
  }
}

// Rows of every x segment of the tile's values Vx and y segment of Vy.
template <int N, int W>
__device__ __forceinline__ void fix_plane_rows(const FixRows& FX, const FixRows& FY, const FixTile& T, const double* Vx,
                                               const double* Vy, FixPlaneRows<N>& R) {
  using L = FixPlane<N>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // y: a warp takes a segment of the tile's TS columns, or up to 32 segments of a
  // wall's last column
  constexpr bool kOwn = W == kFixWideWarps;   // the tile's own number of x segments
  const int div = kOwn ? fix_x_div(T.ekx) : 0;
  const int wx = fix_x_tasks(T.oy, kOwn ? T.ekx : L::E), y0 = T.hyl ? 0 : 1, ns = T.eky + 1 - y0;
  const int wy = ns + (T.ox > L::TS ? (ns + 31) / 32 : 0);
  for (int w = warp; w < wx + wy; w += W) {
    double a[N + 1];
    fix2 v[N + 1];
    if (w < wx) {
      int o, s;
      if (kOwn) fix_x_slot(w, lane, T.ekx, div, o, s);
      else fix_x_slot<L::E>(w, lane, o, s);
      const bool act = o >= 0 && o < T.oy && s < T.ekx && (s >= 0 || T.hxl);
      int u = 0;
      if (act) {
        const double* p = Vx + (o + N) * L::PV + (s + 1) * N;
#pragma unroll
        for (int l = 0; l <= N; ++l) a[l] = p[l];
        u = fix_values<N>(a, FX.sc, v);
      }
      long long* r = R.x + o * L::PR + s * N;
      int* ur = R.ux + o * (2 * L::E + 1) + 2 * s;
      fix_x_rows<N>(FX, v, u, act, act && s >= 0 && lane > 0, s > 0 || T.hxl, T.ox > T.ekx * N && s == T.ekx - 1,
                    [&](int k, FixSum x) {
                      r[k] = x.r;
                      if (k < 2 || k == N) ur[k == N ? 2 : k] = x.u;
                    });
    } else {
      const bool edge = w - wx >= ns;
      const int s = y0 + (edge ? 32 * (w - wx - ns) + lane : w - wx), o = edge ? L::TS : lane;   // s - 1: the segment
      if (s > T.eky || o >= (edge ? T.ox : min(T.ox, L::TS))) continue;
      const double* p = Vy + s * N * L::PV + o + N;
#pragma unroll
      for (int l = 0; l <= N; ++l) a[l] = p[l * L::PV];
      R.uy[s * L::LO + o] = fix_values<N>(a, FY.sc, v);
      R.yn[s * L::LO + o] = fix_row<N>(FY, N, v);
      if (s > 0) {
#pragma unroll
        for (int k = 0; k < N; ++k) R.y[((s - 1) * N + k) * L::PR + o] = fix_row<N>(FY, k, v);
      }
    }
  }
}

// The assembled x and y rows of the tile's node (i, j).
template <int N>
__device__ __forceinline__ FixSum fix_plane_x(const FixPlaneRows<N>& R, int i, int j) {
  using L = FixPlane<N>;
  return {R.x[j * L::PR + i], R.ux[j * (2 * L::E + 1) + fix_unit_slot<N>(i)]};
}

template <int N>
__device__ __forceinline__ FixSum fix_plane_y(const FixTile& T, const FixPlaneRows<N>& R, int i, int j) {
  using L = FixPlane<N>;
  const int s = j / N;
  const FixSum before = {R.yn[s * L::LO + i], R.uy[s * L::LO + i]};
  if (s == T.eky) return fix_twice(before);              // a wall's last node: its row twice
  const FixSum r = {R.y[j * L::PR + i], R.uy[(s + 1) * L::LO + i]};
  if (j != s * N) return r;
  return s > 0 || T.hyl ? fix_add(r, before) : fix_twice(r);
}

// node(i, j) for every owned node of the tile: a warp takes a row, a lane a
// column; a wall's last column (i = TS) goes to the threads of its own.
template <int N, int W, typename F>
__device__ __forceinline__ void fix_plane_nodes(const FixTile& T, F node) {
  using L = FixPlane<N>;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane < min(T.ox, L::TS)) {
    for (int j = warp; j < T.oy; j += W) node(lane, j);
  }
  if (T.ox > L::TS && (int)threadIdx.x < T.oy) node(L::TS, (int)threadIdx.x);
}

// ---------------------------------------------------------------- nodes
// The assembled row of one node along one line, by one thread: the same segments,
// units and sums as the tiles', bit for bit, at a conversion per value and node.
// It serves levels that leave most of a tile empty.  R: the line's matrix in shared
// memory (fix_stage_rows).
template <int N>
struct FixTable {
  int2 c[N + 1][N + 1];
  int sc;
};

template <int N>
__device__ __forceinline__ void fix_stage_rows(const FixRows& F, FixTable<N>& R) {
  for (int k = threadIdx.x; k < (N + 1) * (N + 1); k += blockDim.x) {
    const int a = k / (N + 1), l = k - a * (N + 1);
    R.c[a][l] = make_int2(F.ch[a][l], F.cl[a][l]);
  }
  if (threadIdx.x == 0) R.sc = F.sc;
}

template <int N>
__device__ __forceinline__ FixSum fix_line_node(const FixTable<N>& R, const double* __restrict__ f, long long base,
                                                long long sd, int g, int nd, int nseg, bool per) {
  const int s = min(g / N, nseg - 1), a = g - s * N;
  auto row = [&](int seg, int k) -> FixSum {
    double x[N + 1];
#pragma unroll
    for (int l = 0; l <= N; ++l) {
      const int at = seg * N + l;
      x[l] = f[base + sd * (at >= nd ? at - nd : at)];
    }
    fix2 v[N + 1];
    const int u = fix_values<N>(x, R.sc, v);
    long long hi = 0, mid = 1ll << 29;
#pragma unroll
    for (int l = 0; l <= N; ++l) {
      const int2 c = R.c[k][l];
      hi += (long long)c.x * v[l].h;
      mid += (long long)c.x * v[l].l;
      mid += (long long)c.y * v[l].h;
    }
    return {hi + (mid >> 30), u};
  };
  const FixSum r = row(s, a);
  if (a == N) return fix_twice(r);
  if (a != 0) return r;
  return s > 0 || per ? fix_add(r, row(s > 0 ? s - 1 : nseg - 1, N)) : fix_twice(r);
}

// Whether the tiles take the x and y sums of a level: where it fills an (N + 1)th
// of them (order 1: nine tenths) and a third of their width, which a warp's lanes
// are.  Two Laplacians over 1 M nodes, tiles against nodes: order 4, levels of 4 x 8
// nodes 1.68 / 0.45 ms, 4 x 128 1.06 / 0.45, 8 x 32 0.58 / 0.45, 32 x 8 0.37 /
// 0.45, 32 x 128 0.25 / 0.45.
inline bool fix_plane_pays(int N, int nx, int ny, int nelx, int nely) {
  const int E = fix_plane_elems(N);
  const long long width = (long long)((nelx + E - 1) / E) * E * N, height = (long long)((nely + E - 1) / E) * E * N;
  if (N == 1) return 10ll * nx * ny >= 9 * width * height;
  return (long long)(N + 1) * nx * ny >= width * height && 3ll * nx >= width;
}

// ---------------------------------------------------------------- z lines
// A block of a marching z pass takes 128 columns of one chunk, or all columns of
// several chunks where there are few.
constexpr int kFixZThreads = 128;
inline int fix_z_columns(long long nxy) {
  int c = kFixZThreads;
  while (c > 1 && c / 2 >= nxy) c /= 2;
  return c;
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
