// fixstencil.cuh -- the binary64 5-point stencil on a warp strip in 64-bit fixed
// point.
//
// Why: the FP64 pipe issues a warp instruction every 64 (multiply-add) to 76
// (addition) cycles on each scheduler, the integer pipe one a cycle.  The four FP64
// operations a point of the mask are 292 cycles of the pipe that bounds the
// binary64 CG passes; in fixed point they are about 45 integer instructions and
// one conversion back (64; the ring kernels do that in integers too, 48).  4096^2, an
// iteration, by itself: classic 302 -> 222 us, NewCG 375 -> 311 us.
//
// How: a row's values are aligned to the largest exponent among the warp's values
// of the row (one redux.sync), as signed multiples of 2^-59 of that exponent's
// power of two, so the mask's sum (below 8 x 2^60) fits 63 bits; rows with different
// exponents are aligned by one common shift.  Values are truncated below 2^-59 of
// the largest one of three rows of the strip and the sum is rounded once, in the
// conversion: an error below 2^-56 of that value's power of two, 2^E, beside the
// result's own rounding.
//
// When: only where FP64 may lose as much at the same point.  Four FP64 operations on
// operands of magnitude M at most round results as large as 5, 6, 7 and 8 M: 26 x 2^-53 M.
// The fixed-point error is at most 2^(E-56) + 8 x 2^-53 M: 24 x 2^-53 M where
// M >= 2^(E - kFixSpan), kFixSpan = 7 (29 in a row whose sum is completed in FP64).  A
// residual adds b, with one bit less: 9 x 2^(E-58), 18 x 2^-53 M with kFixSpanRes = 6,
// and its own rounding.  So every point needs an operand within kFixSpan binades of the
// largest value of the warp's rows; those of a point's operands are looked at that its
// lane holds (in the ring march, the larger one of two neighbouring columns).  A row
// that fails -- values beside ones a hundred times larger, zeros, infinities, NaN, the ends
// of the exponent range -- is formed with FP64 operations.  On noise that is one row in
// fifty to two hundred, on smooth fields none.
#pragma once

#include "ring.cuh"

namespace lap5 {

// A fixed-point value q of exponent field E is q 2^(E - 1075 - B): B bits below a
// double's significand, 7 for the mask's eight values, 6 with a ninth.
constexpr int kFixB = 7, kFixBRes = 6;
constexpr int kFixLow = 70, kFixHigh = 0x7fa;  // exponent fields for which no result leaves the normal range
constexpr int kFixSpan = 7, kFixSpanRes = 6;

// v as a fixed-point value of exponent E >= the exponent field of v, truncated.
// (A zero or subnormal v, taken with an implicit leading bit, is shifted out for
// E >= kFixLow.)
template <int B>
__device__ __forceinline__ long long fix_of(double v, int E) {
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
  const int d = min(E - ((hi >> 20) & 0x7ff), 63);
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const uint32_t xh = __funnelshift_l(lo, mh, B), xl = lo << B;
  const bool far = d >= 32;
  const uint32_t a = far ? 0u : xh, b = far ? xh : xl;
  const uint32_t rl = __funnelshift_r(b, a, d), rh = a >> (d & 31);
  const unsigned long long s = (unsigned long long)(long long)(hi >> 31);
  return (long long)(((((unsigned long long)rh << 32) | rl) ^ s) - s);
}
// back, rounded to nearest
template <int B>
__device__ __forceinline__ double fix_to(long long q, int E) {
  const double v = (double)q;
  const int hi = __double2hiint(v);
  return __hiloint2double(hi == 0 ? 0 : hi + ((E - 1075 - B) << 20), __double2loint(v));
}

// The same on the integer pipe (about 40 instructions; the conversion above is one
// slot of the FP64 pipe, 64 cycles), |q| < 2^63: the magnitude with its leading bit
// moved to bit 62 (nothing lost), rounded to 53 bits half to even, the carry running
// into the exponent field.  For the ring kernels, which the FP64 pipe bounds (80-85 %
// busy) at half the issue slots: 4096^2, classic 211 -> 195 us an iteration, NewCG 302
// -> 288.  The resident and multigrid kernels, whose warps wait on a chain rather than
// on the pipe, are faster with the conversion (1024^2 f64 20.5 against 20.9 us).
template <int B>
__device__ __forceinline__ double fix_to_int(long long q, int E) {
  const unsigned long long s = (unsigned long long)(q >> 63), a = ((unsigned long long)q ^ s) - s;
  const int lz = __clzll((long long)a);
  const unsigned long long t = a << ((lz - 1) & 63);
  const unsigned long long m = (t + 0x1ffull + ((t >> 10) & 1ull)) >> 10;
  unsigned long long b = m + ((unsigned long long)(unsigned)(E + 10 - B - lz) << 52);
  if (a == 0ull) b = 0ull;
  return __longlong_as_double((long long)(b | (s << 63)));
}

// One row of a strip: the lane's V values at the row's exponent.
template <int V> struct FixRow {
  long long q[V];
  int E;
};

// Align x (exponent Ex) down to the larger exponent E.
template <int V>
__device__ __forceinline__ void fix_align(long long (&x)[V], int Ex, int E) {
  const int d = E - Ex;  // uniform in the warp
  if (d > 0) {
    const int s = min(d, 63);
#pragma unroll
    for (int k = 0; k < V; ++k) x[k] >>= s;
  }
}

__device__ __forceinline__ unsigned fix_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// The stencil of a row march: rows arrive one after another, the two horizontal
// neighbours and the row behind enter a row's partial sum when it arrives, the
// row ahead completes it.  A sum is fixed point or FP64 (its bits then lie in the
// same registers).  OK = true is the usual way alone: the new row may be added to the
// current row's sum, and begin one of its own, in fixed point; false looks at each.
// The ring march takes a whole step one way or the other: one branch a row (4096^2
// classic, 200 iterations: 39.5 ms against 40.2 with a branch around each half, 38.8
// with none and truncated small values; NewCG 59.0, 59.0, 57.7).
template <int V> struct FixMarch {
  FixRow<V> prev, sum;   // the row behind; the current row's partial sum
  double c[V];           // the current row
  int top = 0x7fffffff;  // the largest exponent the sum may take; < 0: it is FP64, its bits in sum.q

  // Row f in fixed point; LO: in lo the smallest exponent over its points of the larger one of
  // two neighbouring columns of the lane (the ring kernels, which have no registers or
  // cycles for a closer look: it stands beside the other reduction).  nval: columns of
  // the grid from the lane's first on.
  template <bool LO>
  __device__ __forceinline__ static void row(const FRow<V, double>& f, int nval, FixRow<V>& a, int& lo) {
    unsigned m = fix_mag(f.hl), n = 0x7fffffffu;
#pragma unroll
    for (int k = 0; k < V; k += 2) {
      const unsigned p = max(fix_mag(f.f[k]), fix_mag(f.f[k + 1]));
      m = max(m, p);
      if (k < nval) n = min(n, p);
    }
    a.E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
    lo = LO ? (int)(__reduce_min_sync(0xffffffffu, n) >> 20) : 0;
#pragma unroll
    for (int k = 0; k < V; ++k) a.q[k] = fix_of<kFixB>(f.f[k], a.E);
  }
  // That exponent with the row behind (c) among the operands looked at.
  __device__ __forceinline__ int lowest(const FRow<V, double>& f, int nval) const {
    unsigned n = 0x7fffffffu;
#pragma unroll
    for (int k = 0; k < V; k += 2) {
      const unsigned p = max(fix_mag(f.f[k]), fix_mag(f.f[k + 1]));
      if (k < nval) n = min(n, max(p, fix_mag(c[k])));
      if (k + 1 < nval) n = min(n, max(p, fix_mag(c[k + 1])));
    }
    return (int)(__reduce_min_sync(0xffffffffu, n) >> 20);
  }
  __device__ __forceinline__ static int top_of(int lo) { return min(lo + kFixSpan, kFixHigh); }
  __device__ __forceinline__ bool ok(const FixRow<V>& a, int lo, bool behind) const {
    const int E = max(behind ? prev.E : 0, a.E);
    return a.E <= top && E <= top_of(lo) && E >= kFixLow;
  }
  // y = A c with row a = f ahead of c.  INT: fix_to_int.
  template <bool OK, bool INT>
  __device__ __forceinline__ void complete(const FRow<V, double>& f, const FixRow<V>& a, double (&y)[V]) {
    const int E = max(sum.E, a.E);
    if (OK || E <= top) {
      fix_align<V>(sum.q, sum.E, E);
      long long t[V];
#pragma unroll
      for (int k = 0; k < V; ++k) t[k] = a.q[k];
      fix_align<V>(t, a.E, E);
#pragma unroll
      for (int k = 0; k < V; ++k) y[k] = INT ? fix_to_int<kFixB>(sum.q[k] - t[k], E) : fix_to<kFixB>(sum.q[k] - t[k], E);
    } else {
#pragma unroll
      for (int k = 0; k < V; ++k)
        y[k] = __dsub_rn(top < 0 ? __longlong_as_double(sum.q[k]) : fix_to<kFixB>(sum.q[k], sum.E), f.f[k]);
    }
  }
  // Row f becomes the current one; behind: it has a row behind it (else it is that row).
  template <bool OK>
  __device__ __forceinline__ void next(const FRow<V, double>& f, const FixRow<V>& a, int lo, int lane, bool behind) {
    if (behind) {
      const int E = max(prev.E, a.E);
      sum.E = E;
      top = top_of(lo);
      if (OK || (E <= top && E >= kFixLow)) {
        const long long h = fix_of<kFixB>(f.hl, a.E);
        long long l = __shfl_up_sync(0xffffffffu, a.q[V - 1], 1), r = __shfl_down_sync(0xffffffffu, a.q[0], 1);
        if (lane == 0) l = h;
        if (lane == 31) r = h;
#pragma unroll
        for (int k = 0; k < V; ++k) {
          const long long w = k == 0 ? l : a.q[k - 1], e = k == V - 1 ? r : a.q[k + 1];
          sum.q[k] = 4 * a.q[k] - w - e;
        }
        fix_align<V>(sum.q, a.E, E);
        fix_align<V>(prev.q, prev.E, E);
#pragma unroll
        for (int k = 0; k < V; ++k) sum.q[k] -= prev.q[k];
      } else {
        double l = shfl_up1(f.f[V - 1]), r = shfl_dn1(f.f[0]);
        if (lane == 0) l = f.hl;
        if (lane == 31) r = f.hl;
#pragma unroll
        for (int k = 0; k < V; ++k) {
          const double w = k == 0 ? l : f.f[k - 1], e = k == V - 1 ? r : f.f[k + 1];
          sum.q[k] = __double_as_longlong(__dsub_rn(__dsub_rn(__fma_rn(4.0, f.f[k], -w), e), c[k]));
        }
        top = -1;
      }
    }
    prev = a;
  }
  // Row t = f arrives: y = A c (t >= 2), and its own sum begins (t >= 1).
  template <bool OK>
  __device__ __forceinline__ void step(const FRow<V, double>& f, const FixRow<V>& a, int lo, int lane, int t,
                                       double (&y)[V]) {
    if (t >= 2) complete<OK, true>(f, a, y);
    next<OK>(f, a, lo, lane, t >= 1);
  }
  __device__ __forceinline__ void current(const FRow<V, double>& f) {
#pragma unroll
    for (int k = 0; k < V; ++k) c[k] = f.f[k];
  }
};

// Row march like march_ring, with the stencil in fixed point: field(j, slot, FRow&)
// builds row j of the operand (hl: the column beyond lane 0's or lane 31's), finish(j,
// slot, c, y) consumes row j with the operand's values c and y = A c.  nval: columns
// of the grid from the lane's first on.
template <int V, int K, class FieldF, class FinishF>
__device__ __forceinline__ void march_ring_fix(WarpRing& ring, int ny, int lane, int xs, int nval, int y0, int y1,
                                               bool rev, const RingVec (&vecs)[K], const int (&off)[K], FieldF& field,
                                               FinishF& finish) {
  if (y0 >= y1) return;
  const int T = y1 - y0;
  const int step = rev ? -1 : 1;
  const int ystart = rev ? y1 - 1 : y0;
  const unsigned q0 = ring.q;
  auto row_of = [&](int t) { return ystart + (t - 1) * step; };
  const int total = T + 2;
  const int pre = min(ring.S, total);
  typename WarpRing::Plan<V, K> P;
  WarpRing::plan<V, K>(P, xs, vecs, off);
  for (int t = 0; t < pre; ++t) ring.produce<V, K>(row_of(t), ny, t >= 1 && t <= T, P);
  FixMarch<V> m;
  const unsigned char* sC = nullptr;
  for (int t = 0; t < total; ++t) {
    FRow<V, double> f;
    const unsigned char* sA = ring.wait(q0 + t);
    const int j = row_of(t);
    if (j < 0 || j >= ny) f.zero();
    else field(j, sA, f);
    FixRow<V> a;
    int lo;
    FixMarch<V>::template row<true>(f, nval, a, lo);
    double y[V];
    if (__builtin_expect(m.ok(a, lo, t >= 1), 1)) m.template step<true>(f, a, lo, lane, t, y);
    else m.template step<false>(f, a, lo, lane, t, y);
    if (t >= 2) {
      finish(row_of(t - 1), sC, m.c, y);
      __syncwarp();
      if (t - 1 + ring.S < total) ring.produce<V, K>(row_of(t - 1 + ring.S), ny, t - 1 + ring.S <= T, P);
    }
    m.current(f);
    if (t == 1) {  // the slot of the row behind the first one is free
      __syncwarp();
      if (ring.S < total) ring.produce<V, K>(row_of(ring.S), ny, ring.S <= T, P);
    }
    sC = sA;
  }
  ring.q = q0 + (unsigned)total;
}

// The same march over rows loaded straight into registers: load(j, Raw&) reads row j
// one step ahead of its use, field(j, raw, FRow&) builds the operand's row from it,
// finish(j, c, y) consumes row j.
template <int V, class Raw, class LoadF, class FieldF, class FinishF>
__device__ __forceinline__ void march_fix(int ny, int lane, int nval, int y0, int y1, bool rev, LoadF& load,
                                          FieldF& field, FinishF& finish) {
  if (y0 >= y1) return;
  const int step = rev ? -1 : 1;
  const int T = y1 - y0, first = rev ? y1 : y0 - 1;
  FixMarch<V> m;
  Raw next;
  load(first, next);
  for (int t = 0; t < T + 2; ++t) {
    const int j = first + t * step;
    const Raw cur = next;
    if (t < T + 1) load(j + step, next);
    FRow<V, double> f;
    if (j < 0 || j >= ny) f.zero();
    else field(j, cur, f);
    FixRow<V> a;
    int none;
    FixMarch<V>::template row<false>(f, nval, a, none);
    if (t >= 2) {
      double y[V];
      m.template complete<false, false>(f, a, y);
      finish(j - step, m.c, y);
    }
    m.template next<false>(f, a, m.lowest(f, nval), lane, t >= 1);
    m.current(f);
  }
}

// Whether points of the warp may be formed in fixed point of exponent E.  n: the smallest over
// the lane's points of the largest operand of the point that is looked at (fix_mag).
template <int SPAN>
__device__ __forceinline__ bool fix_fits(unsigned n, int E) {
  const bool far = __any_sync(0xffffffffu, n < (unsigned)(E - SPAN) << 20);
  return !far && (unsigned)(E - kFixLow) <= (unsigned)(kFixHigh - kFixLow);
}

// r = b - A c on a lane vector from its neighbours (up, dn: rows; w, e: columns), all
// aligned to the warp's largest exponent: nine values below 2^59 stay below 2^63.
// Every lane of the warp calls.
template <int W>
__device__ __forceinline__ void fix_residual(const double (&c)[W], const double (&up)[W], const double (&dn)[W],
                                             double w, double e, const double (&b)[W], double (&r)[W]) {
  static_assert(W == 2, "a point's row neighbour in the lane");
  unsigned m = max(fix_mag(w), fix_mag(e)), n = 0x7fffffffu;
  const unsigned cc = max(fix_mag(c[0]), fix_mag(c[1]));
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const unsigned p = max(cc, max(fix_mag(up[k]), fix_mag(dn[k])));
    n = min(n, p);
    m = max(m, max(p, fix_mag(b[k])));
  }
  const int E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
  if (fix_fits<kFixSpanRes>(n, E)) {
    long long f[W];
#pragma unroll
    for (int k = 0; k < W; ++k) f[k] = fix_of<kFixBRes>(c[k], E);
    const long long l = fix_of<kFixBRes>(w, E), h = fix_of<kFixBRes>(e, E);
#pragma unroll
    for (int k = 0; k < W; ++k)
      r[k] = fix_to<kFixBRes>(fix_of<kFixBRes>(b[k], E) - 4 * f[k] + (k == 0 ? l : f[k - 1]) +
                                  (k == W - 1 ? h : f[k + 1]) + fix_of<kFixBRes>(up[k], E) + fix_of<kFixBRes>(dn[k], E),
                              E);
  } else {
#pragma unroll
    for (int k = 0; k < W; ++k) {
      double a = __fma_rn(4.0, c[k], -(k == 0 ? w : c[k - 1]));
      a = __dsub_rn(a, k == W - 1 ? e : c[k + 1]);
      a = __dsub_rn(__dsub_rn(a, up[k]), dn[k]);
      r[k] = __dsub_rn(b[k], a);
    }
  }
}

}  // namespace lap5
