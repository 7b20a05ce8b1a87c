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
// of the row (one redux.sync), as signed multiples of 2^-58 of that exponent's
// power of two, so the mask's sum (8 times the largest value at most) fits 63
// bits; rows with different exponents are aligned by one common shift.  Values are
// truncated below 2^-58 of the largest one of three rows of the strip and the sum
// is rounded once, in the conversion.  The error a point is then below 2^-56 of
// the largest value of the strip's rows; the FP64 sum rounds three times to 2^-53
// of intermediate results as large as 3, 2 and 1 values.  In the 2-norm of a strip
// row (128 columns at most: the largest value is at most 11.4 times the root mean
// square) the fixed-point error is the smaller one whatever the data.
//
// Rows with exponents beyond 2^1019 (the CG's dot products overflow long before)
// give NaN, rows below 2^-953 (their squares underflow to zero) give 0.
#pragma once

#include "ring.cuh"

namespace lap5 {

constexpr int kFixBias = 1081;   // a fixed-point value q of exponent E is q 2^(E - 1081)
constexpr int kFixLow = 70, kFixHigh = 0x7fa;

// v as a multiple of 2^(E - 1081), truncated; E >= the exponent field of v.  (A
// zero or subnormal v, taken with an implicit leading bit, is shifted out for
// E >= 70.)
__device__ __forceinline__ long long fix_of(double v, int E) {
  const int hi = __double2hiint(v);
  const uint32_t lo = (uint32_t)__double2loint(v);
  const int d = min(E - ((hi >> 20) & 0x7ff), 63);
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const uint32_t xh = __funnelshift_l(lo, mh, 6), xl = lo << 6;
  const bool far = d >= 32;
  const uint32_t a = far ? 0u : xh, b = far ? xh : xl;
  const uint32_t rl = __funnelshift_r(b, a, d), rh = a >> (d & 31);
  const unsigned long long s = (unsigned long long)(long long)(hi >> 31);
  return (long long)(((((unsigned long long)rh << 32) | rl) ^ s) - s);
}
// q 2^(E - 1081), rounded to nearest
__device__ __forceinline__ double fix_to(long long q, int E) {
  const double v = (double)q;
  const int hi = __double2hiint(v);
  return __hiloint2double(hi == 0 ? 0 : hi + ((E - kFixBias) << 20), __double2loint(v));
}

// The same on the integer pipe (about 40 instructions; the conversion above is one
// slot of the FP64 pipe, 64 cycles), |q| < 2^63: the magnitude with its leading bit
// moved to bit 62 (nothing lost), rounded to 53 bits half to even, the carry running
// into the exponent field.  For the ring kernels, which the FP64 pipe bounds (80-85 %
// busy) at half the issue slots: 4096^2, classic 211 -> 195 us an iteration, NewCG 302
// -> 288.  The resident and multigrid kernels, whose warps wait on a chain rather than
// on the pipe, are faster with the conversion (1024^2 f64 20.5 against 20.9 us).
__device__ __forceinline__ double fix_to_int(long long q, int E) {
  const unsigned long long s = (unsigned long long)(q >> 63), a = ((unsigned long long)q ^ s) - s;
  const int lz = __clzll((long long)a);
  const unsigned long long t = a << ((lz - 1) & 63);
  const unsigned long long m = (t + 0x1ffull + ((t >> 10) & 1ull)) >> 10;
  unsigned long long b = m + ((unsigned long long)(unsigned)(E + 4 - lz) << 52);
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

// Row march like march_ring, with the stencil in fixed point: field(j, slot, FRow&)
// builds row j of the operand, finish(j, slot, c, y) consumes row j with the
// operand's values c and y = A c.  The two horizontal neighbours and the row
// behind enter a row's partial sum when it arrives, the row ahead completes it.
template <int V, int K, class FieldF, class FinishF>
__device__ __forceinline__ void march_ring_fix(WarpRing& ring, int ny, int lane, int xs, int y0, int y1, bool rev,
                                               const RingVec (&vecs)[K], const int (&off)[K], FieldF& field,
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
  FixRow<V> prev, sum;  // the row behind; the current row's partial sum
  double c[V];          // the current row
  const unsigned char* sC = nullptr;
  for (int t = 0; t < total; ++t) {
    FRow<V, double> f;
    const unsigned char* sA = ring.wait(q0 + t);
    const int j = row_of(t);
    if (j < 0 || j >= ny) f.zero();
    else field(j, sA, f);
    FixRow<V> a;
    unsigned m = (unsigned)__double2hiint(f.hl) & 0x7fffffffu;
#pragma unroll
    for (int k = 0; k < V; ++k) m = max(m, (unsigned)__double2hiint(f.f[k]) & 0x7fffffffu);
    a.E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
#pragma unroll
    for (int k = 0; k < V; ++k) a.q[k] = fix_of(f.f[k], a.E);
    if (t >= 2) {
      const int E = max(sum.E, a.E);
      fix_align<V>(sum.q, sum.E, E);
      long long n[V];
#pragma unroll
      for (int k = 0; k < V; ++k) n[k] = a.q[k];
      fix_align<V>(n, a.E, E);
      double y[V];
#pragma unroll
      for (int k = 0; k < V; ++k) y[k] = fix_to_int(sum.q[k] - n[k], E);
      if (E < kFixLow || E > kFixHigh) {
#pragma unroll
        for (int k = 0; k < V; ++k) y[k] = E < kFixLow ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
      }
      finish(row_of(t - 1), sC, c, y);
      __syncwarp();
      if (t - 1 + ring.S < total) ring.produce<V, K>(row_of(t - 1 + ring.S), ny, t - 1 + ring.S <= T, P);
    }
    if (t >= 1 && t <= T) {
      const long long h = fix_of(f.hl, a.E);
      long long l = __shfl_up_sync(0xffffffffu, a.q[V - 1], 1), r = __shfl_down_sync(0xffffffffu, a.q[0], 1);
      if (lane == 0) l = h;
      if (lane == 31) r = h;
      const int E = max(prev.E, a.E);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        const long long w = k == 0 ? l : a.q[k - 1], e = k == V - 1 ? r : a.q[k + 1];
        sum.q[k] = 4 * a.q[k] - w - e;
        c[k] = f.f[k];
      }
      fix_align<V>(sum.q, a.E, E);
      fix_align<V>(prev.q, prev.E, E);
#pragma unroll
      for (int k = 0; k < V; ++k) sum.q[k] -= prev.q[k];
      sum.E = E;
      if (t == 1) {  // the slot of the row behind the first one is free
        __syncwarp();
        if (ring.S < total) ring.produce<V, K>(row_of(ring.S), ny, ring.S <= T, P);
      }
    }
    prev = a;
    sC = sA;
  }
  ring.q = q0 + (unsigned)total;
}

// The same march over rows loaded straight into registers: load(j, Raw&) reads row j
// one step ahead of its use, field(j, raw, FRow&) builds the operand's row from it,
// finish(j, c, y) consumes row j.
template <int V, class Raw, class LoadF, class FieldF, class FinishF>
__device__ __forceinline__ void march_fix(int ny, int lane, int y0, int y1, bool rev, LoadF& load, FieldF& field,
                                          FinishF& finish) {
  if (y0 >= y1) return;
  const int step = rev ? -1 : 1;
  const int T = y1 - y0, first = rev ? y1 : y0 - 1;
  FixRow<V> prev, sum;
  double c[V];
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
    unsigned m = (unsigned)__double2hiint(f.hl) & 0x7fffffffu;
#pragma unroll
    for (int k = 0; k < V; ++k) m = max(m, (unsigned)__double2hiint(f.f[k]) & 0x7fffffffu);
    a.E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
#pragma unroll
    for (int k = 0; k < V; ++k) a.q[k] = fix_of(f.f[k], a.E);
    if (t >= 2) {
      const int E = max(sum.E, a.E);
      fix_align<V>(sum.q, sum.E, E);
      long long n[V];
#pragma unroll
      for (int k = 0; k < V; ++k) n[k] = a.q[k];
      fix_align<V>(n, a.E, E);
      double y[V];
#pragma unroll
      for (int k = 0; k < V; ++k) y[k] = fix_to(sum.q[k] - n[k], E);
      if (E < kFixLow || E > kFixHigh) {
#pragma unroll
        for (int k = 0; k < V; ++k) y[k] = E < kFixLow ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
      }
      finish(j - step, c, y);
    }
    const long long h = fix_of(f.hl, a.E);
    long long l = __shfl_up_sync(0xffffffffu, a.q[V - 1], 1), r = __shfl_down_sync(0xffffffffu, a.q[0], 1);
    if (lane == 0) l = h;
    if (lane == 31) r = h;
    const int E = t == 0 ? a.E : max(prev.E, a.E);
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const long long w = k == 0 ? l : a.q[k - 1], e = k == V - 1 ? r : a.q[k + 1];
      sum.q[k] = 4 * a.q[k] - w - e;
      c[k] = f.f[k];
    }
    if (t > 0) {
      fix_align<V>(sum.q, a.E, E);
      fix_align<V>(prev.q, prev.E, E);
#pragma unroll
      for (int k = 0; k < V; ++k) sum.q[k] -= prev.q[k];
    }
    sum.E = E;
    prev = a;
  }
}

__device__ __forceinline__ unsigned fix_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// r of fixed-point sums q at exponent E (uniform in the warp), the range's ends included.
template <int V>
__device__ __forceinline__ void fix_results(const long long (&q)[V], int E, double (&r)[V]) {
#pragma unroll
  for (int k = 0; k < V; ++k) r[k] = fix_to(q[k], E);
  if (E < kFixLow || E > kFixHigh) {
#pragma unroll
    for (int k = 0; k < V; ++k) r[k] = E < kFixLow ? 0.0 : __longlong_as_double(0x7ff8000000000000ll);
  }
}

// r = b - A c on a lane vector from its neighbours (up, dn: rows; w, e: columns), all
// aligned to the warp's largest exponent: nine values of that size at most stay
// below 2^63.  Every lane of the warp calls.
template <int W>
__device__ __forceinline__ void fix_residual(const double (&c)[W], const double (&up)[W], const double (&dn)[W],
                                             double w, double e, const double (&b)[W], double (&r)[W]) {
  unsigned m = max(fix_mag(w), fix_mag(e));
#pragma unroll
  for (int k = 0; k < W; ++k) m = max(max(m, max(fix_mag(c[k]), fix_mag(b[k]))), max(fix_mag(up[k]), fix_mag(dn[k])));
  const int E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
  long long q[W], f[W];
#pragma unroll
  for (int k = 0; k < W; ++k) f[k] = fix_of(c[k], E);
  const long long l = fix_of(w, E), h = fix_of(e, E);
#pragma unroll
  for (int k = 0; k < W; ++k)
    q[k] = fix_of(b[k], E) - 4 * f[k] + (k == 0 ? l : f[k - 1]) + (k == W - 1 ? h : f[k + 1]) + fix_of(up[k], E) +
           fix_of(dn[k], E);
  fix_results<W>(q, E, r);
}

}  // namespace lap5
