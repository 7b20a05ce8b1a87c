// exchange.cuh -- sums and messages between the CTAs of a persistent solve.
//
// The reductions of a CG iteration are latency: both parts are built for that.
//
//  * Messages carry their own flags.  A value travels as 64-bit words of 32 data
//    and 32 tag bits (relaxed 64-bit accesses are single-copy atomic), so a
//    receiver polls the data itself: no fence, no separate flag, one L2 round trip.
//    (The idea is that of NCCL's low-latency (LL) protocol: 8-byte stores of 4 bytes of
//    data and a 4-byte flag.)
//    An exchange of one value among 152 CTAs, one 256-byte slot a CTA polled by one
//    lane each, measured 1.1 us (1.6 us with five slots a lane; 4.1 us with 16-byte
//    slots, whose lines writers and pollers share; 1.9 us with an inbox a CTA).
//  * Sums over lanes are integer.  An FP64 addition takes 64 to 76 cycles of its
//    scheduler's pipe whatever the number of active lanes, so a five-step shuffle
//    tree in each of 16 warps costs 1500 cycles.  warp_sum aligns the addends to the
//    largest exponent of the warp and adds fixed-point pieces with redux.sync: 290
//    cycles of latency and one FP64 operation (the conversion back).  The result
//    is within one rounding of the exact sum (bits below 2^-63 of the largest
//    addend are dropped) and does not depend on the order.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace lap5 {

using u64 = unsigned long long;

constexpr int kPollWarps = 5;               // a CTA's last warps wait for the other CTAs' sums
constexpr int kMaxPeers = 32 * kPollWarps;  // one slot a lane
constexpr int kSlotWords = 32;              // 64-bit words between slots (256 bytes)

// ---------------------------------------------------------------------------
// Sums over a warp, in fixed point.
// ---------------------------------------------------------------------------

// One addend: mant is its magnitude's significand with the leading bit of a normal
// number at bit 63, ex its biased exponent (1 for subnormals), neg its sign mask.
struct FixTerm {
  u64 mant;
  int ex, neg;
};
__device__ __forceinline__ FixTerm fix_term(double v) {
  const u64 b = (u64)__double_as_longlong(v);
  const int e = (int)((b >> 52) & 0x7ff);
  FixTerm t;
  t.mant = ((b & 0xfffffffffffffull) | (e ? (1ull << 52) : 0ull)) << 11;
  t.ex = max(e, 1);
  t.neg = (int)((long long)b >> 63);
  return t;
}
__device__ __forceinline__ FixTerm fix_term(float v) {
  const uint32_t b = __float_as_uint(v);
  const int e = (int)((b >> 23) & 0xff);
  FixTerm t;
  t.mant = (u64)(((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 8) << 32;
  t.ex = max(e, 1);
  t.neg = (int)b >> 31;
  return t;
}

// M sums at once, each of N terms of every lane (N <= 7), so that their latencies
// overlap; all lanes return them.  kBias: a term is worth mant * 2^(ex - kBias).
// lo, hi: the exponents for which a result's exponent field cannot leave
// [1, 2046]; false when a largest one is outside (sums of zeros, infinities, NaN
// and values near the ends of the range: the caller adds with FP64 operations).
template <int M, int N>
__device__ __forceinline__ bool fix_sums(const FixTerm (&t)[M][N], int kBias, int lo, int hi, double (&out)[M]) {
  int em[M];
  bool ok = true;
#pragma unroll
  for (int m = 0; m < M; ++m) {
    em[m] = t[m][0].ex;
#pragma unroll
    for (int k = 1; k < N; ++k) em[m] = max(em[m], t[m][k].ex);
    em[m] = __reduce_max_sync(0xffffffffu, em[m]);
  }
#pragma unroll
  for (int m = 0; m < M; ++m) ok = ok && em[m] >= lo && em[m] <= hi;
  if (!ok) return false;
  int p[M][3];  // pieces of 23, 23 and 18 bits below the largest term's leading bit
#pragma unroll
  for (int m = 0; m < M; ++m) {
    p[m][0] = p[m][1] = p[m][2] = 0;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const int d = em[m] - t[m][k].ex;
      const u64 w = d > 63 ? 0ull : t[m][k].mant >> d;
      const int pa = (int)(w >> 41), pb = (int)((w >> 18) & 0x7fffffu), pc = (int)(w & 0x3ffffu);
      p[m][0] += (pa ^ t[m][k].neg) - t[m][k].neg;
      p[m][1] += (pb ^ t[m][k].neg) - t[m][k].neg;
      p[m][2] += (pc ^ t[m][k].neg) - t[m][k].neg;
    }
  }
#pragma unroll
  for (int m = 0; m < M; ++m)
#pragma unroll
    for (int i = 0; i < 3; ++i) p[m][i] = __reduce_add_sync(0xffffffffu, p[m][i]);  // < N * 32 * 2^23 < 2^31
#pragma unroll
  for (int m = 0; m < M; ++m) {
    // v in units of 2^9 of the terms' last bit, |v| < 2^63: rounded to nearest once
    // here and once in the conversion
    const long long v = ((long long)p[m][0] << 32) + ((long long)p[m][1] << 9) + ((p[m][2] + 256) >> 9);
    const double s = (double)v;
    out[m] = v == 0 ? s : __hiloint2double(__double2hiint(s) + ((em[m] - kBias + 9) << 20), __double2loint(s));
  }
  return true;
}

// The rare cases are calls, out of the way of the usual path.
static __device__ __noinline__ double shfl_sum(double s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
__device__ __forceinline__ double warp_sum(double v) {
  const FixTerm t[1][1] = {{fix_term(v)}};
  double out[1];
  if (fix_sums<1, 1>(t, 1086, 80, 2030, out)) return out[0];
  return __any_sync(0xffffffffu, !(v == 0.0)) ? shfl_sum(v) : 0.0;
}
__device__ __forceinline__ double2 warp_sum2(double v, double w) {
  const FixTerm t[2][1] = {{fix_term(v)}, {fix_term(w)}};
  double out[2];
  if (fix_sums<2, 1>(t, 1086, 80, 2030, out)) return make_double2(out[0], out[1]);
  return make_double2(warp_sum(v), warp_sum(w));
}
__device__ __forceinline__ double warp_sum(float s, float c) {
  const FixTerm t[1][2] = {{fix_term(s), fix_term(c)}};
  double out[1];
  if (fix_sums<1, 2>(t, 190, 2, 254, out)) return out[0];
  return __any_sync(0xffffffffu, !(s == 0.f) || !(c == 0.f)) ? shfl_sum((double)s + (double)c) : 0.0;
}
static __device__ __noinline__ double plain_quotient(double a, double b) { return a / b; }

// a / b from r = 1 / b (correctly rounded): one residual correction (Markstein,
// IBM J. Res. Dev. 34, 1990), a chain of three FP64 operations (200 cycles)
// instead of a division's 570; where r has left the range, the division.
__device__ __forceinline__ double quotient(double a, double b, double r) {
  const double q0 = __dmul_rn(a, r);
  double q = __fma_rn(__fma_rn(-q0, b, a), r, q0);
  if ((__double2hiint(q) & 0x7ff00000) == 0x7ff00000) q = plain_quotient(a, b);
  return q;
}

// ---------------------------------------------------------------------------
// Messages: 32 data and 32 tag bits a word.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void ll_store(u64* p, u64 x, u64 y) {
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}
__device__ __forceinline__ void ll_load(const u64* p, u64& x, u64& y) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
}
__device__ __forceinline__ u64 ll_word(uint32_t data, uint32_t tag) { return (u64)data | ((u64)tag << 32); }
__device__ __forceinline__ bool ll_is(u64 w, uint32_t tag) { return (uint32_t)(w >> 32) == tag; }

__device__ __forceinline__ void ll_send(u64* p, double v, uint32_t tag) {
  ll_store(p, ll_word((uint32_t)__double2loint(v), tag), ll_word((uint32_t)__double2hiint(v), tag));
}
__device__ __forceinline__ bool ll_recv(const u64* p, double& v, uint32_t tag) {
  u64 x, y;
  ll_load(p, x, y);
  v = __hiloint2double((int)(uint32_t)y, (int)(uint32_t)x);
  return ll_is(x, tag) && ll_is(y, tag);
}
__device__ __forceinline__ void ll_send(u64* p, const double (&v)[2], uint32_t tag) {
  ll_send(p, v[0], tag);
  ll_send(p + 2, v[1], tag);
}
__device__ __forceinline__ bool ll_recv(const u64* p, double (&v)[2], uint32_t tag) {
  const bool a = ll_recv(p, v[0], tag), b = ll_recv(p + 2, v[1], tag);
  return a && b;
}
__device__ __forceinline__ void ll_send(u64* p, const float (&v)[4], uint32_t tag) {
  ll_store(p, ll_word(__float_as_uint(v[0]), tag), ll_word(__float_as_uint(v[1]), tag));
  ll_store(p + 2, ll_word(__float_as_uint(v[2]), tag), ll_word(__float_as_uint(v[3]), tag));
}
__device__ __forceinline__ bool ll_recv(const u64* p, float (&v)[4], uint32_t tag) {
  u64 w[4];
  ll_load(p, w[0], w[1]);
  ll_load(p + 2, w[2], w[3]);
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = __uint_as_float((uint32_t)w[k]);
    ok = ok && ll_is(w[k], tag);
  }
  return ok;
}

// Comparisons on the bits, off the FP64 pipe.
__device__ __forceinline__ bool bits_finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool bits_positive(double v) { return __double_as_longlong(v) > 0; }  // NaN with sign 0: true
// a <= b for a >= 0 (not NaN), b >= 0
__device__ __forceinline__ bool bits_le(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }

}  // namespace lap5
