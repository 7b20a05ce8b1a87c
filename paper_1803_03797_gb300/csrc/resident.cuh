// resident.cuh -- chip-resident CG: solves whose state vectors fit in the
// registers and shared memory of a team of CTAs (one CTA an SM, up to the whole
// chip).
//
// CTA c of a team owns a block of rows.  Every thread keeps its points of r,
// z = A p and x (NewCG: r, z, q, p, x) in registers for the whole solve; the
// stencil operand (p; NewCG: w) lives in shared memory with one halo row above
// and below.  Global memory is read for b and x0 and written with x; per
// iteration only two rows a CTA and one partial sum a CTA cross SMs.
//
// What bounds it: an iteration moves nothing through HBM, so the time is the
// latency of the reductions (classic: two an iteration, NewCG: one) plus the
// FP64 pipe (2 operations an SM a clock) in binary64.  Both are built for that:
//
//  * Messages carry their own flags.  A value travels as 64-bit words of 32
//    data and 32 tag bits (relaxed 64-bit accesses are single-copy atomic), so
//    a receiver polls the data itself: no fence, no separate flag, one L2 round
//    trip.  An exchange of one value among 152 CTAs measured 1.6 us with a
//    256-byte slot a CTA (4.1 us with 16-byte slots: writers and pollers then
//    share lines); the streaming kernels' counter barrier and slot sum take
//    about 3 us.
//  * Sums over lanes are integer.  An FP64 addition takes 64 cycles of its
//    scheduler's pipe whatever the number of active lanes, so a five-step
//    shuffle tree over 16 warps costs 1280 cycles an SM sub-partition.  warp_sum aligns
//    the addends to the largest exponent of the warp and adds 64-bit
//    fixed-point pieces with redux.sync: one FP64 operation (the conversion
//    back).  The result is within one rounding of the exact sum (bits below
//    2^-63 of the largest addend are dropped) and does not depend on the order.
//
// Arithmetic per point is that of the streaming kernels (Algorithm 1 with
// z = A p stored and the x update deferred to the next direction update;
// Algorithm 2); dot products differ in summation order only.
#pragma once

#include "cg_kernels.cuh"

namespace lap5 {

constexpr int kResPollWarps = 5;    // a CTA's last warps wait for the other CTAs' sums
constexpr int kResMaxTeam = 32 * kResPollWarps;  // one slot a lane
constexpr int kResMinThreads = 256, kResMaxThreads = 512;
constexpr int kResMaxVals = 4;      // values of one reduction
constexpr int kResSlotWords = 32;   // 64-bit words between slots (256 bytes)
constexpr int kResItemWords = 4;    // 64-bit words of one lane vector in a halo message

using u64 = unsigned long long;

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
__device__ __forceinline__ double warp_sum(const Acc64& a) { return warp_sum(a.s); }
__device__ __forceinline__ double warp_sum(const Acc32& a) { return warp_sum(a.s, a.c); }
__device__ __forceinline__ void warp_sum2(const Acc64& a, const Acc64& b, double (&w)[2]) {
  const double2 t = warp_sum2(a.s, b.s);
  w[0] = t.x;
  w[1] = t.y;
}
__device__ __forceinline__ void warp_sum2(const Acc32& a, const Acc32& b, double (&w)[2]) {
  w[0] = warp_sum(a);
  w[1] = warp_sum(b);
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

// ---------------------------------------------------------------------------
// A team of CTAs.  All message memory is zero when the solve starts; tags start
// at 1 and rise by one a reduction (tag) and a halo exchange (htag).
//
// Buffers are reused without further synchronisation.  Slots alternate between
// two sets: a CTA writes set s again two reductions later, after it has
// gathered the one between, to which every CTA contributed only after it had
// gathered the first.  Halo rows alternate the same way (htag parity): a CTA
// sends exchange h + 2 after a reduction to which its neighbours contributed
// after they had received exchange h.
// ---------------------------------------------------------------------------
// The scalars of an iteration are formed, compared and converted by one warp alone:
// a comparison of doubles or a conversion takes the FP64 pipe as long as an
// addition, and in every one of 16 warps 300 cycles.
struct ResShared {
  double wp[kResMaxVals * 16];  // warp sums
  double gp[kResMaxVals * kResPollWarps];  // sums of 32 CTAs
  double tot[kResMaxVals];      // totals
  double sc[4];                 // scalars kept from one reduction to the next (that warp)
  double ab[2];                 // alpha, beta in the solve's type
  int code, fail;
};
template <class T> __device__ __forceinline__ void res_set(ResShared* s, int i, double v) {
  *reinterpret_cast<T*>(&s->ab[i]) = (T)v;
}
template <class T> __device__ __forceinline__ T res_get(const ResShared* s, int i) {
  return *reinterpret_cast<const T*>(&s->ab[i]);
}

// Comparisons on the bits, off the FP64 pipe.
__device__ __forceinline__ bool bits_finite(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool bits_positive(double v) { return __double_as_longlong(v) > 0; }  // NaN with sign 0: true
// a <= b for a >= 0 (not NaN), b >= 0
__device__ __forceinline__ bool bits_le(double a, double b) { return __double_as_longlong(a) <= __double_as_longlong(b); }

// How a solve goes on after a reduction.
enum { RES_GO = 0, RES_CONVERGED, RES_MAXIT, RES_CURVATURE, RES_NONFINITE, RES_ABORTED };

struct ResTeam {
  int rank, size;
  uint32_t tag, htag;
  u64 *slots, *halos;
  int groups;  // lane vectors a row
  int *err, *abort_flag;
  long long timeout_ns;
  ResShared* sh;

  __device__ __forceinline__ void init(u64* slots_, u64* halos_, int rank_, int size_, int groups_, int* err_,
                                       int* abort_, long long timeout, ResShared* s) {
    rank = rank_;
    size = size_;
    tag = 1;
    htag = 1;
    slots = slots_;
    halos = halos_;
    groups = groups_;
    err = err_;
    abort_flag = abort_;
    timeout_ns = timeout;
    sh = s;
  }
  __device__ __forceinline__ u64* slot(int cta) const {
    return slots + ((size_t)(tag & 1u) * size + cta) * kResSlotWords;
  }
  // message row of exchange h at CTA cta: side 0 arrives from the CTA above (its
  // last row), side 1 from the one below (its first row)
  __device__ __forceinline__ u64* halo(uint32_t h, int cta, int side) const {
    return halos + (((size_t)(h & 1u) * size + cta) * 2 + side) * (size_t)groups * kResItemWords;
  }
  // After a poll that failed: true when the wait must end (time limit; the abort
  // flag, an L2 round trip, is looked at now and then only).
  __device__ __forceinline__ bool give_up(unsigned& spins, u64& t0) const {
    const u64 now = global_ns();
    if (spins++ == 0u) t0 = now;
    if ((spins & 31u) == 0u && ld_relaxed_i32(abort_flag)) return true;
    if ((long long)(now - t0) <= timeout_ns) return false;
    atomicCAS(err, 0, LAP5CG_ERR_SYNC_TIMEOUT);
    __threadfence();
    atomicExch(abort_flag, 1);
    return true;
  }
  template <class V>
  __device__ __forceinline__ void wait_halo(const u64* p, V& v, uint32_t h) const {
    unsigned spins = 0;
    u64 t0 = 0;
    while (!ll_recv(p, v, h)) {
      if (give_up(spins, t0)) {
        sh->fail = 1;  // seen by the next gather
        return;
      }
    }
  }

  // Contribute this CTA's sums of the NV warp sums w (same in every lane of a
  // warp); warp k sums and sends value k.  fence: order this CTA's earlier global
  // writes before the message.
  template <int NV>
  __device__ __forceinline__ void publish(const double (&w)[NV], bool fence = false) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    if (lane == 0) {
#pragma unroll
      for (int k = 0; k < NV; ++k) sh->wp[k * 16 + warp] = w[k];
    }
    __syncthreads();
    if (warp < NV) {
      const double s = warp_sum(lane < nw ? sh->wp[warp * 16 + lane] : 0.0);
      if (fence) __threadfence();
      if (lane == 0) ll_send(slot(rank) + 2 * warp, s, tag);
    }
  }
  // Wait for every CTA's contribution.  The CTA's last kResPollWarps warps poll,
  // one slot a lane (152 slots: 1.1 us an exchange, against 1.6 us with five
  // slots a lane of one warp).  The last warp forms the totals (the same bits in
  // every CTA), hands them to post(totals), which returns how to go on and may
  // set the scalars in *sh (lane 0's stores count), and leaves them in sh->tot.
  // Returns post's code in every thread, or RES_ABORTED when the solve must stop:
  // a wait ran out here, or in a CTA that then stopped contributing.
  template <int NV, class Post>
  __device__ __forceinline__ int gather(Post post, bool fence = false) {
    const int lane = threadIdx.x & 31;
    const int pw = ((int)threadIdx.x >> 5) - ((int)(blockDim.x >> 5) - kResPollWarps);
    if (pw >= 0) {
      double v[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) v[k] = 0.0;
      const int c = 32 * pw + lane;
      unsigned spins = 0;
      u64 t0 = 0;
      for (;;) {
        bool ok = true;
        if (c < size) {
#pragma unroll
          for (int k = 0; k < NV; ++k) ok = ll_recv(slot(c) + 2 * k, v[k], tag) && ok;
        }
        if (__all_sync(0xffffffffu, ok)) break;
        if (__any_sync(0xffffffffu, give_up(spins, t0))) {
          sh->fail = 1;
          break;
        }
      }
      if (fence) __threadfence();
      if constexpr (NV == 2) {
        const double2 u = warp_sum2(v[0], v[1]);
        v[0] = u.x;
        v[1] = u.y;
      } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k] = warp_sum(v[k]);
      }
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) sh->gp[k * kResPollWarps + pw] = v[k];
      }
    }
    __syncthreads();
    if (pw == kResPollWarps - 1) {
      double s[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        s[k] = sh->gp[k * kResPollWarps];
#pragma unroll
        for (int j = 1; j < kResPollWarps; ++j)
          if (32 * j < size) s[k] += sh->gp[k * kResPollWarps + j];
      }
      const int code = post(s);
      if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) sh->tot[k] = s[k];
        sh->code = sh->fail ? (int)RES_ABORTED : code;
      }
    }
    __syncthreads();
    ++tag;
    return sh->code;
  }
  template <int NV>
  __device__ __forceinline__ bool reduce(const double (&w)[NV], double (&o)[NV], bool fence = false) {
    publish<NV>(w, fence);
    const int code = gather<NV>([](const double (&)[NV]) { return (int)RES_GO; }, fence);
#pragma unroll
    for (int k = 0; k < NV; ++k) o[k] = sh->tot[k];
    return code == RES_GO;
  }
};

// ---------------------------------------------------------------------------
// A CTA's rows and a thread's items.  Item e (a lane vector of W columns) is
// row e / groups, columns W (e % groups) ...; a thread's items are tid + k nt,
// K of them at most.  In binary64, where an item's work is FP64 pipe time, a warp
// without a last item skips it, and the CTA has a multiple of four warps so that
// the schedulers share the items evenly; in binary32 all K run, masked.
// ---------------------------------------------------------------------------
template <class T> struct ResVec;
template <> struct ResVec<double> { static constexpr int W = 2; };
template <> struct ResVec<float> { static constexpr int W = 4; };

template <class T, int K>
struct ResItems {
  static constexpr int W = ResVec<T>::W;
  int off[K];       // element offset of item k in the operand's shared rows (row 0 is the upper halo)
  unsigned valid, top, bot, first, last;  // bit k: item exists, in the first / last own row, first / last of its row
  bool full;        // this warp has a last item
  int nr, r0;       // own rows
  int nx, groups, ldp, tail;  // tail: columns of the last lane vector (1 .. W)

  __device__ __forceinline__ void init(int nx_, int ny, int rank, int size) {
    nx = nx_;
    groups = (nx + W - 1) / W;
    ldp = groups * W;
    tail = nx - (groups - 1) * W;
    const int q = ny / size, rem = ny % size;
    nr = q + (rank < rem ? 1 : 0);
    r0 = rank * q + min(rank, rem);
    const int nt = blockDim.x, n = nr * groups;
    full = ((int)threadIdx.x & ~31) + (K - 1) * nt < n;
    valid = top = bot = first = last = 0u;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = (int)threadIdx.x + k * nt;
      const bool v = e < n;
      const int i = v ? e / groups : 0, g = v ? e - i * groups : 0;
      off[k] = (i + 1) * ldp + g * W;
      valid |= (unsigned)v << k;
      top |= (unsigned)(v && i == 0) << k;
      bot |= (unsigned)(v && i == nr - 1) << k;
      first |= (unsigned)(!v || g == 0) << k;
      last |= (unsigned)(!v || g == groups - 1) << k;
    }
  }
  __device__ __forceinline__ bool has(int k) const { return sizeof(T) == 4 || k < K - 1 || full; }  // warp-uniform
  __device__ __forceinline__ bool is(unsigned m, int k) const { return (m >> k) & 1u; }
  __device__ __forceinline__ int row(int k) const { return off[k] / ldp - 1; }       // own row
  __device__ __forceinline__ int col(int k) const { return off[k] % ldp; }
  // columns past nx hold zero in every vector
  template <class M>
  __device__ __forceinline__ void mask_tail(int k, M (&v)[W]) const {
    if (is(last, k) && tail < W) {
#pragma unroll
      for (int q = 1; q < W; ++q)
        if (q >= tail) v[q] = M(0);
    }
  }
};

// y = A c on item k from the shared rows sm (c: the item itself), in the order
// 4C - W - E - S - N.  up / dn: rows above / below.  Whole-warp call.
template <class T, int K, class M>
__device__ __forceinline__ void res_stencil(const ResItems<T, K>& it, int k, const T* sm, const M (&c)[ResVec<T>::W],
                                            const M (&up)[ResVec<T>::W], const M (&dn)[ResVec<T>::W],
                                            M (&y)[ResVec<T>::W]) {
  constexpr int W = ResVec<T>::W;
  const int lane = threadIdx.x & 31, o = it.off[k];
  M l = shfl_up1(c[W - 1]), r = shfl_dn1(c[0]);
  if (it.is(it.first, k)) l = M(0);
  else if (lane == 0) l = (M)sm[o - 1];
  if (it.is(it.last, k)) r = M(0);
  else if (lane == 31) r = (M)sm[o + W];
#pragma unroll
  for (int q = 0; q < W; ++q) {
    M a = M(4) * c[q];
    a -= q == 0 ? l : c[q - 1];
    a -= q == W - 1 ? r : c[q + 1];
    a -= up[q];
    a -= dn[q];
    y[q] = a;
  }
  it.mask_tail(k, y);
}

template <class T>
__device__ __forceinline__ void res_ld(const T* sm, int o, T (&v)[ResVec<T>::W]) {
  VecIO<ResVec<T>::W, T>::load(sm + o, v);
}
template <class T>
__device__ __forceinline__ void res_st(T* sm, int o, const T (&v)[ResVec<T>::W]) {
  VecIO<ResVec<T>::W, T>::store(sm + o, v);
}

// Send item k where it is the CTA's first or last row (exchange h).
template <class T, int K>
__device__ __forceinline__ void res_send(const ResTeam& tm, const ResItems<T, K>& it, int k,
                                         const T (&v)[ResVec<T>::W], uint32_t h) {
  constexpr int W = ResVec<T>::W;
  if (it.is(it.top, k) && tm.rank > 0)
    ll_send(tm.halo(h, tm.rank - 1, 1) + (it.off[k] - it.ldp) / W * kResItemWords, v, h);
  if (it.is(it.bot, k) && tm.rank + 1 < tm.size)
    ll_send(tm.halo(h, tm.rank + 1, 0) + (it.off[k] - it.nr * it.ldp) / W * kResItemWords, v, h);
}

// Receive both halo rows of exchange h, shared by the threads t0 = 0 .. nt - 1;
// f(offset, values) consumes each lane vector.
template <class T, int K, class F>
__device__ __forceinline__ void res_halos(const ResTeam& tm, const ResItems<T, K>& it, uint32_t h, int t0, int nt,
                                          F f) {
  constexpr int W = ResVec<T>::W;
  for (int e = t0; e < 2 * it.groups; e += nt) {
    const int side = e >= it.groups, g = e - side * it.groups;
    if (side ? tm.rank + 1 >= tm.size : tm.rank == 0) continue;
    T v[W];
    tm.wait_halo(tm.halo(h, tm.rank, side) + g * kResItemWords, v, h);
    f((side ? (it.nr + 1) * it.ldp : 0) + g * W, v);
  }
}

// Global rows: item k's lane vector at row pitch ld (columns >= nx read as zero).
template <class T, int K, class U>
__device__ __forceinline__ void res_load(const ResItems<T, K>& it, int k, const U* g, int ld, U (&v)[ResVec<T>::W]) {
  constexpr int W = ResVec<T>::W;
  const int c = it.col(k);
  if (it.is(it.valid, k)) load_group<W, U, U>(g + (size_t)(it.r0 + it.row(k)) * ld + c, c, it.nx, v);
  else {
#pragma unroll
    for (int q = 0; q < W; ++q) v[q] = U(0);
  }
}
template <class T, int K, class U>
__device__ __forceinline__ void res_store(const ResItems<T, K>& it, int k, U* g, int ld, const U (&v)[ResVec<T>::W]) {
  constexpr int W = ResVec<T>::W;
  const int c = it.col(k);
  if (it.is(it.valid, k)) store_group<W, U, U>(g + (size_t)(it.r0 + it.row(k)) * ld + c, c, it.nx, v);
}

// A g on item k straight from global memory (whole grid at pitch ld; L2 reads,
// since other CTAs write g during the solve).
template <class T, int K, class U>
__device__ __forceinline__ void res_global_stencil(const ResItems<T, K>& it, int k, const U* g, int ld, int ny,
                                                   U (&y)[ResVec<T>::W]) {
  constexpr int W = ResVec<T>::W;
#pragma unroll
  for (int q = 0; q < W; ++q) y[q] = U(0);
  if (!it.is(it.valid, k)) return;
  const int j = it.r0 + it.row(k), c = it.col(k);
#pragma unroll
  for (int q = 0; q < W; ++q) {
    const int x = c + q;
    if (x < it.nx) {
      const U* p = g + (size_t)j * ld + x;
      U a = U(4) * __ldcg(p);
      a -= x > 0 ? __ldcg(p - 1) : U(0);
      a -= x + 1 < it.nx ? __ldcg(p + 1) : U(0);
      a -= j > 0 ? __ldcg(p - ld) : U(0);
      a -= j + 1 < ny ? __ldcg(p + ld) : U(0);
      y[q] = a;
    }
  }
}

struct ResArgs {
  int nx, ny, ld;
  const void* b;
  void* x;
  lap5cg_info* info;
  double* history;
  double tol;
  int maxit, true_res;
  int max_outer, maxit_inner;  // mixed precision
  double tol_inner;
};

__device__ __forceinline__ void res_info(const ResArgs& a, const ResTeam& tm, int status, bool aborted, int iters,
                                         int outer, double gamma, double bb, double relres_true) {
  if (tm.rank != 0 || threadIdx.x != 0) return;
  lap5cg_info inf;
  int st = status;
  const int e = atomicAdd(tm.err, 0);
  if (e != 0) st = e;
  else if (aborted) st = LAP5CG_ERR_SYNC_TIMEOUT;
  inf.status = st;
  inf.iters = iters;
  inf.outer_iters = outer;
  inf.pad = 0;
  inf.relres_recursive = (bb > 0.0) ? sqrt(gamma / bb) : 0.0;
  inf.relres_true = relres_true;
  *a.info = inf;
}

// ---------------------------------------------------------------------------
// Algorithm 1 on the resident state: r holds the residual and its first and
// last rows were sent (exchange tm.htag - 1); x accumulates alpha p.  Returns
// why it ended; x is complete (deferred update applied) unless aborted.
// ---------------------------------------------------------------------------
template <class T, int K>
__device__ __forceinline__ int res_classic_loop(ResTeam& tm, const ResItems<T, K>& it, T* sm,
                                                T (&r)[K][ResVec<T>::W], T (&x)[K][ResVec<T>::W], double& gamma,
                                                double thr, int maxit, int& iters, double* history, double bb) {
  constexpr int W = ResVec<T>::W;
  using Acc = typename AccOf<T>::type;
  if (!(gamma > thr)) return RES_CONVERGED;
  if (iters >= maxit) return RES_MAXIT;
  ResShared* sh = tm.sh;
  T z[K][W];
  T am = T(0), bm = T(0);
  const int start = iters;
  int why;
  // the neighbours' rows of r land beside the operand's halo rows while the
  // reduction that forms beta is under way (its polling warps are busy)
  T* hst = sm + (size_t)(it.nr + 2) * it.ldp;
  auto stage_halos = [&]() {
    if ((int)threadIdx.x < (int)blockDim.x - 32 * kResPollWarps)
      res_halos<T, K>(tm, it, tm.htag - 1u, (int)threadIdx.x, (int)blockDim.x - 32 * kResPollWarps,
                      [&](int o, const T (&v)[W]) { res_st(hst, o < it.ldp ? o : o - it.nr * it.ldp, v); });
  };
  stage_halos();
  if (threadIdx.x == 0) {
    sh->sc[0] = gamma;
    sh->sc[1] = 1.0 / gamma;
  }
  __syncthreads();
  do {
    const bool first = iters == start;
    // p = r + beta p on the own rows (x += alpha p of the last iteration with
    // it) and on the halo rows, whose r has arrived
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (!it.has(k)) break;
      T p[W];
      if (first) {
#pragma unroll
        for (int q = 0; q < W; ++q) p[q] = r[k][q];
      } else {
        res_ld(sm, it.off[k], p);
#pragma unroll
        for (int q = 0; q < W; ++q) {
          x[k][q] = fmx(am, p[q], x[k][q]);
          p[q] = fmx(bm, p[q], r[k][q]);
        }
      }
      if (it.is(it.valid, k)) res_st(sm, it.off[k], p);
    }
    for (int e = threadIdx.x; e < 2 * it.groups; e += blockDim.x) {
      const int side = e >= it.groups, o = (side ? it.nr * it.ldp : 0) + e * W;
      T p[W], rv[W];
      res_ld(hst, e * W, rv);
      if (first) {
#pragma unroll
        for (int q = 0; q < W; ++q) p[q] = rv[q];
      } else {
        res_ld(sm, o, p);
#pragma unroll
        for (int q = 0; q < W; ++q) p[q] = fmx(bm, p[q], rv[q]);
      }
      res_st(sm, o, p);
    }
    __syncthreads();
    {
      Acc acc;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        T c[W], up[W], dn[W];
        res_ld(sm, it.off[k], c);
        res_ld(sm, it.off[k] - it.ldp, up);
        res_ld(sm, it.off[k] + it.ldp, dn);
        if (!it.is(it.valid, k)) {
#pragma unroll
          for (int q = 0; q < W; ++q) c[q] = T(0);
        }
        res_stencil<T, K, T>(it, k, sm, c, up, dn, z[k]);
        if (!it.is(it.valid, k)) {
#pragma unroll
          for (int q = 0; q < W; ++q) z[k][q] = T(0);
        }
        acc.add_block(c, z[k]);
      }
      const double w[1] = {warp_sum(acc)};
      tm.publish<1>(w);
    }
    // alpha = gamma / (p, A p), and beside it in lane 1 the reciprocal that the
    // next quotient by gamma starts from
    why = tm.gather<1>([sh](const double (&s)[1]) {
      const bool l1 = (threadIdx.x & 31) == 1;
      const double gm = sh->sc[0];
      const double q = (l1 ? 1.0 : gm) / (l1 ? gm : s[0]);
      const double rg = __shfl_sync(0xffffffffu, q, 1);
      if ((threadIdx.x & 31) == 0) {
        sh->sc[1] = rg;
        res_set<T>(sh, 0, q);
      }
      return bits_positive(s[0]) && bits_finite(s[0]) ? (int)RES_GO : (int)RES_CURVATURE;
    });
    if (why != RES_GO) break;
    am = res_get<T>(sh, 0);
    {
      Acc acc;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
#pragma unroll
        for (int q = 0; q < W; ++q) r[k][q] = fmx(-am, z[k][q], r[k][q]);
        res_send<T, K>(tm, it, k, r[k], tm.htag);
        acc.add_block(r[k], r[k]);
      }
      ++tm.htag;
      const double w[1] = {warp_sum(acc)};
      tm.publish<1>(w);
      stage_halos();
    }
    why = tm.gather<1>([sh, thr](const double (&s)[1]) {
      const double be = quotient(s[0], sh->sc[0], sh->sc[1]);
      __syncwarp();
      if ((threadIdx.x & 31) == 0) {
        sh->sc[0] = s[0];
        res_set<T>(sh, 1, be);
      }
      return !bits_finite(s[0]) ? (int)RES_NONFINITE : bits_le(s[0], thr) ? (int)RES_CONVERGED : (int)RES_GO;
    });
    if (why == RES_ABORTED) break;
    ++iters;
    bm = res_get<T>(sh, 1);
    if (history && tm.rank == 0 && threadIdx.x == 0) history[iters] = sqrt(sh->tot[0] / bb);
  } while (why == RES_GO && iters < maxit);
  if (why == RES_ABORTED) return why;
  if (why == RES_GO) why = RES_MAXIT;
  gamma = sh->sc[0];
  // The deferred update.  It is pending after an iteration whose direction pass
  // has not been followed by another one; after a curvature failure that pass
  // has already applied the last update.
  if (iters > start && why != RES_CURVATURE) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (!it.has(k)) break;
      T p[W];
      res_ld(sm, it.off[k], p);
#pragma unroll
      for (int q = 0; q < W; ++q) x[k][q] = fmx(am, p[q], x[k][q]);
    }
  }
  return why;
}

// r = b - A x0 with (b, b) and (r, r) as warp sums.
template <class T, int K>
__device__ __forceinline__ void res_start(const ResItems<T, K>& it, const ResArgs& a, T (&r)[K][ResVec<T>::W],
                                          T (&x)[K][ResVec<T>::W], double (&w)[2]) {
  constexpr int W = ResVec<T>::W;
  using Acc = typename AccOf<T>::type;
  Acc abb, arr;
#pragma unroll
  for (int k = 0; k < K; ++k) {
#pragma unroll
    for (int q = 0; q < W; ++q) r[k][q] = x[k][q] = T(0);
    if (!it.has(k)) break;
    T b[W], ax[W];
    res_load<T, K>(it, k, static_cast<const T*>(a.b), a.ld, b);
    res_load<T, K>(it, k, static_cast<const T*>(a.x), a.ld, x[k]);
    res_global_stencil<T, K>(it, k, static_cast<const T*>(a.x), a.ld, a.ny, ax);
#pragma unroll
    for (int q = 0; q < W; ++q) r[k][q] = b[q] - ax[q];
    it.mask_tail(k, r[k]);
    abb.add_block(b, b);
    arr.add_block(r[k], r[k]);
  }
  warp_sum2(abb, arr, w);
}

// ||b - A x||^2 of the resident x (its rows travel like any operand's).
template <class T, int K>
__device__ __forceinline__ bool res_true_residual(ResTeam& tm, const ResItems<T, K>& it, const ResArgs& a, T* sm,
                                                  const T (&x)[K][ResVec<T>::W], double& rr) {
  constexpr int W = ResVec<T>::W;
  using Acc = typename AccOf<T>::type;
  __syncthreads();  // every read of the operand rows is done
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (!it.has(k)) break;
    if (it.is(it.valid, k)) res_st(sm, it.off[k], x[k]);
    res_send<T, K>(tm, it, k, x[k], tm.htag);
  }
  res_halos<T, K>(tm, it, tm.htag, threadIdx.x, blockDim.x, [&](int o, const T (&v)[W]) { res_st(sm, o, v); });
  ++tm.htag;
  __syncthreads();
  Acc acc;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (!it.has(k)) break;
    T b[W], up[W], dn[W], ax[W];
    res_load<T, K>(it, k, static_cast<const T*>(a.b), a.ld, b);
    res_ld(sm, it.off[k] - it.ldp, up);
    res_ld(sm, it.off[k] + it.ldp, dn);
    res_stencil<T, K, T>(it, k, sm, x[k], up, dn, ax);
    if (it.is(it.valid, k)) {
      T rv[W];
#pragma unroll
      for (int q = 0; q < W; ++q) rv[q] = b[q] - ax[q];
      acc.add_block(rv, rv);
    }
  }
  const double w[1] = {warp_sum(acc)};
  double o[1];
  if (!tm.reduce<1>(w, o)) return false;
  rr = o[0];
  return true;
}

template <class T, int K>
__device__ __forceinline__ void res_zero_rows(const ResItems<T, K>& it, T* sm) {
  __syncthreads();
  for (int e = threadIdx.x; e < (it.nr + 4) * it.ldp; e += blockDim.x) sm[e] = T(0);
  __syncthreads();
}

// A whole classic solve (a.x, a.b of type T).
template <class T, int K>
__device__ __forceinline__ void res_classic(const ResArgs& a, ResTeam& tm, T* sm) {
  constexpr int W = ResVec<T>::W;
  ResItems<T, K> it;
  it.init(a.nx, a.ny, tm.rank, tm.size);
  res_zero_rows<T, K>(it, sm);
  T r[K][W], x[K][W];
  int status = LAP5CG_NOT_CONVERGED, iters = 0;
  double bb = 0.0, gamma = 0.0, relres_true = nan("");
  bool aborted = false, store = false;
  double w[2], o[2];
  res_start<T, K>(it, a, r, x, w);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (it.has(k)) res_send<T, K>(tm, it, k, r[k], tm.htag);
  ++tm.htag;
  if (!tm.reduce<2>(w, o)) { aborted = true; goto done; }
  bb = o[0];
  gamma = o[1];
  if (!isfinite(bb)) { status = LAP5CG_ERR_NONFINITE; gamma = 0.0; goto done; }
  store = true;
  if (bb == 0.0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int q = 0; q < W; ++q) x[k][q] = T(0);
    status = LAP5CG_OK;
    gamma = 0.0;
    relres_true = 0.0;
    goto done;
  }
  if (a.history && tm.rank == 0 && threadIdx.x == 0) a.history[0] = sqrt(gamma / bb);
  if (!isfinite(gamma)) {
    status = LAP5CG_ERR_NONFINITE;
  } else {
    const double thr = a.tol > 0.0 ? a.tol * a.tol * bb : 0.0;
    const int why = res_classic_loop<T, K>(tm, it, sm, r, x, gamma, thr, a.maxit, iters, a.history, bb);
    if (why == RES_ABORTED) { aborted = true; goto done; }
    status = why == RES_CONVERGED ? LAP5CG_OK
             : why == RES_CURVATURE ? LAP5CG_ERR_BREAKDOWN
             : why == RES_NONFINITE ? LAP5CG_ERR_NONFINITE
                                    : LAP5CG_NOT_CONVERGED;
  }
  if (a.true_res) {
    double rr;
    if (!res_true_residual<T, K>(tm, it, a, sm, x, rr)) { aborted = true; goto done; }
    relres_true = sqrt(rr / bb);
  }
done:
  if (store) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (it.has(k)) res_store<T, K>(it, k, static_cast<T*>(a.x), a.ld, x[k]);
  }
  res_info(a, tm, status, aborted, iters, 0, gamma, bb, relres_true);
}

// ---------------------------------------------------------------------------
// Algorithm 2: one reduction an iteration.  n = A w (halo rows included) is
// formed between contributing (gamma, delta) and gathering them, so the
// reduction's latency covers the stencil (Sec. II, Fig. NewCG).
// ---------------------------------------------------------------------------
template <class T, int K>
__device__ __forceinline__ void res_newcg(const ResArgs& a, ResTeam& tm, T* sm) {
  constexpr int W = ResVec<T>::W;
  using Acc = typename AccOf<T>::type;
  ResItems<T, K> it;
  it.init(a.nx, a.ny, tm.rank, tm.size);
  res_zero_rows<T, K>(it, sm);
  T r[K][W], x[K][W], z[K][W], q[K][W], p[K][W];
  int status = LAP5CG_NOT_CONVERGED, iters = 0;
  double bb = 0.0, gamma = 0.0, relres_true = nan("");
  bool aborted = false, store = false;
  // A times the operand in the shared rows; the rows across the CTA's edges come
  // straight out of the messages of exchange h
  auto apply = [&](int k, uint32_t h, T (&c)[W], T (&y)[W]) {
    T up[W], dn[W];
    res_ld(sm, it.off[k], c);
    if (it.is(it.top, k) && tm.rank > 0)
      tm.wait_halo(tm.halo(h, tm.rank, 0) + (it.off[k] - it.ldp) / W * kResItemWords, up, h);
    else res_ld(sm, it.off[k] - it.ldp, up);
    if (it.is(it.bot, k) && tm.rank + 1 < tm.size)
      tm.wait_halo(tm.halo(h, tm.rank, 1) + (it.off[k] - it.nr * it.ldp) / W * kResItemWords, dn, h);
    else res_ld(sm, it.off[k] + it.ldp, dn);
    __syncwarp();
    if (!it.is(it.valid, k)) {
#pragma unroll
      for (int e = 0; e < W; ++e) c[e] = T(0);
    }
    res_stencil<T, K, T>(it, k, sm, c, up, dn, y);
    if (!it.is(it.valid, k)) {
#pragma unroll
      for (int e = 0; e < W; ++e) y[e] = T(0);
    }
  };
  {
    double w[2], o[1];
    res_start<T, K>(it, a, r, x, w);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (!it.has(k)) break;
      if (it.is(it.valid, k)) res_st(sm, it.off[k], r[k]);
      res_send<T, K>(tm, it, k, r[k], tm.htag);
    }
    ++tm.htag;
    const double w1[1] = {w[0]};
    if (!tm.reduce<1>(w1, o)) { aborted = true; goto done; }
    bb = o[0];
  }
  if (!isfinite(bb)) { status = LAP5CG_ERR_NONFINITE; goto done; }
  store = true;
  if (bb == 0.0) {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int e = 0; e < W; ++e) x[k][e] = T(0);
    status = LAP5CG_OK;
    relres_true = 0.0;
    goto done;
  }
  {
    const double thr = a.tol > 0.0 ? a.tol * a.tol * bb : 0.0;
    Acc ag, ad;
    {  // w = A r (kept in z until every read of r's rows is done), (r, r), (w, r)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        T c[W];
        apply(k, tm.htag - 1u, c, z[k]);
        ag.add_block(c, c);
        ad.add_block(z[k], c);
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        if (it.is(it.valid, k)) res_st(sm, it.off[k], z[k]);
        res_send<T, K>(tm, it, k, z[k], tm.htag);
      }
      ++tm.htag;
    }
    ResShared* sh = tm.sh;
    for (;;) {
      const bool first = iters == 0;
      {
        double w[2];
        warp_sum2(ag, ad, w);
        tm.publish<2>(w);
      }
      T n[K][W], c[K][W];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        apply(k, tm.htag - 1u, c[k], n[k]);
      }
      const bool cap = iters >= a.maxit;
      const int why = tm.gather<2>([sh, first, cap, thr](const double (&s)[2]) {
        // Algorithm 2's alpha = 1 / (delta/gamma - beta/alpha_old), as
        // gamma / (delta - gamma beta / alpha_old): an FP64 division is a chain of
        // ~560 cycles, so one is left on the way to alpha, with 1 / alpha and
        // 1 / gamma (for the next iteration) beside it in lanes 1 and 2.
        // sc: gamma, 1 / gamma and 1 / alpha of the last iteration
        const int lane = threadIdx.x & 31;
        const double g = s[0], d = s[1];
        double be = 0.0, dn = d;
        if (!first) {
          be = quotient(g, sh->sc[0], sh->sc[1]);
          dn = __fma_rn(-g, __dmul_rn(be, sh->sc[2]), d);
        }
        const double q = (lane == 0 ? g : lane == 1 ? dn : 1.0) / (lane == 0 ? dn : g);
        const double ra = __shfl_sync(0xffffffffu, q, 1), rg = __shfl_sync(0xffffffffu, q, 2);
        if (lane == 0) {
          sh->sc[0] = g;
          sh->sc[1] = rg;
          sh->sc[2] = ra;
          res_set<T>(sh, 0, q);
          res_set<T>(sh, 1, be);
        }
        return !bits_finite(g)                             ? (int)RES_NONFINITE
               : bits_le(g, thr)                           ? (int)RES_CONVERGED
               : cap                                       ? (int)RES_MAXIT
               : !(bits_positive(dn) && bits_finite(dn))   ? (int)RES_CURVATURE
                                                           : (int)RES_GO;
      });
      if (why == RES_ABORTED) {
        aborted = true;
        goto done;
      }
      if (a.history && tm.rank == 0 && threadIdx.x == 0) a.history[iters] = sqrt(sh->tot[0] / bb);
      if (why != RES_GO) {
        gamma = sh->tot[0];
        status = why == RES_CONVERGED ? LAP5CG_OK
                 : why == RES_MAXIT   ? LAP5CG_NOT_CONVERGED
                 : why == RES_CURVATURE ? LAP5CG_ERR_BREAKDOWN
                                        : LAP5CG_ERR_NONFINITE;
        break;
      }
      const T am = res_get<T>(sh, 0), bm = res_get<T>(sh, 1);
      ag = Acc();
      ad = Acc();
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        T wv[W];
#pragma unroll
        for (int e = 0; e < W; ++e) {
          z[k][e] = first ? n[k][e] : fmx(bm, z[k][e], n[k][e]);
          wv[e] = fmx(-am, z[k][e], c[k][e]);
        }
        if (it.is(it.valid, k)) res_st(sm, it.off[k], wv);
        res_send<T, K>(tm, it, k, wv, tm.htag);
#pragma unroll
        for (int e = 0; e < W; ++e) {
          q[k][e] = first ? c[k][e] : fmx(bm, q[k][e], c[k][e]);
          p[k][e] = first ? r[k][e] : fmx(bm, p[k][e], r[k][e]);
          r[k][e] = fmx(-am, q[k][e], r[k][e]);
          x[k][e] = fmx(am, p[k][e], x[k][e]);
        }
        ag.add_block(r[k], r[k]);
        ad.add_block(wv, r[k]);
      }
      ++tm.htag;
      ++iters;
    }
  }
  if (a.true_res) {
    double rr;
    if (!res_true_residual<T, K>(tm, it, a, sm, x, rr)) { aborted = true; goto done; }
    relres_true = sqrt(rr / bb);
  }
done:
  if (store) {
#pragma unroll
    for (int k = 0; k < K; ++k)
      if (it.has(k)) res_store<T, K>(it, k, static_cast<T*>(a.x), a.ld, x[k]);
  }
  res_info(a, tm, status, aborted, iters, 0, gamma, bb, relres_true);
}

// ---------------------------------------------------------------------------
// Mixed precision: the FP64 refinement of ir_kernels.cuh (the same steps, tests
// and guard) around the resident binary32 loop.  The binary64 x and b stay in
// global memory; the correction d is the loop's resident x.
// ---------------------------------------------------------------------------
template <int K>
__device__ __forceinline__ void res_ir(const ResArgs& a, ResTeam& tm, float* sm) {
  constexpr int W = ResVec<float>::W;
  ResItems<float, K> it;
  it.init(a.nx, a.ny, tm.rank, tm.size);
  res_zero_rows<float, K>(it, sm);
  const double* gb = static_cast<const double*>(a.b);
  double* gx = static_cast<double*>(a.x);
  float r[K][W], d[K][W];
  int status = LAP5CG_NOT_CONVERGED, total = 0, outer = 0;
  double bb = 0.0, rr = 0.0, rr_prev = 0.0, relres_true = nan(""), thr = 0.0, dad = 0.0;
  bool aborted = false, have_d = false, reverting = false;
#pragma unroll
  for (int k = 0; k < K; ++k)
#pragma unroll
    for (int q = 0; q < W; ++q) d[k][q] = r[k][q] = 0.f;
  for (;;) {
    double drn = 0.0, g_in;
    if (have_d) {  // x <- x + d (or back), with (d, A d) in binary64
      Acc64 aad;
      if (!reverting) {
        __syncthreads();  // every read of the direction's rows is done
#pragma unroll
        for (int k = 0; k < K; ++k) {
          if (!it.has(k)) break;
          if (it.is(it.valid, k)) res_st(sm, it.off[k], d[k]);
          res_send<float, K>(tm, it, k, d[k], tm.htag);
        }
        res_halos<float, K>(tm, it, tm.htag, threadIdx.x, blockDim.x, [&](int o, const float (&v)[W]) { res_st(sm, o, v); });
        ++tm.htag;
        __syncthreads();
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        double xv[W];
        res_load<float, K>(it, k, gx, a.ld, xv);
        if (!reverting) {
          float up[W], dn[W];
          double c[W], u[W], n[W], ad[W];
          res_ld(sm, it.off[k] - it.ldp, up);
          res_ld(sm, it.off[k] + it.ldp, dn);
#pragma unroll
          for (int q = 0; q < W; ++q) {
            c[q] = (double)d[k][q];
            u[q] = (double)up[q];
            n[q] = (double)dn[q];
          }
          res_stencil<float, K, double>(it, k, sm, c, u, n, ad);
          if (it.is(it.valid, k)) aad.add_block(c, ad);
        }
#pragma unroll
        for (int q = 0; q < W; ++q) xv[q] = reverting ? xv[q] - (double)d[k][q] : xv[q] + (double)d[k][q];
        res_store<float, K>(it, k, gx, a.ld, xv);
      }
      // the neighbours read this CTA's rows of x after this reduction
      const double w[1] = {warp_sum(aad)};
      double o[1];
      if (!tm.reduce<1>(w, o, true)) { aborted = true; goto done; }
      if (!reverting) dad = o[0];
    }
    {  // r = b - A x in binary64, rounded to the inner right-hand side
      Acc64 abb, arr, adr;
      Acc32 agi;
      const bool with_d = have_d && !reverting;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (!it.has(k)) break;
        double b[W], ax[W], rv[W], dv[W];
        res_load<float, K>(it, k, gb, a.ld, b);
        res_global_stencil<float, K>(it, k, gx, a.ld, a.ny, ax);
#pragma unroll
        for (int q = 0; q < W; ++q) {
          rv[q] = b[q] - ax[q];
          dv[q] = (double)d[k][q];
          r[k][q] = __double2float_rn(rv[q]);
        }
        if (outer == 0) abb.add_block(b, b);
        arr.add_block(rv, rv);
        agi.add_block(r[k], r[k]);
        if (with_d) adr.add_block(dv, rv);
        res_send<float, K>(tm, it, k, r[k], tm.htag);
      }
      ++tm.htag;
      const double w[4] = {warp_sum(abb), warp_sum(arr), warp_sum(agi), warp_sum(adr)};
      double o[4];
      if (!tm.reduce<4>(w, o)) { aborted = true; goto done; }
      drn = o[3];
      if (outer == 0) {
        bb = o[0];
        if (!isfinite(bb)) { status = LAP5CG_ERR_NONFINITE; goto done; }
        if (bb == 0.0) {
#pragma unroll
          for (int k = 0; k < K; ++k) {
            const double zero[W] = {0.0, 0.0, 0.0, 0.0};
            if (it.has(k)) res_store<float, K>(it, k, gx, a.ld, zero);
          }
          status = LAP5CG_OK;
          rr = 0.0;
          relres_true = 0.0;
          goto done;
        }
        thr = a.tol > 0.0 ? a.tol * a.tol * bb : 0.0;
      }
      rr = o[1];
      g_in = o[2];
      relres_true = sqrt(rr / bb);
      if (a.history && outer <= a.maxit && tm.rank == 0 && threadIdx.x == 0) a.history[outer] = relres_true;
    }
    if (!isfinite(rr)) { status = LAP5CG_ERR_NONFINITE; goto done; }
    if (reverting) { status = LAP5CG_NOT_CONVERGED; goto done; }
    if (rr <= thr) { status = LAP5CG_OK; goto done; }
    if (outer > 0 && !(rr < rr_prev)) {  // the refinement's energy test (ir_kernels.cuh)
      if (!have_d) { status = LAP5CG_NOT_CONVERGED; goto done; }
      const double dro = drn + dad;
      if (!(dro > 0.0 && drn >= -0.5 * dro)) {
        reverting = true;
        continue;
      }
    }
    rr_prev = rr;
    if (outer >= a.max_outer || total >= a.maxit) { status = LAP5CG_NOT_CONVERGED; goto done; }
    {  // inner classic CG on A d = r from d = 0
      double gamma = g_in;
      const int cap = min(a.maxit, total + min(a.maxit_inner, a.maxit - total)), before = total;
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int q = 0; q < W; ++q) d[k][q] = 0.f;
      const int why = res_classic_loop<float, K>(tm, it, sm, r, d, gamma, a.tol_inner * a.tol_inner * g_in, cap, total,
                                                 nullptr, 1.0);
      if (why == RES_ABORTED) { aborted = true; goto done; }
      if (why == RES_CURVATURE || why == RES_NONFINITE) { status = LAP5CG_ERR_BREAKDOWN; goto done; }
      have_d = total > before;
    }
    ++outer;
  }
done:
  res_info(a, tm, status, aborted, total, outer, rr, bb, relres_true);
}

}  // namespace lap5
