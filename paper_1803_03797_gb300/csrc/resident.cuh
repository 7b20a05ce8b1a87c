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
// latency of the reductions (classic: two an iteration, NewCG: one; exchange.cuh)
// plus the FP64 pipe (2 operations an SM a clock) in binary64.
//
// Arithmetic per point is that of the streaming kernels (Algorithm 1 with
// z = A p stored and the x update deferred to the next direction update;
// Algorithm 2).  The sums of dot products differ in order, and binary64 stencils in
// rounding: fixed point (fixstencil.cuh) aligned to the largest value of a warp's items,
// which may lie in several rows, where the row-ring kernels align a strip's rows
// and the register marches add in FP64.
#pragma once

#include "cg_kernels.cuh"
#include "fixstencil.cuh"

namespace lap5 {

constexpr int kResMinThreads = 256, kResMaxThreads = 512;
constexpr int kResMaxVals = 4;      // values of one reduction
constexpr int kResItemWords = 4;    // 64-bit words of one lane vector in a halo message

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
  double gp[kResMaxVals * kPollWarps];  // sums of 32 CTAs
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
    return slots + ((size_t)(tag & 1u) * size + cta) * kSlotWords;
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
  // Wait for every CTA's contribution.  The CTA's last kPollWarps warps poll,
  // one slot a lane (152 slots: 1.1 us an exchange, against 1.6 us with five
  // slots a lane of one warp).  The last warp forms the totals (the same bits in
  // every CTA), hands them to post(totals), which returns how to go on and may
  // set the scalars in *sh (lane 0's stores count), and leaves them in sh->tot.
  // Returns post's code in every thread, or RES_ABORTED when the solve must stop:
  // a wait ran out here, or in a CTA that then stopped contributing.
  template <int NV, class Post>
  __device__ __forceinline__ int gather(Post post, bool fence = false) {
    const int lane = threadIdx.x & 31;
    const int pw = ((int)threadIdx.x >> 5) - ((int)(blockDim.x >> 5) - kPollWarps);
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
        for (int k = 0; k < NV; ++k) sh->gp[k * kPollWarps + pw] = v[k];
      }
    }
    __syncthreads();
    if (pw == kPollWarps - 1) {
      double s[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        s[k] = sh->gp[k * kPollWarps];
#pragma unroll
        for (int j = 1; j < kPollWarps; ++j)
          if (32 * j < size) s[k] += sh->gp[k * kPollWarps + j];
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

// y = A c on item k from the shared rows sm (c: the item itself; up / dn: rows above
// / below), binary32 in the order 4C - W - E - S - N, binary64 in fixed point
// (fixstencil.cuh; one FP64 operation a point instead of four).  Whole-warp call.
template <class T, int K, class M>
__device__ __forceinline__ void res_stencil(const ResItems<T, K>& it, int k, const T* sm, const M (&c)[ResVec<T>::W],
                                            const M (&up)[ResVec<T>::W], const M (&dn)[ResVec<T>::W],
                                            M (&y)[ResVec<T>::W]) {
  constexpr int W = ResVec<T>::W;
  const int lane = threadIdx.x & 31, o = it.off[k];
  const bool lh = lane == 0 && !it.is(it.first, k), rh = lane == 31 && !it.is(it.last, k);
  if constexpr (sizeof(T) == 8) {
    double h = 0.0;  // the column beyond the warp's first or last item
    if (lh) h = sm[o - 1];
    if (rh) h = sm[o + W];
    unsigned m = fix_mag(h), n = 0x7fffffffu;
    const unsigned cc = max(fix_mag(c[0]), fix_mag(c[1]));
#pragma unroll
    for (int q = 0; q < W; ++q) {
      const unsigned p = max(cc, max(fix_mag(up[q]), fix_mag(dn[q])));
      m = max(m, p);
      if (it.is(it.valid, k) && !(q > 0 && it.tail < W && it.is(it.last, k))) n = min(n, p);
    }
    const int E = (int)(__reduce_max_sync(0xffffffffu, m) >> 20);
    if (fix_fits<kFixSpan>(n, E)) {
      long long f[W];
#pragma unroll
      for (int q = 0; q < W; ++q) f[q] = fix_of<kFixB>(c[q], E);
      const long long e = fix_of<kFixB>(h, E);
      long long l = __shfl_up_sync(0xffffffffu, f[W - 1], 1), r = __shfl_down_sync(0xffffffffu, f[0], 1);
      if (it.is(it.first, k)) l = 0;
      else if (lane == 0) l = e;
      if (it.is(it.last, k)) r = 0;
      else if (lane == 31) r = e;
#pragma unroll
      for (int q = 0; q < W; ++q)
        y[q] = fix_to<kFixB>(4 * f[q] - (q == 0 ? l : f[q - 1]) - (q == W - 1 ? r : f[q + 1]) -
                                 fix_of<kFixB>(up[q], E) - fix_of<kFixB>(dn[q], E),
                             E);
    } else {
      double l = shfl_up1(c[W - 1]), r = shfl_dn1(c[0]);
      if (it.is(it.first, k)) l = 0.0;
      else if (lane == 0) l = h;
      if (it.is(it.last, k)) r = 0.0;
      else if (lane == 31) r = h;
#pragma unroll
      for (int q = 0; q < W; ++q) {
        double a = __fma_rn(4.0, c[q], -(q == 0 ? l : c[q - 1]));
        a = __dsub_rn(a, q == W - 1 ? r : c[q + 1]);
        y[q] = __dsub_rn(__dsub_rn(a, up[q]), dn[q]);
      }
    }
  } else {
    M l = shfl_up1(c[W - 1]), r = shfl_dn1(c[0]);
    if (it.is(it.first, k)) l = M(0);
    else if (lh) l = (M)sm[o - 1];
    if (it.is(it.last, k)) r = M(0);
    else if (rh) r = (M)sm[o + W];
#pragma unroll
    for (int q = 0; q < W; ++q) {
      M a = M(4) * c[q];
      a -= q == 0 ? l : c[q - 1];
      a -= q == W - 1 ? r : c[q + 1];
      a -= up[q];
      a -= dn[q];
      y[q] = a;
    }
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
    if ((int)threadIdx.x < (int)blockDim.x - 32 * kPollWarps)
      res_halos<T, K>(tm, it, tm.htag - 1u, (int)threadIdx.x, (int)blockDim.x - 32 * kPollWarps,
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
