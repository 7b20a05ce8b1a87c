// mg_mid.cuh -- the middle and small levels of the V-cycle (nu = 2) as one kernel
// of at most one CTA an SM, their right-hand sides and iterates resident in
// shared memory.
//
// What it replaces and why: as kernels of their own the levels below the first
// take four to six dependent launches each (5 us a launch and the gap before it,
// whatever the size), 190 of the 270 us of an iteration at 2048^2.  Here a level
// costs two exchanges between neighbouring CTAs (one flag each way, 2 us) and five
// passes over shared memory: 1023^2 and below 65 us (binary32), an iteration at
// 512^2 107 -> 71 us, at 2048^2 275 -> 227 us.
//
// Every level is split into blocks of rows, R_l rows a CTA.  A CTA loads b of its
// rows and three halo rows on each side, and then needs nothing from its
// neighbours until the coarse correction arrives: the sweeps before and after
// are formed on the halo rows too (two rows, one row), instead of being
// exchanged.  Down: u = c b + c (b - A c b) on two halo rows, the residual on one,
// restriction of the coarse rows whose centre row (2J + 1) the CTA owns into the
// coarse level's b in global memory, then the CTA's flag.  Up: the owners' coarse
// rows from global memory, u += P e on two halo rows, one sweep on one, the last
// on the own rows, stored for the finer level, then the flag.  The last CTA owns
// no rows; it runs the levels below the distributed ones on its own.
//
// Flags count V-cycles (zeroed at the start of a solve, so no value repeats);
// every wait is bounded (opts.timeout_s), after which the solve ends with
// LAP5CG_ERR_SYNC_TIMEOUT.  The launch is cooperative: the CTAs wait for one another.
#pragma once

#include "fixstencil.cuh"
#include "mg_kernels.cuh"

namespace lap5 {

constexpr int kMidThreads = 512;
constexpr int kMidMaxCtas = 160;
constexpr int kMidMaxLevels = 12;                 // distributed levels
constexpr int kMidStages = 2 * kMidMaxLevels + 2; // flag rows: down, small, up
constexpr size_t kMidFlagOffset = 160 * 1024;     // flags in the workspace's control block
constexpr size_t kMidFlagBytes = (size_t)(kMidStages * kMidMaxCtas + 1) * sizeof(int);  // and the abort flag
// Levels of at most this many points run on the last CTA alone: below, a level's
// passes between CTA barriers cost less than two exchanges (binary64: FP64 pipe time
// of one SM, 4 us per 400 points and V-cycle).
template <class TM> constexpr int kMidSmallPoints = sizeof(TM) == 4 ? 1100 : 400;

template <class TM>
struct MidLevel {
  MgLevel<TM> g;
  int R, G;        // rows a CTA, CTAs with rows
  int ldp;         // shared row pitch: the columns in vectors, four zeros before and after
  int offB, offU;  // element offsets of the level's shared rows
};

template <class TM>
struct MidArgs {
  MidLevel<TM> lv[kMidMaxLevels];
  int n;           // distributed levels (the finest is lv[0])
  int offT, offE;  // sweep rows; coarse correction of the last distributed level
  int* flags;      // [kMidStages][kMidMaxCtas]
  int* abort_flag;
};

template <class TM>
__host__ __device__ inline int mid_pitch(int nx) { return (nx + 3) / 4 * 4 + 8; }

// Shared rows of the levels: b on R + 6 rows, u on R + 4; sweep rows R + 4 of the
// widest level; and the coarse correction of the last level.
template <class TM>
inline size_t mid_layout(MidArgs<TM>* a, const MgLevel<TM>& below) {
  int off = 0, t = 0;
  for (int m = 0; m < a->n; ++m) {
    MidLevel<TM>& L = a->lv[m];
    L.ldp = mid_pitch<TM>(L.g.nx);
    L.offB = off;
    off += (L.R + 6) * L.ldp;
    L.offU = off;
    off += (L.R + 4) * L.ldp;
    t = t > (L.R + 4) * L.ldp ? t : (L.R + 4) * L.ldp;
  }
  a->offT = off;
  off += t;
  a->offE = off;
  off += ((a->lv[a->n - 1].R + 4) / 2 + 4) * mid_pitch<TM>(below.nx);
  return (size_t)off * sizeof(TM);
}

template <class TM> struct MidVec { static constexpr int W = 16 / (int)sizeof(TM); };

__device__ __forceinline__ float mid_ldcg(const float* p) { return __ldcg(p); }
__device__ __forceinline__ double mid_ldcg(const double* p) { return __ldcg(p); }
__device__ __forceinline__ void mid_ldcg(const float* p, float (&v)[4]) {
  const float4 t = __ldcg(reinterpret_cast<const float4*>(p));
  v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
}
__device__ __forceinline__ void mid_ldcg(const double* p, double (&v)[2]) {
  const double2 t = __ldcg(reinterpret_cast<const double2*>(p));
  v[0] = t.x; v[1] = t.y;
}

// f(row, group, live) for every lane vector of `rows` rows of `groups` vectors: a
// warp takes 32 consecutive vectors of one row; all its lanes call, those past the
// row's end with the last vector and live = false.
template <class F>
__device__ __forceinline__ void mid_items(int rows, int groups, F f) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int seg = (groups + 31) / 32;
  for (int q = warp; q < rows * seg; q += nw) {
    const int i = q / seg, g = (q - i * seg) * 32 + lane;
    f(i, min(g, groups - 1), g < groups);
  }
}

// r = b - A c, c the lane vector at p of the operand's shared rows (binary32: the
// order of stencil_row; binary64: in fixed point).  Every lane of the warp calls.
template <class TM>
__device__ __forceinline__ void mid_residual(const TM* p, int ldp, const TM (&b)[MidVec<TM>::W],
                                             TM (&c)[MidVec<TM>::W], TM (&r)[MidVec<TM>::W]) {
  constexpr int W = MidVec<TM>::W;
  TM s[W], n[W];
  VecIO<W, TM>::load(p, c);
  VecIO<W, TM>::load(p - ldp, s);
  VecIO<W, TM>::load(p + ldp, n);
  const TM w = p[-1], e = p[W];
  if constexpr (sizeof(TM) == 8) {
    fix_residual<W>(c, s, n, w, e, b, r);
  } else {
#pragma unroll
    for (int k = 0; k < W; ++k) {
      TM a = TM(4) * c[k];
      a -= k == 0 ? w : c[k - 1];
      a -= k == W - 1 ? e : c[k + 1];
      a -= s[k];
      a -= n[k];
      r[k] = b[k] - a;
    }
  }
}

template <class TM>
__device__ __forceinline__ void mid_store(TM* p, int x, int nx, bool live, TM (&v)[MidVec<TM>::W]) {
  constexpr int W = MidVec<TM>::W;
  if (!live) return;
#pragma unroll
  for (int k = 1; k < W; ++k)
    if (x + k >= nx) v[k] = TM(0);
  VecIO<W, TM>::store(p, v);
}

// Waits for flags [c0, c1] of a stage to reach tag.  False (in every thread) when
// the solve must stop.
__device__ __forceinline__ bool mid_wait(const int* flags, int c0, int c1, int tag, int* abort_flag,
                                         long long timeout_ns) {
  bool fail = false;
  for (int c = c0 + (int)threadIdx.x; c <= c1 && !fail; c += blockDim.x) {
    unsigned spins = 0;
    unsigned long long t0 = 0;
    while (ld_relaxed_i32(flags + c) != tag) {
      const unsigned long long now = global_ns();
      if (spins++ == 0u) t0 = now;
      if (((spins & 31u) == 0u && ld_relaxed_i32(abort_flag)) || (long long)(now - t0) > timeout_ns) {
        atomicExch(abort_flag, 1);
        fail = true;
        break;
      }
    }
  }
  if (c0 + (int)threadIdx.x <= c1) __threadfence();
  return !__syncthreads_or(fail);
}
__device__ __forceinline__ void mid_signal(int* flag, int tag) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(flag), "r"(tag) : "memory");
  }
}

// The columns before and after the vectors of a level's rows, zero for good (the next
// CTA barrier publishes them).
template <class TM>
__device__ __forceinline__ void mid_zero_pads(const MidLevel<TM>& L, TM* sm) {
  constexpr int W = MidVec<TM>::W;
  const int used = (L.g.nx + W - 1) / W * W, rows = 2 * L.R + 10, pads = L.ldp - used;  // b and u rows are adjacent
  for (int i = threadIdx.x; i < rows * pads; i += blockDim.x) {
    const int r = i / pads, k = i - r * pads;
    sm[L.offB + r * L.ldp + (k < 4 ? k : used + k)] = TM(0);
  }
}

// Down one level: loads b, forms u (kept), restricts the residual.
template <class TM>
__device__ __forceinline__ void mid_down(const MidLevel<TM>& L, const MgLevel<TM>& C, TM* sm, int offT, int cta) {
  constexpr int W = MidVec<TM>::W;
  const int s = cta * L.R, e = min(L.g.ny, s + L.R), n = e - s;
  const int nx = L.g.nx, ny = L.g.ny, ldp = L.ldp, groups = (nx + W - 1) / W;
  TM *B = sm + L.offB + 4, *U = sm + L.offU + 4, *T = sm + offT + 4;
  const TM c = (TM)kMgC;
  mid_items(n + 6, groups, [&](int i, int g, bool live) {
    const int j = s - 3 + i;
    TM v[W];
#pragma unroll
    for (int k = 0; k < W; ++k) v[k] = TM(0);
    if (j >= 0 && j < ny) mid_ldcg(L.g.b + (size_t)j * L.g.ld + g * W, v);
    mid_store(B + i * ldp + g * W, g * W, nx, live, v);
  });
  __syncthreads();
  mid_items(n + 4, groups, [&](int i, int g, bool live) {  // the second sweep from zero: u = c b + c (b - A c b)
    const int j = s - 2 + i;
    TM u[W];
    if (j < 0 || j >= ny) {
#pragma unroll
      for (int k = 0; k < W; ++k) u[k] = TM(0);
    } else {
      TM b[W], d[W], zero[W];  // d = -A b
#pragma unroll
      for (int k = 0; k < W; ++k) zero[k] = TM(0);
      mid_residual(B + (i + 1) * ldp + g * W, ldp, zero, b, d);
#pragma unroll
      for (int k = 0; k < W; ++k)
        u[k] = sizeof(TM) == 8 ? mg_fma(c * c, d[k], (c + c) * b[k]) : mg_fma(c, mg_fma(c, d[k], b[k]), c * b[k]);
    }
    mid_store(U + i * ldp + g * W, g * W, nx, live, u);
  });
  __syncthreads();
  mid_items(n + 2, groups, [&](int i, int g, bool live) {  // the residual
    const int j = s - 1 + i;
    TM r[W];
    if (j < 0 || j >= ny) {
#pragma unroll
      for (int k = 0; k < W; ++k) r[k] = TM(0);
    } else {
      TM u[W], b[W];
      VecIO<W, TM>::load(B + (i + 2) * ldp + g * W, b);
      mid_residual(U + (i + 1) * ldp + g * W, ldp, b, u, r);
    }
    mid_store(T + i * ldp + g * W, g * W, nx, live, r);
  });
  __syncthreads();
  const int J0 = s >> 1, J1 = min(e >> 1, C.ny);  // centre rows 2J + 1 in [s, e)
  mid_items(J1 - J0, C.nx, [&](int i, int I, bool live) {
    if (!live) return;
    const TM* lo = T + (2 * (J0 + i) - (s - 1)) * ldp + 2 * I;
    const TM *mid = lo + ldp, *hi = mid + ldp;
    const TM s1 = ((mid[0] + mid[2]) + lo[1]) + hi[1];
    const TM s2 = ((lo[0] + lo[2]) + hi[0]) + hi[2];
    C.b[(size_t)(J0 + i) * C.ld + I] = TM(0.25) * ((TM(4) * mid[1] + TM(2) * s1) + s2);
  });
}

// Up one level: u += P e, two sweeps, the result to out (global).  eg: the coarse
// iterate; E: shared rows for it.
template <class TM>
__device__ __forceinline__ void mid_up(const MidLevel<TM>& L, const MgLevel<TM>& C, const TM* eg, TM* E, TM* sm,
                                       int offT, TM* out, int cta) {
  constexpr int W = MidVec<TM>::W;
  const int s = cta * L.R, e = min(L.g.ny, s + L.R), n = e - s;
  const int nx = L.g.nx, ny = L.g.ny, ldp = L.ldp, groups = (nx + W - 1) / W;
  TM *B = sm + L.offB + 4, *U = sm + L.offU + 4, *T = sm + offT + 4;
  const int ldc = mid_pitch<TM>(C.nx), Jl = ((s - 2) >> 1) - 1, Jh = (e + 1) >> 1;
  E += 4;
  const TM c = (TM)kMgC;
  mid_items(Jh - Jl + 1, (C.nx + W - 1) / W, [&](int i, int g, bool live) {
    const int J = Jl + i;
    TM v[W];
#pragma unroll
    for (int k = 0; k < W; ++k) v[k] = TM(0);
    if (J >= 0 && J < C.ny) mid_ldcg(eg + (size_t)J * C.ld + g * W, v);
    mid_store(E + i * ldc + g * W, g * W, C.nx, live, v);
  });
  // the columns past the last vector (E lies where wider rows were)
  for (int i = threadIdx.x; i <= Jh - Jl; i += blockDim.x) {
    E[i * ldc - 1] = TM(0);
    E[i * ldc + (C.nx + W - 1) / W * W] = TM(0);
  }
  __syncthreads();
  mid_items(n + 4, groups, [&](int i, int g, bool live) {
    const int j = s - 2 + i;
    if (j < 0 || j >= ny) return;
    const int I = g * W / 2;  // the vector's first column, even: between coarse I - 1 and I
    TM u[W];
    TM* p = U + i * ldp + g * W;
    VecIO<W, TM>::load(p, u);
    const TM* a = E + ((j >> 1) - Jl) * ldc + I;  // odd row: coarse row (j - 1) / 2; even row: j / 2 and the one before
    TM v[W];
    if (j & 1) {
#pragma unroll
      for (int k = 0; k < W; k += 2) {
        v[k] = TM(0.5) * (a[k / 2 - 1] + a[k / 2]);
        v[k + 1] = a[k / 2];
      }
    } else {
      const TM* b = a - ldc;
#pragma unroll
      for (int k = 0; k < W; k += 2) {
        v[k] = TM(0.25) * ((b[k / 2 - 1] + b[k / 2]) + (a[k / 2 - 1] + a[k / 2]));
        v[k + 1] = TM(0.5) * (b[k / 2] + a[k / 2]);
      }
    }
#pragma unroll
    for (int k = 0; k < W; ++k) u[k] += v[k];
    mid_store(p, g * W, nx, live, u);
  });
  __syncthreads();
  mid_items(n + 2, groups, [&](int i, int g, bool live) {
    const int j = s - 1 + i;
    TM t[W];
    if (j < 0 || j >= ny) {
#pragma unroll
      for (int k = 0; k < W; ++k) t[k] = TM(0);
    } else {
      TM d[W], b[W];
      VecIO<W, TM>::load(B + (i + 2) * ldp + g * W, b);
      mid_residual(U + (i + 1) * ldp + g * W, ldp, b, t, d);
#pragma unroll
      for (int k = 0; k < W; ++k) t[k] = mg_fma(c, d[k], t[k]);
    }
    mid_store(T + i * ldp + g * W, g * W, nx, live, t);
  });
  for (int i = threadIdx.x; i < n + 2; i += blockDim.x) {  // (other levels' rows lay here)
    T[i * ldp - 1] = TM(0);
    T[i * ldp + groups * W] = TM(0);
  }
  __syncthreads();
  mid_items(n, groups, [&](int i, int g, bool live) {
    TM t[W], d[W], b[W];
    VecIO<W, TM>::load(B + (i + 3) * ldp + g * W, b);
    mid_residual(T + (i + 1) * ldp + g * W, ldp, b, t, d);
#pragma unroll
    for (int k = 0; k < W; ++k) t[k] = mg_fma(c, d[k], t[k]);
    if (live) store_group<W, TM, TM>(out + (size_t)(s + i) * L.g.ld + g * W, g * W, nx, t);
  });
}

// ---------------------------------------------------------------------------
// The levels below the distributed ones, on one CTA.  Rows have a border of zeros
// all around, so no pass looks at the grid's edges; a thread's points of a level
// are found once a pass group, not by a division a pass.  (The generic point-wise
// passes of mg_kernels.cuh took 15 us for 31^2 and below, 0.4 us a pass.)
// ---------------------------------------------------------------------------
constexpr int kTinyMost = 3;  // points a thread of a level: 3 x 512 >= kMidSmallPoints

struct TinyPts {
  int off[kTinyMost];  // offsets in the bordered array; n of them
  int i[kTinyMost], j[kTinyMost];
  int n, pitch;
  __device__ __forceinline__ void init(int nx, int ny) {
    pitch = nx + 2;
    n = 0;
#pragma unroll
    for (int k = 0; k < kTinyMost; ++k) {
      const int p = (int)threadIdx.x + k * (int)blockDim.x;
      if (p < nx * ny) {
        j[k] = p / nx;
        i[k] = p - j[k] * nx;
        off[k] = (j[k] + 1) * pitch + i[k] + 1;
        n = k + 1;
      }
    }
  }
  template <class F>
  __device__ __forceinline__ void each(F f) const {
#pragma unroll
    for (int k = 0; k < kTinyMost; ++k)
      if (k < n) f(off[k], i[k], j[k]);
  }
};

template <class TM>
__device__ __forceinline__ TM tiny_at(const TM* u, int o, int pitch) {  // A u, the order of stencil_row
  TM a = TM(4) * u[o];
  a -= u[o - 1];
  a -= u[o + 1];
  a -= u[o - pitch];
  a -= u[o + pitch];
  return a;
}

// Elements of the bordered b, u and sweep arrays of levels [first, nlev).
template <class TM>
__host__ __device__ inline int tiny_elems(const MgLevel<TM>* lv, int first, int nlev) {
  int s = 0;
  for (int l = first; l < nlev; ++l) s += 3 * (lv[l].nx + 2) * (lv[l].ny + 2);
  return s;
}

// V(2, 2) from level `first` (b in global memory) down to the coarsest and back;
// the result goes to out (level first's pitch).  sm: zero on entry.
template <class TM>
__device__ void tiny_levels(const MgLevel<TM>* lv, int first, int nlev, int nu_c, TM* sm, TM* out) {
  const TM c = (TM)kMgC;
  TinyPts pt;
  pt.init(lv[first].nx, lv[first].ny);
  TM* B = sm;
  pt.each([&](int o, int i, int j) { B[o] = mid_ldcg(lv[first].b + (size_t)j * lv[first].ld + i); });
  __syncthreads();
  int l = first;
  for (; l < nlev - 1; ++l) {
    const int sz = (lv[l].nx + 2) * (lv[l].ny + 2), w = pt.pitch;
    TM *U = B + sz, *T = U + sz, *Bc = T + sz;
    pt.each([&](int o, int, int) { U[o] = mg_fma(c, mg_fma(-c, tiny_at(B, o, w), B[o]), c * B[o]); });
    __syncthreads();
    pt.each([&](int o, int, int) { T[o] = B[o] - tiny_at(U, o, w); });
    __syncthreads();
    pt.init(lv[l + 1].nx, lv[l + 1].ny);
    pt.each([&](int o, int i, int j) {
      const TM* lo = T + (2 * j + 1) * w + 2 * i + 1;
      const TM *mid = lo + w, *hi = mid + w;
      const TM s1 = ((mid[0] + mid[2]) + lo[1]) + hi[1];
      const TM s2 = ((lo[0] + lo[2]) + hi[0]) + hi[2];
      Bc[o] = TM(0.25) * ((TM(4) * mid[1] + TM(2) * s1) + s2);
    });
    __syncthreads();
    B = Bc;
  }
  {  // the coarsest: nu_c sweeps from zero
    const int sz = (lv[l].nx + 2) * (lv[l].ny + 2), w = pt.pitch;
    TM *U = B + sz, *T = U + sz;
    pt.each([&](int o, int, int) { U[o] = c * B[o]; });
    if (lv[l].nx * lv[l].ny > 1) __syncthreads();
    for (int k = 1; k < nu_c; ++k) {
      if (lv[l].nx * lv[l].ny == 1) {  // one point: no neighbour to wait for
        pt.each([&](int o, int, int) { U[o] = mg_fma(c, B[o] - TM(4) * U[o], U[o]); });
        continue;
      }
      pt.each([&](int o, int, int) { T[o] = mg_fma(c, B[o] - tiny_at(U, o, w), U[o]); });
      __syncthreads();
      TM* t = U;
      U = T;
      T = t;
    }
    if (l == first) {  // (also the only level here)
      pt.each([&](int o, int i, int j) { out[(size_t)j * lv[l].ld + i] = U[o]; });
      return;
    }
    if (U != B + sz) pt.each([&](int o, int, int) { B[sz + o] = U[o]; });
    __syncthreads();
  }
  for (--l; l >= first; --l) {
    const int sz = (lv[l].nx + 2) * (lv[l].ny + 2);
    const TM* E = B + (lv[l + 1].nx + 2) * (lv[l + 1].ny + 2);  // the coarse iterate
    const int wc = lv[l + 1].nx + 2;
    B -= 3 * sz;
    TM *U = B + sz, *T = U + sz;
    pt.init(lv[l].nx, lv[l].ny);
    const int w = pt.pitch;
    pt.each([&](int o, int i, int j) {
      // bordered coarse point (I, J) at (J + 1) wc + I + 1; column i = 2I + 1 or between
      const TM* a = E + ((j >> 1) + 1) * wc + (i >> 1) + 1;
      const TM* b = a - wc;
      TM v;
      if (j & 1) v = (i & 1) ? a[0] : TM(0.5) * (a[-1] + a[0]);
      else v = (i & 1) ? TM(0.5) * (b[0] + a[0]) : TM(0.25) * ((b[-1] + b[0]) + (a[-1] + a[0]));
      U[o] += v;
    });
    __syncthreads();
    pt.each([&](int o, int, int) { T[o] = mg_fma(c, B[o] - tiny_at(U, o, w), U[o]); });
    __syncthreads();
    if (l == first) {
      pt.each([&](int o, int i, int j) {
        out[(size_t)j * lv[l].ld + i] = mg_fma(c, B[o] - tiny_at(T, o, w), T[o]);
      });
    } else {
      pt.each([&](int o, int, int) { U[o] = mg_fma(c, B[o] - tiny_at(T, o, w), T[o]); });
      __syncthreads();
    }
  }
}

}  // namespace lap5
