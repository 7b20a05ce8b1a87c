// resident_kernels.cuh -- the kernels of the chip-resident solves (resident.cuh),
// single and batched, instantiated one solve kind a translation unit.
#pragma once

#include "batch_teams.h"
#include "launch.h"
#include "resident.cuh"

namespace lap5 {

enum { RK_F64_CLASSIC = 0, RK_F64_NEWCG, RK_F32_CLASSIC, RK_IR_F32, RK_NONE };

template <int KIND> struct ResKind { using T = double; };
template <> struct ResKind<RK_F32_CLASSIC> { using T = float; };
template <> struct ResKind<RK_IR_F32> { using T = float; };

struct ResLaunch {
  ResArgs a;
  u64 *slots, *halos;
  int *err, *abort_flag;
  long long timeout_ns;
};

template <int KIND, int K>
__device__ __forceinline__ void res_body(const ResArgs& a, ResTeam& tm, typename ResKind<KIND>::T* sm) {
  if constexpr (KIND == RK_F64_NEWCG) res_newcg<double, K>(a, tm, sm);
  else if constexpr (KIND == RK_IR_F32) res_ir<K>(a, tm, sm);
  else res_classic<typename ResKind<KIND>::T, K>(a, tm, sm);
}

template <int KIND, int K>
__global__ void __launch_bounds__(kResMaxThreads, 1) k_resident(const ResLaunch l) {
  using T = typename ResKind<KIND>::T;
  __shared__ ResShared sh;
  extern __shared__ __align__(16) unsigned char dsm[];
  if (threadIdx.x == 0) sh.fail = 0;  // published by the solve's first CTA barrier
  ResTeam tm;
  constexpr int W = ResVec<T>::W;
  tm.init(l.slots, l.halos, (int)blockIdx.x, (int)gridDim.x, (l.a.nx + W - 1) / W, l.err, l.abort_flag, l.timeout_ns,
          &sh);
  res_body<KIND, K>(l.a, tm, reinterpret_cast<T*>(dsm));
}

// The most items a thread whose state fits 128 registers (classic: r, z, x of
// each; NewCG: five vectors, n and w).
static constexpr int res_most_items(int kind) { return kind == RK_F64_NEWCG ? 3 : 7; }

template <int KIND, int K = 1>
static const void* res_kernel(int k) {
  if (k == K) return reinterpret_cast<const void*>(&k_resident<KIND, K>);
  if constexpr (K < res_most_items(KIND)) return res_kernel<KIND, K + 1>(k);
  else return nullptr;
}

// CTAs of a grid on a team of `team`: at least min_rows rows each.
__host__ __device__ inline int res_rows(int ny, int team, int min_rows) {
  const int rows = (ny + team - 1) / team;
  return rows > min_rows ? rows : (min_rows < ny ? min_rows : ny);
}

// ---------------------------------------------------------------------------
// Batched: teams of equal size over the chip take instances from a queue,
// largest first.  An instance smaller than its team leaves the last CTAs idle.
// ---------------------------------------------------------------------------
struct ResBatchLaunch {
  const BatchEntry* tab;  // ws_off: the instance's message memory
  unsigned char* ws;
  unsigned* next;         // queue head (zero)
  u64* item;              // one message word a team, 256 bytes apart (zero)
  int *errs, *abort_flag;
  lap5cg_info* info;
  int count, team, min_rows;
  long long timeout_ns;
  ResArgs a;              // what all instances share
};

template <int KIND, int K = 1>
__device__ __forceinline__ void res_body_of(int k, const ResArgs& a, ResTeam& tm, typename ResKind<KIND>::T* sm) {
  if (k == K) res_body<KIND, K>(a, tm, sm);
  else if constexpr (K < res_most_items(KIND)) res_body_of<KIND, K + 1>(k, a, tm, sm);
}

template <int KIND>
__global__ void __launch_bounds__(kResMaxThreads, 1) k_resident_batch(const ResBatchLaunch l) {
  using T = typename ResKind<KIND>::T;
  constexpr int W = ResVec<T>::W;
  __shared__ ResShared sh;
  __shared__ int s_item;
  extern __shared__ __align__(16) unsigned char dsm[];
  const int team = (int)blockIdx.x / l.team, rank = (int)blockIdx.x - team * l.team;
  u64* word = l.item + (size_t)team * kTeamWordStride;
  uint32_t seq = 0;
  for (;;) {
    // The team's first CTA draws an item and passes it on.  A CTA that an
    // instance did not need may find a later one here; it cannot miss one that
    // needs it, since the first CTA cannot end that one alone.
    if (threadIdx.x == 0) {
      int item;
      if (rank == 0) {
        item = (int)atomicAdd(l.next, 1u);
        asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(word), "l"(ll_word((uint32_t)item, ++seq)) : "memory");
      } else {
        // as long as the instance before takes; ends with the launch's abort
        // flag, and after an hour in any case
        const u64 t0 = global_ns();
        for (;;) {
          u64 w;
          asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(word) : "memory");
          item = (int)(uint32_t)w;
          if ((uint32_t)(w >> 32) != seq) {
            seq = (uint32_t)(w >> 32);
            break;
          }
          if (ld_relaxed_i32(l.abort_flag) || global_ns() - t0 > 3600000000000ull) {
            item = l.count;
            break;
          }
          __nanosleep(200);
        }
      }
      s_item = item;
      sh.fail = 0;
    }
    __syncthreads();
    const int item = s_item;
    if (item >= l.count) return;
    const BatchEntry e = l.tab[item];
    const int rows = res_rows(e.ny, l.team, l.min_rows), ctas = (e.ny + rows - 1) / rows;
    if (rank < ctas) {
      ResArgs a = l.a;
      a.nx = e.nx;
      a.ny = e.ny;
      a.ld = e.ld;
      a.b = e.b;
      a.x = e.x;
      a.info = l.info + e.idx;
      if (a.maxit_inner == 0) a.maxit_inner = 4 * (e.nx + e.ny) + 50;
      const int groups = (e.nx + W - 1) / W;
      u64* mem = reinterpret_cast<u64*>(l.ws + e.ws_off);
      ResTeam tm;
      tm.init(mem, mem + (size_t)2 * ctas * kSlotWords, rank, ctas, groups, l.errs + e.idx, l.abort_flag,
              l.timeout_ns, &sh);
      res_body_of<KIND>((rows * groups + kResMaxThreads - 1) / kResMaxThreads, a, tm, reinterpret_cast<T*>(dsm));
    }
    __syncthreads();  // the shared rows and scalars are the next instance's
  }
}

// The kernel of a kind for k items a thread (nullptr: too many), and its batched form.
#define LAP5_RESIDENT_KERNELS(NAME, KIND)                                                       \
  const void* res_single_##NAME(int k) { return res_kernel<KIND>(k); }                          \
  const void* res_batch_##NAME() { return reinterpret_cast<const void*>(&k_resident_batch<KIND>); }
const void* res_single_f64(int k);
const void* res_single_newcg(int k);
const void* res_single_f32(int k);
const void* res_single_ir(int k);
const void* res_batch_f64();
const void* res_batch_newcg();
const void* res_batch_f32();
const void* res_batch_ir();

}  // namespace lap5
