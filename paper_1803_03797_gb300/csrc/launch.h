// launch.h -- host-side launch interface between the C ABI (api.cu) and the
// kernel translation units.  Internal to liblap5cg.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <vector>

#include "../../include/lap5cg.h"
#include "ring.cuh"

namespace lap5 {

// Launch geometry chosen on the host.
struct LaunchCfg {
  int ctas;           // persistent CTAs (all co-resident)
  int threads;        // threads per CTA
  size_t dyn_smem;    // dynamic shared memory per CTA (row ring)
  int ns, nseg, seg_rows, nunits;  // warp-unit decomposition
};

// One solve on device buffers that already satisfy the vector-path layout:
// every row 16-byte aligned, ld a multiple of the lane vector width.
struct SolvePlan {
  int nx, ny, ld;              // ld of b and x (user or staged)
  int ldw;                     // ld of workspace vectors
  const void* b;
  void* x;
  unsigned char* ws;           // workspace base (control block first)
  size_t ws_bytes;
  lap5cg_info* info;
  double tol;
  int maxit;
  int variant, precision;
  lap5cg_opts opts;
};

int apply_dispatch(int nx, int ny, int ld, int dtype, const void* x, void* y, cudaStream_t st);

// Workspace layout queries (bytes), per precision family.
size_t ws_bytes_f64(int nx, int ny, int ldw, int variant);
size_t ws_bytes_f32(int nx, int ny, int ldw, int variant);
size_t ws_bytes_ir(int nx, int ny, int variant, int precision);
size_t ws_bytes_mg(int nx, int ny, int ldw, int variant, int precision);

// One instance of a batched solve, as the device-side queue's table holds it.
struct BatchEntry {
  const void* b;
  void* x;
  long long ws_off;  // byte offset of this instance's memory in the workspace
  int nx, ny, ld;
  int idx;           // position in the caller's arrays (info slot)
};
int fill_batch_table(BatchEntry* dst, const BatchEntry* src, int n, cudaStream_t st);
// Workspace bytes of one instance's state vectors.
size_t batched_instance_bytes(int nx, int ny, int ld, int variant, int precision);

// Batched solves: the instances whose state fits on a team of SMs are solved by
// the chip-resident kernels; taken[k] is set for them (count entries).  dtab:
// device table of count entries; their memory starts at first_off of the
// workspace and ends at *end_off.
int resident_batched(int count, const int* nx, const int* ny, const int* ld, const void* const* b, void* const* x,
                     double tol, int maxit, int variant, int precision, unsigned char* ws, size_t ws_bytes,
                     BatchEntry* dtab, size_t first_off, int* errs, lap5cg_info* info, const lap5cg_opts& o,
                     cudaStream_t st, std::vector<char>& taken, size_t* end_off);

size_t batched_ws(int count, const int* nx, const int* ny, const int* ld, int variant, int precision);
int solve_batched(int count, const int* nx, const int* ny, const int* ld, const void* const* b, void* const* x,
                  double tol, int maxit, int variant, int precision, void* workspace, size_t ws_bytes,
                  lap5cg_info* info, const lap5cg_opts& o, cudaStream_t st);

// Chip-resident solve (F64, F32 classic, IR_F32): *used = false when the state
// does not fit on the chip or the options ask for other kernels.
int try_resident(const SolvePlan& p, cudaStream_t st, bool* used);

// Cluster-resident solve of a small grid (F64 / F32): *used = false when the
// grid does not fit or the options ask for the streaming kernels.
int try_small(const SolvePlan& p, cudaStream_t st, bool* used);

// Batched solves: the instances that fit in one cluster's shared memory are
// solved by the cluster-resident kernel (one cluster an instance); taken[k]
// is set for them (count entries).
int small_batched(int count, const int* nx, const int* ny, const int* ld, const void* const* b, void* const* x,
                  double tol, int maxit, int variant, int precision, lap5cg_info* info, const lap5cg_opts& o,
                  cudaStream_t st, std::vector<char>& taken);

int solve_f64(const SolvePlan& p, cudaStream_t st);
int solve_f32(const SolvePlan& p, cudaStream_t st);
int solve_ir(const SolvePlan& p, cudaStream_t st);
int solve_mg(const SolvePlan& p, cudaStream_t st);

// Device properties cached per device.
struct DevProps {
  int sms;
  int max_smem_optin;
};
int dev_props(DevProps* out);

// Lets launches of fn use `bytes` of dynamic shared memory.  The limit belongs to the
// function, not to a launch, so every call sets the same value (all that fn's static
// shared memory leaves): a size of its own would lower the limit under a launch of
// another thread, or under graph nodes recorded with more.
int allow_dyn_smem(const void* fn, size_t bytes);

// Grid sizing shared by the persistent kernels: fills cfg from the occupancy
// of kernel func at the requested warps per CTA.
int plan_units(const void* func, int nx, int ny, int V, const lap5cg_opts& o, size_t dyn_smem, LaunchCfg* cfg,
               int row_align = 1);

// Row-ring geometry for a kernel whose largest ring slot is slot_bytes: sets
// the kernel's dynamic shared memory limit and returns the bytes per CTA
// (S = 0 and 0 bytes when the ring is off or does not fit).  auto_on: whether
// ring_slots = 0 (automatic) turns the ring on for this kernel family.
// wpc: the warps per CTA the kernel will be launched with (every warp gets a
// ring of its own in the dynamic shared memory).
int choose_ring(const void* func, int slot_bytes, const lap5cg_opts& o, int wpc, RingGeom* g, size_t* dyn_smem,
                bool auto_on);

// Warps per CTA of the single-grid kernels for these options.
int warps_of(const lap5cg_opts& o);
// The options with warps_per_cta filled in for a kernel of V columns a lane with ring
// slots of slot_bytes: the default; fewer where an explicit ring_slots would not fit,
// and on grids with fewer units than the SMs hold warps, which are then spread over the
// SMs (kPollWarps at least: the reductions' messages need them).  Us an iteration with 16
// warps, on 2 to 50 SMs, and so: NewCG with residual replacement 64^2 15.1 and 9.9, 300^2
// 15.7 and 10.9; classic 64^2 12.8 and 9.8; the spare FP64 pipes are what it gains.
lap5cg_opts with_warps(const lap5cg_opts& o, int slot_bytes, int nx, int ny, int V);

// Largest ring slot (bytes) of each kernel family, V = lane vector width.
inline int ring_slot_classic(int V, int es) {
  const int M = 32 * V * es;
  const int p = 2 * (M + 32) + M, rz = 2 * M, rr = (M + 32) + 2 * M;  // phase P carries x for the deferred update
  return p > rz ? (p > rr ? p : rr) : (rz > rr ? rz : rr);
}
inline int ring_slot_newcg(int V, int es) { return (32 * V * es + 32) + 5 * 32 * V * es; }
inline int ring_slot_ir(int V, int es_r) {
  const int Mr = 32 * V * es_r, Mf = 32 * V * 4;
  const int p = 2 * (Mr + 32), r = (Mr + 32) + Mf + Mr;
  return p > r ? p : r;
}

// Launch defaults (measured on GB300; the autotuner can override them).
constexpr int kDefaultWarps = 16;         // warps per CTA: one CTA an SM, the reductions' peers
// The same in the reproducible mode, whose warps add blocks to accumulators that their CTA
// shares (us an iteration with 4 and 16 warps: classic 100^2 41 and 56, 500^2 41 and
// 67, 1500^2 68 and 68; NewCG 100^2 48 and 66, 500^2 48 and 79, 4096^2 449 and 449).
constexpr int kExactWarps = 4;
constexpr int kDefaultMinRows = 2;        // shortest warp unit (rows) on small grids
constexpr int kRingBytesPerWarp = 12800;  // 16 warps per SM fit 228 KB of shared memory
constexpr int kRingMinRows = 8;           // automatic ring only for units at least this tall

// Wide lanes (eight binary32 columns, four binary64) are only built with the
// ring; half as many columns mean twice the row steps a point.  Chosen by the
// library (not by lane_vec) they are worth it from units of five rows on, where
// the narrow choice has eight and a ring too (us an iteration, narrow -> wide:
// binary32 classic 2048^2, 7 rows, 32.6 -> 26.3; 1600^2, 5 rows, 25.0 -> 21.3;
// IR_F32 1600^2 26.8 -> 21.7; binary64 classic 1300^2, 6 rows, 38.4 -> 33.0; 1100^2,
// 5 rows, 31.7 -> 29.7).  At four rows the narrow register march can be the faster
// (IR_F32 1300^2 17.5 against 19.3).
constexpr int kRingMinRowsWide = 5;
inline int ring_min_rows(bool wide, const lap5cg_opts& o) {
  return wide && o.lane_vec == 0 ? kRingMinRowsWide : kRingMinRows;
}

constexpr size_t kCtlBytes = 256 * 1024;  // control block region at the workspace start
constexpr size_t kAlign = 256;
__host__ __device__ inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace lap5
