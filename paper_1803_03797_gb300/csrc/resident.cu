// resident.cu -- host launch of the chip-resident solves (resident.cuh).
#include <algorithm>
#include <vector>

#include "resident_kernels.cuh"

namespace lap5 {

static int res_kind(int variant, int precision) {
  if (precision == LAP5CG_PREC_F64) return variant == LAP5CG_NEWCG ? RK_F64_NEWCG : RK_F64_CLASSIC;
  if (precision == LAP5CG_PREC_F32 && variant == LAP5CG_CLASSIC) return RK_F32_CLASSIC;
  if (precision == LAP5CG_PREC_IR_F32 && variant == LAP5CG_CLASSIC) return RK_IR_F32;
  return RK_NONE;
}

// Geometry of a resident solve: CTAs, items a thread, bytes.
struct ResPlan {
  int ctas, rows, k, items;
  long long groups;
  size_t smem, slot_bytes, halo_bytes;
};

static bool res_is_f64(int kind) { return kind == RK_F64_CLASSIC || kind == RK_F64_NEWCG; }

// At least two rows a CTA: the message rows (two sets of two rows a CTA, twice
// the element size) then take no more than the state vectors they replace.
static bool res_plan(int kind, int nx, int ny, int team, int min_rows, ResPlan* p) {
  const int w = res_is_f64(kind) ? 2 : 4, es = res_is_f64(kind) ? 8 : 4;
  p->groups = ((long long)nx + w - 1) / w;
  p->rows = res_rows(ny, std::min(team, kMaxPeers), min_rows);
  const long long items = p->groups * p->rows;
  if (items > (long long)res_most_items(kind) * kResMaxThreads) return false;
  p->items = (int)items;
  p->ctas = (ny + p->rows - 1) / p->rows;
  p->k = (int)((items + kResMaxThreads - 1) / kResMaxThreads);
  p->smem = (size_t)(p->rows + 4) * p->groups * w * es;  // two halo rows, two more staged
  p->slot_bytes = (size_t)2 * p->ctas * kSlotWords * 8;
  p->halo_bytes = (size_t)4 * p->ctas * p->groups * kResItemWords * 8;
  return true;
}

static const void* res_kernel_of(int kind, int k) {
  switch (kind) {
    case RK_F64_CLASSIC: return res_single_f64(k);
    case RK_F64_NEWCG: return res_single_newcg(k);
    case RK_F32_CLASSIC: return res_single_f32(k);
    default: return res_single_ir(k);
  }
}

static const void* res_batch_kernel_of(int kind) {
  switch (kind) {
    case RK_F64_CLASSIC: return res_batch_f64();
    case RK_F64_NEWCG: return res_batch_newcg();
    case RK_F32_CLASSIC: return res_batch_f32();
    default: return res_batch_ir();
  }
}

// Options that shape or select the other kernels keep them.
static bool res_wanted(const lap5cg_opts& o) {
  return o.resident == 0 && o.ring_slots == 0 && o.rr_period == 0 && !o.reproducible && !o.stabilized && o.ctas == 0 &&
         o.warps_per_cta == 0 && o.min_rows == 0 && o.lane_vec == 0 && o.store_z < 0 && o.team_ctas == 0;
}

constexpr size_t kResSlotOffset = 4096;  // the slots' place in the control block's region

int try_resident(const SolvePlan& p, cudaStream_t st, bool* used) {
  *used = false;
  const lap5cg_opts& o = p.opts;
  const int kind = res_kind(p.variant, p.precision);
  if (kind == RK_NONE || !res_wanted(o)) return LAP5CG_OK;
  DevProps dp;
  int rc = dev_props(&dp);
  if (rc != LAP5CG_OK) return rc;
  ResPlan g;
  if (!res_plan(kind, p.nx, p.ny, dp.sms, 2, &g)) return LAP5CG_OK;
  // A wide, flat grid gives rows to few SMs (two rows a CTA at least): past twice the
  // even share of the items the streaming kernels, which also split columns, are
  // faster (3000 x 100 binary64: 14.9 against 23.2 us an iteration; 1024 x 24, with 1024
  // items a CTA, 14.2 against 8.5)
  if (g.items > 1024 && (long long)g.items * dp.sms > 2 * g.groups * p.ny) return LAP5CG_OK;
  const void* fn = res_kernel_of(kind, g.k);
  if (!fn || g.smem + sizeof(ResShared) + 1024 > (size_t)dp.max_smem_optin) return LAP5CG_OK;
  if (kResSlotOffset + g.slot_bytes > kCtlBytes || kCtlBytes + g.halo_bytes > p.ws_bytes) return LAP5CG_OK;
  if (g.smem + sizeof(ResShared) > 48 * 1024 &&  // beyond the size every launch may use
      (rc = allow_dyn_smem(fn, g.smem)) != LAP5CG_OK)
    return rc;
  // tags of an earlier solve in this workspace must not be taken for this one's
  if (cudaMemsetAsync(p.ws, 0, kResSlotOffset + g.slot_bytes, st) != cudaSuccess ||
      cudaMemsetAsync(p.ws + kCtlBytes, 0, g.halo_bytes, st) != cudaSuccess)
    return LAP5CG_ERR_CUDA;
  Ctl* ctl = reinterpret_cast<Ctl*>(p.ws);
  ResLaunch l;
  l.a.nx = p.nx;
  l.a.ny = p.ny;
  l.a.ld = p.ld;
  l.a.b = p.b;
  l.a.x = p.x;
  l.a.info = p.info;
  l.a.history = o.history;
  l.a.tol = p.tol;
  l.a.maxit = p.maxit;
  l.a.true_res = o.true_residual;
  l.a.max_outer = o.max_outer > 0 ? o.max_outer : 60;
  l.a.maxit_inner = o.maxit_inner > 0 ? o.maxit_inner : 4 * (p.nx + p.ny) + 50;
  l.a.tol_inner = o.tol_inner > 0.0 ? o.tol_inner : 1e-4;
  l.slots = reinterpret_cast<u64*>(p.ws + kResSlotOffset);
  l.halos = reinterpret_cast<u64*>(p.ws + kCtlBytes);
  l.err = &ctl->status;
  l.abort_flag = &ctl->abort;
  l.timeout_ns = (long long)((o.timeout_s > 0.0 ? o.timeout_s : 2.0) * 1e9);
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(g.ctas);
  // a multiple of four warps: one scheduler's share of the items each
  lc.blockDim = dim3(std::max(kResMinThreads, (g.items + 128 * g.k - 1) / (128 * g.k) * 128));
  lc.dynamicSmemBytes = g.smem;
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // every CTA resident: they wait for one another
  attr[0].val.cooperative = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  void* args[] = {&l};
  if (cudaLaunchKernelExC(&lc, fn, args) != cudaSuccess) return LAP5CG_ERR_CUDA;
  *used = true;
  return LAP5CG_OK;
}

// Time of one iteration of an instance on a team, in us, for choosing the team
// size only: two exchanges (NewCG: one) and the items' work, from single solves
// of 100^2 .. 1024^2.  Binary64 work is FP64 pipe time, a step of it every four
// warps; binary32 work goes with the items a thread.
static double res_us(int kind, const ResPlan& g) {
  const double warps4 = (g.items + 127) / 128;
  switch (kind) {
    case RK_F64_CLASSIC: return 3.6 + 0.65 * warps4;
    case RK_F64_NEWCG: return 2.6 + 0.8 * warps4;
    default: return 3.8 + 0.45 * g.k;
  }
}

struct ResPick {
  int index;     // in the caller's arrays
  int team_min;  // smallest team it fits on
  double iters;  // relative iteration count
};

// Makespan of the picks on `n` teams of `team` CTAs (longest first).
static double res_makespan(int kind, const std::vector<ResPick>& v, const int* nx, const int* ny, int team, int n,
                           int min_rows) {
  std::vector<double> t;
  ResPlan g;
  for (const ResPick& p : v)
    if (res_plan(kind, nx[p.index], ny[p.index], team, min_rows, &g)) t.push_back(p.iters * res_us(kind, g));
  std::sort(t.rbegin(), t.rend());
  std::vector<double> load(std::max(1, n), 0.0);
  for (double x : t) *std::min_element(load.begin(), load.end()) += x;
  return *std::max_element(load.begin(), load.end());
}

static int res_launch_batch(const void* fn, ResBatchLaunch l, int teams, size_t smem, cudaStream_t st) {
  if (smem + sizeof(ResShared) > 48 * 1024 - 64) {
    const int rc = allow_dyn_smem(fn, smem);
    if (rc != LAP5CG_OK) return rc;
  }
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(teams * l.team);
  lc.blockDim = dim3(kResMaxThreads);
  lc.dynamicSmemBytes = smem;
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  lc.attrs = attr;
  lc.numAttrs = 1;
  void* args[] = {&l};
  return cudaLaunchKernelExC(&lc, fn, args) == cudaSuccess ? LAP5CG_OK : LAP5CG_ERR_CUDA;
}

int resident_batched(int count, const int* nx, const int* ny, const int* ld, const void* const* b, void* const* x,
                     double tol, int maxit, int variant, int precision, unsigned char* ws, size_t ws_bytes,
                     BatchEntry* dtab, size_t first_off, int* errs, lap5cg_info* info, const lap5cg_opts& o,
                     cudaStream_t st, std::vector<char>& taken, size_t* end_off) {
  taken.assign(count, 0);
  *end_off = first_off;
  const int kind = res_kind(variant, precision);
  if (kind == RK_NONE || !res_wanted(o)) return LAP5CG_OK;
  DevProps dp;
  int rc = dev_props(&dp);
  if (rc != LAP5CG_OK) return rc;
  const int sms = std::min(dp.sms, kMaxPeers);
  const int min_rows = 3;  // the message memory then fits in the place of the state vectors
  const size_t smem_cap = (size_t)dp.max_smem_optin - sizeof(ResShared) - 1024;
  std::vector<ResPick> picks;
  for (int i = 0; i < count; ++i) {
    ResPlan g;
    if (!res_plan(kind, nx[i], ny[i], sms, min_rows, &g) || g.smem > smem_cap ||
        g.slot_bytes + g.halo_bytes > batched_instance_bytes(nx[i], ny[i], ld[i], variant, precision))
      continue;
    const long long most_rows = (long long)res_most_items(kind) * kResMaxThreads / g.groups;
    picks.push_back({i, (int)((ny[i] + most_rows - 1) / most_rows), (double)(nx[i] + ny[i])});
  }
  if (picks.empty()) return LAP5CG_OK;
  // Team sizes: the instances that fit on a team of the base size share one
  // launch, larger ones a launch of the next size they fit on; the base with the
  // least total time.
  std::vector<int> sizes;
  for (int n : kTeamSplits) sizes.push_back(team_size(sms, n));
  auto classes = [&](int base) {
    std::vector<std::vector<ResPick>> c(sizes.size());
    for (const ResPick& p : picks) {
      int s = base;
      while (s + 1 < (int)sizes.size() && sizes[s] < p.team_min) ++s;
      c[s].push_back(p);
    }
    return c;
  };
  int best = 0;
  double best_us = 0.0;
  for (int base = 0; base < (int)sizes.size(); ++base) {
    const auto c = classes(base);
    double us = 0.0;
    for (size_t s = 0; s < c.size(); ++s)
      if (!c[s].empty()) us += res_makespan(kind, c[s], nx, ny, sizes[s], team_count(sms, sizes[s]), min_rows);
    if (base == 0 || us < best_us) {
      best = base;
      best_us = us;
    }
  }
  const auto c = classes(best);
  // message memory: the abort flag, per launch a queue head and a word a team, then
  // the instances'; all of it starts at zero
  size_t off = first_off + kAlign;
  std::vector<size_t> launch_off(c.size(), 0);
  for (size_t s = 0; s < c.size(); ++s)
    if (!c[s].empty()) {
      launch_off[s] = off;
      off += kTeamLaunchBytes;
    }
  std::vector<BatchEntry> tab;
  std::vector<int> first(c.size(), 0);
  std::vector<size_t> smem(c.size(), 0);
  std::vector<char> mine(count, 0);
  for (size_t s = 0; s < c.size(); ++s) {
    first[s] = (int)tab.size();
    std::vector<ResPick> v = c[s];
    std::stable_sort(v.begin(), v.end(), [&](const ResPick& p, const ResPick& q) {
      return p.iters * nx[p.index] * ny[p.index] > q.iters * nx[q.index] * ny[q.index];
    });
    for (const ResPick& p : v) {
      ResPlan g;
      if (!res_plan(kind, nx[p.index], ny[p.index], sizes[s], min_rows, &g) || g.smem > smem_cap) continue;
      BatchEntry e;
      e.b = b[p.index];
      e.x = x[p.index];
      e.ws_off = (long long)off;
      e.nx = nx[p.index];
      e.ny = ny[p.index];
      e.ld = ld[p.index];
      e.idx = p.index;
      tab.push_back(e);
      mine[p.index] = 1;
      off += align_up(g.slot_bytes + g.halo_bytes, kAlign);
      smem[s] = std::max(smem[s], g.smem);
    }
  }
  // the others' state vectors need their place too
  size_t rest = 0;
  for (int i = 0; i < count; ++i)
    if (!mine[i]) rest += batched_instance_bytes(nx[i], ny[i], ld[i], variant, precision);
  if (off + rest > ws_bytes) return LAP5CG_OK;
  rc = fill_batch_table(dtab, tab.data(), (int)tab.size(), st);
  if (rc != LAP5CG_OK) return rc;
  if (cudaMemsetAsync(ws + first_off, 0, off - first_off, st) != cudaSuccess) return LAP5CG_ERR_CUDA;
  for (size_t s = 0; s < c.size(); ++s) {
    const int n = (s + 1 < c.size() ? first[s + 1] : (int)tab.size()) - first[s];
    if (n == 0) continue;
    ResBatchLaunch l;
    l.tab = dtab + first[s];
    l.ws = ws;
    l.next = reinterpret_cast<unsigned*>(ws + launch_off[s]);
    l.item = reinterpret_cast<u64*>(ws + launch_off[s] + kTeamWordOffset);
    l.errs = errs;
    l.abort_flag = reinterpret_cast<int*>(ws + first_off);
    l.info = info;
    l.count = n;
    l.team = sizes[s];
    l.min_rows = min_rows;
    l.timeout_ns = (long long)((o.timeout_s > 0.0 ? o.timeout_s : 2.0) * 1e9);
    l.a = ResArgs();
    l.a.history = nullptr;
    l.a.tol = tol;
    l.a.maxit = maxit;
    l.a.true_res = o.true_residual;
    l.a.max_outer = o.max_outer > 0 ? o.max_outer : 60;
    l.a.maxit_inner = o.maxit_inner;
    l.a.tol_inner = o.tol_inner > 0.0 ? o.tol_inner : 1e-4;
    const int teams = std::min(team_count(sms, sizes[s]), n);
    rc = res_launch_batch(res_batch_kernel_of(kind), l, teams, smem[s], st);
    if (rc != LAP5CG_OK) return rc;
  }
  taken = mine;
  *end_off = off;
  return LAP5CG_OK;
}

}  // namespace lap5
