// FUSED engine, host side: launch planning (variants, team size, cost
// model), workspace layout and launches. The kernel is in lr_fused_kernel.cuh;
// its rotating-frame instantiations are compiled in lr_fused_rwa.cu.
#include <mutex>
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>

#include "lr_fused_kernel.cuh"

namespace lr {

// ----------------------------------------------------------------- host side

namespace {

struct SmemLayout {
  int o_zs, o_slot, slot_bytes, s_gp, s_tp, s_pop, o_gd, o_w, o_tred, o_xs, o_misc, o_tab;
  int o_ta, o_tb, npad, o_gs, total;
};

int al16(int x) { return (x + 15) / 16 * 16; }
int al128(int x) { return (x + 127) / 128 * 128; }

// gs: the two bf16 slice buffers of the tensor-core Gram
SmemLayout layout(int R, int Mp, int zs_smem, size_t es, int tc, int gs) {
  SmemLayout L{};
  int o = 0;
  L.o_zs = o;
  if (zs_smem) o += al16((int)(2 * (size_t)R * (Mp + 1) * es));
  L.s_gp = 0;
  L.s_tp = al16(Mp * Mp * (int)sizeof(double2));
  L.s_pop = L.s_tp + al16(2 * Mp * Mp * (int)es);
  L.slot_bytes = L.s_pop + al16((LR_MAX_NT + 2) * (int)sizeof(double));
  L.o_slot = o;
  o += 2 * L.slot_bytes;
  L.o_gd = o;
  o += al16(Mp * (Mp + 1) * (int)sizeof(double2));
  L.o_w = o;
  o += al16(Mp * (Mp + 1) * (int)sizeof(double2));
  L.o_tred = o;
  o += al16(2 * Mp * Mp * (int)es);
  L.o_xs = o;
  o += al16(2 * Mp * Mp * (int)es);
  L.o_misc = o;
  o += al16(168 * (int)sizeof(double));
  L.o_tab = o;
  o += al16(fz::TAB * 7 * (int)(es / 2));
  L.o_ta = L.o_tb = o;
  L.npad = (2 * Mp + 15) / 16 * 16;
  if (tc > 0) {
    const int nbuf = tc == 3 ? 2 : 1;   // big (and small) halves of the TF32 split
    const int K = 4 * Mp;
    o = al128(o);
    L.o_ta = o;
    o += nbuf * fz::TC_ROWS * K * 4;
    L.o_tb = o;
    o += al128(nbuf * L.npad * K * 4);
  }
  L.o_gs = o;
  if (gs) {
    o = al128(o);
    L.o_gs = o;
    o += 2 * GS_BUF;
  }
  L.total = o;
  return L;
}

// tc: tensor-core passes of the projection (0: CUDA cores; 3 or 1: tcgen05,
// L2-resident stage state and FP32 state with the double-word Gram only)
const void* kernel_ptr(lr_precision prec, int zs_smem, int tc, int frame, int gram_mode) {
  if (frame) return fz::rwa_kernel_ptr(prec, zs_smem);
  if (gram_mode == 2) return (const void*)fz::fused_kernel<float2, 2, 0, 0, 0>;
  if (tc == 3) return (const void*)fz::fused_kernel<float2, 1, 0, 3, 0>;
  if (tc == 1) return (const void*)fz::fused_kernel<float2, 1, 0, 1, 0>;
  if (zs_smem) {
    if (prec == LR_PREC_FP64) return (const void*)fz::fused_kernel<double2, 0, 1, 0, 0>;
    if (prec == LR_PREC_FP32) return (const void*)fz::fused_kernel<float2, 0, 1, 0, 0>;
    return (const void*)fz::fused_kernel<float2, 1, 1, 0, 0>;
  }
  if (prec == LR_PREC_FP64) return (const void*)fz::fused_kernel<double2, 0, 0, 0, 0>;
  if (prec == LR_PREC_FP32) return (const void*)fz::fused_kernel<float2, 0, 0, 0, 0>;
  return (const void*)fz::fused_kernel<float2, 1, 0, 0, 0>;
}

// Raise (never lower) a kernel's dynamic shared-memory limit, so that contexts
// planned later cannot shrink it under a context (or a captured graph) that
// needs more.
cudaError_t raise_smem_limit(const void* kern, int bytes) {
  // one lock around the read and the write: two host threads planning at
  // once must not let the smaller request land last
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  cudaFuncAttributes fa{};
  cudaError_t e = cudaFuncGetAttributes(&fa, kern);
  if (e != cudaSuccess) return e;
  if (fa.maxDynamicSharedSizeBytes >= bytes) return cudaSuccess;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

int rows_per_cta(const TrajDev& d, int C) {
  return d.Nt * ((d.Nr + C - 1) / C) * d.Nf;
}

// Trajectories of costs t on n teams, in rows of n: the largest first, and in every row
// the largest to the team with the least so far. Returns the largest team's sum; order
// (unless null) lists them as the kernel takes them, team c = entries c, c + n, ...
double assign_teams(const std::vector<double>& t, int n, std::vector<int>* order) {
  const int T = (int)t.size();
  std::vector<int> by(T), team(n);
  for (int j = 0; j < T; ++j) by[j] = j;
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return t[a] > t[b]; });
  std::vector<double> load(n, 0.0);
  std::vector<std::vector<int>> list(n);
  for (int r = 0; r < T; r += n) {
    for (int c = 0; c < n; ++c) team[c] = c;
    std::stable_sort(team.begin(), team.end(), [&](int a, int b) { return load[a] < load[b]; });
    for (int c = 0; c < std::min(n, T - r); ++c) {
      load[team[c]] += t[by[r + c]];
      list[team[c]].push_back(by[r + c]);
    }
  }
  if (order) {   // the teams with an entry in the last, partial row first
    std::stable_sort(list.begin(), list.end(),
                     [](const std::vector<int>& a, const std::vector<int>& b) { return a.size() > b.size(); });
    order->clear();
    for (size_t r = 0; r < list[0].size(); ++r)
      for (int c = 0; c < n && r < list[c].size(); ++c) order->push_back(list[c][r]);
  }
  return *std::max_element(load.begin(), load.end());
}

// The wide schedule (four launches per RK4 stage, each over the whole chip) against the
// teams: a team holds a trajectory on at most min(16, N_r) SMs, so a batch of one or
// two candidates leaves most of the chip idle. Estimates in us per stage, fitted on
// GB300 to 1 to 16 candidates of 13 models (M = 4 .. 32, N = 40 .. 9600):
//   teams: 2.05 M (1.5 M on one CTA; the M x M phase and the barrier) + rows per CTA x
//          M (M + 11) x 1.7e-4 (stage state in L2: 2.3e-4; two modes, shared memory: 1e-4),
//          the sum over a team's trajectories;
//   wide:  20 + 1.1 M (launches and the M x M phase) + 4.6e-6 x sum N M (M + 11).
// FP64 state, bound by the FP64 pipe (18 M^2 + 47 M FMAs a row at 2.05 per clock and SM):
//   teams: 3 M + rows per CTA x (M^2 + 2.6 M) x 4.5e-3, likewise;
//   wide:  25 + 1.5 M + 4.5e-3 / 152 x sum N (M^2 + 2.6 M).
// Measured, teams / wide: N = 2000, M = 20, 1 candidate 62 / 47, 2 candidates 62 / 61;
// N = 480, M = 32 (two modes) 202 / 62, 8 candidates 203 / 114; N = 8000, M = 32 269 /
// 148; N = 2000, M = 10 32 / 35; N = 40, M = 4 10 / 28. The line lies at 0.9, where no
// measured batch lost more than 1%. Both sides launched from the host; in the device loop
// of a long run the wide schedule takes less (N = 2000, M = 20: 38), and contexts side by side
// on streams of their own too (teams / wide, us a stage of all: 2 contexts 63 / 46, 4
// contexts 63 / 57, 8 contexts 123 / 119).
bool wide_is_faster(const std::vector<TrajDev>& traj, const FusedPlan& plan) {
  double wide = 0.0;
  std::vector<double> team;
  const bool fp64 = plan.es == (int)sizeof(double2);
  for (const TrajDev& d : traj) {
    const double w = fp64 ? d.M * (d.M + 2.6) : d.M * (d.M + 11.0);
    const double slope = fp64 ? 4.5e-3 : (!plan.zs_smem ? 2.3e-4 : (d.n_modes == 2 ? 1.0e-4 : 1.7e-4));
    team.push_back((fp64 ? 3.0 : (plan.C > 1 ? 2.05 : 1.5)) * d.M + slope * w * rows_per_cta(d, plan.C));
    wide = std::max(wide, fp64 ? 25.0 + 1.5 * d.M : 20.0 + 1.1 * d.M);
  }
  for (const TrajDev& d : traj)
    wide += d.N * (fp64 ? 4.5e-3 / SMS * d.M * (d.M + 2.6) : 4.6e-6 * d.M * (d.M + 11.0));
  return wide < 0.9 * assign_teams(team, plan.n_clusters, nullptr);
}

// Wide schedule: two stage buffers and the accumulator, partial sums, a loop counter, from
// `off` (X_k has a place of its own in every context).
struct WideLayout {
  size_t za, zb, acc, part, loop, total;
};
WideLayout wide_layout(const FusedPlan& plan, size_t off) {
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  WideLayout L{};
  L.za = take(plan.es * (size_t)plan.tot);
  L.zb = take(plan.es * (size_t)plan.tot);
  L.acc = take(plan.es * (size_t)plan.tot);
  L.part = take(sizeof(double) * plan.part);
  L.loop = take(3 * sizeof(long long));
  L.total = off;
  return L;
}
size_t order_bytes(int n_traj) { return ((sizeof(int) * n_traj + 255) / 256) * 256; }

}  // namespace

bool fused_plan(const std::vector<TrajDev>& traj, lr_precision prec, int frame, FusedPlan* plan) {
  *plan = FusedPlan{};
  int dev = 0;
  cudaDeviceProp prop{};
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (prop.major < 10) return false;
  const size_t es = prec == LR_PREC_FP64 ? sizeof(double2) : sizeof(float2);
  int Mmax = 0, Nmax = 0, min_nr = 1 << 30;
  bool two = false;
  double max_work = 0.0, tot_work = 0.0;
  for (const TrajDev& d : traj) {
    Mmax = std::max(Mmax, d.M);
    Nmax = std::max(Nmax, d.N);
    if (d.n_modes == 2) two = true;
    min_nr = std::min(min_nr, d.Nr);
    if (d.Nt >= fz::TAB || d.Nr >= fz::TAB || d.Nf >= fz::TAB) return false;
    const double w = (double)d.N * d.M * (d.M + 11.0);
    max_work = std::max(max_work, w);
    tot_work += w;
  }
  const int Mp = (Mmax + 3) / 4 * 4;
  // Variants (stage state placement, tensor-core passes of the projection).
  // Overrides for tuning and tests: LR_FUSED_WIDE = 0 / 1 (teams / wide schedule, the latter
  // also under capture; FP32_G64 and FP64), LR_FUSED_C = cluster size, LR_FUSED_ZS =
  // "global" keeps the stage state in L2, LR_FUSED_TC = 0 keeps the FP32_G64
  // projection on the CUDA cores (3: only the tensor-core variant).
  int force_c = 0, force_global = 0, force_tc = -1, gram_dw = 0;
  if (const char* e = getenv("LR_FUSED_C")) force_c = atoi(e);
  if (const char* e = getenv("LR_FUSED_GRAM")) gram_dw = strcmp(e, "dw") == 0;
  if (const char* e = getenv("LR_FUSED_ZS")) force_global = strcmp(e, "global") == 0;
  if (const char* e = getenv("LR_FUSED_TC")) force_tc = atoi(e);
  struct Variant {
    int zs_smem, tc, gs;
  };
  std::vector<Variant> vars;
  if (prec == LR_PREC_TF32_G64) {
    if (frame) return false;   // the tensor-core variants are built for the lab frame only
    vars.push_back({0, 1, 0});
  } else {
    if (force_tc != 3) {
      if (!force_global) vars.push_back({1, 0, 0});
      // FP32_G64 in the lab frame at Mp = 20: the Gram matrix on the tensor cores
      // (LR_FUSED_GRAM=dw keeps the double-word CUDA-core sums; 2% slower on the
      // N = 2000, M = 20 batch)
      if (prec == LR_PREC_FP32_G64 && !frame && Mp == 20 && !gram_dw)
        vars.push_back({0, 0, 1});
      else
        vars.push_back({0, 0, 0});
    }
    if (prec == LR_PREC_FP32_G64 && force_tc != 0 && !frame) vars.push_back({0, 3, 0});
  }
  double best = 1e300;
  for (const Variant& v : vars) {
    const int zs_smem = v.zs_smem, tc = v.tc, gs = v.gs;
    const int gmode = gs ? 2 : (prec == LR_PREC_FP32_G64 || prec == LR_PREC_TF32_G64 ? 1 : 0);
    const void* kern = kernel_ptr(prec, zs_smem, tc, frame, gmode);
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, kern) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    const int smem_max = (int)prop.sharedMemPerBlockOptin - (int)fa.sharedSizeBytes;
    cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int C = 1; C <= 16; ++C) {
      if (two && C > 1) break;
      if (C > min_nr) break;
      if (force_c > 0 && C != force_c) continue;
      int R = 0;
      for (const TrajDev& d : traj) R = std::max(R, rows_per_cta(d, C));
      if (gs && R > GS_MAXR) continue;   // the slice sums stay exact for <= GS_MAXR rows
      const SmemLayout L = layout(R, Mp, zs_smem, es, tc, gs);
      if (L.total > smem_max) continue;
      if (raise_smem_limit(kern, L.total) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(C * 32);
      cfg.blockDim = dim3(fz::threads_for(tc));
      cfg.dynamicSmemBytes = L.total;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = C;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int ncl = 0;
      if (cudaOccupancyMaxActiveClusters(&ncl, kern, &cfg) != cudaSuccess || ncl <= 0) {
        cudaGetLastError();
        continue;
      }
      // Cost model, fitted to measurements on GB300 (N = 2000, M = 20 batch):
      // a stage costs ~0.16 us per row per CTA with the stage state in shared
      // memory (x1.3 in L2; x1.7 and x1.55 in L2 with the projection on the
      // tensor cores in 3 and 1 passes: per 128-row tile the operand staging
      // and two block barriers cost more than the FMAs they replace), plus a
      // fixed ~60 us per team (the M x M phase and the cluster barrier, ~M
      // sequential elimination steps) that does not shrink with C; teams run
      // trajectories in waves.
      const double row_cost = zs_smem ? 1.0 : (tc == 3 ? 1.7 : tc == 1 ? 1.55 : gs ? 1.0 : 1.3);
      std::vector<double> cost;
      for (const TrajDev& d : traj) {
        const double rows = (double)rows_per_cta(d, C) * row_cost * (d.M * d.M) / 400.0;
        const double fixed = 375.0 * d.M / 20.0 * (C > 1 ? 1.0 : 0.95);
        cost.push_back(rows + fixed);
      }
      // Only as many teams as the waves need (the same number of waves, less scratch), or
      // all that fit where an uneven batch gains by it. 256 trajectories of N = 1000 ..
      // 4000, M = 10 .. 30: their mean cost times the waves chose single CTAs, whose
      // largest pair took 1548 us a stage; the largest team's sum, and the assignment
      // that keeps it small, take 935 us.
      const int n_traj = (int)traj.size();
      const int waves_needed = (n_traj + ncl - 1) / ncl;
      int used = std::min((n_traj + waves_needed - 1) / waves_needed, n_traj);
      const int all = std::min(ncl, n_traj);
      double sum = 0.0, lo = cost[0], hi = cost[0];
      for (double c : cost) {
        sum += c;
        lo = std::min(lo, c);
        hi = std::max(hi, c);
      }
      if (std::max(hi, sum / all) >= best) continue;
      double t = hi == lo ? waves_needed * hi : assign_teams(cost, used, nullptr);
      if (all > used && hi > lo) {
        const double ta = assign_teams(cost, all, nullptr);
        if (ta < 0.99 * t) {
          t = ta;
          used = all;
        }
      }
      if (t < best) {
        best = t;
        assign_teams(cost, used, &plan->order);
        plan->ok = 1;
        plan->C = C;
        plan->n_clusters = used;
        plan->threads = fz::threads_for(tc);
        plan->smem = L.total;
        plan->zs_smem = zs_smem;
        plan->tc = tc;
        plan->frame = frame;
        plan->Mp = Mp;
        plan->R = R;
        plan->Nmax = Nmax;
        plan->gram_mode = gmode;
        plan->es = (int)es;
      }
    }
  }
  if (!plan->ok) return false;
  for (const TrajDev& d : traj) {
    plan->max_nblk = std::max(plan->max_nblk, d.nblk);
    plan->tot += (long long)d.N * d.M;
    plan->part += (long long)d.nblk * (long long)plain_pstride(d.M);
  }
  const bool has_wide = prec == LR_PREC_FP32_G64 || prec == LR_PREC_FP64;
  plan->wide = has_wide && !force_c && !force_global && force_tc < 0 && !gram_dw && wide_is_faster(traj, *plan);
  if (const char* e = getenv("LR_FUSED_WIDE")) plan->wide = has_wide && atoi(e) ? 2 : 0;
  return true;
}

size_t fused_scratch_bytes(const FusedPlan& plan, int n_traj) {
  // order list, then global stage buffers (only without smem residency) and accumulators per team
  size_t b = order_bytes(n_traj);
  const size_t wide = plan.wide ? wide_layout(plan, b).total : 0;   // in the place of the teams' buffers
  const size_t es = plan.es;
  if (!plan.zs_smem)
    b += ((2 * (size_t)plan.R * (plan.Mp + 1) * es * plan.C * plan.n_clusters + 255) / 256) * 256;
  b += (((size_t)plan.Nmax * plan.Mp * es * plan.n_clusters + 255) / 256) * 256;
  return std::max(b, wide);
}

cudaError_t fused_prepare(const FusedPlan& plan, lr_precision prec, void* scratch, int n_traj) {
  cudaError_t e = cudaMemcpy(scratch, plan.order.data(), sizeof(int) * n_traj, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  const size_t es = prec == LR_PREC_FP64 ? sizeof(double2) : sizeof(float2);
  const SmemLayout L = layout(plan.R, plan.Mp, plan.zs_smem, es, plan.tc, plan.gram_mode == 2);
  const void* kern = kernel_ptr(prec, plan.zs_smem, plan.tc, plan.frame, plan.gram_mode);
  e = raise_smem_limit(kern, L.total);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

cudaError_t fused_integrate(const FusedPlan& plan, const DevPtrs& p, const RunParams& rp, lr_precision prec,
                            long step0, long n_steps, int capturing, LoopCache& loops, cudaStream_t s) {
  // a capture holds the teams' one kernel: the wide schedule is 16 nodes a step
  if (plan.wide == 2 || (plan.wide && !capturing)) {
    const WideLayout L = wide_layout(plan, order_bytes(rp.n_traj));
    char* sc = static_cast<char*>(p.scratch);
    DevPtrs q = p;
    q.Za = sc + L.za;
    q.Zb = sc + L.zb;
    q.acc = sc + L.acc;
    q.part = reinterpret_cast<double*>(sc + L.part);
    return wide_integrate(q, rp, plan.max_nblk, plan.Nmax, n_steps, prec != LR_PREC_FP64,
                          LoopRef{&loops, capturing ? nullptr : reinterpret_cast<long long*>(sc + L.loop)}, s);
  }
  const size_t es = prec == LR_PREC_FP64 ? sizeof(double2) : sizeof(float2);
  const SmemLayout L = layout(plan.R, plan.Mp, plan.zs_smem, es, plan.tc, plan.gram_mode == 2);
  fz::Args a{};
  a.p = p;
  a.rp = rp;
  a.step0 = step0;
  a.n_steps = n_steps;
  a.C = plan.C;
  a.n_clusters = plan.n_clusters;
  a.Mp = plan.Mp;
  a.R = plan.R;
  a.Nmax = plan.Nmax;
  a.zs_smem = plan.zs_smem;
  a.o_zs = L.o_zs;
  a.o_slot = L.o_slot;
  a.slot_bytes = L.slot_bytes;
  a.s_gp = L.s_gp;
  a.s_tp = L.s_tp;
  a.s_pop = L.s_pop;
  a.o_gd = L.o_gd;
  a.o_w = L.o_w;
  a.o_tred = L.o_tred;
  a.o_xs = L.o_xs;
  a.o_misc = L.o_misc;
  a.o_tab = L.o_tab;
  a.o_ta = L.o_ta;
  a.o_tb = L.o_tb;
  a.npad = L.npad;
  a.o_gs = L.o_gs;
  char* sc = static_cast<char*>(p.scratch);
  size_t off = order_bytes(rp.n_traj);
  a.order = reinterpret_cast<const int*>(sc);
  if (!plan.zs_smem) {
    a.zs_glob = sc + off;
    off += ((2 * (size_t)plan.R * (plan.Mp + 1) * es * plan.C * plan.n_clusters + 255) / 256) * 256;
  }
  a.acc_glob = sc + off;
  // test hook of the device-wait timeout path (see Args::debug_wait)
  if (const char* e = getenv("LR_DEBUG_WAIT_CYCLES")) a.debug_wait = atoll(e);
  // the trajectory order is in the scratch since fused_prepare; the kernel's
  // attributes are raised here only outside a stream capture
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return e;
  if (cap == cudaStreamCaptureStatusNone) {
    const void* kern = kernel_ptr(prec, plan.zs_smem, plan.tc, plan.frame, plan.gram_mode);
    e = raise_smem_limit(kern, L.total);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(plan.C * plan.n_clusters);
  cfg.blockDim = dim3(plan.threads);
  cfg.dynamicSmemBytes = L.total;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = plan.C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (plan.frame) return fz::rwa_launch(cfg, prec, plan.zs_smem, a);
  if (plan.gram_mode == 2) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 2, 0, 0, 0>, a);
  if (plan.tc == 3) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 1, 0, 3, 0>, a);
  if (plan.tc == 1) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 1, 0, 1, 0>, a);
  if (plan.zs_smem) {
    if (prec == LR_PREC_FP64) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<double2, 0, 1, 0, 0>, a);
    if (prec == LR_PREC_FP32) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 0, 1, 0, 0>, a);
    return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 1, 1, 0, 0>, a);
  }
  if (prec == LR_PREC_FP64) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<double2, 0, 0, 0, 0>, a);
  if (prec == LR_PREC_FP32) return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 0, 0, 0, 0>, a);
  return cudaLaunchKernelEx(&cfg, fz::fused_kernel<float2, 1, 0, 0, 0>, a);
}

}  // namespace lr
