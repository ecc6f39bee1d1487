// plan.cu -- the plan kernels of the predictor-corrector step and their
// enqueue functions (plan.h).  Each kernel maps its block to a grid through
// the class's block table and runs the per-thread body of that grid.
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "../../include/grmhd.h"
#include "grmhd_impl.h"
#include "ff_bodies.cuh"
#include "mixed_bodies.cuh"
#include "elec_bodies.cuh"
#include "plan.h"
#include "step_bodies.cuh"

namespace grmhd {

namespace {

struct BView {
  const StageItem *__restrict__ items;
  const int *__restrict__ map;  // grid of each block of this class
  const int *__restrict__ loc;  // index of each block within its grid
};

__device__ __forceinline__ int block_grid(const BView &V) { return __ldg(V.map + blockIdx.x); }
__device__ __forceinline__ long long block_tid(const BView &V, int) {
  return (long long)__ldg(V.loc + blockIdx.x) * blockDim.x + threadIdx.x;
}
// the stage arrays: 0 = P, 1 = Ph
__device__ __forceinline__ double *arr(const StageItem &it, int which) { return which ? it.Ph : it.P; }
// their electron entropies (null without electrons)
__device__ __forceinline__ double *karr(const StageItem &it, int which) {
  return it.A.elec ? (which ? it.Kh : it.K) : nullptr;
}

template <int X>
__global__ void kp_bounds(BView V, int which) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  double *P = arr(it, which);
  double *K = karr(it, which);
  if (X == 0) bounds_x1_body(it.A, P, K, t);
  if (X == 1) bounds_x2_body(it.A, P, K, t);
  if (X == 2) bounds_x3_body(it.A, P, K, t);
}

// all ghosts; end: and the clock's advance and the signal speeds' reset, which close
// a cycle, in one thread per grid
__global__ void kp_bounds_all(BView V, int which, int end) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  bounds_all_body(it.A, arr(it, which), karr(it, which), t);
  if (end && t == 0) {
    advance_body(it.A);
    reset_ctop_body(it.A.clk);
  }
}

template <int DIR>
__global__ void __launch_bounds__(BS_MAX) kp_recon(BView V, int in) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  const double *Ps = arr(it, in);
  if (it.A.recon == 1) {
    if (DIR == 0)
      recon_x1_body<1>(it.A, Ps, it.Lf[DIR], it.Rf[DIR], t);
    else
      recon_body<DIR, 1>(it.A, Ps, it.Lf[DIR], it.Rf[DIR], t);
  } else {
    if (DIR == 0)
      recon_x1_body<0>(it.A, Ps, it.Lf[DIR], it.Rf[DIR], t);
    else
      recon_body<DIR, 0>(it.A, Ps, it.Lf[DIR], it.Rf[DIR], t);
  }
}

// ELEC: the grids of the launch evolve electron entropies (a class of their own)
// at most 72 registers: 28 warps per SM, whose integer and FP64 work overlap,
// against the spills (per cycle of a 128^3 grid: 168 registers 3.37 ms, 128 2.88,
// 96 2.92, 80 2.80, 72 2.77, 64 2.83)
template <int DIR, bool ELEC = false>
__global__ void __maxnreg__(72) kp_face(BView V, int in) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  const double *Lf = it.Lf[DIR], *Rf = it.Rf[DIR];
  if (DIR == 2 && it.A.flat3) Lf = Rf = arr(it, in);  // flat X3: the primitives
  face_body<DIR, ELEC>(it.A, Lf, Rf, it.F[DIR], t);
}

__global__ void kp_to_f32(BView V, int in) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  to_f32_state_body(arr(it, in), it.Pf, (long long)NV * it.A.D.ntot, block_tid(V, g));
}

// fused FP32 reconstruction + face fluxes (mixed-precision grids)
template <int DIR>
__global__ void __launch_bounds__(BS_MAX) kp_flux_f32(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  if (DIR == 0) {
    if (it.A.recon == 1)
      flux_f32_x1_body<1>(it.A, it.geomf, it.Pf, it.F[0], t);
    else
      flux_f32_x1_body<0>(it.A, it.geomf, it.Pf, it.F[0], t);
  } else {
    if (it.A.recon == 1)
      flux_f32_walk_body<DIR, 1>(it.A, it.geomf, it.Pf, it.F[DIR], t);
    else
      flux_f32_walk_body<DIR, 0>(it.A, it.geomf, it.Pf, it.F[DIR], t);
  }
}

__global__ void kp_to_ff(BView V, int in) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  to_ff_body(arr(it, in), it.Pff, (long long)NV * it.A.D.ntot, block_tid(V, g));
}

template <int DIR>
__global__ void __launch_bounds__(BS_MAX) kp_recon_ff(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  float *Lf = (float *)it.Lf[DIR], *Rf = (float *)it.Rf[DIR];
  if (it.A.recon == 1)
    recon_ff_body<DIR, 1>(it.A, it.Pff, Lf, Rf, t);
  else
    recon_ff_body<DIR, 0>(it.A, it.Pff, Lf, Rf, t);
}

// at most 128 registers: 4 blocks of 128 threads per SM (a few bytes spill)
template <int DIR>
__global__ void __maxnreg__(128) kp_face_ff(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  const float *Lf = (const float *)it.Lf[DIR], *Rf = (const float *)it.Rf[DIR];
  if (DIR == 2 && it.A.flat3) Lf = Rf = it.Pff;
  face_ff_body<DIR>(it.A, it.geomff, Lf, Rf, it.F[DIR], t);
}

__global__ void kp_replicate(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  replicate_body(it.A, it.F[0], it.F[1], it.F[2], block_tid(V, g));
}

__global__ void kp_fix(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const bool e = it.A.elec != 0;
  fix_flux_body(it.A, it.F[0], it.F[1], e ? it.FK[0] : nullptr, e ? it.FK[1] : nullptr,
                block_tid(V, g));
}

// step: within a step (a flat X3 on its one layer); take_dt: and the CFL step, in one
// thread per grid (the update after this reads it)
__global__ void kp_emf(BView V, int step, int take_dt) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  const long long t = block_tid(V, g);
  emf_body(it.A, it.F[0], it.F[1], it.F[2], it.emf, step && it.A.flat3, t);
  if (take_dt && t == 0) dt_body(it.A);
}

__global__ void kp_ct(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  ct_body(it.A, it.F[0], it.F[1], it.F[2], it.emf, block_tid(V, g));
}

// The update's two passes.  PRED: the predictor (in = 0).
// 20 and 24 warps per SM against some spills (both passes per cycle of a 128^3
// grid: 168 and 128 registers 1.74 ms, 128 and 112 1.66, 96 and 80 1.58).
template <bool PRED>
__global__ void __maxnreg__(96) kp_source(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  source_body<PRED>(it.A, PRED ? it.P : it.Ph, it.Uc, it.scr, block_tid(V, g));
}

// the source pass of the float-float modes
template <bool PRED>
__global__ void __maxnreg__(96) kp_source_ff(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  source_ff_body<PRED>(it.A, PRED ? it.P : it.Ph, it.Pff, it.Uc, it.scr, block_tid(V, g));
}

__global__ void __maxnreg__(80) kp_invert(BView V, int in, double dtfac) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  invert_body(it.A, it.F[0], it.F[1], it.F[2], it.emf, it.Uc, it.scr, dtfac, it.P, arr(it, 1 - in), it.pflag,
              it.fflag, block_tid(V, g));
}

template <int DIR>
__global__ void kp_elec_recon(BView V, int in) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  elec_recon_body<DIR>(it.A, karr(it, in), it.KLf, it.KRf, block_tid(V, g));
}

template <int DIR>
__global__ void kp_elec_flux(BView V) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  elec_flux_body<DIR>(it.A, it.KLf, it.KRf, it.FK[DIR], block_tid(V, g));
}

// stage in: P_s = arr(in), output arr(1 - in); kappa_i is always K (of P^n)
__global__ void __maxnreg__(96) kp_elec_post(BView V, int in, double dtfac) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  elec_post_body(it.A, arr(it, in), arr(it, 1 - in), it.F[0], it.F[1], it.F[2], it.FK[0],
                 it.FK[1], it.FK[2], it.K, karr(it, in), karr(it, 1 - in), it.Uc, it.scr, it.pflag,
                 it.fflag, dtfac, block_tid(V, g));
}

__global__ void kp_elec_fix(BView V, int out) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  elec_fix_body(it.A, arr(it, out), karr(it, out), it.pflag, it.fflag, block_tid(V, g));
}

__global__ void __maxnreg__(128) kp_floor_drift(BView V, int out) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  floor_drift_body(it.A, arr(it, out), it.scr, it.pflag, it.fflag, block_tid(V, g));
}

__global__ void kp_fixup(BView V, int out) {
  const int g = block_grid(V);
  const StageItem &it = V.items[g];
  fixup_body(it.A, arr(it, out), it.pflag, it.fflag, block_tid(V, g));
}

// one thread per grid
__global__ void kp_clock(const StageItem *__restrict__ items, int ngrid, int op) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= ngrid) return;
  const StageItem &it = items[g];
  if (op == 0) reset_ctop_body(it.A.clk);
  if (op == 1) dt_body(it.A);
  if (op == 2) advance_body(it.A);
}

long long nblk(long long n, int bs) { return (n + bs - 1) / bs; }

BView view(const Plan &p, int cls) {
  BView V;
  V.items = p.items;
  V.map = p.tab + p.map_base[cls];
  V.loc = p.tab + p.loc_base[cls];
  return V;
}

// NVTX range names of the kernel classes (GRMHD_K_*): a timeline tool sees
// every launch under its class; without a tool the ranges cost a pointer test.
const char *const KCLASS_NAME[GRMHD_NKCLASS] = {"grmhd:flux",  "grmhd:dt",     "grmhd:ct",
                                                 "grmhd:update", "grmhd:fixup", "grmhd:bounds",
                                                 "grmhd:other", "grmhd:recon"};

// Launch one kernel of class cls (skipped when no grid has blocks in it),
// bracketed for the hook and an NVTX range as kernel class kclass.
template <typename L>
int launch(const Plan &p, int cls, int kclass, PlanHook *h, L &&body) {
  if (p.nblocks[cls] <= 0) return 0;
  nvtxRangePushA(KCLASS_NAME[kclass]);
  if (h) h->begin(kclass, 1);
  body((unsigned)p.nblocks[cls], (unsigned)p.bs[cls], view(p, cls));
  if (h) h->end(kclass);
  nvtxRangePop();
  return 1;
}

// Block tables of every class, laid out for p.bs / p.sched and uploaded.
int upload_tables(Plan &p) {
  std::vector<int> host;
  host.reserve((size_t)p.tab_cap);
  const int n = p.ngrid;
  for (int q = 0; q < PC_N; q++) {
    std::vector<long long> nb(n);
    long long tot = 0;
    for (int g = 0; g < n; g++) {
      nb[g] = nblk(p.count[(size_t)q * n + g], p.bs[q]);
      tot += nb[g];
    }
    if (tot >= (1ll << 31) - 1) return GRMHD_ERR_INVALID;
    p.nblocks[q] = (int)tot;
    std::vector<int> map, loc;
    map.reserve((size_t)tot);
    loc.reserve((size_t)tot);
    if (p.sched[q] == PLAN_SCHED_RR) {
      for (long long r = 0; (long long)map.size() < tot; r++)
        for (int g = 0; g < n; g++)
          if (r < nb[g]) {
            map.push_back(g);
            loc.push_back((int)r);
          }
    } else {
      std::vector<int> order(n);
      for (int g = 0; g < n; g++) order[g] = g;
      if (p.sched[q] == PLAN_SCHED_LPT)
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return nb[a] > nb[b]; });
      for (int g : order)
        for (long long r = 0; r < nb[g]; r++) {
          map.push_back(g);
          loc.push_back((int)r);
        }
    }
    p.map_base[q] = (int)host.size();
    host.insert(host.end(), map.begin(), map.end());
    p.loc_base[q] = (int)host.size();
    host.insert(host.end(), loc.begin(), loc.end());
  }
  if ((long long)host.size() > p.tab_cap) return GRMHD_ERR_INVALID;
  if (!host.empty() &&
      cudaMemcpy(p.tab, host.data(), sizeof(int) * host.size(), cudaMemcpyHostToDevice) != cudaSuccess)
    return GRMHD_ERR_CUDA;
  return GRMHD_OK;
}

}  // namespace

void plan_counts(const Dims &D, int flat3, int prec, int drift, int elec, int rwalk,
                 int x1_split, long long c[PC_N]) {
  const int fl = flat3;
  // the flux stage: FP64, FP32 or float-float
  const bool f64 = prec == GRMHD_PREC_FP64, fx = prec == GRMHD_PREC_FF;
  const bool mx = prec == GRMHD_PREC_MIXED || prec == GRMHD_PREC_MIXED_FF;
  c[PC_BX1] = n_bounds_x1(D);
  c[PC_BX2] = n_bounds_x2(D);
  c[PC_BX3] = n_bounds_x3(D);
  c[PC_BALL] = n_bounds_all(D);
  c[PC_RECON0] = f64 ? (x1_split ? NV : 1) * n_recon_walk(D, 0, fl, rwalk) : 0;
  c[PC_RECON1] = f64 ? NV * n_recon_walk(D, 1, fl, rwalk) : 0;
  c[PC_RECON2] = (f64 && !fl) ? NV * n_recon_walk(D, 2, 0, rwalk) : 0;
  for (int d = 0; d < 3; d++) {
    c[PC_FACE0 + d] = (f64 && !elec) ? n_face_threads(D, d, fl) : 0;
    c[PC_FACE0E + d] = (f64 && elec) ? n_face_threads(D, d, fl) : 0;
    c[PC_FACE0F + d] = mx ? (d == 0 ? n_flux_f32_x1(D, fl) : n_flux_f32_walk(D, d, fl)) : 0;
    c[PC_FACE0X + d] = fx ? n_face(D, d, fl) : 0;
  }
  c[PC_TOF32] = mx ? (long long)NV * D.ntot / 2 : 0;  // two elements per thread (NV even)
  c[PC_TOFF] = fx ? (long long)NV * D.ntot : 0;
  c[PC_RECON01X] = fx ? n_recon(D, fl) : 0;
  c[PC_RECON2X] = (fx && !fl) ? n_recon(D, 0) : 0;
  c[PC_REPL] = fl ? n_replicate(D) : 0;
  c[PC_FIX] = f64 ? 0 : n_fix(D);  // (the FP64 face fluxes fix their own)
  c[PC_EDGE] = n_edge(D, 0);
  c[PC_EDGES] = n_edge(D, fl);
  c[PC_ZONE] = n_fixup(D);
  const bool ux = fx || prec == GRMHD_PREC_MIXED_FF;  // the source pass in float-float
  c[PC_SRC64] = ux ? 0 : n_update(D);
  c[PC_SRCX] = ux ? n_update(D) : 0;
  c[PC_UPD] = n_update(D);
  c[PC_FLOORD] = (drift && !elec) ? n_update(D) : 0;
  for (int d = 0; d < 3; d++) c[PC_EFACE0 + d] = elec ? n_face(D, d, fl) : 0;
  c[PC_EREC01] = elec ? n_recon(D, fl) : 0;
  c[PC_EREC2] = (elec && !fl) ? n_recon(D, 0) : 0;
  c[PC_EZONE] = elec ? n_update(D) : 0;
  c[PC_EFIX] = elec ? n_fixup(D) : 0;
}

long long plan_bytes(const Dims &D, int flat3, int prec, int drift, int elec) {
  long long c[PC_N], ints = 0;
  plan_counts(D, flat3, prec, drift, elec, 1, 1, c);  // one thread per zone: the most blocks
  for (int q = 0; q < PC_N; q++) ints += 2 * nblk(c[q], 64);
  return (long long)sizeof(StageItem) + 4 * ints;
}

int plan_rwalk(const StageItem *items, int n) {
  for (int rw = RWALK; rw >= 2; rw /= 2) {
    long long least = -1, zones = 0;  // of the FP64 walk launch (X2 or X3) with the fewest threads
    bool any = false;
    for (int d = 1; d < 3; d++) {
      long long tot = 0, one = 0;
      for (int g = 0; g < n; g++) {
        const StepArgs &A = items[g].A;
        if (items[g].prec != GRMHD_PREC_FP64 || (d == 2 && A.flat3)) continue;
        tot += NV * n_recon_walk(A.D, d, A.flat3, rw);
        one += n_recon_walk(A.D, d, A.flat3, 1);
        any = true;
      }
      if (tot > 0 && (least < 0 || tot < least)) {
        least = tot;
        zones = one;
      }
    }
    if (!any || (least >= RWALK_MIN_THREADS && zones >= RWALK_MIN_ZONES)) return rw;
  }
  return 1;
}

int plan_x1_split(const StageItem *items, int n) {
  long long tot = 0;
  for (int g = 0; g < n; g++)
    if (items[g].prec == GRMHD_PREC_FP64) tot += n_recon_walk(items[g].A.D, 0, items[g].A.flat3, 1);
  return tot < X1_MIN_THREADS;
}

int plan_build(Plan &p, const StageItem *items, int n) {
  memset(&p, 0, sizeof(p));
  if (!items || n < 1) return GRMHD_ERR_INVALID;
  p.ngrid = n;
  p.count = new (std::nothrow) long long[(size_t)PC_N * n];
  p.host_items = new (std::nothrow) StageItem[n];
  if (!p.count || !p.host_items) {
    plan_free(p);
    return GRMHD_ERR_NOMEM;
  }
  memcpy(p.host_items, items, sizeof(StageItem) * n);
  const int rw = plan_rwalk(items, n);
  const int xs = plan_x1_split(items, n);
  for (int g = 0; g < n; g++) {
    p.host_items[g].A.rwalk = rw;
    p.host_items[g].A.x1_split = xs;
  }
  long long zones = 0, cap = 0;
  for (int g = 0; g < n; g++) {
    long long c[PC_N], c1[PC_N];
    const StepArgs &A = items[g].A;
    plan_counts(A.D, A.flat3, items[g].prec, A.floor_drift, A.elec, rw, xs, c);
    plan_counts(A.D, A.flat3, items[g].prec, A.floor_drift, A.elec, 1, 1, c1);
    for (int q = 0; q < PC_N; q++) {
      p.count[(size_t)q * n + g] = c[q];
      // room for the smallest block the tuner tries and any walk length
      cap += 2 * nblk(c1[q] > c[q] ? c1[q] : c[q], 64);
    }
    zones += n_zone(items[g].A.D);
  }
  for (int q = 0; q < PC_N; q++) {
    p.bs[q] = BS;
    p.sched[q] = PLAN_SCHED_GRID;
  }
  p.zones = zones;
  p.tab_cap = cap;
  p.may_split = zones <= SPLIT_ZONES;
  for (int g = 0; g < n; g++) p.may_split = p.may_split && items[g].split;
  if (cudaMalloc(&p.items, sizeof(StageItem) * n) != cudaSuccess ||
      cudaMalloc(&p.tab, sizeof(int) * (size_t)(cap > 0 ? cap : 1)) != cudaSuccess) {
    cudaGetLastError();
    plan_free(p);
    return GRMHD_ERR_NOMEM;
  }
  if (cudaMemcpy(p.items, p.host_items, sizeof(StageItem) * n, cudaMemcpyHostToDevice) != cudaSuccess) {
    plan_free(p);
    return GRMHD_ERR_CUDA;
  }
  const int rc = upload_tables(p);
  if (rc != GRMHD_OK) plan_free(p);
  return rc;
}

void plan_free(Plan &p) {
  if (p.items) cudaFree(p.items);
  if (p.tab) cudaFree(p.tab);
  for (int q = 0; q < 3; q++) {
    if (p.side[q]) cudaStreamDestroy(p.side[q]);
    if (p.join[q]) cudaEventDestroy(p.join[q]);
    p.side[q] = nullptr;
    p.join[q] = nullptr;
  }
  if (p.fork) cudaEventDestroy(p.fork);
  p.fork = nullptr;
  p.concurrent = 0;
  delete[] p.count;
  delete[] p.host_items;
  p.items = nullptr;
  p.tab = nullptr;
  p.count = nullptr;
  p.host_items = nullptr;
  p.ngrid = 0;
}

int plan_set_rwalk(Plan &p, int rw) {
  if (rw < 0 || rw > RWALK || (rw > 1 && (rw & (rw - 1)))) return GRMHD_ERR_INVALID;
  if (rw == 0) rw = plan_rwalk(p.host_items, p.ngrid);
  // kernels still in flight may read the items and tables
  if (cudaDeviceSynchronize() != cudaSuccess) return GRMHD_ERR_CUDA;
  const int n = p.ngrid;
  for (int g = 0; g < n; g++) {
    StageItem &it = p.host_items[g];
    it.A.rwalk = rw;
    long long c[PC_N];
    plan_counts(it.A.D, it.A.flat3, it.prec, it.A.floor_drift, it.A.elec, rw, it.A.x1_split, c);
    for (int q = PC_RECON0; q <= PC_RECON2; q++) p.count[(size_t)q * n + g] = c[q];
  }
  if (cudaMemcpy(p.items, p.host_items, sizeof(StageItem) * n, cudaMemcpyHostToDevice) != cudaSuccess)
    return GRMHD_ERR_CUDA;
  return upload_tables(p);
}

int plan_set_class(Plan &p, int cls, int bs, int sched) {
  if (cls < 0 || cls >= PC_N || bs < 64 || bs > BS_MAX || bs % 32 || sched < 0 || sched >= PLAN_SCHED_N)
    return GRMHD_ERR_INVALID;
  // kernels still in flight may read the tables
  if (cudaDeviceSynchronize() != cudaSuccess) return GRMHD_ERR_CUDA;
  const int obs = p.bs[cls], osc = p.sched[cls];
  p.bs[cls] = bs;
  p.sched[cls] = sched;
  const int rc = upload_tables(p);
  if (rc != GRMHD_OK) {
    p.bs[cls] = obs;
    p.sched[cls] = osc;
    upload_tables(p);
  }
  return rc;
}

int plan_clock(const Plan &p, int op, cudaStream_t st, PlanHook *h) {
  const int kc = (op == 1) ? GRMHD_K_DT : GRMHD_K_OTHER;
  if (h) h->begin(kc, 1);
  kp_clock<<<(unsigned)nblk(p.ngrid, BS), BS, 0, st>>>(p.items, p.ngrid, op);
  if (h) h->end(kc);
  return 1;
}

void plan_side_streams(Plan &p) {
  if (!p.may_split || p.concurrent) return;
  bool ok = p.fork || cudaEventCreateWithFlags(&p.fork, cudaEventDisableTiming) == cudaSuccess;
  for (int q = 0; q < 3 && ok; q++)
    ok = (p.side[q] || cudaStreamCreateWithFlags(&p.side[q], cudaStreamNonBlocking) == cudaSuccess) &&
         (p.join[q] || cudaEventCreateWithFlags(&p.join[q], cudaEventDisableTiming) == cudaSuccess);
  if (!ok) cudaGetLastError();  // one after the other, then
  p.concurrent = ok;
}

namespace {

// reconstruction and face fluxes along one direction, in every precision
template <int DIR>
int flux_dir(const Plan &p, int in, cudaStream_t st, PlanHook *h) {
  const int R = GRMHD_K_RECON, F = GRMHD_K_FLUX;
  int nl = launch(p, PC_RECON0 + DIR, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_recon<DIR><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_FACE0 + DIR, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_face<DIR><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_FACE0E + DIR, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_face<DIR, true><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_FACE0F + DIR, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_flux_f32<DIR><<<nb, bs, 0, st>>>(V); });
  nl += launch(p, (DIR == 2) ? PC_RECON2X : PC_RECON01X, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_recon_ff<DIR><<<nb, bs, 0, st>>>(V); });
  nl += launch(p, PC_FACE0X + DIR, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_face_ff<DIR><<<nb, bs, 0, st>>>(V); });
  return nl;
}

// the update's source pass
int source_pass(const Plan &p, int in, cudaStream_t st, PlanHook *h) {
  int nl = launch(p, PC_SRCX, GRMHD_K_UPDATE, h, [&](unsigned nb, unsigned bs, BView V) {
    if (in == 0)
      kp_source_ff<true><<<nb, bs, 0, st>>>(V);
    else
      kp_source_ff<false><<<nb, bs, 0, st>>>(V);
  });
  nl += launch(p, PC_SRC64, GRMHD_K_UPDATE, h, [&](unsigned nb, unsigned bs, BView V) {
    if (in == 0)
      kp_source<true><<<nb, bs, 0, st>>>(V);
    else  // the predictor before it kept U(P^n)
      kp_source<false><<<nb, bs, 0, st>>>(V);
  });
  return nl;
}

}  // namespace

int plan_fluxes(const Plan &p, int in, bool with_source, cudaStream_t st, PlanHook *h) {
  const int R = GRMHD_K_RECON;
  // the FP32 and the split copies of the stage input
  int nl = launch(p, PC_TOF32, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_to_f32<<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_TOFF, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_to_ff<<<nb, bs, 0, st>>>(V, in); });
  if (p.concurrent && !(h && h->serial())) {
    // nothing below reads what another of the four writes
    cudaEventRecord(p.fork, st);
    for (int q = 0; q < 3; q++)
      if (q < 2 || with_source) cudaStreamWaitEvent(p.side[q], p.fork, 0);
    nl += flux_dir<0>(p, in, p.side[0], h);
    nl += flux_dir<1>(p, in, p.side[1], h);
    if (with_source) nl += source_pass(p, in, p.side[2], h);
    nl += flux_dir<2>(p, in, st, h);
    for (int q = 0; q < 3; q++) {
      if (q == 2 && !with_source) continue;
      cudaEventRecord(p.join[q], p.side[q]);
      cudaStreamWaitEvent(st, p.join[q], 0);
    }
  } else {
    nl += flux_dir<0>(p, in, st, h);
    nl += flux_dir<1>(p, in, st, h);
    nl += flux_dir<2>(p, in, st, h);
    if (with_source) nl += source_pass(p, in, st, h);  // its scratch may be face values' space
  }
  // electron entropies (grids with electrons, any precision): per direction,
  // reconstruction and the fluxes from the face kernels' weights
  const int F = GRMHD_K_FLUX;
  nl += launch(p, PC_EREC01, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_recon<0><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_EFACE0, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_flux<0><<<nb, bs, 0, st>>>(V); });
  nl += launch(p, PC_EREC01, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_recon<1><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_EFACE1, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_flux<1><<<nb, bs, 0, st>>>(V); });
  nl += launch(p, PC_EREC2, R, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_recon<2><<<nb, bs, 0, st>>>(V, in); });
  nl += launch(p, PC_EFACE2, F, h, [&](unsigned nb, unsigned bs, BView V) { kp_elec_flux<2><<<nb, bs, 0, st>>>(V); });
  // boundary flux fixes
  nl += launch(p, PC_FIX, GRMHD_K_CT, h, [&](unsigned nb, unsigned bs, BView V) { kp_fix<<<nb, bs, 0, st>>>(V); });
  return nl;
}

int plan_emf(const Plan &p, int take_dt, cudaStream_t st, PlanHook *h) {
  return launch(p, PC_EDGES, GRMHD_K_CT, h, [&](unsigned nb, unsigned bs, BView V) { kp_emf<<<nb, bs, 0, st>>>(V, 1, take_dt); });
}

int plan_whole_fluxes(const Plan &p, int in, cudaStream_t st, PlanHook *h) {
  const int C = GRMHD_K_CT;
  int nl = plan_fluxes(p, in, false, st, h);
  nl += launch(p, PC_REPL, GRMHD_K_OTHER, h,
               [&](unsigned nb, unsigned bs, BView V) { kp_replicate<<<nb, bs, 0, st>>>(V); });
  nl += launch(p, PC_EDGE, C, h, [&](unsigned nb, unsigned bs, BView V) { kp_emf<<<nb, bs, 0, st>>>(V, 0, 0); });
  nl += launch(p, PC_EDGE, C, h, [&](unsigned nb, unsigned bs, BView V) { kp_ct<<<nb, bs, 0, st>>>(V); });
  return nl;
}

int plan_invert(const Plan &p, int in, double dtfac, cudaStream_t st, PlanHook *h) {
  int nl = launch(p, PC_UPD, GRMHD_K_UPDATE, h, [&](unsigned nb, unsigned bs, BView V) { kp_invert<<<nb, bs, 0, st>>>(V, in, dtfac); });
  nl += launch(p, PC_FLOORD, GRMHD_K_UPDATE, h, [&](unsigned nb, unsigned bs, BView V) {
    kp_floor_drift<<<nb, bs, 0, st>>>(V, 1 - in);
  });
  nl += launch(p, PC_EZONE, GRMHD_K_UPDATE, h, [&](unsigned nb, unsigned bs, BView V) {
    kp_elec_post<<<nb, bs, 0, st>>>(V, in, dtfac);
  });
  return nl;
}

int plan_fixup(const Plan &p, int out, cudaStream_t st, PlanHook *h) {
  int nl = launch(p, PC_ZONE, GRMHD_K_FIXUP, h,
                  [&](unsigned nb, unsigned bs, BView V) { kp_fixup<<<nb, bs, 0, st>>>(V, out); });
  nl += launch(p, PC_EFIX, GRMHD_K_FIXUP, h,
               [&](unsigned nb, unsigned bs, BView V) { kp_elec_fix<<<nb, bs, 0, st>>>(V, out); });
  return nl;
}

int plan_bounds_pass(const Plan &p, int which, int pass, cudaStream_t st, PlanHook *h) {
  const int B = GRMHD_K_BOUNDS;
  if (pass == 0)
    return launch(p, PC_BX1, B, h, [&](unsigned nb, unsigned bs, BView V) { kp_bounds<0><<<nb, bs, 0, st>>>(V, which); });
  if (pass == 1)
    return launch(p, PC_BX2, B, h, [&](unsigned nb, unsigned bs, BView V) { kp_bounds<1><<<nb, bs, 0, st>>>(V, which); });
  return launch(p, PC_BX3, B, h, [&](unsigned nb, unsigned bs, BView V) { kp_bounds<2><<<nb, bs, 0, st>>>(V, which); });
}

int plan_bounds(const Plan &p, int which, int end, cudaStream_t st, PlanHook *h) {
  return launch(p, PC_BALL, GRMHD_K_BOUNDS, h, [&](unsigned nb, unsigned bs, BView V) { kp_bounds_all<<<nb, bs, 0, st>>>(V, which, end); });
}

// Six launches on a stage's critical chain (reconstruction and face fluxes per
// direction on streams of their own, EMFs, inversion, fixup, ghosts).  With the
// flux fixes, the flux copies of a flat X3, the CFL step, flux-CT's flux update, the
// three ghost passes and the clock as launches of their own it was twelve and a
// half: by that alone a cycle went from 114 to 85 us at 64 x 64, 281 to 239 at 217 x 217,
// 640 to 563 at 61 x 45 x 37, 6990 to 6040 for a batch of 64 flat grids of 32^2
// to 256^2.
int plan_stage(const Plan &p, int stage, cudaStream_t st, PlanHook *h) {
  int nl = plan_fluxes(p, stage, true, st, h);
  nl += plan_emf(p, stage == 0, st, h);
  nl += plan_invert(p, stage, stage ? 1.0 : 0.5, st, h);
  nl += plan_fixup(p, 1 - stage, st, h);
  nl += plan_bounds(p, 1 - stage, stage, st, h);
  return nl;
}

int plan_steps(const Plan &p, int nsteps, cudaStream_t st, PlanHook *h) {
  int nl = 0;
  for (int n = 0; n < nsteps; n++) {
    nl += plan_stage(p, 0, st, h);  // predictor: keeps U(P^n)
    nl += plan_stage(p, 1, st, h);  // corrector: reads it back
  }
  return nl;
}

namespace {

// Device time (ms) of `trials` passes of run() on st, after one warm-up pass.
template <typename R>
double time_passes(cudaStream_t st, int trials, R &&run) {
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  run();
  cudaEventRecord(e0, st);
  for (int q = 0; q < trials; q++) run();
  cudaEventRecord(e1, st);
  cudaEventSynchronize(e1);
  float ms = 0.0f;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return (double)ms / trials;
}

}  // namespace

int plan_autotune(Plan &p, int trials, cudaStream_t st, double *ms_before, double *ms_after) {
  if (p.ngrid < 1 || trials < 1) return GRMHD_ERR_INVALID;
  if (cudaDeviceSynchronize() != cudaSuccess) return GRMHD_ERR_CUDA;
  const int n = p.ngrid;
  std::vector<Clock> saved(n);
  for (int g = 0; g < n; g++)
    if (cudaMemcpy(&saved[g], p.host_items[g].A.clk, sizeof(Clock), cudaMemcpyDeviceToHost) !=
        cudaSuccess)
      return GRMHD_ERR_CUDA;
  // representative scratch: fluxes, EMFs and a CFL dt of the current state
  plan_fluxes(p, 0, false, st, nullptr);
  plan_emf(p, 1, st, nullptr);
  struct Group {
    int cls;
    int which;  // what one pass launches
  };
  const Group groups[] = {{PC_RECON0, 0},   {PC_RECON1, 6},  {PC_RECON2, 1},   {PC_FACE0, 2},
                          {PC_FACE1, 3},    {PC_FACE2, 4},   {PC_UPD, 5},
                          {PC_FACE0F, 8},   {PC_FACE1F, 9},  {PC_FACE2F, 10},  {PC_RECON01X, 11},
                          {PC_RECON2X, 12}, {PC_FACE0X, 13}, {PC_FACE1X, 14},  {PC_FACE2X, 15},
                          {PC_SRC64, 16},   {PC_SRCX, 17}};
  auto pass = [&](int which) {
    auto L = [&](int cls, auto &&body) { launch(p, cls, 0, nullptr, body); };
    switch (which) {
      case 0:
        L(PC_RECON0, [&](unsigned nb, unsigned bs, BView V) { kp_recon<0><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 6:
        L(PC_RECON1, [&](unsigned nb, unsigned bs, BView V) { kp_recon<1><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 1:
        L(PC_RECON2, [&](unsigned nb, unsigned bs, BView V) { kp_recon<2><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 2:
        L(PC_FACE0, [&](unsigned nb, unsigned bs, BView V) { kp_face<0><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 3:
        L(PC_FACE1, [&](unsigned nb, unsigned bs, BView V) { kp_face<1><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 4:
        L(PC_FACE2, [&](unsigned nb, unsigned bs, BView V) { kp_face<2><<<nb, bs, 0, st>>>(V, 0); });
        break;
      case 5:
        L(PC_UPD, [&](unsigned nb, unsigned bs, BView V) { kp_invert<<<nb, bs, 0, st>>>(V, 0, 0.5); });
        break;
      case 8:
        L(PC_FACE0F, [&](unsigned nb, unsigned bs, BView V) { kp_flux_f32<0><<<nb, bs, 0, st>>>(V); });
        break;
      case 9:
        L(PC_FACE1F, [&](unsigned nb, unsigned bs, BView V) { kp_flux_f32<1><<<nb, bs, 0, st>>>(V); });
        break;
      case 10:
        L(PC_FACE2F, [&](unsigned nb, unsigned bs, BView V) { kp_flux_f32<2><<<nb, bs, 0, st>>>(V); });
        break;
      case 11:
        L(PC_RECON01X, [&](unsigned nb, unsigned bs, BView V) { kp_recon_ff<0><<<nb, bs, 0, st>>>(V); });
        L(PC_RECON01X, [&](unsigned nb, unsigned bs, BView V) { kp_recon_ff<1><<<nb, bs, 0, st>>>(V); });
        break;
      case 12:
        L(PC_RECON2X, [&](unsigned nb, unsigned bs, BView V) { kp_recon_ff<2><<<nb, bs, 0, st>>>(V); });
        break;
      case 13:
        L(PC_FACE0X, [&](unsigned nb, unsigned bs, BView V) { kp_face_ff<0><<<nb, bs, 0, st>>>(V); });
        break;
      case 14:
        L(PC_FACE1X, [&](unsigned nb, unsigned bs, BView V) { kp_face_ff<1><<<nb, bs, 0, st>>>(V); });
        break;
      case 15:
        L(PC_FACE2X, [&](unsigned nb, unsigned bs, BView V) { kp_face_ff<2><<<nb, bs, 0, st>>>(V); });
        break;
      case 16:
        L(PC_SRC64, [&](unsigned nb, unsigned bs, BView V) { kp_source<true><<<nb, bs, 0, st>>>(V); });
        break;
      case 17:
        L(PC_SRCX, [&](unsigned nb, unsigned bs, BView V) { kp_source_ff<true><<<nb, bs, 0, st>>>(V); });
        break;
    }
  };
  const int sizes[] = {64, 128, 256};
  double before = 0.0, after = 0.0;
  int rc = GRMHD_OK;
  for (const Group &gr : groups) {
    if (p.nblocks[gr.cls] <= 0) continue;
    const int bs0 = p.bs[gr.cls], sc0 = p.sched[gr.cls];
    // the inversion's scratch, which the reconstructions before it may share
    if (gr.cls == PC_UPD) source_pass(p, 0, st, nullptr);
    double best = time_passes(st, trials, [&] { pass(gr.which); });
    before += best;
    int best_bs = bs0, best_sc = sc0;
    for (int bs : sizes)
      for (int sc = 0; sc < (n > 1 ? PLAN_SCHED_N : 1); sc++) {
        if (bs == bs0 && sc == sc0) continue;
        rc = plan_set_class(p, gr.cls, bs, sc);
        if (rc != GRMHD_OK) break;
        const double t = time_passes(st, trials, [&] { pass(gr.which); });
        if (t < 0.99 * best) {  // a change must gain more than the timing noise
          best = t;
          best_bs = bs;
          best_sc = sc;
        }
      }
    if (rc != GRMHD_OK) break;
    rc = plan_set_class(p, gr.cls, best_bs, best_sc);
    if (rc != GRMHD_OK) break;
    after += best;
  }
  if (cudaDeviceSynchronize() != cudaSuccess && rc == GRMHD_OK) rc = GRMHD_ERR_CUDA;
  for (int g = 0; g < n; g++)
    if (cudaMemcpy(p.host_items[g].A.clk, &saved[g], sizeof(Clock), cudaMemcpyHostToDevice) !=
            cudaSuccess &&
        rc == GRMHD_OK)
      rc = GRMHD_ERR_CUDA;
  if (rc == GRMHD_OK) p.tuned = 1;
  if (ms_before) *ms_before = before;
  if (ms_after) *ms_after = after;
  return rc;
}

}  // namespace grmhd
