// plan.h -- the launch plan of the step over one or more grids (host side).
//
// Every grid of the step, whether a simulation stepped alone or a member of
// a batch, is advanced by the same plan kernels (plan.cu): one launch per
// kernel of the stage covers every grid of the plan, each block works on one
// grid, found through a per-class block -> grid table, and runs the per-thread
// body of step_bodies.cuh / mixed_bodies.cuh for its thread index within that
// grid.  Since the machine code is the same whatever the plan holds, a
// grid's results are bitwise independent of the grids it is stepped with.
#pragma once

#include <cuda_runtime.h>

#include "../../include/grmhd.h"
#include "grmhd_impl.h"

namespace grmhd {

// One grid as the plan kernels see it.
struct StageItem {
  StepArgs A;
  double *P, *Ph;  // stage arrays: P^n / P^{n+1} and P^{n+1/2}
  double *F[3], *emf, *Uc;
  // face values along each direction, and the update's scratch (SCR_*, [8][ntot]):
  // arrays of their own where split is set, else one pair, which the directions
  // use in turn and whose low half is the scratch when they have done
  double *Lf[3], *Rf[3], *scr;
  int split;
  int *pflag, *fflag;
  float *Pf;           // mixed precision: FP32 primitives (8 x ntot)
  const float *geomf;  // mixed precision: FP32 geometry
  float *Pff;          // float-float: split primitives ([2][8][ntot])
  const float *geomff; // float-float: split geometry ([2][NLOC][G_NCOMP][n2d])
  int prec;            // GRMHD_PREC_*: the flux stage's arithmetic
  // electrons (A.elec): (kappa_tot, kappa_e) of the stage arrays ([2][ntot]
  // each, with P and Ph) and their fluxes
  double *K, *Kh, *FK[3];
  double *KLf, *KRf;  // their face values along the current direction
};

// launch classes, each with its own block table
enum {
  PC_BX1,
  PC_BX2,
  PC_BX3,
  PC_BALL,  // all ghosts in one pass (grids that share no side)
  PC_RECON0,  // FP64 reconstruction along X1 (a lane per pair of differences)
  PC_RECON1,  // along X2
  PC_RECON2,  // along X3 (none for flat-X3 grids)
  PC_FACE0,
  PC_FACE1,
  PC_FACE2,
  PC_FACE0E,  // FP64 face fluxes of grids with electrons (they also store the entropy weights)
  PC_FACE1E,
  PC_FACE2E,
  PC_TOF32,  // mixed: FP32 copy of the stage input
  PC_FACE0F, // mixed: fused FP32 reconstruction + face fluxes per direction
  PC_FACE1F,
  PC_FACE2F,
  PC_TOFF,  // float-float: split copy of the stage input
  PC_RECON01X,
  PC_RECON2X,
  PC_FACE0X,
  PC_FACE1X,
  PC_FACE2X,
  PC_REPL,  // flat-X3 flux copies (for callers who want F)
  PC_FIX,
  PC_EDGE,   // EMFs and CT, every layer
  PC_EDGES,  // EMFs within a step (flat X3: one layer)
  PC_ZONE,   // fixup (every grid)
  PC_SRC64,  // the update's source pass (FP64 and mixed-precision grids)
  PC_SRCX,   // in float-float (float-float and mixed + float-float grids)
  PC_UPD,    // its inversion pass (every grid)
  PC_FLOORD, // drift-frame bounds (grids with bounds in the drift frame, no electrons)
  PC_EREC01, // electron entropy reconstruction along X1, X2 (grids with electrons)
  PC_EREC2,  // along X3
  PC_EFACE0, // electron entropy fluxes per direction
  PC_EFACE1,
  PC_EFACE2,
  PC_EZONE,  // electron heating + bounds (grids with electrons)
  PC_EFIX,   // and their fixup
  PC_N
};

// block order of a launch class
enum {
  PLAN_SCHED_GRID = 0,  // grids in plan order, each grid's blocks contiguous
  PLAN_SCHED_LPT = 1,   // grids by decreasing block count (largest first), contiguous
  PLAN_SCHED_RR = 2,    // round robin: one block of each grid that has blocks left, in turn
  PLAN_SCHED_N
};

struct Plan {
  int ngrid;
  StageItem *items;  // device
  StageItem *host_items;  // host copy of items
  int *tab;          // device: per class, the grid of each block, then its index within that grid
  long long tab_cap; // ints allocated for tab (enough for 64-thread blocks in every class)
  long long *count;  // host: threads of each grid per class, [PC_N][ngrid]
  int bs[PC_N];      // threads per block of each class (multiple of 32, <= 256)
  int sched[PC_N];   // block order of each class (SCHED_*)
  int map_base[PC_N], loc_base[PC_N], nblocks[PC_N];
  long long zones;  // interior zones over all grids
  // every grid split, and few enough zones: the directions' flux kernels and the
  // source pass may run on streams of their own, forked from and joined to the
  // plan's; concurrent once those exist (plan_side_streams)
  int may_split, concurrent;
  cudaStream_t side[3];
  cudaEvent_t fork, join[3];
  int tuned;        // 1 after plan_autotune
};

// Observer of the launches, per kernel class GRMHD_K_* (profiling).
struct PlanHook {
  virtual void begin(int kclass, int nlaunch) = 0;
  virtual void end(int kclass) = 0;
  virtual bool serial() const { return false; }  // times every launch: one after the other
  virtual ~PlanHook() {}
};

// Build the tables and upload the items (device memory of the plan);
// GRMHD_OK, GRMHD_ERR_INVALID (more than 2^31 - 1 blocks in a launch),
// GRMHD_ERR_NOMEM or GRMHD_ERR_CUDA.
int plan_build(Plan &p, const StageItem *items, int n);
// threads per launch class of one grid (dimensions, flat X3, GRMHD_PREC_*,
// bounds in the drift frame, electrons evolved, the plan's reconstruction
// walk length and whether its X1 pass takes a thread per primitive)
void plan_counts(const Dims &D, int flat3, int prec, int drift, int elec, int rwalk,
                 int x1_split, long long c[PC_N]);
// Largest number of interior zones, of a grid and of a plan, whose directions get
// face arrays of their own and run side by side.  A small grid's kernels leave
// most of the GPU idle, each waiting for its threads' chains of work; side by side
// a cycle of a 64x64 mode takes 82 us against 119, of 217x217 zones 227 against
// 264, of 64^3 1.02 against 1.13 ms for 0.11 GB more memory; of larger grids, where only
// the kernels' tails overlap, 100^3 3.36 against 3.46 ms (0.38 GB), 128^3 6.79 against
// 6.89 (0.77), 136^3 8.07 against 8.16 (0.92), 160^3 12.95 against 13.05 (1.46), 192^3
// 22.15 against 22.23 (2.48).  The line lies where the gain, 1.4% there, has come down to
// 1%; the arrays are left out where they do not fit (sim_create).
constexpr long long SPLIT_ZONES = 1 << 21;
constexpr int SPLIT_SETS = 5;  // arrays of [8][ntot] they take
// (FP32 fluxes need no face arrays: their space is the update's scratch at once)
inline bool splits(const Dims &D, int prec) {
  return prec != GRMHD_PREC_MIXED && prec != GRMHD_PREC_MIXED_FF &&
         (long long)D.n[0] * D.n[1] * D.n[2] <= SPLIT_ZONES;
}
// The FP64 reconstruction's walk length along X2 and X3 for a plan of these grids: the
// longest of 16, 8, 4, 2 zones per thread that still gives each of those launches
// RWALK_MIN_THREADS threads, 12 warps per SM; 1 (one thread per zone and primitive,
// which forms each pair of differences three times) where a primitive has fewer
// than RWALK_MIN_ZONES zones, which walks gain 3% at most.  A cycle with 1, 2, 4, 8
// and 16 zones per thread: 217x217 zones 236, 238, 229, 233, 236 us; 61x45x37 534, 542,
// 514, 499, 491; 400x400 611, 606, 605, 587, 592; 32^3 247, 248, 241, 239, 249; 128^3 7.26,
// 7.43, 7.06, 6.88, 6.77 ms.  (A thread that walked all 8 primitives left the last
// wave nearly empty: a 128^3 launch took 0.45 ms, 0.40 so; a 61x45x37 cycle 550 and 508
// us.)
constexpr long long RWALK_MIN_THREADS = 152 * 384;
constexpr long long RWALK_MIN_ZONES = 152 * 256;
int plan_rwalk(const StageItem *items, int n);
// Whether a plan's X1 reconstruction takes a thread per primitive: where threads for all 8
// would be fewer than X1_MIN_THREADS, 8 warps per SM (a cycle of 64x64 zones 83 against
// 89 us, of 128x128 110 against 117, of 217x217 238 against 239, of 61x45x37 519
// against 501: each primitive repeats the index arithmetic).
constexpr long long X1_MIN_THREADS = 152 * 256;
int plan_x1_split(const StageItem *items, int n);
// Set the plan's reconstruction walk length (1, 2, 4, 8 or 16 zones per
// thread; 0: plan_rwalk's choice) and re-lay the reconstruction's block
// tables.  The values do not depend on it.
int plan_set_rwalk(Plan &p, int rw);
// device bytes a one-grid plan of such a grid holds (item + block tables)
long long plan_bytes(const Dims &D, int flat3, int prec, int drift, int elec);
void plan_free(Plan &p);
// Create the streams of a plan that may split, before its first step (and outside
// a capture); without them it runs in sequence.
void plan_side_streams(Plan &p);
// Re-lay the block tables of class cls for bs threads per block and block
// order sched (the results of every grid do not depend on either).
int plan_set_class(Plan &p, int cls, int bs, int sched);
// Pick, by timing on st, the block size and block order of each heavy
// launch class (reconstruction, face fluxes, update + fixup, in both
// precisions) among 64/128/256 threads and the SCHED_* orders.  Leaves
// every grid's state and clock as it found them: the trial launches write
// only scratch (face values, fluxes, the interior of the half-step array)
// and the failure/bound flags of the last stage, and the clocks are saved
// and restored.  Waits for the device before and after.  ms_before / ms_after (may be NULL): one
// pass of the tuned kernels with the previous and the chosen settings.
int plan_autotune(Plan &p, int trials, cudaStream_t st, double *ms_before, double *ms_after);

// The functions below enqueue on st and return the number of kernels
// launched; launch errors are left for cudaGetLastError().
// stage input: 0 = P, 1 = Ph.  Reconstruction + face fluxes (FP64, FP32 or
// float-float per grid) with their boundary fixes; with_source: and the update's
// source pass.  The signal speeds' maxima add to what the clocks hold, which is
// zero between the library's calls: whoever calls this resets them after reading (a
// decomposed grid, whose blocks nothing else steps, before its next step).
int plan_fluxes(const Plan &p, int in, bool with_source, cudaStream_t st, PlanHook *h);
// the fluxes of every layer and flux-CT in place of the induction fluxes: F as
// grmhd_get_fluxes returns it
int plan_whole_fluxes(const Plan &p, int in, cudaStream_t st, PlanHook *h);
// per-grid clock: 0 reset the signal-speed maxima, 1 CFL time step, 2 advance
int plan_clock(const Plan &p, int op, cudaStream_t st, PlanHook *h);
// edge EMFs; take_dt: and the CFL step
int plan_emf(const Plan &p, int take_dt, cudaStream_t st, PlanHook *h);
// U(P^n) + dtfac dt (S - div F) of the source pass's scratch -> inversion -> bounds
// into the other array (in 0: Ph, in 1: P), and the passes that close the state
// (drift-frame bounds, electrons)
int plan_invert(const Plan &p, int in, double dtfac, cudaStream_t st, PlanHook *h);
int plan_fixup(const Plan &p, int out, cudaStream_t st, PlanHook *h);
// ghost fill of P (which 0) or Ph (which 1); end: and the clock's advance and the
// maxima's reset
int plan_bounds(const Plan &p, int which, int end, cudaStream_t st, PlanHook *h);
// one ghost-fill pass (0: X1, 1: X2, 2: X3), for a decomposed grid that exchanges
// block edges between them
int plan_bounds_pass(const Plan &p, int which, int pass, cudaStream_t st, PlanHook *h);
// one stage: stage 0 predictor (P -> Ph, dt/2, with the CFL step), stage 1 corrector
// (Ph -> P, dt, then the clock's advance and the maxima's reset)
int plan_stage(const Plan &p, int stage, cudaStream_t st, PlanHook *h);
// full predictor-corrector steps (U(P^n) kept between the stages)
int plan_steps(const Plan &p, int nsteps, cudaStream_t st, PlanHook *h);

}  // namespace grmhd
