// step_bodies.cuh -- the per-thread bodies of the kernels of one
// predictor-corrector stage of the HARM scheme (iharm3D, arXiv:2110.10191):
//   zone-centric reconstruction -> face fluxes (LLF, with their boundary fixes and
//   a warp/block max of the signal speed for the CFL step) -> flux-CT EMFs (Toth
//   2000; paper, "Implementation Notes", first paragraph), dt -> update (its source
//   pass may run beside the fluxes) + 1D_W inversion + bounds (same section) ->
//   fixup of failed zones -> ghost fill.
//
// Each body takes the step arguments of one grid and the linear index t of
// its thread within that grid's launch range.  The plan kernels (plan.cu)
// run them for one grid or many (t from the block's index within its grid);
// the allocation-free flux entry point's kernels (step.cu) for one.  A block
// never spans two grids: the block reductions (signal speed maxima, warp
// counts) see the threads of one grid only.
//
// A thread owns an edge, a zone, half a face or a stretch of one primitive's column;
// fields are SoA float64 in HBM with i fastest, so warps read and write contiguous runs.
//
// Flat X3 (A.flat3: n3 = 1 with periodic X3): every k layer of the
// primitives is an exact copy of the single interior layer, so the fluxes
// along X1 and X2 are computed on that layer only, the update takes the layer's X3
// differences as zero, and the X3 faces read the primitives themselves as their
// face states (reconstruction of constant data returns the data exactly).  Callers
// who want the fluxes get them copied to the layers above and below (replicate_body).
#pragma once

#include "grmhd_dev.cuh"
#include "grmhd_impl.h"
#include "wide_face.cuh"
#include "wide_update.cuh"

namespace grmhd {

constexpr int BS = 128;      // default threads per block of the stage kernels
constexpr int BS_MAX = 256;  // largest block the plan kernels are compiled for

__device__ __forceinline__ int wrap(int g, int n) {  // periodic image of ghost index g
  int q = (g - NG) % n;
  if (q < 0) q += n;
  return NG + q;
}

// t as (i, j, k) of a range n0 x n1 x ..., i fastest.  Every range of a grid has
// fewer than 2^32 entries (the library refuses grids of 2^31 zones, ghosts
// included), so that two 32-bit divisions do, a fifth of the instructions of the
// 64-bit ones.
struct Idx3 {
  int i, j, k;
};
__device__ __forceinline__ Idx3 unflatten(long long t, int n0, int n1) {
  const u32 u = (u32)t, q = u / (u32)n0, k = q / (u32)n1;
  return {(int)(u - q * n0), (int)(q - k * n1), (int)k};
}

// Warps over columns along X3: a warp takes `lanes` consecutive points of the
// (X1, X2) plane of a range n0 x n1 x n2 at one k, the next warp the same points at
// the next k, so that the warps of a block share the points' geometry in L1.
__host__ __device__ inline long long n_column_threads(int lanes, int n0, int n1, int n2) {
  return 32 * (((long long)n0 * n1 + lanes - 1) / lanes) * n2;
}
struct Column {
  bool active;
  int i, j, k;  // inactive lanes: of the plane's last point
};
__device__ __forceinline__ Column column_of(long long t, int lane, int lanes, int n0, int n1, int n2) {
  const u32 w = (u32)(t >> 5), chunk = w / (u32)n2, plane = (u32)(n0 * n1);
  u32 p = chunk * lanes + lane;
  Column q;
  q.k = (int)(w - chunk * n2);
  q.active = p < plane;
  if (!q.active) p = plane - 1;
  q.j = (int)(p / (u32)n0);
  q.i = (int)(p - q.j * n0);
  return q;
}

// ---------------------------------------------------------------------------
// Launch extents (threads per grid) of each body
// ---------------------------------------------------------------------------
__host__ __device__ inline long long n_bounds_x1(const Dims &D) {
  return (long long)D.n[1] * D.n[2] * 2 * NG;
}
__host__ __device__ inline long long n_bounds_x2(const Dims &D) {
  return (long long)D.s[0] * D.n[2] * 2 * NG;
}
__host__ __device__ inline long long n_bounds_x3(const Dims &D) { return D.n2d * 2 * NG; }
// zones whose two face values are reconstructed along one direction
__host__ __device__ inline long long n_recon(const Dims &D, int flat3) {
  return (long long)(D.n[0] + 2) * (D.n[1] + 2) * (flat3 ? 1 : D.n[2] + 2);
}
// longest FP64 reconstruction walk (zones per thread)
constexpr int RWALK = 16;
// pairs that a warp of recon_x1_body finishes
constexpr int X1_LANES = 30;
// threads of one variable of the FP64 reconstruction along dir: along X1 a warp per
// X1_LANES pairs (recon_x1_body); else one per column and segment of rw zones along
// dir (rw >= 2), or one per zone (rw = 1)
__host__ __device__ inline long long n_recon_walk(const Dims &D, int dir, int flat3, int rw) {
  const long long e[3] = {D.n[0] + 2, D.n[1] + 2, flat3 ? 1 : D.n[2] + 2};
  if (dir == 0) return 32 * (((e[0] + 2) * e[1] * e[2] - 2 + X1_LANES - 1) / X1_LANES);
  if (rw <= 1) return e[0] * e[1] * e[2];
  return e[0] * e[1] * e[2] / e[dir] * ((e[dir] + rw - 1) / rw);
}
// thread t of NV per -> the variable, t within it (per threads a variable)
__device__ __forceinline__ int split_var(long long &t, long long per) {
  int v = 0;
#pragma unroll
  for (int b = NV / 2; b >= 1; b /= 2)
    if (t >= b * per) {
      t -= b * per;
      v += b;
    }
  return v;
}
// faces along dir: dir index NG .. n+NG, transverse NG-1 .. n+NG (flux-CT
// needs one transverse layer on each side); flat X3 keeps the k = NG layer
__host__ __device__ inline void face_box(const Dims &D, int dir, int flat3, int lo[3], int ext[3]) {
  for (int e = 0; e < 3; e++) {
    lo[e] = (e == dir) ? NG : NG - 1;
    ext[e] = (e == dir) ? D.n[e] + 1 : D.n[e] + 2;
  }
  if (flat3) {
    lo[2] = NG;
    ext[2] = 1;
  }
}
__host__ __device__ inline long long n_face(const Dims &D, int dir, int flat3) {
  int lo[3], ext[3];
  face_box(D, dir, flat3, lo, ext);
  return (long long)ext[0] * ext[1] * ext[2];
}
__host__ __device__ inline long long n_replicate(const Dims &D) { return D.n2d * NV; }
__host__ __device__ inline long long n_fix(const Dims &D) {
  return (long long)((D.n[0] > D.n[1]) ? D.n[0] + 2 : D.n[1] + 2) * (D.n[2] + 2);
}
__host__ __device__ inline long long n_edge(const Dims &D, int flat3) {
  return (long long)(D.n[0] + 1) * (D.n[1] + 1) * (flat3 ? 1 : D.n[2] + 1);
}
__host__ __device__ inline long long n_zone(const Dims &D) {
  return (long long)D.n[0] * D.n[1] * D.n[2];
}
// threads of the update's passes
__host__ __device__ inline long long n_update(const Dims &D) {
  return n_column_threads(32, D.n[0], D.n[1], D.n[2]);
}

// ---------------------------------------------------------------------------
// Boundary conditions
// ---------------------------------------------------------------------------
// K (null without electrons): the two electron entropies, copied as scalars
__device__ __forceinline__ void copy_zone(const Dims &D, double *P, double *K, long long dst,
                                          long long src) {
#pragma unroll
  for (int v = 0; v < NV; v++) P[v * D.ntot + dst] = P[v * D.ntot + src];
  if (K) {
    K[dst] = K[src];
    K[D.ntot + dst] = K[D.ntot + src];
  }
}

// X1 ghosts for interior (j, k); one thread per (ghost layer, side, j, k)
__device__ __forceinline__ void bounds_x1_body(const StepArgs &A, double *P, double *K,
                                               long long t) {
  const Dims &D = A.D;
  if (t >= n_bounds_x1(D)) return;
  const Idx3 q3 = unflatten(t, 2 * NG, D.n[1]);
  const int g = q3.i % NG, side = q3.i / NG, j = NG + q3.j, k = NG + q3.k;
  const int bc = A.bc[0][side];
  const int ig = side ? D.n[0] + NG + g : g;
  const long long d = zid(D, ig, j, k);
  if (bc == 0) {
    copy_zone(D, P, K, d, zid(D, wrap(ig, D.n[0]), j, k));
  } else if (bc == 1) {
    const int ia = side ? D.n[0] + NG - 1 : NG;
    copy_zone(D, P, K, d, zid(D, ia, j, k));
    const double *gd = A.geom + (LOC_CENT * G_NCOMP + G_GDET) * D.n2d;
    const double rs = gd[(long long)j * D.s[0] + ia] / gd[(long long)j * D.s[0] + ig];
    P[B1 * D.ntot + d] *= rs;
    P[B2 * D.ntot + d] *= rs;
    P[B3 * D.ntot + d] *= rs;
    const double u1 = P[U1 * D.ntot + d];
    if (side == 0 ? (u1 > 0.0) : (u1 < 0.0)) P[U1 * D.ntot + d] = 0.0;
  }
}

// X2 ghosts for all i and interior k
__device__ __forceinline__ void bounds_x2_body(const StepArgs &A, double *P, double *K,
                                               long long t) {
  const Dims &D = A.D;
  if (t >= n_bounds_x2(D)) return;
  const Idx3 q3 = unflatten(t, D.s[0], 2 * NG);
  const int i = q3.i, g = q3.j % NG, side = q3.j / NG, k = NG + q3.k;
  const int bc = A.bc[1][side];
  const int jg = side ? D.n[1] + NG + g : NG - 1 - g;
  const long long d = zid(D, i, jg, k);
  if (bc == 0) {
    copy_zone(D, P, K, d, zid(D, i, wrap(jg, D.n[1]), k));
  } else if (bc == 2) {
    const int jm = side ? D.n[1] + NG - 1 - g : NG + g;
    copy_zone(D, P, K, d, zid(D, i, jm, k));
    P[U2 * D.ntot + d] = -P[U2 * D.ntot + d];
    P[B2 * D.ntot + d] = -P[B2 * D.ntot + d];
  } else if (bc == 1) {
    copy_zone(D, P, K, d, zid(D, i, side ? D.n[1] + NG - 1 : NG, k));
  }
}

// X3 ghosts for all i, j
__device__ __forceinline__ void bounds_x3_body(const StepArgs &A, double *P, double *K,
                                               long long t) {
  const Dims &D = A.D;
  if (t >= n_bounds_x3(D)) return;
  const Idx3 q3 = unflatten(t, (int)D.n2d, NG);
  const long long ij = q3.i;
  const int g = q3.j, side = q3.k;
  const int bc = A.bc[2][side];
  const int kg = side ? D.n[2] + NG + g : NG - 1 - g;
  const long long d = (long long)kg * D.n2d + ij;
  if (bc == 0) {
    copy_zone(D, P, K, d, (long long)wrap(kg, D.n[2]) * D.n2d + ij);
  } else if (bc == 1) {
    copy_zone(D, P, K, d, (long long)(side ? D.n[2] + NG - 1 : NG) * D.n2d + ij);
  }
}

// All ghosts in one pass, each from the zones that the three passes above would
// carry to it (X3's from X2's from X1's), for grids whose sides are all their own:
// every value read is an interior zone's or a fixed ghost's, which nothing here
// writes.  Same values bit for bit.
__host__ __device__ inline long long n_bounds_all(const Dims &D) {
  return n_bounds_x1(D) + n_bounds_x2(D) + n_bounds_x3(D);
}
__device__ __forceinline__ void bounds_all_body(const StepArgs &A, double *P, double *K,
                                                long long t) {
  const Dims &D = A.D;
  if (t >= n_bounds_all(D)) return;
  int i, j, k;
  if (t < n_bounds_x3(D)) {
    const Idx3 q3 = unflatten(t, D.s[0], D.s[1]);
    i = q3.i;
    j = q3.j;
    k = (q3.k < NG) ? q3.k : D.n[2] + q3.k;
  } else if ((t -= n_bounds_x3(D)) < n_bounds_x2(D)) {
    const Idx3 q3 = unflatten(t, D.s[0], 2 * NG);
    i = q3.i;
    j = (q3.j < NG) ? q3.j : D.n[1] + q3.j;
    k = NG + q3.k;
  } else {
    t -= n_bounds_x2(D);
    const Idx3 q3 = unflatten(t, 2 * NG, D.n[1]);
    i = (q3.i < NG) ? q3.i : D.n[0] + q3.i;
    j = NG + q3.j;
    k = NG + q3.k;
  }
  const long long d = zid(D, i, j, k);
  int si = i, sj = j, sk = k;
  if (k < NG || k >= D.n[2] + NG) {
    const int side = k >= NG, bc = A.bc[2][side];
    if (bc == 0)
      sk = wrap(k, D.n[2]);
    else if (bc == 1)
      sk = side ? D.n[2] + NG - 1 : NG;
    else
      return;  // fixed
  }
  bool mirror = false, out = false;
  if (j < NG || j >= D.n[1] + NG) {
    const int side = j >= NG, bc = A.bc[1][side];
    if (bc == 0) {
      sj = wrap(j, D.n[1]);
    } else if (bc == 2) {
      sj = side ? 2 * (D.n[1] + NG) - 1 - j : 2 * NG - 1 - j;
      mirror = true;
    } else if (bc == 1) {
      sj = side ? D.n[1] + NG - 1 : NG;
    } else if (sk == k) {
      return;  // fixed
    }
  }
  const bool own_row = sj >= NG && sj < D.n[1] + NG;  // else a fixed X2 ghost, whatever its i
  if (own_row && (i < NG || i >= D.n[0] + NG)) {
    const int bc = A.bc[0][i >= NG];
    if (bc == 0) {
      si = wrap(i, D.n[0]);
    } else if (bc == 1) {
      si = (i >= NG) ? D.n[0] + NG - 1 : NG;
      out = true;
    } else if (sk == k && sj == j) {
      return;  // fixed
    }
  }
  const long long c = zid(D, si, sj, sk), N = D.ntot;
  double p[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) p[v] = P[v * N + c];
  if (out) {
    const double *gd = A.geom + (LOC_CENT * G_NCOMP + G_GDET) * D.n2d + (long long)sj * D.s[0];
    const double rs = gd[si] / gd[i];
    p[B1] *= rs;
    p[B2] *= rs;
    p[B3] *= rs;
    if (i >= NG ? (p[U1] < 0.0) : (p[U1] > 0.0)) p[U1] = 0.0;
  }
  if (mirror) {
    p[U2] = -p[U2];
    p[B2] = -p[B2];
  }
#pragma unroll
  for (int v = 0; v < NV; v++) P[v * N + d] = p[v];
  if (K) {
    K[d] = K[c];
    K[N + d] = K[N + c];
  }
}

// ---------------------------------------------------------------------------
// Face fluxes
// ---------------------------------------------------------------------------
// Block maximum of v >= 0 (any block size that is a multiple of 32, up to
// 1024), one atomicMax per block; every thread of the block must call it.
__device__ __forceinline__ void warp_block_max(double v, unsigned long long *dst) {
  // v >= 0: its bit pattern orders like the value; high words first, then the
  // low words of the lanes that have the highest
  const u64 b = w_bits(v);
  const u32 hi = __reduce_max_sync(0xffffffffu, w_hi(b));
  const u32 lo = __reduce_max_sync(0xffffffffu, (w_hi(b) == hi) ? w_lo(b) : 0u);
  __shared__ unsigned long long sm[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sm[w] = (u64)hi << 32 | lo;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    unsigned long long m = sm[0];
    for (int q = 1; q < nw; q++) m = (sm[q] > m) ? sm[q] : m;
    if (m) atomicMax(dst, m);
  }
}

// Zone-centric reconstruction along X2 or X3: both face values of each zone's
// 8 primitives (zones NG-1 .. n+NG along DIR and the extended transverse range),
// each zone's WENO smoothness indicators formed once.  A thread takes one primitive:
// with A.rwalk >= 2 it walks a segment of A.rwalk zones of one column along DIR, so
// that consecutive zones share their differences and indicators (WenoWalk); with
// A.rwalk = 1 (grids too small to fill the GPU with walks) it takes one zone.
// Consecutive threads take neighbouring columns along X1, the primitives follow
// one another.  Same values either way.  Lf = value at the zone's low face, Rf = at
// its high face.
template <int DIR, int RECON>
__device__ __forceinline__ void recon_body(const StepArgs &A, const double *__restrict__ P,
                                           double *__restrict__ Lf, double *__restrict__ Rf,
                                           long long t) {
  const Dims &D = A.D;
  const int e0 = D.n[0] + 2, e1 = D.n[1] + 2, e2 = A.flat3 ? 1 : D.n[2] + 2;
  const int kb = A.flat3 ? NG : NG - 1;
  const long long st = (DIR == 1) ? D.s[0] : D.n2d;
  const int rw = A.rwalk;
  const int v = split_var(t, n_recon_walk(D, DIR, A.flat3, rw));
  if (rw <= 1) {
    if (t >= (long long)e0 * e1 * e2) return;
    const Idx3 q3 = unflatten(t, e0, e1);
    const long long o = v * D.ntot + zid(D, NG - 1 + q3.i, NG - 1 + q3.j, kb + q3.k);
    const double *p = P + o;
    double lo, hi;
    if (RECON == 1) {
      weno5_wide_pair(__ldg(p - 2 * st), __ldg(p - st), __ldg(p), __ldg(p + st), __ldg(p + 2 * st),
                      lo, hi);
    } else {
      const double x1 = __ldg(p), h = mc_half_slope(x1 - __ldg(p - st), __ldg(p + st) - x1);
      lo = x1 - h;
      hi = x1 + h;
    }
    Lf[o] = lo;
    Rf[o] = hi;
    return;
  }
  const int ed = (DIR == 1) ? e1 : e2;
  const int eb = (DIR == 2) ? e1 : e2;
  const int nseg = (ed + rw - 1) / rw;
  if (t >= (long long)e0 * eb * nseg) return;
  const Idx3 q3 = unflatten(t, e0, eb);
  const int i = NG - 1 + q3.i, cb = q3.j, m0 = q3.k * rw;
  const int j = NG - 1 + ((DIR == 1) ? m0 : cb);
  const int k = (DIR == 2) ? NG - 1 + m0 : kb + cb;
  const int n = min(rw, ed - m0);
  const long long o = v * D.ntot + zid(D, i, j, k);
  const double *p = P + o;
  double *lf = Lf + o, *rf = Rf + o;
  if (RECON == 1) {
    weno5_walk(p, lf, rf, st, n);
  } else {
    double x1 = __ldg(p), dm = x1 - __ldg(p - st);
    for (int m = 0; m < n; m++) {
      const double x2 = __ldg(p + (m + 1) * st), dp = x2 - x1, h = mc_half_slope(dm, dp);
      lf[m * st] = x1 - h;
      rf[m * st] = x1 + h;
      x1 = x2;
      dm = dp;
    }
  }
}

// The reconstruction along X1, for every A.rwalk.  A lane takes one pair of
// neighbouring first differences of a row, (x1 - x0, x2 - x1) from zone x0 on,
// forms the substencil's indicators in its three roles and gets the two
// substencils below from the two lanes below by warp shuffles, so that each
// pair is formed once, as along a walk, and loads and stores stay coalesced.  The
// pairs of all rows (n1 + 4 per row) are numbered through; a warp takes 32
// consecutive ones, 30 of them its own (lanes 0 and 1 only serve the lanes
// above).  Against walks of 32 rows per warp staged in shared memory, whose 152
// registers and tile left 10 warps per SM waiting for loads, a 128x128x64 grid's
// launch went from 446 to 220 us.  A thread takes all 8 primitives, or one of them
// (A.x1_split: small grids).  Same values as recon_body's.  Every thread of the warp
// must call it.
template <int RECON>
__device__ __forceinline__ void recon_x1_body(const StepArgs &A, const double *__restrict__ P,
                                              double *__restrict__ Lf, double *__restrict__ Rf,
                                              long long t) {
  const Dims &D = A.D;
  const int e1 = D.n[1] + 2, e2 = A.flat3 ? 1 : D.n[2] + 2, row = D.n[0] + 4;
  const int lane = (int)(t & 31);
  const long long npair = (long long)row * e1 * e2;
  // whole warps of one variable, or of all of them
  const int v0 = A.x1_split ? split_var(t, n_recon_walk(D, 0, A.flat3, 1)) : 0;
  const long long g = (t >> 5) * X1_LANES + lane;
  const long long h = (g < npair) ? g : npair - 1;
  const Idx3 q3 = unflatten(h, row, e1);
  const int q = q3.i;  // zone NG - 3 + q: the row's first two lie below the range
  const long long c = zid(D, NG - 3 + q, NG - 1 + q3.j, (A.flat3 ? NG : NG - 1) + q3.k);
  const bool own = g < npair && lane >= 2 && q >= 2;
#pragma unroll 1
  for (int v = v0; v < (A.x1_split ? v0 + 1 : NV); v++) {
    const double *p = P + v * D.ntot + c;
    const double x0 = __ldg(p), x1 = __ldg(p + 1);
    double lo, hi;
    if (RECON == 1) {
      const WidePair p2 = wide_pair(wide_diff(x1 - x0), wide_diff(__ldg(p + 2) - x1));
      const u64 D13 = wide_D13(p2);
      const WideNum low = wide_q_low(p2, D13), mid = wide_q_mid(p2, D13);
      const unsigned all = 0xffffffffu;
      WidePair p0, p1;
      WideNum q0, q1;
      p1.a = __shfl_up_sync(all, p2.a, 1);
      p1.b = __shfl_up_sync(all, p2.b, 1);
      p1.x = __shfl_up_sync(all, p2.x, 1);
      q1.m = __shfl_up_sync(all, mid.m, 1);
      q1.x = __shfl_up_sync(all, mid.x, 1);
      p0.a = __shfl_up_sync(all, p2.a, 2);
      p0.b = __shfl_up_sync(all, p2.b, 2);
      p0.x = __shfl_up_sync(all, p2.x, 2);
      q0.m = __shfl_up_sync(all, low.m, 2);
      q0.x = __shfl_up_sync(all, low.x, 2);
      if (own) weno5_wide(x0, p0, p1, p2, q0, q1, wide_q_high(p2, D13), lo, hi);
    } else if (own) {
      const double d = mc_half_slope(x0 - __ldg(p - 1), x1 - x0);
      lo = x0 - d;
      hi = x0 + d;
    }
    if (own) {
      Lf[v * D.ntot + c] = lo;
      Rf[v * D.ntot + c] = hi;
    }
  }
}

// The two threads of a face: lanes 0..15 of a warp take the left states of 16
// faces, lanes 16..31 their right states.
__host__ __device__ inline long long n_face_threads(const Dims &D, int dir, int flat3) {
  int lo[3], ext[3];
  face_box(D, dir, flat3, lo, ext);
  return n_column_threads(16, ext[0], ext[1], ext[2]);
}
struct FaceLane {
  bool active, right;
  int i, j, k;
  long long c;  // zone above the face
};
template <int DIR>
__device__ __forceinline__ FaceLane face_lane(const Dims &D, int flat3, long long t) {
  int lo[3], ext[3];
  face_box(D, DIR, flat3, lo, ext);
  // a block's last warps may lie past the last column
  const long long n = n_column_threads(16, ext[0], ext[1], ext[2]);
  const Column q = column_of((t < n) ? t : t & 31, (int)(t & 15), 16, ext[0], ext[1], ext[2]);
  FaceLane L;
  L.active = q.active && t < n;
  L.right = (t & 16) != 0;
  L.i = lo[0] + q.i;
  L.j = lo[1] + q.j;
  L.k = lo[2] + q.k;
  L.c = zid(D, L.i, L.j, L.k);
  return L;
}

// The larger of two signal speeds; one that is not a number loses, as in fmax.
__device__ __forceinline__ double speed_max(double a, double b) {
  const s64 x = (s64)w_bits(a), y = (s64)w_bits(b), inf = 0x7ffll << 52;
  return (x > inf || x < 0) ? b : (y > inf || y < 0 || x > y) ? a : b;
}

// LLF flux of a face from its two states P, one per lane (face_lane): each lane
// forms its state and signal speed, takes the pair's larger speed ct, forms
// 1/2 sqrt(-g) (F +- ct U) and adds the other lane's for half of the variables.
// The states' and fluxes' dot products run in Wide numbers on the integer pipes
// (wide_face.cuh), the signal speeds (about 30 instructions) beside them on the
// FP64 unit, whose 241 instructions a face bound the former all-FP64 form (0.937 ms
// per launch on a 128^3 grid; 0.462 ms so).  Two lanes a face, so that a thread
// keeps one state's values and the warps are many; the FP64 unit and the ALU are
// each busy about 60% of the time.
// ELEC: the grid evolves electron entropies, whose flux weights it stores.
// Every thread of the block must call it.
template <int DIR, bool ELEC>
__device__ __forceinline__ void face_flux(const StepArgs &A, const FaceLane &L, const double P[NV],
                                          double *__restrict__ F) {
  const Dims &D = A.D;
  const int loc = (DIR == 0) ? LOC_FACE1 : (DIR == 1) ? LOC_FACE2 : LOC_CENT;
  const double *g = A.geom + (long long)loc * G_NCOMP * D.n2d + (long long)L.j * D.s[0] + L.i;
  const auto geo = [g, &D](int comp) { return __ldg(g + comp * D.n2d); };
  WideState s;
  if (A.clk->coupled)
    wide_state<false>(P, geo, s);
  else
    wide_state<true>(P, geo, s);
  const double bsq = w_to_double(s.bsq), ee = bsq + fma(A.gam, P[UU], P[RHO]);
  const double ut = w_to_double(s.ucon[0]), ud = w_to_double(s.ucon[DIR + 1]);
  const double own = mhd_cmax(fma(A.ggm1, P[UU], bsq), ee, ut, ud, geo(G_GCON + SY(0, 0)),
                              geo(G_GCON + SY(DIR + 1, DIR + 1)), geo(G_GCON + SY(0, DIR + 1)));
  // c_top = max(0, vmax_L, vmax_R, -vmin_L, -vmin_R): the larger root
  // magnitude of either side
  const double ct = speed_max(own, __shfl_xor_sync(0xffffffffu, own, 16));
  double out[NV];
  wide_flux(P, s, ee, A.gm1, DIR + 1, L.right ? -ct : ct, 0.5 * geo(G_GDET), out);
  // boundary flux fixes (fix_flux_body): no flux through the axis, no mass in
  // through an outflow boundary
  const bool axis = DIR == 1 && ((A.bc[1][0] == 2 && L.j == NG) ||
                                 (A.bc[1][1] == 2 && L.j == D.n[1] + NG));
  bool dry = false;
#pragma unroll
  for (int q = 0; q < NV / 2; q++) {
    const double keep = L.right ? out[q + NV / 2] : out[q];
    const double got = __shfl_xor_sync(0xffffffffu, L.right ? out[q] : out[q + NV / 2], 16);
    double f = axis ? 0.0 : keep + got;
    if (DIR == 0 && q == RHO && !L.right) {
      dry = (A.bc[0][0] == 1 && L.i == NG && less(0.0, f)) ||
            (A.bc[0][1] == 1 && L.i == D.n[0] + NG && less(f, 0.0));
      if (dry) f = 0.0;
    }
    if (L.active) F[(q + (L.right ? NV / 2 : 0)) * D.ntot + L.c] = f;
  }
  // the electron entropies' flux weights (LLF of rho u^d K, rho u^t K), none
  // where the mass flux is fixed to zero
  if (ELEC) {
    const bool none = axis || (DIR == 0 && __shfl_sync(0xffffffffu, dry, threadIdx.x & 15));
    if (L.active) A.elec_w[(2 * DIR + (L.right ? 1 : 0)) * D.ntot + L.c] = none ? 0.0 : out[RHO];
  }
  bool interior = L.active;
#pragma unroll
  for (int e = 0; e < 3; e++) {
    if (e == DIR) continue;
    const int q = (e == 0) ? L.i : (e == 1) ? L.j : L.k;
    interior = interior && (q >= NG) && (q < D.n[e] + NG);
  }
  warp_block_max(interior ? ct : 0.0, &A.clk->ctop_bits[DIR]);
}

// The face's left state is Rf of zone c-1, the right state Lf of zone c; every
// thread of the block must call it.
template <int DIR, bool ELEC = false>
__device__ __forceinline__ void face_body(const StepArgs &A, const double *__restrict__ Lf,
                                          const double *__restrict__ Rf, double *__restrict__ F,
                                          long long t) {
  const Dims &D = A.D;
  const FaceLane L = face_lane<DIR>(D, A.flat3, t);
  const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
  const double *p = L.right ? Lf + L.c : Rf + L.c - st;
  double P[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) P[v] = __ldg(p + v * D.ntot);
  face_flux<DIR, ELEC>(A, L, P, F);
}

// Flat X3: copy the k = NG layer of F1 and F2 to k = NG-1 and NG+1, and of
// F3 to k = NG+1 (one thread per (variable, i, j)).
__device__ __forceinline__ void replicate_body(const StepArgs &A, double *F1, double *F2, double *F3,
                                               long long t) {
  const Dims &D = A.D;
  if (t >= n_replicate(D)) return;
  const Idx3 q3 = unflatten(t, (int)D.n2d, NV);
  const long long c = q3.j * D.ntot + NG * D.n2d + q3.i;
  const double f1 = F1[c], f2 = F2[c], f3 = F3[c];
  F1[c - D.n2d] = f1;
  F1[c + D.n2d] = f1;
  F2[c - D.n2d] = f2;
  F2[c + D.n2d] = f2;
  F3[c + D.n2d] = f3;
}

__device__ __forceinline__ void reset_ctop_body(Clock *clk) {
  clk->ctop_bits[0] = clk->ctop_bits[1] = clk->ctop_bits[2] = 0ull;
}

// ---------------------------------------------------------------------------
// Time step: ndt_d = cfl dx_d / max ctop_d over directions with n_d > 1,
// dt = 1/sum(1/ndt_d), dt <= 1.3 dt_prev, last step lands on t_final.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void dt_body(const StepArgs &A) {
  Clock *c = A.clk;
  double inv = 0.0;
  for (int d = 0; d < 3; d++) {
    if (A.D.n[d] <= 1) continue;
    const double ct = __longlong_as_double((long long)c->ctop_bits[d]);
    if (ct > 0.0) {
      const double ndt = __ddiv_rn(A.cfl * A.dx[d], ct);
      inv = __dadd_rn(inv, __ddiv_rn(1.0, ndt));
    }
  }
  double dt = (inv > 0.0) ? __ddiv_rn(1.0, inv) : __longlong_as_double(0x7ff0000000000000ll);
  if (c->dt_prev > 0.0 && dt > 1.3 * c->dt_prev) dt = 1.3 * c->dt_prev;
  if (c->t_final > 0.0 && __dadd_rn(c->t, dt) > c->t_final) dt = __dadd_rn(c->t_final, -c->t);
  if (!isfinite(dt)) {  // every signal speed zero: no CFL step exists
    c->counters[3] += 1;
    dt = 0.0;
  }
  if (!(dt > 0.0)) dt = 0.0;
  c->dt = dt;
}

__device__ __forceinline__ void advance_body(const StepArgs &A) {
  Clock *c = A.clk;
  if (c->dt > 0.0 && isfinite(c->dt)) {
    c->t = __dadd_rn(c->t, c->dt);
    c->dt_prev = c->dt;
    c->steps += 1;
  }
}

// ---------------------------------------------------------------------------
// Boundary flux fixes and flux-CT
// ---------------------------------------------------------------------------
// FK1, FK2 (null without electrons): the electron entropy fluxes of X1 and
// X2 faces, zeroed with the polar fluxes and with a zeroed mass inflow.
__device__ __forceinline__ void fix_flux_body(const StepArgs &A, double *F1, double *F2,
                                              double *FK1, double *FK2, long long t) {
  const Dims &D = A.D;
  // polar faces: (i, k) over the extended ranges
  const long long np = (long long)(D.n[0] + 2) * (D.n[2] + 2);
  const long long nr = (long long)(D.n[1] + 2) * (D.n[2] + 2);
  if (t < np) {
    const int i = NG - 1 + (int)(t % (D.n[0] + 2));
    const int k = NG - 1 + (int)(t / (D.n[0] + 2));
    if (A.bc[1][0] == 2) {
      const long long c = zid(D, i, NG, k);
      for (int v = 0; v < NV; v++) F2[v * D.ntot + c] = 0.0;
      if (FK2) FK2[c] = FK2[D.ntot + c] = 0.0;
    }
    if (A.bc[1][1] == 2) {
      const long long c = zid(D, i, D.n[1] + NG, k);
      for (int v = 0; v < NV; v++) F2[v * D.ntot + c] = 0.0;
      if (FK2) FK2[c] = FK2[D.ntot + c] = 0.0;
    }
  }
  if (t < nr) {
    const int j = NG - 1 + (int)(t % (D.n[1] + 2));
    const int k = NG - 1 + (int)(t / (D.n[1] + 2));
    if (A.bc[0][0] == 1) {
      const long long c = zid(D, NG, j, k);
      double *f = F1 + RHO * D.ntot + c;
      if (*f > 0.0) {
        *f = 0.0;
        if (FK1) FK1[c] = FK1[D.ntot + c] = 0.0;
      }
    }
    if (A.bc[0][1] == 1) {
      const long long c = zid(D, D.n[0] + NG, j, k);
      double *f = F1 + RHO * D.ntot + c;
      if (*f < 0.0) {
        *f = 0.0;
        if (FK1) FK1[c] = FK1[D.ntot + c] = 0.0;
      }
    }
  }
}

// Edge EMFs, four times over (the factor goes to 1/dx in flux_ct_div and to the
// half in ct_body, exactly), over i, j, k in [NG, n+NG]:
// 4 e3 = F1[B2] + F1[B2](j-1) - F2[B1] - F2[B1](i-1), cyclic for e1, e2.
// flat3: on the layer k = NG alone, whose neighbours along X3 are itself.
__device__ __forceinline__ void emf_body(const StepArgs &A, const double *__restrict__ F1,
                                         const double *__restrict__ F2,
                                         const double *__restrict__ F3, double *__restrict__ emf,
                                         int flat3, long long t) {
  const Dims &D = A.D;
  const int e0 = D.n[0] + 1, e1 = D.n[1] + 1;
  if (t >= n_edge(D, flat3)) return;
  const Idx3 q3 = unflatten(t, e0, e1);
  const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
  const long long c = zid(D, i, j, k), N = D.ntot;
  const long long im = c - 1, jm = c - D.s[0], km = flat3 ? c : c - D.n2d;
  emf[2 * N + c] = F1[B2 * N + c] + F1[B2 * N + jm] - F2[B1 * N + c] - F2[B1 * N + im];
  emf[1 * N + c] = F3[B1 * N + c] + F3[B1 * N + im] - F1[B3 * N + c] - F1[B3 * N + km];
  emf[0 * N + c] = F2[B3 * N + c] + F2[B3 * N + km] - F3[B2 * N + c] - F3[B2 * N + jm];
}

// Induction fluxes from the EMFs on every face next to a zone (flux_ct_div takes
// their differences from the EMFs themselves; this is for callers who want F).
__device__ __forceinline__ void ct_body(const StepArgs &A, double *F1, double *F2, double *F3,
                                        const double *__restrict__ emf, long long t) {
  const Dims &D = A.D;
  const int e0 = D.n[0] + 1, e1 = D.n[1] + 1;
  if (t >= n_edge(D, 0)) return;
  const Idx3 q3 = unflatten(t, e0, e1);
  const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
  const long long c = zid(D, i, j, k), N = D.ntot;
  const double *E1 = emf, *E2 = emf + N, *E3 = emf + 2 * N;
  const bool in1 = i < D.n[0] + NG, in2 = j < D.n[1] + NG, in3 = k < D.n[2] + NG;
  if (in2 && in3) {  // X1 face
    F1[B1 * N + c] = 0.0;
    F1[B2 * N + c] = 0.125 * (E3[c] + E3[c + D.s[0]]);
    F1[B3 * N + c] = -0.125 * (E2[c] + E2[c + D.n2d]);
  }
  if (in1 && in3) {  // X2 face
    F2[B1 * N + c] = -0.125 * (E3[c] + E3[c + 1]);
    F2[B2 * N + c] = 0.0;
    F2[B3 * N + c] = 0.125 * (E1[c] + E1[c + D.n2d]);
  }
  if (in1 && in2) {  // X3 face
    F3[B1 * N + c] = 0.125 * (E2[c] + E2[c + 1]);
    F3[B2 * N + c] = -0.125 * (E1[c] + E1[c + D.s[0]]);
    F3[B3 * N + c] = 0.0;
  }
}

// ---------------------------------------------------------------------------
// Update + inversion + floors, one thread per interior zone.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void count_warp(bool pred, unsigned long long *ctr) {
  const unsigned m = __ballot_sync(0xffffffffu, pred);
  if (m && (threadIdx.x & 31) == 0) atomicAdd(ctr, (unsigned long long)__popc(m));
}

// S_nu = sqrt(-g) T^k_l Gamma^l_{nu k}
__device__ __forceinline__ void geo_source(const double T[4][4], double gdet,
                                           const double *__restrict__ conn, long long n2d,
                                           long long ij, double S[4]) {
#pragma unroll
  for (int nu = 0; nu < 4; nu++) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 4; k++)
#pragma unroll
      for (int l = 0; l < 4; l++) acc += T[k][l] * __ldg(conn + (l * 10 + SY(nu, k)) * n2d + ij);
    S[nu] = acc * gdet;
  }
}

// sqrt(-g)-weighted sum of a variable's flux differences over the zone at c (o = v
// ntot + c).  On a flat X3 both X3 faces are the same.
__device__ __forceinline__ double flux_div(const StepArgs &A, const double *__restrict__ F1,
                                           const double *__restrict__ F2,
                                           const double *__restrict__ F3, long long o) {
  double s = (F1[o + 1] - F1[o]) * A.idx[0];
  s = fma(F2[o + A.D.s[0]] - F2[o], A.idx[1], s);
  return A.flat3 ? s : fma(F3[o + A.D.n2d] - F3[o], A.idx[2], s);
}

// The same of the induction fluxes of flux-CT, straight from the EMFs: with each
// flux the mean of the two EMFs that bound its face (ct_body), B^1's through
// an X2 face is -(E3(i) + E3(i+1))/2, through an X3 face (E2(i) + E2(i+1))/2, and
// cyclically (B^d has no flux along d).  The four EMFs of one kind around the
// zone enter two such differences each, as p + q and p - q of their differences over
// the diagonals p = E(0,0) - E(1,1), q = E(1,0) - E(0,1).
__device__ __forceinline__ void flux_ct_div(const StepArgs &A, const double *__restrict__ emf,
                                            long long c, double div[3]) {
  const long long N = A.D.ntot, y = A.D.s[0], z = A.flat3 ? 0 : A.D.n2d;
  const double *E1 = emf + c, *E2 = emf + N + c, *E3 = emf + 2 * N + c;
  const double h1 = 0.125 * A.idx[0], h2 = 0.125 * A.idx[1], h3 = 0.125 * A.idx[2];
  const double p3 = E3[0] - E3[y + 1], q3 = E3[1] - E3[y];
  const double p2 = E2[0] - E2[z + 1], q2 = E2[z] - E2[1];
  const double p1 = E1[0] - E1[y + z], q1 = E1[y] - E1[z];
  // B^2 through X1 faces: E3(1,.) - E3(0,.); B^1 through X2 faces: E3(.,0) - E3(.,1)
  const double d21 = q3 - p3, d12 = q3 + p3;
  const double d31 = q2 + p2, d32 = q1 - p1;
  div[2] = fma(d32, h2, d31 * h1);
  if (A.flat3) {
    div[0] = d12 * h2;
    div[1] = d21 * h1;
  } else {
    const double d13 = q2 - p2, d23 = q1 + p1;  // through X3 faces
    div[0] = fma(d13, h3, d12 * h2);
    div[1] = fma(d23, h3, d21 * h1);
  }
}

// U(P), the stress-energy tensor, the Lorentz factor squared and b^2 of a state
// in FP64: metrics that couple X2.
static __device__ __noinline__ void tensor_fp64(const StepArgs &A, const double *__restrict__ Ps,
                                                long long c, long long ij, double U[NV],
                                                double T[4][4], double &g2, double &bsq) {
  Geo G;
  load_geo(A.geom, A.D.n2d, ij, G);
  double p[NV];
  for (int v = 0; v < NV; v++) p[v] = Ps[v * A.D.ntot + c];
  FState s;
  fluid_state(p, G, s);
  prim_flux(p, s, G, A.gam, 0, U);
  const double pg = (A.gam - 1.0) * p[UU];
  const double w = p[RHO] + p[UU] + pg + s.bsq;
  for (int m = 0; m < 4; m++) {
    for (int n = 0; n < 4; n++) T[m][n] = w * s.ucon[m] * s.ucov[n] - s.bcon[m] * s.bcov[n];
    T[m][m] += pg + 0.5 * s.bsq;
  }
  const double g = s.ucon[0] * G.alpha;
  g2 = g * g;
  bsq = s.bsq;
}

// The bounds of a zone that needs the Lorentz-factor cap.
static __device__ __noinline__ int floors_capped(const StepArgs &A, long long ij, double P[NV]) {
  Geo G;
  load_geo(A.geom, A.D.n2d, ij, G);
  return apply_floors(P, G, __ldg(A.floors + ij), __ldg(A.floors + A.D.n2d + ij), A.gk);
}
// The fluid-frame bounds of a zone whose b^2 and Lorentz factor are known.
__device__ __forceinline__ int floors_fluid(const StepArgs &A, long long ij, double P[NV],
                                            double bsq, double lorentz) {
  if (!less(FL_GAMMA, lorentz))
    return apply_floors_known(P, __ldg(A.floors + ij), __ldg(A.floors + A.D.n2d + ij), A.gk, bsq);
  double p[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) p[v] = P[v];
  const int ff = floors_capped(A, ij, p);
#pragma unroll
  for (int v = 0; v < NV; v++) P[v] = p[v];
  return ff;
}

// The drift-frame bounds in FP64: zones that need the Lorentz-factor cap, metrics
// that couple X2, sums that wide_invert gives no answer for.
static __device__ __noinline__ int floors_drift_fp64(const StepArgs &A, long long ij, double P[NV]) {
  Geo G;
  load_geo(A.geom, A.D.n2d, ij, G);
  return apply_floors_drift(P, G, __ldg(A.floors + ij), __ldg(A.floors + A.D.n2d + ij), A.gk);
}
// The drift-frame bounds (apply_floors_drift) of a zone whose b^2 and Lorentz
// factor are known, the sum with the parcel and its inversion in Wide numbers.
__device__ __forceinline__ int floors_drift(const StepArgs &A, long long ij, double P[NV],
                                            double bsq, double lorentz) {
  int ff = 0;
  if (!A.clk->coupled && !less(FL_GAMMA, lorentz)) {
    double Pf[NV];
#pragma unroll
    for (int v = 0; v < NV; v++) Pf[v] = P[v];
    ff = apply_floors_known(Pf, __ldg(A.floors + ij), __ldg(A.floors + A.D.n2d + ij), A.gk, bsq);
    if (!ff) return 0;
    const double *g = A.geom + ij;
    const long long n2d = A.D.n2d;
    const auto geo = [g, n2d](int comp) { return __ldg(g + comp * n2d); };
    double U[NV], pn[NV], guess, b, l;
    wide_drift_sum(P, geo, A.gam, Pf[RHO] - P[RHO], Pf[UU] - P[UU], FL_DRIFT_BSQ * Pf[RHO], Pf[RHO],
                   Pf[UU], U, guess);
    if (wide_invert<true>(U, geo, A.gk, guess, pn, b, l)) {
#pragma unroll
      for (int v = 0; v < NV; v++) P[v] = pn[v];
      return ff | FF_DRIFT | floors_fluid(A, ij, P, b, l);
    }
  }
  double p[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) p[v] = P[v];
  ff = floors_drift_fp64(A, ij, p);
#pragma unroll
  for (int v = 0; v < NV; v++) P[v] = p[v];
  return ff;
}

// The inversion in FP64 from the guess P_i: zones for which wide_invert gives
// no answer.
static __device__ __noinline__ int invert_fp64(const StepArgs &A, const double U[NV],
                                               const double *Pi, long long c, long long ij,
                                               double P[NV], double &bsq, double &lorentz) {
  Geo G;
  load_geo(A.geom, A.D.n2d, ij, G);
  double p[NV];
  for (int v = 0; v < NV; v++) p[v] = Pi[v * A.D.ntot + c];
  return invert_1dw(U, G, A.gk, p, P, bsq, lorentz);
}

// The update is two passes, so that each keeps its registers and its code in
// the SM's instruction cache: source_body forms U(P^n), the source and the
// inversion's guess W, invert_body the new conserved vector, its primitives and
// their bounds.  The states' products and the inversion run in Wide numbers
// (wide_update.cuh); the source's contraction (64 instructions) in the one pass
// and the flux divergence (60) in the other run on the FP64 unit beside them,
// whose 577 instructions a zone bound the former single pass of FP64 (per launch on
// a 128^3 grid 2.26 ms; 0.79 ms for both passes, 1.03 as one pass of Wide numbers
// with the source among them, which waited for spills and instructions).
//
// The predictor (PRED: P_s = P_i = P^n) keeps U(P^n) in Ucache for both stages.
// scratch ([8][ntot]): S_0 .. S_3 and the guess; b^2 of P_s (for electron grids);
// then, from invert_body, b^2 and the Lorentz factor of the result, where a later
// pass takes the bounds.
enum { SCR_GUESS = 4, SCR_BSQ_S, SCR_BSQ, SCR_LORENTZ };
template <bool PRED>
__device__ __forceinline__ void source_body(const StepArgs &A, const double *__restrict__ Ps,
                                            double *__restrict__ Ucache,
                                            double *__restrict__ scratch, long long t) {
  const Dims &D = A.D;
  if (t >= n_update(D)) return;
  const Column q3 = column_of(t, (int)(t & 31), 32, D.n[0], D.n[1], D.n[2]);
  if (!q3.active) return;
  const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
  const long long c = zid(D, i, j, k), N = D.ntot;
  const long long ij = (long long)j * D.s[0] + i;
  const double *g = A.geom + ij;
  const auto geo = [g, &D](int comp) { return __ldg(g + comp * D.n2d); };
  double p[NV], U[NV], T[4][4], S[4], g2, bsq;
#pragma unroll
  for (int v = 0; v < NV; v++) p[v] = __ldg(Ps + v * N + c);
  if (A.clk->coupled) {
    double Uc[NV], Tc[4][4], gc, bc;
    tensor_fp64(A, Ps, c, ij, Uc, Tc, gc, bc);
#pragma unroll
    for (int v = 0; v < NV; v++) U[v] = Uc[v];
#pragma unroll
    for (int m = 0; m < 4; m++)
#pragma unroll
      for (int n = 0; n < 4; n++) T[m][n] = Tc[m][n];
    g2 = gc;
    bsq = bc;
  } else {
    wide_tensor<true, PRED>(p, geo, A.gm1, U, T, g2, bsq);
  }
  const double gd = geo(G_GDET);
  if (PRED) {  // U^t has no field part: b^i u^t - b^t u^i = B^i
#pragma unroll
    for (int v = 0; v < NV; v++) Ucache[v * N + c] = (v < B1) ? U[v] : gd * p[v];
  }
  geo_source(T, gd, A.conn, D.n2d, ij, S);
#pragma unroll
  for (int n = 0; n < 4; n++) scratch[n * N + c] = S[n];
  scratch[SCR_GUESS * N + c] = fma(A.gam, p[UU], p[RHO]) * g2;
  if (A.elec) scratch[SCR_BSQ_S * N + c] = bsq;
}

// U(P^n) + dt' (S - div F), its inversion and the bounds; Pi: the guess of the
// FP64 iteration.  Every thread of the block must call it (warp counters).
__device__ __forceinline__ void invert_body(const StepArgs &A, const double *__restrict__ F1,
                                            const double *__restrict__ F2,
                                            const double *__restrict__ F3,
                                            const double *__restrict__ emf,
                                            const double *__restrict__ Ucache, double *scratch,
                                            double dtfac, const double *Pi, double *Pout, int *pflag, int *fflag,
                                            long long t) {
  const Dims &D = A.D;
  const double dt = A.clk->dt;
  if (!less(0.0, dt)) return;  // uniform across the grid: no warp divergence
  const double dtp = dtfac * dt;
  const bool in = t < n_update(D);
  const Column q3 = column_of(in ? t : t & 31, (int)(t & 31), 32, D.n[0], D.n[1], D.n[2]);
  const bool active = in && q3.active;
  int pf = 0, ff = 0;
  if (active) {
    const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
    const long long c = zid(D, i, j, k), N = D.ntot;
    const long long ij = (long long)j * D.s[0] + i;
    const double *g = A.geom + ij;
    const auto geo = [g, &D](int comp) { return __ldg(g + comp * D.n2d); };
    double Un[NV], pn[NV], bsq_n = 0.0, lor_n = 1.0, divB[3];
    flux_ct_div(A, emf, c, divB);
#pragma unroll
    for (int v = 0; v < NV; v++) {
      const long long o = v * N + c;
      const double div = (v < B1) ? flux_div(A, F1, F2, F3, o) : divB[v < B1 ? 0 : v - B1];
      const double u = __ldg(Ucache + o);
      // the source enters the energy and momentum rows only
      Un[v] = (v >= UU && v <= U3) ? fma(dtp, scratch[(v - UU) * N + c] - div, u)
                                   : fma(-dtp, div, u);
    }
    const double guess = scratch[SCR_GUESS * N + c];
    if (A.clk->coupled || !wide_invert<true>(Un, geo, A.gk, guess, pn, bsq_n, lor_n)) {
      double u[NV], p[NV], b = 0.0, l = 1.0;
#pragma unroll
      for (int v = 0; v < NV; v++) u[v] = Un[v];
      pf = invert_fp64(A, u, Pi, c, ij, p, b, l);
#pragma unroll
      for (int v = 0; v < NV; v++) pn[v] = p[v];
      bsq_n = b;
      lor_n = l;
    }
    if (A.floor_drift || A.elec) {  // the bounds are a later pass's
      scratch[SCR_BSQ * N + c] = bsq_n;
      scratch[SCR_LORENTZ * N + c] = lor_n;
    } else if (pf == PF_OK && A.floors_on) {
      ff = floors_fluid(A, ij, pn, bsq_n, lor_n);
    }
#pragma unroll
    for (int v = 0; v < NV; v++) Pout[v * N + c] = pn[v];
    pflag[c] = pf;
    fflag[c] = ff;
  }
  count_warp(active && pf != 0, &A.clk->counters[0]);
  count_warp(active && ff != 0, &A.clk->counters[1]);
}

// ---------------------------------------------------------------------------
// Drift-frame bounds of the zones whose inversion succeeded (the update
// leaves their bounds to this pass when A.floor_drift is set).  Every thread
// of the block must call it (warp counters).
// ---------------------------------------------------------------------------
__device__ __forceinline__ void floor_drift_body(const StepArgs &A, double *P,
                                                 const double *__restrict__ scratch,
                                                 const int *__restrict__ pflag, int *fflag,
                                                 long long t) {
  const Dims &D = A.D;
  if (!less(0.0, A.clk->dt)) return;
  const bool in = t < n_update(D);
  const Column q3 = column_of(in ? t : t & 31, (int)(t & 31), 32, D.n[0], D.n[1], D.n[2]);
  const bool active = in && q3.active;
  int ff = 0;
  if (active) {
    const int i = NG + q3.i, j = NG + q3.j, k = NG + q3.k;
    const long long c = zid(D, i, j, k), N = D.ntot;
    if (pflag[c] == 0) {
      double p[NV];
#pragma unroll
      for (int v = 0; v < NV; v++) p[v] = P[v * N + c];
      ff = floors_drift(A, (long long)j * D.s[0] + i, p, scratch[SCR_BSQ * N + c],
                        scratch[SCR_LORENTZ * N + c]);
      if (ff) {
#pragma unroll
        for (int v = 0; v < NV; v++) P[v * N + c] = p[v];
        fflag[c] = ff;
      }
    }
  }
  count_warp(active && ff != 0, &A.clk->counters[1]);
}

// ---------------------------------------------------------------------------
// Fixup: a failed zone takes the mean of rho, u, utilde over the non-failed
// interior zones of its 3x3x3 neighbourhood (B is kept), then the bounds.
// ---------------------------------------------------------------------------
// 1: a bound acted, 2: no valid neighbour
__device__ __forceinline__ int fixup_zone(const StepArgs &A, double *P, const int *__restrict__ pflag,
                                          int *fflag, int i, int j, int k) {
  const Dims &D = A.D;
  const long long c = zid(D, i, j, k), N = D.ntot;
  double sum[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  int cnt = 0;
  for (int dk = -1; dk <= 1; dk++)
    for (int dj = -1; dj <= 1; dj++)
      for (int di = -1; di <= 1; di++) {
        if (di == 0 && dj == 0 && dk == 0) continue;
        const int ii = i + di, jj = j + dj, kk = k + dk;
        if (ii < NG - A.xlo[0] || ii >= D.n[0] + NG + A.xhi[0] || jj < NG - A.xlo[1] ||
            jj >= D.n[1] + NG + A.xhi[1] || kk < NG - A.xlo[2] || kk >= D.n[2] + NG + A.xhi[2])
          continue;
        const long long nb = zid(D, ii, jj, kk);
        if (pflag[nb] != 0) continue;
#pragma unroll
        for (int v = 0; v < 5; v++) sum[v] += P[v * N + nb];
        cnt++;
      }
  if (cnt == 0) return 2;
  double p[NV];
#pragma unroll
  for (int v = 0; v < NV; v++) p[v] = P[v * N + c];
#pragma unroll
  for (int v = 0; v < 5; v++) p[v] = sum[v] / (double)cnt;
  int f = 0;
  if (A.floors_on) {
    const long long ij = (long long)j * D.s[0] + i;
    Geo G;
    load_geo(A.geom, D.n2d, ij, G);
    f = apply_floors(p, G, __ldg(A.floors + ij), __ldg(A.floors + D.n2d + ij), A.gk);
    if (f) fflag[c] |= f;
  }
#pragma unroll
  for (int v = 0; v < NV; v++) P[v * N + c] = p[v];
  return f != 0;
}

// A thread looks at the failure flags of FIXUP_ZONES zones along X3, loaded together:
// next to no zone fails, and with a zone a thread the passes over the flags waited
// for them one wave after another (35 us a launch on a 128^3 grid, 14 so).  The
// failed ones, which come in clusters (an axisymmetric state fails along all of X3), are
// listed in shared memory and dealt out to the block's threads.
constexpr int FIXUP_ZONES = 8;
__host__ __device__ inline long long n_fixup(const Dims &D) {
  return (long long)D.n[0] * D.n[1] * ((D.n[2] + FIXUP_ZONES - 1) / FIXUP_ZONES);
}
// Calls zone(i, j, k), whose result's bits 0 and 1 are counted, for each failed zone of
// the block's threads.  Every thread of the block must call it.
template <class ZoneFn>
__device__ __forceinline__ void for_failed_zones(const StepArgs &A, const int *__restrict__ pflag,
                                                 long long t, const ZoneFn &zone) {
  __shared__ unsigned short list[BS_MAX * FIXUP_ZONES];
  __shared__ unsigned count;
  const Dims &D = A.D;
  if (threadIdx.x == 0) count = 0;
  u32 bad = 0;
  if (t < n_fixup(D)) {
    const Idx3 q3 = unflatten(t, D.n[0], D.n[1]);
    const int k = NG + FIXUP_ZONES * q3.k;
    const long long c = zid(D, NG + q3.i, NG + q3.j, k);
#pragma unroll
    for (int m = 0; m < FIXUP_ZONES; m++)
      if (k + m < D.n[2] + NG) bad |= (pflag[c + m * D.n2d] != 0 ? 1u : 0u) << m;
  }
  if (!__syncthreads_or(bad != 0)) return;
  if (bad) {
    unsigned at = atomicAdd(&count, (unsigned)__popc(bad));
    for (; bad; bad &= bad - 1)
      list[at++] = (unsigned short)(threadIdx.x * FIXUP_ZONES + __ffs((int)bad) - 1);
  }
  __syncthreads();
  const unsigned n = count;
  for (unsigned e = threadIdx.x; e < n; e += blockDim.x) {
    const Idx3 q3 = unflatten(t - threadIdx.x + list[e] / FIXUP_ZONES, D.n[0], D.n[1]);
    const int f = zone(NG + q3.i, NG + q3.j, NG + FIXUP_ZONES * q3.k + list[e] % FIXUP_ZONES);
    if (f & 1) atomicAdd(&A.clk->counters[1], 1ull);
    if (f & 2) atomicAdd(&A.clk->counters[2], 1ull);
  }
}
__device__ __forceinline__ void fixup_body(const StepArgs &A, double *P, const int *__restrict__ pflag,
                                           int *fflag, long long t) {
  if (!less(0.0, A.clk->dt)) return;
  for_failed_zones(A, pflag, t, [&](int i, int j, int k) {
    return fixup_zone(A, P, pflag, fflag, i, j, k);
  });
}

}  // namespace grmhd
