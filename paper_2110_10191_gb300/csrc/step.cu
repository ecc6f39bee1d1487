// step.cu -- the single-grid kernels of the allocation-free flux entry
// point (noalloc.cu): fused reconstruction + LLF face fluxes, the
// signal-speed reset, the boundary flux fixes and flux-CT; and the
// interior <-> ghost layout copies.  The step itself runs the plan kernels
// (plan.cu) on the same per-thread bodies (step_bodies.cuh).
#include "grmhd_dev.cuh"
#include "grmhd_impl.h"
#include "step_bodies.cuh"

namespace grmhd {

__device__ __forceinline__ long long gtid() { return blockIdx.x * (long long)blockDim.x + threadIdx.x; }

static unsigned nblk(long long n) { return (unsigned)((n + BS - 1) / BS); }

// ---------------------------------------------------------------------------
// Fused face fluxes (reconstruction and LLF in one pass per face; used by
// the allocation-free flux entry point, which has no room for the face-value
// scratch of the split stage).  Face box for direction d: d-index NG .. n_d+NG,
// transverse NG-1 .. n_e+NG.
// ---------------------------------------------------------------------------
template <int DIR, int RECON>
__global__ void __launch_bounds__(BS) k_flux(StepArgs A, const double *__restrict__ P,
                                             double *__restrict__ F) {
  const Dims &D = A.D;
  const FaceLane L = face_lane<DIR>(D, 0, gtid());
  const long long st = (DIR == 0) ? 1 : (DIR == 1) ? D.s[0] : D.n2d;
  // the lane's state: the high face of the zone below, or the low face of the
  // zone above, whose mirrored stencil gives it as a high face
  const long long up = L.right ? -st : st;
  const double *p = P + (L.right ? L.c : L.c - st);
  double S[NV];
#pragma unroll 1
  for (int v = 0; v < NV; v++, p += D.ntot) {
    const double x = __ldg(p), xm = __ldg(p - up), xp = __ldg(p + up);
    if (RECON == 1) {
      double other;
      weno5_wide_pair(__ldg(p - 2 * up), xm, x, xp, __ldg(p + 2 * up), other, S[v]);
    } else {
      S[v] = x + mc_half_slope(x - xm, xp - x);
    }
  }
  face_flux<DIR, false>(A, L, S, F);
}

template <int DIR>
static void launch_flux_dir(const StepArgs &A, const double *P, double *F, cudaStream_t st) {
  const unsigned nb = nblk(n_face_threads(A.D, DIR, 0));
  if (A.recon == 1)
    k_flux<DIR, 1><<<nb, BS, 0, st>>>(A, P, F);
  else
    k_flux<DIR, 0><<<nb, BS, 0, st>>>(A, P, F);
}

void launch_fluxes(const StepArgs &A, const double *P, double *F[3], cudaStream_t st) {
  launch_flux_dir<0>(A, P, F[0], st);
  launch_flux_dir<1>(A, P, F[1], st);
  launch_flux_dir<2>(A, P, F[2], st);
}

// (the entry point builds its own metric, which does not couple X2)
__global__ void k_reset_ctop(Clock *clk) {
  reset_ctop_body(clk);
  clk->coupled = 0;
}

void launch_ctop_reset(const StepArgs &A, cudaStream_t st) { k_reset_ctop<<<1, 1, 0, st>>>(A.clk); }

// ---------------------------------------------------------------------------
// Flux-CT
// ---------------------------------------------------------------------------
__global__ void k_emf(StepArgs A, const double *__restrict__ F1, const double *__restrict__ F2,
                      const double *__restrict__ F3, double *__restrict__ emf) {
  emf_body(A, F1, F2, F3, emf, 0, gtid());
}

__global__ void k_ct(StepArgs A, double *F1, double *F2, double *F3, const double *__restrict__ emf) {
  ct_body(A, F1, F2, F3, emf, gtid());
}

void launch_ct(const StepArgs &A, double *F[3], double *emf, cudaStream_t st) {
  const Dims &D = A.D;
  k_emf<<<nblk(n_edge(D, 0)), BS, 0, st>>>(A, F[0], F[1], F[2], emf);
  k_ct<<<nblk(n_edge(D, 0)), BS, 0, st>>>(A, F[0], F[1], F[2], emf);
}

// ---------------------------------------------------------------------------
// Interior <-> ghost layout copies
// ---------------------------------------------------------------------------
__global__ void k_pack(Dims D, const double *__restrict__ src, double *__restrict__ dst,
                       int to_ghost, int nvar) {
  const long long nz = (long long)D.n[0] * D.n[1] * D.n[2];
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t >= nz * nvar) return;
  const long long v = t / nz, r = t % nz;
  const int i = (int)(r % D.n[0]);
  const int j = (int)((r / D.n[0]) % D.n[1]);
  const int k = (int)(r / ((long long)D.n[0] * D.n[1]));
  const long long g = v * D.ntot + zid(D, i + NG, j + NG, k + NG);
  if (to_ghost)
    dst[g] = src[t];
  else
    dst[t] = src[g];
}

void launch_pack(const Dims &D, const double *src, double *dst, int to_ghost, cudaStream_t st,
                 int nvar) {
  const long long n = (long long)D.n[0] * D.n[1] * D.n[2] * nvar;
  k_pack<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(D, src, dst, to_ghost, nvar);
}

}  // namespace grmhd
