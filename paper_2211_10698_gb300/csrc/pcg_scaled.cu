// The symmetrically Jacobi-scaled pressure Poisson system (Eq. pm_poisson) that the FP64 conjugate
// gradients of pcg_fused.cu, pcg_cluster.cu and pcg_batch.cu solve.
//
// With D the diagonal of K, Jacobi-preconditioned CG on K x = b and plain CG on
//     K~ x~ = b~,   K~ = D^-1/2 K D^-1/2,   x~ = D^1/2 x,   b~ = D^-1/2 b
// produce the same iterates in exact arithmetic (x = D^-1/2 x~ at every step), so the method is
// the Jacobi-PCG of the pressure step.  The scaled form saves FP64 work on a part whose FP64
// pipe is narrow: K~ has a unit diagonal, the preconditioned residual is the residual itself,
// and on cells whose four neighbours are uncut the row of K~ is one constant stencil
// x~_c - ax (x~_W + x~_E) - ay (x~_S + x~_N).  Per cell and iteration that leaves 4 FMA in the
// vector updates, 4 in the stencil and 2 in the dot products.
//
// The recurrences are the single-reduction arrangement of Chronopoulos and Gear: with w = K~ r
// and s = K~ p carried along, one grid reduction per iteration yields gamma = (r, r),
// delta = (w, r) and the convergence norm ||r_K||^2 = ||D^1/2 r~||^2 of the unscaled residual,
// so the stopping test ||r|| <= tol ||b|| is the one of the unscaled system.
//
// This file sets the scaling up; the iterations are in pcg_fused.cu (one barrier per iteration),
// pcg_cluster.cu (one thread-block cluster) and pcg_batch.cu (many cases in one launch).
#include "pcg_common.cuh"

namespace ccm {

namespace {

// Set-up: sqrt(d), 1/sqrt(d), the scaled face coefficients and the scaled row kinds.
// d is the diagonal of K on active cells, 1 on inactive cells (identity rows) and 0 outside
// the domain, where every iterate is zero; 1/sqrt(d) is taken as 0 there so that faces to
// ghost cells get a zero scaled coefficient.
__global__ void k_scaling(Geom g, CoefPtrs o) {
  const int i = (int)(blockIdx.x * blockDim.x + threadIdx.x) - 1;
  const int j = (int)(blockIdx.y * blockDim.y + threadIdx.y) - 1;
  if (i > g.nx + 1 || j > g.ny + 1) return;
  const size_t k = g.idx(i, j);
  auto isd_at = [&](size_t q) {
    const double d = o.diagk[q];
    return d > 0.0 ? 1.0 / sqrt(d) : 0.0;
  };
  const double d = o.diagk[k];
  const double sd = d > 0.0 ? sqrt(d) : 0.0;
  const double isd = isd_at(k);
  o.sdk[k] = sd;
  o.isdk[k] = isd;
  o.isdk32[k] = (float)isd;
  const double cus = i >= 0 ? o.cu[k] * isd * isd_at(k - 1) : 0.0;
  const double cvs = j >= 0 ? o.cv[k] * isd * isd_at(k - g.pitch) : 0.0;
  o.cus[k] = cus;
  o.cvs[k] = cvs;
  o.cus32[k] = (float)cus;
  o.cvs32[k] = (float)cvs;
  int8_t ks = 0;
  if (i >= 0 && i < g.nx && j >= 0 && j < g.ny && o.kind[k] != 0) {
    ks = 2;
    if (o.kind[k] == 1) {
      // uncut row; the scaled row is the constant stencil when every in-domain neighbour has
      // the uncut diagonal too (ghost neighbours hold zero in every iterate)
      const double cx = g.hy / g.hx, cy = g.hx / g.hy, dreg = 2.0 * (cx + cy), e = 1e-14 * dreg;
      bool uni = true;
      if (i > 0) uni = uni && fabs(o.diagk[k - 1] - dreg) <= e;
      if (i < g.nx - 1) uni = uni && fabs(o.diagk[k + 1] - dreg) <= e;
      if (j > 0) uni = uni && fabs(o.diagk[k - g.pitch] - dreg) <= e;
      if (j < g.ny - 1) uni = uni && fabs(o.diagk[k + g.pitch] - dreg) <= e;
      if (uni) ks = 1;
    }
  }
  o.kinds[k] = ks;
  if (ks == 2) {
    const double cx = g.hy / g.hx, cy = g.hx / g.hy, dreg = 2.0 * (cx + cy);
    const float ax = (float)(cx / dreg), ay = (float)(cy / dreg);
    // (the E and N neighbours form their W and S faces like this)
    if ((float)cus == ax && (float)cvs == ay && (float)(o.cu[k + 1] * isd_at(k + 1) * isd) == ax &&
        (float)(o.cv[k + g.pitch] * isd_at(k + g.pitch) * isd) == ay)
      ks = 3;
  }
  o.kindq[k] = ks;
}

}  // namespace

void launch_scaling(const Geom& g, const CoefPtrs& o, cudaStream_t st) {
  const dim3 b(32, 8);
  const dim3 grid((g.nx + 3 + b.x - 1) / b.x, (g.ny + 3 + b.y - 1) / b.y);
  k_scaling<<<grid, b, 0, st>>>(g, o);
}

}  // namespace ccm
