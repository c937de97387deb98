// clot_eta.cu -- K2: the virtual-substance solve of App. A, Eq. eta,
//     (I - (L_eta^2 / 4) lap_h) eta = theta_B,   zero-flux boundaries,
// by conjugate gradients in one persistent cooperative launch, on meshes whose
// extents or coupling the direct solver (clot_eta_dct.cu) does not take.  Vectors are
// FP32; every dot product and norm is accumulated in FP64 and reduced in a
// fixed order, so all blocks see bit-identical scalars and the iteration is
// deterministic.  The solve is warm-started from the eta passed in and stops
// when max|r| <= max(tol * max|theta_B|, atol); since the operator is an
// M-matrix with unit row sums, max|eta - eta_exact| <= max|r|.
//
// Blocks synchronise through a grid barrier whose waits are bounded
// (clot_eta_ops.cuh).
//
// A predicted eta (from the fused step) that misses the stopping rule is first
// corrected on a box.  Its residual r is large only where theta_B changed in a
// way the linear extrapolation did not follow -- around the clot -- and the
// correction d of A d = r decays away from there like exp(-mu n) per cell along
// an axis, cosh(mu) = 1 + 1 / (2 c_a) (the 1D Green's function of I - c_a lap_h).
// So CG runs on the bounding box of the cells with |r| > stop / (2 (1 + c)),
// c the largest c_a, widened by ln(2 c_a max|r| / stop) / mu_a cells per axis,
// with d = 0 outside, until its residual meets the stopping rule.  Then the
// true residual theta_B - A eta is recomputed on the layer of cells around the
// box, where the cut-off correction leaves its mark; every cell further out
// keeps the residual the fused step computed, below stop / 2.  If the layer
// also meets the rule the solve is done; if not, the residual is recomputed
// everywhere and CG continues on the whole mesh.  Either way the rule holds at
// exit in the same sense as without the box (the iteration's residual where
// CG ran, the computed residual elsewhere).
#include "clot_eta_cg.cuh"

namespace clot {

__global__ void __launch_bounds__(ETA_BLOCK, 1) eta_cg_kernel(const __grid_constant__ EtaArgs a) {
  const bool v4 = (a.g.nx & 3) == 0 && (a.g.pitch & 3) == 0 && al16(a.c) && al16(a.eta) && al16(a.r) && al16(a.p) &&
                  al16(a.q) && al16(a.p2);
  Team T{(int)gridDim.x, 0u, 0, true};
  EtaOut o;
  float pr = 0.0f, pb = 0.0f;
  double s_rr = 0.0;
  float s_rmax, s_bmax;
  bool ok = true;
  if (a.predicted) {
    if (prediction_accepted(a, pr, pb)) return;
    s_rmax = pr;
    s_bmax = pb;
  } else {
    ok = residual_reduce<ETA_BLOCK>(a, T, v4, s_rr, s_bmax, s_rmax);
  }
  if (ok) ok = eta_iterate<ETA_BLOCK>(a, T, v4, a.predicted != 0, s_rr, s_rmax, s_bmax, o);
  eta_note(a, o, ok);
  team_leave(a);
}

int eta_sms() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 152;
  return sms;
}

int eta_max_grid(int* grid_out) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return -1;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return -1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, eta_cg_kernel, ETA_BLOCK, 0) != cudaSuccess)
    return -1;
  *grid_out = sms * (per_sm < 1 ? 1 : per_sm);
  return 0;
}

cudaError_t launch_eta_solve(const EtaArgs& a, int grid, cudaStream_t s) {
  EtaArgs copy = a;
  void* args[] = {&copy};
  return cudaLaunchCooperativeKernel((const void*)eta_cg_kernel, dim3(grid), dim3(ETA_BLOCK), args, 0, s);
}

}  // namespace clot
