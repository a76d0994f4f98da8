// Angular-flux prefactor of one side of the angle grid in one column
// (Eq. flux_angle): len (V . nu) n_0 with V . nu = -nu_i omega^ihat_{AB} n^A
// n^B at the side's midpoint.  Shared by the kernel that tabulates it per
// column (sides.cu) and by the kernels that compute it themselves where
// there is no table; every rounding is written out (fused or not), so that
// both give the same bits.
#pragma once

#include "rad_internal.h"

namespace rad {

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Prefactor of the side with geometry eg (edge_geo row) in the orientation
// from the side's cell p to its cell q, and whether p is the upwind cell.
template <typename R, typename Col>
__device__ __forceinline__ R side_prefactor(const Col &cg, const double *eg, bool &upp) {
  const R x = (R)eg[0], y = (R)eg[1], z = (R)eg[2], len = (R)eg[6];
  const R pr[10] = {R(1),         x,            y,            z,            mul_rn(x, x),
                    mul_rn(x, y), mul_rn(x, z), mul_rn(y, y), mul_rn(y, z), mul_rn(z, z)};
  R q[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    q[c] = (R)cg.K[c][0];
#pragma unroll
    for (int p = 1; p < 10; ++p) q[c] = fma_rn((R)cg.K[c][p], pr[p], q[c]);
  }
  const R sp = -fma_rn((R)eg[5], q[2], fma_rn((R)eg[3], q[0], mul_rn((R)eg[4], q[1])));   // V . nu
  const R n0 = fma_rn((R)cg.M[0][3], z, fma_rn((R)cg.M[0][2], y, fma_rn((R)cg.M[0][1], x, (R)cg.M[0][0])));
  upp = sp >= R(0);
  return mul_rn(mul_rn(len, sp), n0);
}

// FP64 prefactor n^d n_0 of a face for a direction, and whether n^d < 0 (the
// upwind cell is the upper one).
template <typename Face>
__device__ __forceinline__ double face_nd_n0(const Face &F, double x, double y, double z, bool &upR) {
  const double na = fma_rn(F.ea[3], z, fma_rn(F.ea[2], y, fma_rn(F.ea[1], x, F.ea[0])));
  upR = na < 0.0;
  return mul_rn(na, fma_rn(F.m0[3], z, fma_rn(F.m0[2], y, fma_rn(F.m0[1], x, F.m0[0]))));
}

// v per solid angle of bin n: a quotient in FP32, a product with the
// tabulated reciprocal in FP64 (a division costs ten operations of the FP64
// pipe).
__device__ __forceinline__ float per_solid_angle(float v, const double *dOmega, const double *, int n) {
  return __fdiv_rn(v, (float)dOmega[n]);
}
__device__ __forceinline__ double per_solid_angle(double v, const double *, const double *rdO, int n) {
  return __dmul_rn(v, rdO[n]);
}

}  // namespace rad
