// Frequency fluxes of multigroup transport (Sec. 2.2, Eq.
// radiation_integral_frequency): per cell, bin and group edge nu_f,
//   F_f = n^nu n_0 I_nu = nu_f s n_0 I_up / dnu_up,   s = n^nu / nu = -omega^0hat_{AB} n^A n^B,
// donor cell in frequency (the lower group where s > 0, the upper one where
// s < 0); the end edges let radiation out of the resolved range and none in,
// and an edge at nu = 0 or nu = infinity carries nothing.  The kernel writes
// each group's divergence F_{g+1} - F_g, which the stage kernel adds to the
// spatial and angular divergences of that group before the stage update.
//
// One CTA per column and chunk of x3 cells; each thread owns bins, keeps
// their frequency symbol for the chunk, and walks the groups of each cell,
// carrying the flux of the previous edge, so every intensity is read once and
// every divergence written once (coalesced rows of n_ap elements).  The
// widths and edge frequencies come in the working precision from a table of
// the context: forming them per bin took five operations of the FP64 pipe per
// bin and group, which bound the kernel (48 x 32 x 30 cells x 92 bins x 6
// groups FP32: 0.220 ms against 0.031 ms for its bytes).
#include <cmath>

#include "rad_internal.h"

namespace rad {

namespace {

constexpr int kFreqChunk = 8;      // x3 cells per CTA

// nu[f]: edge frequency, 0 for an edge that carries nothing (0 or infinity);
// dnu[g]: group width (infinite for a group reaching infinity, whose mean is 0)
template <typename R, typename Col>
__global__ void k_freq_div(const R *__restrict__ I, R *__restrict__ D, const Col *__restrict__ cols,
                           const double *__restrict__ dir, const R *__restrict__ nu, const R *__restrict__ dnu,
                           int ngroup, int nang, int nap, int ncol, int n3, size_t gstride) {
  const int nchunk = (n3 + kFreqChunk - 1) / kFreqChunk;
  const int col = blockIdx.x / nchunk, k0 = blockIdx.x % nchunk * kFreqChunk, k1 = min(n3, k0 + kFreqChunk);
  const Col &cg = cols[col];
  for (int n = threadIdx.x; n < nap; n += blockDim.x) {
    R s = R(0), sn0 = R(0);
    if (n < nang) {
      const R x = (R)dir[3 * n], y = (R)dir[3 * n + 1], z = (R)dir[3 * n + 2];
      const R pr[10] = {R(1), x, y, z, x * x, x * y, x * z, y * y, y * z, z * z};
      R q0 = R(0);
#pragma unroll
      for (int p = 0; p < 10; ++p) q0 += (R)cg.K0[p] * pr[p];
      s = -q0;                                                     // n^nu / nu
      const R n0 = (R)cg.M[0][0] + (R)cg.M[0][1] * x + (R)cg.M[0][2] * y + (R)cg.M[0][3] * z;
      sn0 = s * n0;
    }
    for (int k = k0; k < k1; ++k) {
      const size_t off = ((size_t)k * ncol + col) * nap + n;
      if (n >= nang) {
        for (int g = 0; g < ngroup; ++g) D[g * gstride + off] = R(0);
        continue;
      }
      // mean specific intensity of group g (0 for a group reaching infinity)
      auto mean = [&](int g) -> R {
        const R d = dnu[g];
        return isinf(d) ? R(0) : I[g * gstride + off] / d;
      };
      auto flux = [&](int f, R below, R above) -> R {
        const R v = nu[f];
        return v == R(0) ? R(0) : v * sn0 * (s > R(0) ? below : above);
      };
      R m_hi = mean(0);
      R F = flux(0, R(0), m_hi);
#pragma unroll 4
      for (int g = 0; g < ngroup; ++g) {
        const R m_lo = m_hi;
        m_hi = g + 1 < ngroup ? mean(g + 1) : R(0);
        const R Fn = flux(g + 1, m_lo, m_hi);
        D[g * gstride + off] = Fn - F;
        F = Fn;
      }
    }
  }
}

}  // namespace

int launch_freq_div(rad_ctx *ctx, const void *I, void *D, int precision, std::string &err) {
  const DevGeom &G = ctx->geom;
  const int ncol = G.n[0] * G.n[1], n3 = G.n[2], ng = ctx->n_groups;
  const size_t gstride = (size_t)ncol * n3 * ctx->ang.n_ap;
  const int threads = std::min(256, (ctx->ang.n_ap + 31) / 32 * 32);
  const unsigned grid = (unsigned)((long long)ncol * ((n3 + kFreqChunk - 1) / kFreqChunk));
  const double *t64 = ctx->grp_tab;
  const float *t32 = (const float *)(ctx->grp_tab + 2 * ng + 1);
  if (precision == RAD_F32)
    k_freq_div<float, ColGeoF><<<grid, threads, 0, ctx->stream>>>((const float *)I, (float *)D, G.colsF, ctx->dang.dir,
                                                                  t32, t32 + ng + 1, ng, ctx->ang.n_ang,
                                                                  ctx->ang.n_ap, ncol, n3, gstride);
  else
    k_freq_div<double, ColGeo><<<grid, threads, 0, ctx->stream>>>((const double *)I, (double *)D, G.cols, ctx->dang.dir,
                                                                  t64, t64 + ng + 1, ng, ctx->ang.n_ang,
                                                                  ctx->ang.n_ap, ncol, n3, gstride);
  const cudaError_t ce = cudaGetLastError();
  if (ce != cudaSuccess) {
    err = std::string("frequency flux launch failed: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  return RAD_OK;
}

}  // namespace rad
