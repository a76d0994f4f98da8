// Table of the angular-flux prefactors of every (column, bin, side).
//
// The prefactor of a side is a quadratic form in its direction with the
// column's rotation coefficients: about 45 operations, six sides per bin.
// The stage kernels used to form it per CTA, i.e. once per column and chunk
// of x3 cells and stage: in a 2D grid (one cell per CTA) that is 270
// operations per bin beside about 100 of the update itself, on the FP64 pipe
// of the FP64 kernels.  It depends on the metric and the angle grid only, so
// it is laid out once per context and precision, in the order the consumer
// threads read it (bin fastest), and read back as one coalesced row per slot.
// Per rad_step: Kerr-Schild 128 x 64 x 64 x 362 bins FP32 6.72 -> 5.15 ms
// (192 x 96 x 96 x 642: 43.5 -> 32.3), 61 x 37 x 34 x 92 FP64 7.09 -> 5.69 ms,
// 256 x 128 x 162 FP64 15.4 -> 5.0 ms.  Building it takes about as long as
// one stage gains by it.
#include <algorithm>

#include "sides.cuh"

namespace rad {

namespace {

// One CTA per column; each thread strides over the bins of the six slots.
template <typename R, typename Col>
__global__ void k_side_table(const Col *__restrict__ cols, int nang, int nap, const int *__restrict__ slot_nbr,
                             const int *__restrict__ slot_edge, const int *__restrict__ edge_pq,
                             const double *__restrict__ edge_geo, const double *__restrict__ dOmega,
                             const double *__restrict__ rdO, R *__restrict__ P, unsigned char *__restrict__ up) {
  const size_t col = blockIdx.x;
  const Col &cg = cols[col];
  for (int n = threadIdx.x; n < nap; n += blockDim.x) {
    unsigned mask = 0;
    R self = R(0);
    for (int s = 0; s < kMaxSlots; ++s) {
      R v = R(0);
      if (n < nang && slot_nbr[6 * n + s] >= 0) {
        const int e = slot_edge[6 * n + s];
        bool upp;
        const R c = side_prefactor<R>(cg, edge_geo + 8 * e, upp);
        const bool isp = edge_pq[2 * e] == n, upn = upp == isp;
        v = isp ? c : -c;
        if (upn) self += v;
        v = per_solid_angle(v, dOmega, rdO, n);
        mask |= (upn ? 1u : 0u) << s;
      }
      P[(col * kSideRows + s) * nap + n] = v;
    }
    P[(col * kSideRows + kMaxSlots) * nap + n] = n < nang ? per_solid_angle(self, dOmega, rdO, n) : R(0);
    up[col * nap + n] = (unsigned char)mask;
  }
}

}  // namespace

// The table's bound: 4 GiB per precision (a 2D grid of 460,000 columns with
// 162 bins in FP64).  Beyond it, or when the allocation fails, or while the
// stream is being captured, the kernels form the prefactors as they go.
constexpr size_t kSideTableMax = (size_t)4 << 30;

void ensure_side_table(rad_ctx *ctx, int precision) {
  DevGeom &G = ctx->geom;
  const int ip = precision == RAD_F32 ? 1 : 0;
  if (G.kind == RAD_MINK_CART || G.side_P[ip]) return;
  const size_t ncol = (size_t)G.n[0] * G.n[1], nap = (size_t)ctx->ang.n_ap;
  const size_t bytes = ncol * nap * kSideRows * (ip ? 4 : 8);
  if (bytes > kSideTableMax) return;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  void *P = nullptr;
  unsigned char *up = nullptr;
  if (cudaMalloc(&P, bytes) != cudaSuccess || cudaMalloc(&up, ncol * nap) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(P);
    return;
  }
  const int threads = std::min(256, (int)(nap + 31) / 32 * 32);
  if (ip)
    k_side_table<float, ColGeoF><<<(unsigned)ncol, threads, 0, ctx->stream>>>(
        G.colsF, ctx->ang.n_ang, (int)nap, ctx->dang.slot_nbr, ctx->dang.slot_edge, ctx->dang.edge_pq,
        ctx->dang.edge_geo, ctx->dang.dOmega, ctx->dang.rdO, (float *)P, up);
  else
    k_side_table<double, ColGeo><<<(unsigned)ncol, threads, 0, ctx->stream>>>(
        G.cols, ctx->ang.n_ang, (int)nap, ctx->dang.slot_nbr, ctx->dang.slot_edge, ctx->dang.edge_pq,
        ctx->dang.edge_geo, ctx->dang.dOmega, ctx->dang.rdO, (double *)P, up);
  if (cudaGetLastError() != cudaSuccess) {
    cudaFree(P);
    cudaFree(up);
    return;
  }
  G.side_P[ip] = P;
  G.side_up[ip] = up;
}

}  // namespace rad
