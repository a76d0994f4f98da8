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
// Step and moments: Kerr-Schild 128 x 64 x 64 x 362 bins FP32 7.01 -> 5.45 ms
// (192 x 96 x 96 x 642: 45.5 -> 34.2), 61 x 37 x 34 x 92 FP64 7.09 -> 5.69 ms,
// 256 x 128 x 162 FP64 gradient over two steps 117.8 -> 47.3.  Building it takes about as long as
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

// One CTA per face; FP64 prefactors n^d n_0 of the spatial fluxes (the stage
// and adjoint kernels' operations, so that they give the same bits with and without).
__global__ void k_face_table(const FaceGeo *__restrict__ faces, int nang, int nap, const double *__restrict__ dir,
                             double *__restrict__ c, unsigned char *__restrict__ up) {
  const size_t f = blockIdx.x;
  const FaceGeo &F = faces[f];
  for (int n = threadIdx.x; n < nap; n += blockDim.x) {
    double v = 0.0;
    bool u = false;
    if (n < nang) v = face_nd_n0(F, dir[3 * n], dir[3 * n + 1], dir[3 * n + 2], u);
    c[f * nap + n] = v;
    up[f * nap + n] = u;
  }
}

}  // namespace

// The tables' bound: 4 GiB per precision, side and face tables and their flags
// together (in FP64 a 2D grid of 350,000 columns with 162 bins).  Face tables
// that do not fit beside the side table are left out.  Beyond the bound, or
// when the allocation fails, or while the stream is being captured, the
// kernels form the prefactors as they go.
constexpr size_t kSideTableMax = (size_t)4 << 30;

void ensure_side_table(rad_ctx *ctx, int precision) {
  DevGeom &G = ctx->geom;
  const int ip = precision == RAD_F32 ? 1 : 0;
  if (G.kind == RAD_MINK_CART || G.side_P[ip] || G.side_refused[ip]) return;
  const size_t ncol = (size_t)G.n[0] * G.n[1], nap = (size_t)ctx->ang.n_ap;
  const size_t nf[2] = {(size_t)G.n[1] * (G.n[0] + 1), (size_t)(G.n[1] + 1) * G.n[0]};
  auto pad = [](size_t b) { return (b + 255) / 256 * 256; };
  const size_t bP = pad(ncol * nap * kSideRows * (ip ? 4 : 8)), bU = pad(ncol * nap);
  // the FP64 kernels also read the faces' prefactors (eight operations of their
  // pipe per bin and face: in a 2D grid, where a CTA has one cell, as much as a
  // third of the update; two gradient steps of 256 x
  // 128 x 162: 27.8 -> 24.3 ms with the adjoint's slopes on fewer operations)
  size_t bF = 0;
  for (int d = 0; d < 2 && !ip; ++d) bF += pad(nf[d] * nap * sizeof(double)) + pad(nf[d] * nap);
  if (bP + bU + bF > kSideTableMax) bF = 0;
  if (bP + bU > kSideTableMax) return;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return;
  }
  unsigned char *buf = nullptr;
  while (cudaMalloc(&buf, bP + bU + bF) != cudaSuccess) {
    cudaGetLastError();
    if (!bF) {
      // not tried again for this metric: steps after the first allocate nothing
      G.side_refused[ip] = true;
      return;
    }
    bF = 0;
  }
  void *P = buf;
  unsigned char *up = buf + bP, *next = up + bU;
  const int threads = std::min(256, (int)(nap + 31) / 32 * 32);
  if (ip)
    k_side_table<float, ColGeoF><<<(unsigned)ncol, threads, 0, ctx->stream>>>(
        G.colsF, ctx->ang.n_ang, (int)nap, ctx->dang.slot_nbr, ctx->dang.slot_edge, ctx->dang.edge_pq,
        ctx->dang.edge_geo, ctx->dang.dOmega, ctx->dang.rdO, (float *)P, up);
  else
    k_side_table<double, ColGeo><<<(unsigned)ncol, threads, 0, ctx->stream>>>(
        G.cols, ctx->ang.n_ang, (int)nap, ctx->dang.slot_nbr, ctx->dang.slot_edge, ctx->dang.edge_pq,
        ctx->dang.edge_geo, ctx->dang.dOmega, ctx->dang.rdO, (double *)P, up);
  double *c[2] = {nullptr, nullptr};
  unsigned char *u[2] = {nullptr, nullptr};
  for (int d = 0; d < 2 && bF; ++d) {
    c[d] = (double *)next;
    u[d] = next + pad(nf[d] * nap * sizeof(double));
    next = u[d] + pad(nf[d] * nap);
    k_face_table<<<(unsigned)nf[d], threads, 0, ctx->stream>>>(d == 0 ? G.f1 : G.f2, ctx->ang.n_ang, (int)nap,
                                                             ctx->dang.dir, c[d], u[d]);
  }
  if (cudaGetLastError() != cudaSuccess) {
    cudaFree(buf);
    return;
  }
  G.side_buf[ip] = buf;
  G.side_P[ip] = P;
  G.side_up[ip] = up;
  for (int d = 0; d < 2 && !ip; ++d) {
    G.face_c[d] = c[d];
    G.face_up[d] = u[d];
  }
}

cudaError_t alloc_scratch(rad_ctx *ctx, void **p, size_t bytes) {
  cudaError_t ce = cudaMalloc(p, bytes);
  if (ce == cudaSuccess) return ce;
  cudaGetLastError();                    // handled here: later launches look at this state too
  DevGeom &G = ctx->geom;
  if (!(G.side_buf[0] || G.side_buf[1]) || G.side_captured) return ce;
  cudaStreamSynchronize(ctx->stream);
  for (int ip = 0; ip < 2; ++ip) {
    cudaFree(G.side_buf[ip]);
    G.side_buf[ip] = G.side_P[ip] = nullptr;
    G.side_up[ip] = nullptr;
    G.face_c[ip] = nullptr;
    G.face_up[ip] = nullptr;
    G.side_refused[ip] = true;
  }
  ce = cudaMalloc(p, bytes);
  if (ce != cudaSuccess) cudaGetLastError();
  return ce;
}

void note_capture(rad_ctx *ctx) {
  DevGeom &G = ctx->geom;
  if (G.side_captured || !(G.side_buf[0] || G.side_buf[1])) return;
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    G.side_captured = true;
  }
}

}  // namespace rad
