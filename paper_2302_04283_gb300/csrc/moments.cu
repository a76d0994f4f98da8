// Moment contraction R^{AB} = sum_n I_n n^A n^B dOmega_n (Sec. 2.5), CUDA
// cores.  k_moments_simt: one warp per cell; lanes stride over the bins with
// ten running sums, a butterfly reduction combines the lanes, and lane 0
// applies the FP64 frame change (coordinate frame e e R; fluid frame Lambda
// Lambda R with the boost of Sec. 2.1).  k_moments_f64: FP64 intensities, up
// to kMomMaxBins bins, in fewer operations of the FP64 pipe.
#include <algorithm>

#include "step_kernel.cuh"

namespace rad {

// out^{ab} = L^a_A L^b_B R^{AB} for the ten components (00 01 02 03 11 12 13
// 22 23 33), written out with fixed indices.
__device__ __forceinline__ void frame_change(const double L[4][4], const double Rt[10], double out[10]) {
  const double R[4][4] = {{Rt[0], Rt[1], Rt[2], Rt[3]},
                          {Rt[1], Rt[4], Rt[5], Rt[6]},
                          {Rt[2], Rt[5], Rt[7], Rt[8]},
                          {Rt[3], Rt[6], Rt[8], Rt[9]}};
  double T[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int B = 0; B < 4; ++B) T[a][B] = L[a][0] * R[0][B] + L[a][1] * R[1][B] + L[a][2] * R[2][B] + L[a][3] * R[3][B];
  auto c = [&](int a, int b) { return T[a][0] * L[b][0] + T[a][1] * L[b][1] + T[a][2] * L[b][2] + T[a][3] * L[b][3]; };
  out[0] = c(0, 0);
  out[1] = c(0, 1);
  out[2] = c(0, 2);
  out[3] = c(0, 3);
  out[4] = c(1, 1);
  out[5] = c(1, 2);
  out[6] = c(1, 3);
  out[7] = c(2, 2);
  out[8] = c(2, 3);
  out[9] = c(3, 3);
}

// Boost Lambda^abar_Bhat to the fluid frame for tetrad-frame u^ihat (Sec. 2.1).
__device__ __forceinline__ void boost_matrix(double ux, double uy, double uz, double L[4][4]) {
  const double u[3] = {ux, uy, uz};
  const double u0 = sqrt(1.0 + ux * ux + uy * uy + uz * uz);
  const double g = 1.0 / (1.0 + u0);
  L[0][0] = u0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    L[0][a + 1] = -u[a];
    L[a + 1][0] = -u[a];
#pragma unroll
    for (int b = 0; b < 3; ++b) L[a + 1][b + 1] = u[a] * u[b] * g + (a == b ? 1.0 : 0.0);
  }
}

template <typename R>
__global__ void k_moments_simt(const R *I, R *out, long long ncell, int ncol, int nap, int nang,
                               const double *dir, const double *dOmega, int frame, const ColGeo *cols,
                               const double *u) {
  long long cell = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5);
  int lane = threadIdx.x & 31;
  if (cell >= ncell) return;
  const R *row = I + cell * nap;
  R acc[10];
#pragma unroll
  for (int p = 0; p < 10; ++p) acc[p] = R(0);
  for (int n = lane; n < nang; n += 32) {
    R v = row[n] * (R)dOmega[n];
    R x = (R)dir[3 * n], y = (R)dir[3 * n + 1], z = (R)dir[3 * n + 2];
    R vx = v * x, vy = v * y, vz = v * z;
    acc[0] += v;
    acc[1] += vx;
    acc[2] += vy;
    acc[3] += vz;
    acc[4] += vx * x;
    acc[5] += vx * y;
    acc[6] += vx * z;
    acc[7] += vy * y;
    acc[8] += vy * z;
    acc[9] += vz * z;
  }
#pragma unroll
  for (int p = 0; p < 10; ++p)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[p] += __shfl_xor_sync(0xffffffffu, acc[p], o);
  if (lane == 0) {
    double Rt[10], Ro[10];
    for (int p = 0; p < 10; ++p) Rt[p] = (double)acc[p];
    if (frame == RAD_FRAME_COORD) {
      double E[4][4];
      const ColGeo &cg = cols[cell % ncol];
#pragma unroll
      for (int m = 0; m < 4; ++m)
#pragma unroll
        for (int A = 0; A < 4; ++A) E[m][A] = cg.e[m][A];
      frame_change(E, Rt, Ro);
    } else if (frame == RAD_FRAME_FLUID) {
      double L[4][4];
      boost_matrix(u[3 * cell], u[3 * cell + 1], u[3 * cell + 2], L);
      frame_change(L, Rt, Ro);
    } else {
      for (int p = 0; p < 10; ++p) Ro[p] = Rt[p];
    }
    for (int p = 0; p < 10; ++p) out[cell * 10 + p] = (R)Ro[p];
  }
}

// FP64: bound by the FP64 pipe (an FP64 warp instruction occupies it for 16
// cycles), so the weights n^A n^B dOmega come from a table in shared memory
// (ten multiply-adds per bin, where forming them takes fourteen operations),
// and a warp takes three cells at a time, whose thirty sums share one
// reduce-scatter (31 additions per lane instead of three butterflies' 150)
// and one frame change in three lanes.  64^3 cells x 162 bins, 2.28 ms before: a
// step with moments 15.07 -> 13.97 ms (48^3: 0.485 ms, FP64 pipe 96 % active).
constexpr int kMomCells = 3;
constexpr int kMomMaxBins = 1024;          // 80 KB of weights per CTA
__global__ void __launch_bounds__(256) k_moments_f64(const double *__restrict__ I, double *__restrict__ out,
                                                     long long ncell, int ncol, int nap, int nang,
                                                     const double *dir, const double *dOmega, int frame,
                                                     const ColGeo *cols, const double *u) {
  extern __shared__ double W[];            // [10][nang]
  for (int n = threadIdx.x; n < nang; n += blockDim.x) {
    const double x = dir[3 * n], y = dir[3 * n + 1], z = dir[3 * n + 2], w = dOmega[n];
    const double wx = w * x, wy = w * y, wz = w * z;
    const double v[10] = {w, wx, wy, wz, wx * x, wx * y, wx * z, wy * y, wy * z, wz * z};
#pragma unroll
    for (int p = 0; p < 10; ++p) W[p * nang + n] = v[p];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const long long nwarp = (long long)gridDim.x * (blockDim.x / 32);
  for (long long g = (long long)blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5); g * kMomCells < ncell; g += nwarp) {
    const long long c0 = g * kMomCells;
    const int nc = (int)min((long long)kMomCells, ncell - c0);
    double v[32];
#pragma unroll
    for (int q = 0; q < 32; ++q) v[q] = 0.0;
    const double *row = I + c0 * nap;
    for (int n = lane; n < nang; n += 32) {
      double x[kMomCells];
#pragma unroll
      for (int c = 0; c < kMomCells; ++c) x[c] = c < nc ? __ldg(row + (size_t)c * nap + n) : 0.0;
#pragma unroll
      for (int p = 0; p < 10; ++p) {
        const double w = W[p * nang + n];
#pragma unroll
        for (int c = 0; c < kMomCells; ++c) v[10 * c + p] = fma(x[c], w, v[10 * c + p]);
      }
    }
    double s = warp_reduce32<double>(v, lane);            // lane 10 c + p: component p of cell c
    if (frame != RAD_FRAME_TETRAD) {
      double Rt[10], Ro[10], L[4][4];
      const int c = min(lane, nc - 1);
#pragma unroll
      for (int p = 0; p < 10; ++p) Rt[p] = __shfl_sync(0xffffffffu, s, 10 * c + p);
      const long long cell = c0 + c;
      if (frame == RAD_FRAME_COORD) {
        const ColGeo &cg = cols[cell % ncol];
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
          for (int A = 0; A < 4; ++A) L[m][A] = cg.e[m][A];
      } else {
        boost_matrix(u[3 * cell], u[3 * cell + 1], u[3 * cell + 2], L);
      }
      frame_change(L, Rt, Ro);
      if (lane < nc)
#pragma unroll
        for (int p = 0; p < 10; ++p) out[cell * 10 + p] = Ro[p];
    } else if (lane < 10 * nc) {
      out[c0 * 10 + lane] = s;
    }
  }
}

int launch_moments_bf16x3(rad_ctx *ctx, const float *I, int frame, const double *u, float *R,
                          cudaStream_t st, std::string &err);

int launch_moments(rad_ctx *ctx, const void *I, int precision, int frame, int method, const rad_gas *gas,
                   void *R, cudaStream_t st, std::string &err) {
  const DevGeom &G = ctx->geom;
  long long ncell = (long long)G.n[0] * G.n[1] * G.n[2];
  const double *u = (frame == RAD_FRAME_FLUID) ? gas->u : nullptr;
  if (method == RAD_MOM_BF16X3) return launch_moments_bf16x3(ctx, (const float *)I, frame, u, (float *)R, st, err);
  const int wpb = 8;
  unsigned blocks = (unsigned)((ncell + wpb - 1) / wpb);
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (precision == RAD_F32)
    k_moments_simt<float><<<blocks, 32 * wpb, 0, st>>>(
        (const float *)I, (float *)R, ncell, G.n[0] * G.n[1], ctx->ang.n_ap, ctx->ang.n_ang, ctx->dang.dir,
        ctx->dang.dOmega, frame, G.cols, u);
  else if (ctx->ang.n_ang <= kMomMaxBins &&
           (ncell > 8ll * nsm || ctx->ang.n_ang <= (frame == RAD_FRAME_TETRAD ? 100 : 256))) {
    const size_t smem = (size_t)ctx->ang.n_ang * 10 * sizeof(double);
    if (smem > 48 * 1024) {
      const cudaError_t ce = cudaFuncSetAttribute(k_moments_f64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (ce != cudaSuccess) {
        err = std::string("moments: ") + cudaGetErrorString(ce);
        return RAD_ECUDA;
      }
    }
    // two CTAs (sixteen warps) per SM keep the FP64 pipe busy; each builds its
    // table once.  Fewer cells than fill them: CTAs of fewer warps, so that the
    // pipes of all SMs share them (fluid frame, one CTA per eight warps -> now, and
    // k_moments_simt: 12^3 cells x 162 bins 30.7 -> 20.7 us, 44.4; 8^3 x 162 30.7 ->
    // 22.6, 24.6).  Of cells that k_moments_simt takes in one wave of CTAs and many
    // bins, the table costs more than it saves: 8^3 x 642 bins 59.0, with fewer warps
    // 46.9, k_moments_simt 38.3; 362 bins 46.6, 34.9, 32.6; without a frame change
    // 162 bins 17.9 with fewer warps, 15.9.
    const long long groups = (ncell + kMomCells - 1) / kMomCells, cta = 2ll * nsm;
    const int wpc = (int)std::min<long long>(wpb, (groups + cta - 1) / cta);
    const unsigned grid = (unsigned)std::min<long long>((groups + wpc - 1) / wpc, cta);
    k_moments_f64<<<grid, 32 * wpc, smem, st>>>((const double *)I, (double *)R, ncell, G.n[0] * G.n[1], ctx->ang.n_ap,
                                               ctx->ang.n_ang, ctx->dang.dir, ctx->dang.dOmega, frame, G.cols, u);
  } else
    k_moments_simt<double><<<blocks, 32 * wpb, 0, st>>>(
        (const double *)I, (double *)R, ncell, G.n[0] * G.n[1], ctx->ang.n_ap, ctx->ang.n_ang, ctx->dang.dir,
        ctx->dang.dOmega, frame, G.cols, u);
  cudaError_t ce = cudaGetLastError();
  if (ce != cudaSuccess) {
    err = std::string("moments launch failed: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  return RAD_OK;
}

}  // namespace rad
