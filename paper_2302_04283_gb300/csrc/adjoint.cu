// Reverse-mode step (hand-written adjoint) and the outgoing-flux loss.
//
// rad_step_adjoint recomputes the two stages of rad_step from the checkpoint
// I_n (keeping I^1 and both pre-coupling primitives I^1*, I^2*) and then
// runs the stages backwards:
//   coupling adjoint   lambda_I+  ->  mu = lambda_U* = lambda_I* / (n^0 n_0),
//                      and dL/d(alpha_a, alpha_s, eta) of this coupling
//                      (k_couple_adj: per-cell reductions, as in the forward);
//                      with thermal coupling also lambda_T+ -> lambda_T-,
//                      through the root of the quartic by the implicit-function
//                      theorem (dT+ = -(T^4 dB4 + T dB1 + dB0) / f'(T+))
//   transport adjoint  mu -> lambda_{I^{s-1}} += b f mu + b beta dt J_L^T mu,
//                      lambda_{I^0} += a f mu
//                      (k_transport_adj: gather form of the transposed
//                      DC / PLM / PPM upwind stencil and of the angular
//                      fluxes; adjoint_kernels.cuh, adjoint_tadj_*.cu)
// with (a, b, beta) = (0, 1, 1) for stage 1 and (1/2, 1/2, 1/2) for stage 2.
// With the optical-depth weighting of Sec. 2.4 every face's lambda weight
// carries the face's factor (1 +- d), and the factor's dependence on
// alpha_E = alpha_a + alpha_s (through f = -expm1(-tau^2)) gives a further
// opacity gradient: each cell reduces over bins the flux derivative of its
// lower face in each dimension (k_transport_adj), and k_tau_grad adds the
// two faces on either side of a cell to dL/dalpha_a and dL/dalpha_s.
// The PLM and PPM limiters are differentiated on their active branches.
// Boundary conditions enter through the transpose of the neighbour map:
// periodic wrap and outflow clamp by matching every stencil position's
// source cell against the target (a face that appears twice in the window
// of a short periodic line counts once), the polar map by explicit terms
// for the faces next to a pole whose upwind stencils reach across it (the
// pole faces themselves have zero area).  No atomics: every output element
// is written by one thread.
#include <type_traits>

#include "adjoint_kernels.cuh"

namespace rad {

// L = sum_{k,j} sum_{n: n^1 > 0 at the outer x1 face} I[k][j][n1-1][n] dOmega_n.
// One block per (j, k) row; the outer-face tetrad row gives the sign of n^1.
template <typename R>
__global__ void k_loss(const R *I, R *dL, double *L, int n1, int n2, int nap, int nang, const FaceGeo *f1,
                       const double *dir, const double *dOmega) {
  int row = blockIdx.x;            // k * n2 + j
  int j = row % n2;
  const FaceGeo &F = f1[j * (n1 + 1) + n1];
  long long base = ((long long)row * n1 + (n1 - 1)) * nap;
  double acc = 0.0;
  for (int n = threadIdx.x; n < nang; n += blockDim.x) {
    double na = F.ea[0] + F.ea[1] * dir[3 * n] + F.ea[2] * dir[3 * n + 1] + F.ea[3] * dir[3 * n + 2];
    double w = na > 0.0 ? dOmega[n] : 0.0;
    acc += w * (double)I[base + n];
    if (dL) dL[base + n] = (R)w;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ double part[32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += part[w];
    L[row] = s;                      // per-row partial; summed in order below
  }
}

// Fixed-order sum of the row partials (deterministic loss).
__global__ void k_sum_rows(const double *part, int rows, double *L) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int r = threadIdx.x; r < rows; r += blockDim.x) s += part[r];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *L = sh[0];
}

int launch_loss(rad_ctx *ctx, const void *I, int precision, double *L, void *dL, std::string &err) {
  const DevGeom &G = ctx->geom;
  size_t ncell = (size_t)G.n[0] * G.n[1] * G.n[2];
  size_t esz = precision == RAD_F32 ? 4 : 8;
  if (dL) cudaMemsetAsync(dL, 0, ncell * ctx->ang.n_ap * esz, ctx->stream);
  unsigned rows = (unsigned)(G.n[1] * G.n[2]);
  if (ctx->loss_rows < (int)rows) {
    cudaStreamSynchronize(ctx->stream);
    cudaFree(ctx->loss_buf);
    ctx->loss_buf = nullptr;
    ctx->loss_rows = 0;
    if (alloc_scratch(ctx, (void **)&ctx->loss_buf, rows * sizeof(double)) != cudaSuccess) {
      err = "loss scratch allocation failed";
      return RAD_ENOMEM;
    }
    ctx->loss_rows = (int)rows;
  }
  if (precision == RAD_F32)
    k_loss<float><<<rows, 256, 0, ctx->stream>>>((const float *)I, (float *)dL, ctx->loss_buf, G.n[0], G.n[1],
                                                 ctx->ang.n_ap, ctx->ang.n_ang, G.f1, ctx->dang.dir,
                                                 ctx->dang.dOmega);
  else
    k_loss<double><<<rows, 256, 0, ctx->stream>>>((const double *)I, (double *)dL, ctx->loss_buf, G.n[0], G.n[1],
                                                  ctx->ang.n_ap, ctx->ang.n_ang, G.f1, ctx->dang.dir,
                                                  ctx->dang.dOmega);
  k_sum_rows<<<1, 256, 0, ctx->stream>>>(ctx->loss_buf, (int)rows, L);
  cudaError_t ce = cudaGetLastError();
  if (ce != cudaSuccess) {
    err = std::string("loss launch failed: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  return RAD_OK;
}

// ---------------------------------------------------------------- adjoint
// Adjoint of the coupling of one stage (MODE: thermal, fixed emissivity or
// none).  One thread per bin; a CTA takes the column's chunk of kc cells in
// phases, like the forward stage kernel:
//   A  per cell the four bin sums of the forward coupling and of lambda_S
//      (warp reduce-scatter, per-warp partials in shared memory);
//   B  one thread per cell: the quartic's root (or the fixed-emissivity
//      closed form) and the reverse sweep through the cell's scalars;
//   C  per bin lambda_I* -> mu, and the bin sums of dL/dalpha_E (and dL/du);
//   D  one thread per cell adds the gradients.
// The kernel is bound by the FP64 pipe (two FP64 lanes per SM and clock on
// this part: one warp instruction costs 16 SM cycles however few lanes are
// active), so what counts is FP64 warp instructions.  Solving the root once
// per cell with one active lane, between the barriers of that cell, cost as
// many of them as the bins themselves; phase B solves a chunk's cells in one
// warp.  Every quotient comes from one reciprocal of n^0bar den in place of
// six correctly rounded divisions of about ten FP64 operations each.  45 x 38 x
// 33 cells x 162 bins, thermal, FP32 intensities: 5.24 -> 1.32 ms per stage; 256
// x 128 x 162, fixed emissivity, FP64: 2.69 -> 1.17 ms.
// The thermal sweep runs in FP64 in both precisions (only I* and
// lambda_I+ are in the working precision): the terms of dL/dalpha_s cancel,
// and FP32 per-bin sums lose percents.
template <typename R, int MODE, int MAXT>
__global__ void __launch_bounds__(MAXT) k_couple_adj(AdjArgs A) {
  constexpr bool THERMAL = MODE == RAD_COUPLE_THERMAL;
  using W = typename std::conditional<THERMAL, double, R>::type;      // type of the sweep
  using Col = typename GeoTypes<W>::Col;
  const StageArgs &a = A.s;
  extern __shared__ __align__(16) unsigned char adj_smem[];
  const int n = threadIdx.x;
  const int nwarp = blockDim.x >> 5, lane = n & 31, warp = n >> 5;
  const bool act = n < a.nang;
  const int nchunk = (a.n3 + a.kc - 1) / a.kc;
  const int col = blockIdx.x / nchunk, chunk = blockIdx.x % nchunk;
  const int k0 = chunk * a.kc, nc = min(a.kc, a.n3 - k0);
  const size_t ncol = (size_t)a.n1 * a.n2, strideK = ncol * a.nap;
  const size_t own = (size_t)k0 * strideK + (size_t)col * a.nap + (act ? n : 0);
  const Col &cg = THERMAL ? ((const Col *)A.cols64)[col] : ((const Col *)a.cols)[col];
  W x = W(0), y = W(0), z = W(0), dOm = W(0);
  if (act) {
    x = (W)a.dir[3 * n];
    y = (W)a.dir[3 * n + 1];
    z = (W)a.dir[3 * n + 2];
    dOm = (W)a.dOmega[n];
  }
  const W n0up = cg.n0up;
  const W nlow0 = cg.M[0][0] + cg.M[0][1] * x + cg.M[0][2] * y + cg.M[0][3] * z;
  // the guard's test in the working precision of the forward kernel
  R g0 = (R)nlow0;
  if (THERMAL && sizeof(R) == 4) {
    const ColGeoF &cf = ((const ColGeoF *)a.cols)[col];
    g0 = (R)(cf.M[0][0] + cf.M[0][1] * (float)x + cf.M[0][2] * (float)y + cf.M[0][3] * (float)z);
  }
  const bool live = act && !(a.zero_guard && fabs((double)g0) < a.n0crit);
  const W inv_f = act ? W(1) / (n0up * nlow0) : W(0);
  const R *lam = (const R *)A.lam, *Isv = (const R *)A.Istar;
  R *mu = (R *)A.mu;
  if (MODE == RAD_COUPLE_NONE) {
    for (int c = 0; c < nc; ++c)
      if (act) mu[own + c * strideK] = live ? (R)((W)lam[own + c * strideK] * inv_f) : R(0);
    return;
  }
  W *gas = (W *)adj_smem;                     // [kc][8]: u, u^0, alpha_E (times dts in FP64)
  W *sc = gas + 8 * a.kc;                     // [kc][8]: scalars of phase B
  W *red = sc + 8 * a.kc;                     // [kc][nwarp][4]
  const W dts = (W)a.dts, c2p = dts / W(kFourPi);
  for (int c = n; c < nc; c += blockDim.x) {
    const size_t cell = (size_t)(k0 + c) * ncol + col;
    const W ux = (W)a.u[3 * cell], uy = (W)a.u[3 * cell + 1], uz = (W)a.u[3 * cell + 2];
    W *g = gas + 8 * c;
    g[0] = ux;
    g[1] = uy;
    g[2] = uz;
    g[3] = sqrt(W(1) + ux * ux + uy * uy + uz * uz);
    g[4] = (W)(a.aa[cell] + a.as[cell]);
    if (sizeof(W) == 8) g[4] *= dts;
  }
  __syncthreads();
  constexpr bool D64 = sizeof(W) == 8;
  // per bin and cell: nb = n^0bar, rden = 1 / (n^0 + nb alpha_E dt), wb = nb^2
  // dOmega.  FP64: r = 1 / (nb den) gives rden = nb r and inb = 1 / nb = den r;
  // factors common to a cell's bins (alpha_E dt, dt, dt / 4 pi, n^0, S) are
  // taken out of the sums, to save operations of the FP64 pipe.  FP32: c2n =
  // c2pre rden / nb^3 and rn = dOmega rden / nb.
  struct Bin { W nb, rden, wb, r, inb, c2n, rn; };
  auto bin = [&](int c) -> Bin {
    const W *g = gas + 8 * c;
    Bin b;
    if (D64) {
      b.nb = fma_rn(-g[0], x, fma_rn(-g[1], y, fma_rn(-g[2], z, g[3])));
      const W den = fma_rn(b.nb, g[4], n0up);
      b.r = inv1(b.nb * den);
      b.rden = b.nb * b.r;
      b.inb = den * b.r;
      b.wb = b.nb * b.nb * dOm;
      b.c2n = b.rn = W(0);
    } else {
      b.nb = g[3] - (g[0] * x + g[1] * y + g[2] * z);
      b.wb = b.nb * b.nb * dOm;
      b.rden = W(1) / (n0up + b.nb * g[4] * dts);
      b.c2n = c2p * b.rden / (b.nb * b.nb * b.nb);
      b.rn = dOm * b.rden / b.nb;
      b.r = b.inb = W(0);
    }
    return b;
  };
  // ---- phase A: thermal D = sum (c1 - 1) I* wbar, sum dOmega rden / nb, Ebar- =
  // sum I* wbar, lambda_S; fixed emissivity A1 = sum c1 I* wbar, the same, lambda_S
#pragma unroll 2
  for (int c = 0; c < nc; ++c) {
    const W Is = act ? (W)Isv[own + c * strideK] : W(0);
    const W lp = live ? (W)lam[own + c * strideK] : W(0);
    const Bin b = bin(c);
    W s;
    if (D64) {
      const W w = Is * b.wb, v3 = b.rden * b.inb * (b.inb * b.inb) * lp;
      s = THERMAL ? warp_reduce4(b.nb * b.rden * w, dOm * b.r, w, v3, lane)
                  : warp_reduce4(b.rden * w, dOm * b.r, v3, W(0), lane);
    } else {
      const W c1 = n0up * b.rden;
      s = warp_reduce4(act ? c1 * Is * b.wb : W(0), act ? b.rn : W(0), act ? b.c2n * lp : W(0), W(0), lane);
    }
    if ((lane & 7) == 0) red[(c * nwarp + warp) * 4 + (lane >> 3)] = s;
  }
  __syncthreads();
  // ---- phase B
  // reports what the forward stage reports of a cell (the recomputation of stage 2
  // stops before its coupling): no root, or a source term S past the range of FP64
  // (no convergence) or of the intensities (they come out non-finite)
  for (int c = n; c < nc; c += blockDim.x) {
    const size_t cell = (size_t)(k0 + c) * ncol + col;
    W t[4] = {W(0), W(0), W(0), W(0)};
    for (int w = 0; w < nwarp; ++w)
#pragma unroll
      for (int r = 0; r < 4; ++r) t[r] += red[(c * nwarp + w) * 4 + r];
    W *o = sc + 8 * c;
    if (D64) {                              // the common factors of the sums
      t[0] *= THERMAL ? -gas[8 * c + 4] : n0up;
      t[THERMAL ? 3 : 2] *= c2p;
    }
    const W A2 = c2p * t[1], lS = THERMAL ? t[3] : t[2];
    if (THERMAL) {
      // the quartic B4 T^4 + B1 T + B0 = 0, Ebar+ = Ebar- - c_v (T+ - T-),
      // S = alpha_a a T+^4 + alpha_s Ebar+, I+ = c1 I* + c2n S
      const double aad = a.aa[cell], asd = a.as[cell], ar = a.a_rad;
      const double D = t[0], Em = t[2];
      const double Tm = a.stage2 ? 0.5 * (a.T0[cell] + a.T1[cell]) : a.T0[cell];
      const double cv = a.rho[cell] * a.inv_gm1;
      const double B4 = A2 * aad * ar, B1 = cv * (1.0 - A2 * asd), B0 = D + A2 * asd * Em - B1 * Tm;
      bool ok = true;
      const double Tp = quartic_root(B4, B1, B0, true, ok, Tm);
      const double T3 = Tp * Tp * Tp, T4 = T3 * Tp;
      const double Ep = Em - cv * (Tp - Tm);
      const double S = aad * ar * T4 + asd * Ep;
      if (!ok || !isfinite(Tp) || exp_ones(S)) atomicOr(a.err, kErrNoConv);      // S off the FP64 pipe
      else if (sizeof(R) == 4 && !isfinite((float)S)) atomicOr(a.err, kErrNonFinite);
      double lT = (A.lamTp ? A.lamTp[cell] : 0.0) + 4.0 * aad * ar * T3 * lS;
      const double lEp = asd * lS;
      double laa = ar * T4 * lS, las = Ep * lS;
      // Ebar+ = Ebar- - c_v T+ + c_v T-
      double lEm = lEp, lTm = cv * lEp;
      lT -= cv * lEp;
      // T+ = root(B4, B1, B0): d/dB = -(T^4, T, 1) / f'(T+)
      const double g = lT / (4.0 * B4 * T3 + B1);
      const double lB4 = -g * T4, lB0 = -g;
      double lB1 = -g * Tp;
      // B0 = D + A2 alpha_s Ebar- - B1 T-
      double lA2 = asd * Em * lB0;
      las += A2 * Em * lB0;
      lEm += A2 * asd * lB0;
      lB1 -= Tm * lB0;
      lTm -= B1 * lB0;
      // B1 = c_v (1 - A2 alpha_s), B4 = A2 alpha_a a
      lA2 += -cv * asd * lB1 + aad * ar * lB4;
      las -= cv * A2 * lB1;
      laa += A2 * ar * lB4;
      o[0] = c2p * S;                        // c2pre S
      o[1] = lB0;                            // lambda_D
      o[2] = lEm;
      o[3] = c2p * lA2;                      // lambda of sum dOmega rden / n^0bar
      o[4] = laa;
      o[5] = las;
      if (A.outTa) A.outTa[cell] = (A.accTa ? A.outTa[cell] : 0.0) + A.wTa * lTm;
      if (A.outTb) A.outTb[cell] = A.wTb * lTm;
    } else {
      const W as = (W)a.as[cell], eta = (W)a.eta[cell], A1 = t[0];
      const W Q = W(1) - A2 * as;
      const W Ep = (A1 + W(kFourPi) * A2 * eta) / Q;
      const W S = W(kFourPi) * eta + as * Ep;
      // (FP32: 1 - A2 alpha_s may round to 0 or below at great depth, which the
      // forward stage, in FP64 there, does not report)
      if ((D64 ? exp_ones((double)S) : !isfinite(S)) && Q > W(0))
        atomicOr(a.err, sizeof(R) == 8 ? kErrNoConv : kErrNonFinite);
      const W lEp = as * lS;
      const W lA1 = lEp / Q;
      const W lQ = -Ep * lEp / Q;
      const W lA2 = W(kFourPi) * eta * lEp / Q - as * lQ;
      const W leta = W(kFourPi) * lS + W(kFourPi) * A2 * lEp / Q;
      const W las = Ep * lS - A2 * lQ;
      o[0] = D64 ? c2p * S : S;
      o[1] = lA1;
      o[3] = D64 ? c2p * lA2 : lA2;
      o[4] = W(0);
      o[5] = las;
      if (A.g_eta) A.g_eta[cell] += (double)leta;
    }
  }
  __syncthreads();
  // ---- phase C: lambda_I* and dL/d(1 / den) of every bin; the sum of
  // dL/dalpha_E of four cells shares one reduce-scatter (with the
  // radiation-dominated substitution a cell's four sums, dL/du among them)
  W held[3] = {W(0), W(0), W(0)};
  for (int c = 0; c < nc; ++c) {
    const size_t e = own + c * strideK;
    const W Is = act ? (W)Isv[e] : W(0);
    const W lp = live ? (W)lam[e] : W(0);
    const Bin b = bin(c);
    const W *o = sc + 8 * c;
    const W S = o[0], lD = o[1], lA2 = o[3];
    const W lEm = THERMAL ? o[2] : W(0);
    W lIs, vE, lrden = W(0);
    if (D64) {
      // lambda of rden = 1 / den; vE without its factor -dt
      const W wl = b.wb * lD, h = lp + wl;
      lrden = fma_rn(n0up * Is, h, fma_rn(S, b.inb * b.inb * b.inb * lp, dOm * b.inb * lA2));
      vE = b.rden * b.rden * b.nb * lrden;
      lIs = THERMAL ? fma_rn(b.rden, fma_rn(-(b.nb * gas[8 * c + 4]), wl, n0up * lp), b.wb * lEm) : n0up * b.rden * h;
    } else {
      const W c1 = n0up * b.rden;
      const W lc1 = Is * lp + Is * b.wb * lD;
      const W lc2n = S * lp;
      lIs = c1 * lp + c1 * b.wb * lD;
      const W lden = -c1 * b.rden * lc1 - b.c2n * b.rden * lc2n - c2p * dOm * b.rden * b.rden / b.nb * lA2;
      vE = b.nb * dts * lden;
    }
    if (!act) vE = W(0);
    if (act) mu[e] = live ? (R)(lIs * inv_f) : R(0);
    if (THERMAL && A.lam_u) {
      // the velocity is itself a function of the intensities: dL/du through
      // every n^0bar = u^0 - u.n
      W du[3] = {W(0), W(0), W(0)};
      if (act) {
        const W *g = gas + 8 * c;
        const W cm1 = -(b.nb * g[4]) * b.rden;
        const W dLdnb = -lrden * g[4] * b.rden * b.rden - W(3) * b.rden * (b.inb * b.inb) * (b.inb * b.inb) * S * lp +
                        (cm1 * Is * lD + Is * lEm) * W(2) * b.nb * dOm - lA2 * dOm * b.r * b.inb;
        const W iu0 = W(1) / g[3];
        du[0] = dLdnb * (g[0] * iu0 - x);
        du[1] = dLdnb * (g[1] * iu0 - y);
        du[2] = dLdnb * (g[2] * iu0 - z);
      }
      const W s = warp_reduce4(vE, du[0], du[1], du[2], lane);
      if ((lane & 7) == 0) red[(c * nwarp + warp) * 4 + (lane >> 3)] = s;
      continue;
    }
    if ((c & 3) == 3 || c == nc - 1) {
      const int q = c & 3, c4 = c - q;
      const W s = warp_reduce4(q == 0 ? vE : held[0], q == 1 ? vE : (q > 1 ? held[1] : W(0)),
                               q == 2 ? vE : (q > 2 ? held[2] : W(0)), q == 3 ? vE : W(0), lane);
      const int r = lane >> 3;
      if ((lane & 7) == 0 && c4 + r < nc) red[((c4 + r) * nwarp + warp) * 4] = s;
    } else if ((c & 3) == 0) {
      held[0] = vE;
    } else if ((c & 3) == 1) {
      held[1] = vE;
    } else {
      held[2] = vE;
    }
  }
  __syncthreads();
  // ---- phase D
  for (int c = n; c < nc; c += blockDim.x) {
    const size_t cell = (size_t)(k0 + c) * ncol + col;
    const int nr = THERMAL && A.lam_u ? 4 : 1;
    W t[4] = {W(0), W(0), W(0), W(0)};
    for (int w = 0; w < nwarp; ++w)
      for (int r = 0; r < nr; ++r) t[r] += red[(c * nwarp + w) * 4 + r];
    if (D64) t[0] *= -dts;
    const W *o = sc + 8 * c;
    A.g_aa[cell] += THERMAL ? (double)(o[4] + t[0]) : (double)t[0];
    A.g_as[cell] += (double)(t[0] + o[5]);
    if (THERMAL && A.lam_u)
      for (int d = 0; d < 3; ++d) A.lam_u[3 * cell + d] = (double)t[1 + d];
  }
}

namespace {

template <typename R>
cudaError_t launch_transport_adj_any(const AdjArgs &A, bool ang, cudaStream_t st) {
  if (ang && A.s.recon_ang == RAD_RECON_PLM) return launch_transport_adj<R, true, 1>(A, st);
  if (ang && A.s.recon_ang == RAD_RECON_MAPR) return launch_transport_adj<R, true, 2>(A, st);
  return ang ? launch_transport_adj<R, true>(A, st) : launch_transport_adj<R, false>(A, st);
}

template <typename R, int MODE>
cudaError_t launch_couple_adj_m(const AdjArgs &A, cudaStream_t st) {
  const int threads = (A.s.nap + 31) / 32 * 32;
  const int nchunk = (A.s.n3 + A.s.kc - 1) / A.s.kc;
  const dim3 grid((unsigned)((long long)A.s.n1 * A.s.n2 * nchunk));
  const size_t esz = MODE == RAD_COUPLE_THERMAL ? 8 : sizeof(R);
  const size_t smem = (size_t)A.s.kc * (16 + 4 * (threads / 32)) * esz;     // kc <= 32: at most 37 KB
  if (threads <= 256) k_couple_adj<R, MODE, 256><<<grid, threads, smem, st>>>(A);
  else if (threads <= 512) k_couple_adj<R, MODE, 512><<<grid, threads, smem, st>>>(A);
  else k_couple_adj<R, MODE, 1024><<<grid, threads, smem, st>>>(A);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_couple_adj(const AdjArgs &A, cudaStream_t st) {
  if (A.s.mode == RAD_COUPLE_THERMAL) return launch_couple_adj_m<R, RAD_COUPLE_THERMAL>(A, st);
  if (A.s.mode == RAD_COUPLE_EMISSIVITY) return launch_couple_adj_m<R, RAD_COUPLE_EMISSIVITY>(A, st);
  return launch_couple_adj_m<R, RAD_COUPLE_NONE>(A, st);
}

}  // namespace

int launch_adjoint(rad_ctx *ctx, const void *I_n, const rad_gas *gas, double dt, const rad_opts *o,
                   const void *lam_np1, void *lam_n, const double *lamT_np1, double *lamT_n, double *g_aa,
                   double *g_as, double *g_eta, std::string &err) {
  const DevGeom &G = ctx->geom;
  const bool f32 = o->precision == RAD_F32;
  const bool ang = G.kind != RAD_MINK_CART;
  const size_t ncell = (size_t)G.n[0] * G.n[1] * G.n[2];
  const size_t esz = f32 ? 4 : 8;
  const size_t ib = (ncell * ctx->ang.n_ap * esz + 255) / 256 * 256;
  const size_t tb = (ncell * sizeof(double) + 255) / 256 * 256;
  const size_t need = 5 * ib + 12 * tb;
  if (ctx->adj_bytes < need) {
    cudaStreamSynchronize(ctx->stream);
    cudaFree(ctx->adj_buf);
    ctx->adj_buf = nullptr;
    ctx->adj_bytes = 0;
    if (alloc_scratch(ctx, &ctx->adj_buf, need) != cudaSuccess) {
      err = "adjoint scratch allocation failed";
      return RAD_ENOMEM;
    }
    ctx->adj_bytes = need;
  }
  ensure_side_table(ctx, o->precision);      // after the scratch: the call runs without the table
  unsigned char *p = (unsigned char *)ctx->adj_buf;
  void *I1 = p, *I1s = p + ib, *I2s = p + 2 * ib, *mu = p + 3 * ib, *lamI1 = p + 4 * ib;
  double *T1 = (double *)(p + 5 * ib), *T2 = (double *)(p + 5 * ib + tb);
  double *lamT1 = (double *)(p + 5 * ib + 2 * tb);   // adjoint of the stage-1 temperature
  double *gtau = (double *)(p + 5 * ib + 3 * tb);    // [cell][3] lower-face sums (optical-depth weighting)
  double *usub = (double *)(p + 5 * ib + 6 * tb);    // [cell][3] substituted velocity (rad_dom)
  double *lamu = (double *)(p + 5 * ib + 9 * tb);    // [cell][3] dL/du of the substituted velocity (rad_dom)
  const bool rd = o->rad_dom != 0;
  const bool thermal = o->coupling == RAD_COUPLE_THERMAL;
  if (!thermal && lamT_n && lamT_n != lamT_np1) {
    // the temperature passes through an uncoupled or fixed-emissivity step
    const cudaError_t te = lamT_np1 ? cudaMemcpyAsync(lamT_n, lamT_np1, ncell * sizeof(double),
                                                      cudaMemcpyDeviceToDevice, ctx->stream)
                                    : cudaMemsetAsync(lamT_n, 0, ncell * sizeof(double), ctx->stream);
    if (te != cudaSuccess) {
      err = std::string("adjoint temperature copy failed: ") + cudaGetErrorString(te);
      return RAD_ECUDA;
    }
  }
  // ---- forward recompute with the pre-coupling primitives kept
  StageArgs s = make_stage_args(ctx, gas, dt, o, nullptr);
  {
    const int rc = check_stage(s, f32, err);
    if (rc != RAD_OK) return rc;
  }
  s.Iprev = I_n;
  s.I0 = I_n;
  s.Iout = I1;
  s.Istar = I1s;
  s.T0 = gas->T;
  s.T1 = nullptr;
  s.Tout = T1;
  s.stage2 = 0;
  s.dts = dt;
  // with the radiation-dominated substitution the forward stage is the
  // transport-only stage kernel followed by the substituted coupling
  if (rd) s.mode = RAD_COUPLE_NONE;
  cudaError_t ce = launch_stage(s, f32, ang, ctx->stream);
  if (ce == cudaSuccess && rd) ce = launch_couple_rd(s, f32, T1, T1, ctx->stream);
  if (ce == cudaSuccess) {
    // stage 2 up to I*: its coupled result is not needed (the coupling adjoint
    // forms its root from I* and T- = (T^0 + T^1) / 2), so the transport-only
    // stage writes I* and T- (gradient of two steps of 256 x 128 x 162 FP64: 24.3
    // -> 23.4 ms)
    s.mode = RAD_COUPLE_NONE;
    s.Iprev = I1;
    s.I0 = I_n;
    s.Iout = I2s;
    s.Istar = nullptr;
    s.T0 = gas->T;
    s.T1 = T1;
    s.Tout = T2;
    s.stage2 = 1;
    s.dts = 0.5 * dt;
    ce = launch_stage(s, f32, ang, ctx->stream);
  }
  s.Istar = nullptr;
  s.mode = o->coupling;
  // ---- stage 2 backwards
  AdjArgs A;
  A.s = s;
  A.g_aa = g_aa;
  A.g_as = g_as;
  A.g_eta = g_eta;
  A.cols64 = G.cols;
  A.gtau = gtau;
  // temperature adjoint (thermal coupling): stage 2 takes lambda_T of the
  // step's output, T- = (T^0 + T^1) / 2 splits its lambda_T- in halves to
  // T^0 (lamT_n) and T^1 (lamT1); stage 1 takes lamT1 and adds its
  // lambda_T- (T- = T^0) to lamT_n
  A.lamTp = lamT_np1;
  A.outTa = lamT_n;
  A.wTa = 0.5;
  A.accTa = 0;
  A.outTb = lamT1;
  A.wTb = 0.5;
  A.lam_u = nullptr;
  // the coupling adjoint of one stage; with rad_dom the coupling ran at the
  // substituted velocity: recompute it, take the coupling back at it (which
  // also gives dL/du), then take dL/du back through the substitution
  auto couple_adj = [&](const void *Istar, const double *Tm) -> cudaError_t {
    cudaError_t e = cudaSuccess;
    if (rd) {
      e = launch_rd_sub(0, A.s, f32, Istar, Tm, usub, nullptr, nullptr, nullptr, nullptr, nullptr, 0.0, nullptr,
                        0.0, ctx->stream);
      A.s.u = usub;
      A.lam_u = lamu;
    }
    if (e == cudaSuccess) e = f32 ? launch_couple_adj<float>(A, ctx->stream) : launch_couple_adj<double>(A, ctx->stream);
    if (rd) {
      A.s.u = gas->u;
      A.lam_u = nullptr;
      if (e == cudaSuccess)
        e = launch_rd_sub(1, A.s, f32, Istar, Tm, nullptr, lamu, A.mu, g_aa, g_as, A.outTa, A.wTa, A.outTb, A.wTb,
                          ctx->stream);
    }
    return e;
  };
  if (ce == cudaSuccess) {
    A.s.dts = 0.5 * dt;
    A.s.stage2 = 1;
    A.lam = lam_np1;
    A.Istar = I2s;
    A.mu = mu;
    ce = couple_adj(I2s, T2);     // T2 holds the stage's T- = (T^0 + T^1) / 2
  }
  if (ce == cudaSuccess) {
    A.Ilin = I1;
    A.outA = lamI1;
    A.wAf = 0.5;
    A.wAL = 0.5 * dt;
    A.accA = 0;
    A.outB = lam_n;
    A.wBf = 0.5;
    A.accB = 0;
    ce = f32 ? launch_transport_adj_any<float>(A, ang, ctx->stream) : launch_transport_adj_any<double>(A, ang, ctx->stream);
  }
  // ---- stage 1 backwards
  if (ce == cudaSuccess) {
    A.s.dts = dt;
    A.s.stage2 = 0;
    A.lamTp = lamT1;
    A.outTa = lamT_n;
    A.wTa = 1.0;
    A.accTa = 1;
    A.outTb = nullptr;
    A.lam = lamI1;
    A.Istar = I1s;
    A.mu = mu;
    ce = couple_adj(I1s, gas->T);
  }
  if (ce == cudaSuccess) {
    A.Ilin = I_n;
    A.outA = lam_n;
    A.wAf = 1.0;
    A.wAL = dt;
    A.accA = 1;
    A.outB = nullptr;
    ce = f32 ? launch_transport_adj_any<float>(A, ang, ctx->stream) : launch_transport_adj_any<double>(A, ang, ctx->stream);
  }
  if (ce != cudaSuccess) {
    err = std::string("adjoint launch failed: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  return RAD_OK;
}

}  // namespace rad
