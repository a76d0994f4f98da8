// Moment contraction on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// R^{AB} = sum_n I_n n^A n^B dOmega_n is the product D[cells x 16] =
// I[cells x K] . W^T[16 x K] with W[n][p] = n^A n^B dOmega_n for the ten
// pairs p (columns 10..15 zero, bins >= n_ang zero).  To keep FP32 accuracy
// on bf16 tensor cores both operands are split, x = hi + lo with hi =
// bf16(x), lo = bf16(x - hi), and D accumulates hi.hi + hi.lo + lo.hi in
// FP32 (the lo.lo term is below 2^-16 relative).
//
// One persistent CTA per SM walks tiles of 128 cells (M = 128, one TMEM lane
// per cell) and K in chunks of 64 bins.  The kernel is bound by HBM (5 flop per
// byte), so no part of the chain from load to output may wait for another:
//   16 converter warps  hold their pieces of the next two chunks in registers
//                       on their way (a warp's load covers two rows x 256
//                       contiguous bytes), convert the arrived chunk into bf16
//                       hi / lo and store it in the no-swizzle K-major
//                       core-matrix layout (8 rows x 16 bytes per core matrix)
//                       of one of two operand buffers;
//   1 issuing warp      one thread issues up to 4 x 3 tcgen05.mma (M=128, N=16,
//                       K=16) per chunk and commits to the buffer's mbarrier;
//   4 epilogue warps    read a finished tile back (tcgen05.ld) from one of two
//                       TMEM tiles, change the frame and write the components.
// The K-direction stride of the core matrices is 2064 bytes (2048 + 16), which
// spreads a warp's operand stores over all banks.  The previous form (four
// CTAs of 128 threads, each loading, converting, issuing and waiting in turn)
// left the memory idle meanwhile: 101 x 67 x 53 cells x 252 bins 0.145 -> 0.092 ms
// (4.1 TB/s), with the same bits.  Tried on the way: all roles in 16 warps 0.146
// ms (the issuing thread and the epilogue hold every chunk's barrier back),
// 16-byte cp.async pieces 0.139 ms (every piece costs a 32-byte sector of L2),
// 256-byte bulk copies 0.412 ms (some 80 cycles of an SM's copy engine each),
// the weights' hi and lo side by side in one N = 32 MMA 0.088 ms (fluid-frame
// components up to 1.3 times further from their 64-bit values: not kept).
// W^T hi/lo is built once on the host; each chunk's 4 KB of it (from L2) travel
// with the chunk, so shared memory does not grow with the bins.
// Every wait is bounded: on timeout the CTA records an error, frees its TMEM
// and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "rad_internal.h"

namespace rad {

constexpr int kTcM = 128;           // cells per tile
constexpr int kTcN = 16;            // moment columns (10 used)
constexpr int kTcKC = 64;           // bins per K chunk
constexpr int kTcConv = 512;         // converter threads
constexpr int kTcThreads = kTcConv + 32 + 128;
constexpr int kTcDepth = 3;         // chunks a thread holds: two on their way, one being converted
constexpr int kTcMaxKp = 2624;      // padded bins taken
constexpr uint32_t kBChunk = kTcKC * kTcN * 2 * 2;     // hi then lo: one 16-byte piece per thread
static_assert(kBChunk == kTcConv / 2 * 16, "one piece of W^T for half the threads");
constexpr int kTcPieces = kTcM * kTcKC / 4 / kTcConv;   // 16-byte pieces per thread and chunk
constexpr int kTcErrTimeout = 1 << 3;  // reported as RAD_ECUDA by rad_check
constexpr long long kTcSpinLimit = 1ll << 24;

// byte offsets of the K-major no-swizzle layouts
//   A (128 x 64 chunk): core (mg, kg) at kg * 2064 + mg * 128  -> SBO 128, LBO 2064
//   B (16 x 64 chunk):  core (ng, kg) at (kg * 2 + ng) * 128   -> SBO 128, LBO 256
constexpr uint32_t kALbo = 2064, kASbo = 128, kBLbo = 256, kBSbo = 128;
constexpr uint32_t kATile = 8 * kALbo;          // one operand half (16 KB and the padding)
static_assert(kATile % 128 == 0, "operand halves start on core matrix boundaries");

__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version for tcgen05; no swizzle, base offset 0
  return d;
}

// kind::f16 instruction descriptor: D f32, A bf16, B bf16, both K-major, N = 16, M = 128
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                            ((uint32_t)(kTcM >> 4) << 24);

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(kIdesc), "r"(acc));
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (long long it = 0; it < kTcSpinLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        "selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    // bounded in time as well as in polls; the global timer takes about a
    // microsecond to read, so only once a wait is long
    if ((it & 63) == 63) {
      unsigned long long now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (it == 63) t0 = now;
      else if (now - t0 > 2000000000ull) return false;
    }
  }
  return false;
}

// bf16 pair (low half a), rounded to nearest
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(b), "f"(a));
  return r;
}

template <bool ONE>
__global__ void __launch_bounds__(kTcThreads, 1) k_moments_tc(const float *__restrict__ I, float *__restrict__ out,
                                                            long long ncell, int nap, int nang, int kp,
                                                            const uint4 *__restrict__ wt, int frame,
                                                            const ColGeoF *cols, int ncol, const double *u,
                                                            int *err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  // operand buffers [2][hi, lo][kATile], W^T chunks [2]
  unsigned char *Aop = sm;
  unsigned char *Bw = sm + 4 * kATile;
  uint64_t *fullA = (uint64_t *)(Bw + 2 * kBChunk);      // per operand buffer: written (one arrival per converter warp)
  uint64_t *emptyA = fullA + 2;                          // ... read by the tensor cores
  uint64_t *fullD = emptyA + 2;                          // per TMEM tile: complete
  uint64_t *emptyD = fullD + 2;                          // ... read back (one arrival per epilogue warp)
  uint32_t *tslot = (uint32_t *)(emptyD + 2);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if (t == 0) {
    auto init = [](uint64_t *b, uint32_t n) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(b)), "r"(n));
    };
    for (int b = 0; b < 2; ++b) {
      init(fullA + b, kTcConv / 32);
      init(emptyA + b, 1);
      init(fullD + b, 1);
      init(emptyD + b, 4);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const uint32_t sA = smem_addr(Aop), sB = smem_addr(Bw);
  auto arrive = [](uint64_t *b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(b)) : "memory");
  };
  auto commit = [](uint64_t *b) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(b))
                 : "memory");
  };

  const long long ntile = (ncell + kTcM - 1) / kTcM;
  const int nk = ONE ? 1 : kp / kTcKC;                              // chunks per tile
  const int mytiles = ntile > blockIdx.x ? (int)((ntile - 1 - blockIdx.x) / gridDim.x) + 1 : 0;
  const int nunit = mytiles * nk;                                   // this CTA's chunks
  const long long row_step = (long long)gridDim.x * kTcM;
  bool ok = true;

  if (warp < kTcConv / 32) {
    // ---- converters.  Piece `it` of a chunk: row it 32 + m0 of the tile, bins
    // pk .. pk + 3 of the chunk (a warp: two rows x sixteen pieces)
    const int m0 = warp * 2 + (lane >> 4), pk = (lane & 15) * 4;
    const size_t prow = (size_t)32 * nap;
    float4 v[kTcDepth][kTcPieces];
    uint4 wv[kTcDepth];
    long long left = ncell - (long long)blockIdx.x * kTcM - m0;     // rows from the first piece's on
    const float *src = I + ((long long)blockIdx.x * kTcM + m0) * nap + pk;
    const size_t tile_step = (size_t)row_step * nap - (size_t)nk * kTcKC;
    const uint4 *wsrc = wt + (size_t)(t >> 7) * kp * kTcN * 2 / 16 + (t & 127);
    int lkq = 0, lun = 0;
    auto load = [&](float4 (&p)[kTcPieces], uint4 &w) {             // the next unit
      if (lun >= nunit) return;
      const bool kin = lkq * kTcKC + pk < nap;
#pragma unroll
      for (int it = 0; it < kTcPieces; ++it)
        p[it] = kin && it * 32 < left ? __ldg((const float4 *)(src + it * prow)) : make_float4(0.f, 0.f, 0.f, 0.f);
      // this chunk's W^T: hi (threads 0 .. 127) and lo (128 .. 255)
      if (t < kTcConv / 2) w = __ldg(wsrc + lkq * (kBChunk / 32));
      ++lun;
      src += kTcKC;
      if (++lkq == nk) {
        lkq = 0;
        src += tile_step;
        left -= row_step;
      }
    };
    const uint32_t off0 = (uint32_t)(pk >> 3) * kALbo + (uint32_t)(m0 >> 3) * 128u + (uint32_t)(m0 & 7) * 16u + (pk & 4) * 2u;
    int kq = 0;
    auto convert = [&](const float4 (&p)[kTcPieces], const uint4 &w, int buf) {
      unsigned char *Ah = Aop + buf * 2 * kATile + off0;
      const int k = kq * kTcKC + pk;
#pragma unroll
      for (int it = 0; it < kTcPieces; ++it) {
        float4 x = p[it];
        if (k + 3 >= nang) {                                // padding bins are not data
          if (k >= nang) x.x = 0.0f;
          if (k + 1 >= nang) x.y = 0.0f;
          if (k + 2 >= nang) x.z = 0.0f;
          x.w = 0.0f;
        }
        const uint32_t h0 = pack_bf16(x.x, x.y), h1 = pack_bf16(x.z, x.w);
        const uint32_t l0 = pack_bf16(x.x - __uint_as_float(h0 << 16), x.y - __uint_as_float(h0 & 0xffff0000u));
        const uint32_t l1 = pack_bf16(x.z - __uint_as_float(h1 << 16), x.w - __uint_as_float(h1 & 0xffff0000u));
        *(uint2 *)(Ah + it * 512) = make_uint2(h0, h1);            // 32 rows on: four core matrices
        *(uint2 *)(Ah + kATile + it * 512) = make_uint2(l0, l1);
      }
      if (t < kTcConv / 2) *(uint4 *)(Bw + buf * kBChunk + t * 16) = w;
    };
#pragma unroll
    for (int s = 0; s < kTcDepth - 1; ++s) load(v[s], wv[s]);
    for (int u0 = 0; u0 < nunit && ok; u0 += kTcDepth) {
#pragma unroll
      for (int s = 0; s < kTcDepth; ++s) {                        // static register slots
        const int un = u0 + s, buf = un & 1;
        if (un >= nunit || !ok) break;
        load(v[(s + kTcDepth - 1) % kTcDepth], wv[(s + kTcDepth - 1) % kTcDepth]);
        // the MMAs that read this operand buffer two units ago are done
        ok = un < 2 || mbar_wait(smem_addr(emptyA + buf), (uint32_t)((un >> 1) - 1) & 1u);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        convert(v[s], wv[s], buf);
        if (++kq == nk) kq = 0;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) arrive(fullA + buf);
      }
    }
  } else if (warp == kTcConv / 32) {
    // ---- issuing thread
    if (lane == 0) {
      int un = 0;
      for (int ti = 0; ti < mytiles && ok; ++ti) {
        const uint32_t tcol = tmem + (uint32_t)(ti & 1) * kTcN;
        // the tile read back from these columns two tiles ago
        ok = ti < 2 || mbar_wait(smem_addr(emptyD + (ti & 1)), (uint32_t)((ti >> 1) - 1) & 1u);
        for (int kq = 0; kq < nk && ok; ++kq, ++un) {
          const int buf = un & 1;
          ok = mbar_wait(smem_addr(fullA + buf), (uint32_t)(un >> 1) & 1u);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int steps = min(kTcKC / 16, (nang - kq * kTcKC + 15) / 16);    // K steps that hold data
          uint64_t ah = umma_desc(sA + (uint32_t)buf * 2u * kATile, kALbo, kASbo);
          uint64_t bh = umma_desc(sB + (uint32_t)buf * kBChunk, kBLbo, kBSbo);
          constexpr uint64_t dl = kATile >> 4, da = (2 * kALbo) >> 4, dbl = (kBChunk / 2) >> 4, db = (2 * kBLbo) >> 4;
          for (int kk = 0; kk < steps; ++kk, ah += da, bh += db) {   // 2 core matrices per K step
            mma_bf16(tcol, ah, bh, (kq == 0 && kk == 0) ? 0u : 1u);
            mma_bf16(tcol, ah, bh + dbl, 1u);
            mma_bf16(tcol, ah + dl, bh, 1u);
          }
          commit(emptyA + buf);
          if (kq == nk - 1) commit(fullD + (ti & 1));
        }
      }
      // let the MMAs in flight end (again with a limit)
      if (!ok && un > 0) mbar_wait(smem_addr(emptyA + ((un - 1) & 1)), (uint32_t)((un - 1) >> 1) & 1u);
    }
  } else {
    // ---- epilogue: lane m of a tile's TMEM columns holds the 16 sums of its cell m
    const int ew = warp & 3;                               // TMEM lanes 32 ew .. + 31 are this warp's
    auto cell_of = [&](int ti) { return (blockIdx.x + (long long)ti * gridDim.x) * kTcM + ew * 32 + lane; };
    // ONE chunk per tile (64 bins or fewer): four warps of this role in place of
    // the previous form's sixteen per SM, each of which did it, are the chain of
    // the whole kernel, so a tile's velocities travel a tile ahead.  Fluid frame,
    // previous form -> without -> with: 96^3 cells x 42 bins 63.6 -> 74.3 -> 64.7 us,
    // 12 bins 59.0 -> 63.6 -> 52.2.  With more chunks there is time, and 92 bins lose
    // by it (101 -> 109 us).
    double un[3] = {0.0, 0.0, 0.0};
    auto fetch = [&](int ti) {
      const long long cell = cell_of(ti);
      if (frame != RAD_FRAME_FLUID || ti >= mytiles || cell >= ncell) return;
#pragma unroll
      for (int q = 0; q < 3; ++q) un[q] = __ldg(u + 3 * cell + q);
    };
    if (ONE) fetch(0);
    for (int ti = 0; ti < mytiles; ++ti) {
      const float nx = (float)un[0], ny = (float)un[1], nz = (float)un[2];
      if (ONE) fetch(ti + 1);
      ok = mbar_wait(smem_addr(fullD + (ti & 1)), (uint32_t)(ti >> 1) & 1u);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      uint32_t r[16];
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
            "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(tmem + (uint32_t)(ti & 1) * kTcN + ((uint32_t)(ew * 32) << 16)));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (lane == 0) arrive(emptyD + (ti & 1));
      const long long cell = cell_of(ti);
      if (cell >= ncell) continue;
      float Rt[10];
#pragma unroll
      for (int p = 0; p < 10; ++p) Rt[p] = __uint_as_float(r[p]);
      float Ro[10];
      if (frame == RAD_FRAME_TETRAD) {
#pragma unroll
        for (int p = 0; p < 10; ++p) Ro[p] = Rt[p];
      } else {
        float L[4][4];
        if (frame == RAD_FRAME_COORD) {
          const ColGeoF &cg = cols[cell % ncol];
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) L[a][b] = cg.e[a][b];
        } else {
          const float ux = ONE ? nx : (float)u[3 * cell], uy = ONE ? ny : (float)u[3 * cell + 1],
                      uz = ONE ? nz : (float)u[3 * cell + 2];
          const float uu[3] = {ux, uy, uz};
          const float u0 = sqrtf(1.0f + ux * ux + uy * uy + uz * uz);
          L[0][0] = u0;
#pragma unroll
          for (int a = 0; a < 3; ++a) {
            L[0][a + 1] = -uu[a];
            L[a + 1][0] = -uu[a];
#pragma unroll
            for (int b = 0; b < 3; ++b) {
              // a zero numerator (gas at rest, or along an axis) would take the
              // division's slow path (64^3 x 32 bins at rest 30.5 -> 20.9 us, 26.1 in the
              // previous form); asm: the compiler would undo the select
              const float w = uu[a] * uu[b];
              float num = w == 0.0f ? 1.0f : w;
              asm("" : "+f"(num));
              const float q = num / (1.0f + u0);
              L[a + 1][b + 1] = (w == 0.0f ? 0.0f : q) + (a == b ? 1.0f : 0.0f);
            }
          }
        }
        const float R4[4][4] = {{Rt[0], Rt[1], Rt[2], Rt[3]},
                                {Rt[1], Rt[4], Rt[5], Rt[6]},
                                {Rt[2], Rt[5], Rt[7], Rt[8]},
                                {Rt[3], Rt[6], Rt[8], Rt[9]}};
        float T4[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int B = 0; B < 4; ++B)
            T4[a][B] = L[a][0] * R4[0][B] + L[a][1] * R4[1][B] + L[a][2] * R4[2][B] + L[a][3] * R4[3][B];
        const int pa[10] = {0, 0, 0, 0, 1, 1, 1, 2, 2, 3}, pb[10] = {0, 1, 2, 3, 1, 2, 3, 2, 3, 3};
#pragma unroll
        for (int p = 0; p < 10; ++p)
          Ro[p] = T4[pa[p]][0] * L[pb[p]][0] + T4[pa[p]][1] * L[pb[p]][1] + T4[pa[p]][2] * L[pb[p]][2] +
                  T4[pa[p]][3] * L[pb[p]][3];
      }
      float *o = out + cell * 10;
#pragma unroll
      for (int p = 0; p < 10; ++p) o[p] = Ro[p];
    }
  }
  if (!ok) atomicOr(err, kTcErrTimeout);
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(tmem));
}

namespace {

uint16_t bf16_bits(float x) {
  // round to nearest even (finite inputs)
  uint32_t b;
  std::memcpy(&b, &x, 4);
  uint32_t rnd = 0x7FFFu + ((b >> 16) & 1u);
  return (uint16_t)((b + rnd) >> 16);
}
float bf16_to_float(uint16_t h) {
  uint32_t b = (uint32_t)h << 16;
  float f;
  std::memcpy(&f, &b, 4);
  return f;
}

}  // namespace

// Build W^T = (n^A n^B dOmega)^T split into bf16 hi / lo in the B layout.
static int build_wt(rad_ctx *ctx, int kp, std::string &err) {
  const AngleGrid &g = ctx->ang;
  const int pa[10] = {0, 0, 0, 0, 1, 1, 1, 2, 2, 3}, pb[10] = {0, 1, 2, 3, 1, 2, 3, 2, 3, 3};
  size_t half = (size_t)kp * kTcN;          // bf16 elements per operand half
  std::vector<uint16_t> buf(2 * half, 0);
  for (int n = 0; n < g.n_ang; ++n) {
    double nv[4] = {1.0, g.dir[3 * n], g.dir[3 * n + 1], g.dir[3 * n + 2]};
    for (int p = 0; p < 10; ++p) {
      float w = (float)(nv[pa[p]] * nv[pb[p]] * g.dOmega[n]);
      uint16_t hi = bf16_bits(w);
      uint16_t lo = bf16_bits(w - bf16_to_float(hi));
      // element (row p, k = n): core (p / 8, n / 8), row p % 8, column n % 8
      size_t off = ((size_t)(n / 8) * 2 + p / 8) * 64 + (p % 8) * 8 + (n % 8);
      buf[off] = hi;
      buf[half + off] = lo;
    }
  }
  cudaFree(ctx->wt_dev);
  ctx->wt_dev = nullptr;
  if (alloc_scratch(ctx, (void **)&ctx->wt_dev, buf.size() * 2) != cudaSuccess) {
    err = "moment weight allocation failed";
    return RAD_ENOMEM;
  }
  cudaMemcpyAsync(ctx->wt_dev, buf.data(), buf.size() * 2, cudaMemcpyHostToDevice, ctx->stream);
  cudaStreamSynchronize(ctx->stream);
  ctx->wt_kp = kp;
  ctx->wt_level = g.level;
  return RAD_OK;
}

int launch_moments_bf16x3(rad_ctx *ctx, const float *I, int frame, const double *u, float *R, cudaStream_t st,
                          std::string &err) {
  const DevGeom &G = ctx->geom;
  const int kp = (ctx->ang.n_ap + kTcKC - 1) / kTcKC * kTcKC;
  if (ctx->wt_dev == nullptr || ctx->wt_kp != kp || ctx->wt_level != ctx->ang.level) {
    int st = build_wt(ctx, kp, err);
    if (st != RAD_OK) return st;
  }
  const long long ncell = (long long)G.n[0] * G.n[1] * G.n[2];
  if (kp > kTcMaxKp) {
    err = "split-bf16 moments: too many bins";
    return RAD_EUNSUPPORTED;
  }
  // two operand buffers (hi, lo), two W^T chunks, barriers and TMEM slot
  constexpr size_t smem = 4 * (size_t)kATile + 2 * kBChunk + 128;
  const auto kernel = kp == kTcKC ? k_moments_tc<true> : k_moments_tc<false>;
  cudaError_t ce = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (ce != cudaSuccess) {
    err = std::string("split-bf16 moments: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  long long ntile = (ncell + kTcM - 1) / kTcM;
  const long long blocks = std::min<long long>(ntile, nsm);        // one persistent CTA per SM
  kernel<<<(unsigned)blocks, kTcThreads, smem, st>>>(I, R, ncell, ctx->ang.n_ap, ctx->ang.n_ang, kp,
                                                     (const uint4 *)ctx->wt_dev, frame, G.colsF, G.n[0] * G.n[1], u,
                                                     ctx->err_word);
  ce = cudaGetLastError();
  if (ce != cudaSuccess) {
    err = std::string("split-bf16 moments launch failed: ") + cudaGetErrorString(ce);
    return RAD_ECUDA;
  }
  return RAD_OK;
}

}  // namespace rad
