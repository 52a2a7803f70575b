// Tensor-core (tcgen05) products of the Fourier neural operator's pointwise
// channel maps: C[b](m, p) = sum_k A(m, k) X[b](k, p) (+ beta C + bias[m]),
// with A a bfloat16 weight matrix (any strides; NC = 64 or 128 rows, K = 64
// or 128) and X the float32 activations [k][p] (p contiguous, P a multiple
// of 128).
//
// The product runs transposed on the tensor cores: each tile is 128 points
// (the MMA's M), NC channels (its N) and K input channels, accumulated in
// tensor memory (TMEM, one 32-bit column per output channel, one lane per
// point).  The weights are exact in bfloat16; each float32 activation x is
// split into three bfloat16 terms, x = h + m + l up to the last bit of its
// 24-bit significand (h = bf16(x), m = bf16(x - h), l = bf16(x - h - m)),
// so that A X = A h + A m + A l with every product exact and float32
// accumulation: three MMA passes per K step instead of one, at float32
// accuracy (the technique of splitting a float32 operand into bfloat16
// terms: Henry, Tang and Heinecke, "Leveraging the bfloat16 artificial
// intelligence datatype for higher-precision computations", ARITH 2019).
//
// Shared-memory operands are K-major with the 128-byte swizzle (rows of 64
// bfloat16, 16-byte chunk c of row r stored at chunk c ^ (r & 7), 1024-byte
// aligned blocks of 8 rows), written by the threads from registers (the
// activations need the split, so no TMA here); one thread issues the MMAs
// and commits them to an mbarrier that every thread waits on (bounded).
// Persistent CTAs of 128 threads loop over tiles; the weights are staged once.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "async_copy.cuh"
#include "fno_internal.h"
#include "fno_umma.cuh"
#include "smem_grant.h"

namespace spgpe {
namespace fno {

namespace {

// Shared memory: three activation terms [term][kb][128 rows][128 B], the
// weights [kb][NC rows][128 B], the mbarrier and the TMEM address slot.
template <int NC, int KB> struct TcSmem {
  static constexpr size_t kTerm = (size_t)KB * kTcRows * kRowBytes;
  static constexpr size_t kA = 3 * kTerm;
  static constexpr size_t kB = (size_t)KB * NC * kRowBytes;
  static constexpr size_t kBytes = 1024 /* alignment slack */ + kA + kB + 16;
};

template <int NC, int KB>
__global__ void __launch_bounds__(128) gemm_tc(int ntiles, int tiles_per_batch, const __nv_bfloat16 *__restrict__ A,
                                               long sAm, long sAk, const float *__restrict__ X, long sXk, long sXb,
                                               float *C, long sCm, long sCb, float beta,
                                               const float *__restrict__ bias, int *flags) {
  constexpr int K = KB * kKBlock;
  using S = TcSmem<NC, KB>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sA = sm;            // activation terms
  unsigned char *sB = sm + S::kA;    // weights
  uint64_t *bar = reinterpret_cast<uint64_t *>(sB + S::kB);
  uint32_t *slot = reinterpret_cast<uint32_t *>(bar + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 0) {
    tmem_alloc(slot, NC);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  // weights, once: row m (output channel), chunk j holds k = 8 j .. 8 j + 7
  for (int e = tid; e < NC * (K / 8); e += blockDim.x) {
    const int m = e / (K / 8), j = e - m * (K / 8);
    const int kb = j / 8, jc = j % 8;
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const long k0 = 8L * j + 2 * i;
      w[i] = pack_bf16(A[m * sAm + k0 * sAk], A[m * sAm + (k0 + 1) * sAk]);
    }
    *reinterpret_cast<uint4 *>(sB + (size_t)kb * NC * kRowBytes + sw128(m, jc)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  constexpr uint32_t idesc = idesc_bf16(kTcRows, NC);
  // Software pipeline: while the tensor cores and the epilogue work on one
  // tile, this thread's activations of the next tile (and, for 64 output
  // channels, the previous C values of the current one) are already in flight.
  float xr[K];
  auto load_x = [&](int tile) {
    const int b = tile / tiles_per_batch;
    const float *xs = X + b * sXb + (long)(tile - b * tiles_per_batch) * kTcRows + tid;
#pragma unroll
    for (int k = 0; k < K; ++k) xr[k] = xs[(long)k * sXk];
  };
  constexpr bool kPreC = NC == 64;
  float cpre[kPreC ? NC : 1];
  bool ok = true;
  int it = 0;
  int tile = blockIdx.x;
  if (tile < ntiles) load_x(tile);
  for (; tile < ntiles && ok; tile += gridDim.x, ++it) {
    const int b = tile / tiles_per_batch;
    const long p0 = (long)(tile - b * tiles_per_batch) * kTcRows;
    // this thread's point p0 + tid: three bfloat16 terms per activation
#pragma unroll
    for (int j = 0; j < K / 8; ++j) {
      uint32_t hw[4], mw[4], lw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        __nv_bfloat16 h[2], md[2], lo[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float v = xr[8 * j + 2 * i + q];
          h[q] = __float2bfloat16_rn(v);
          const float r1 = v - __bfloat162float(h[q]);
          md[q] = __float2bfloat16_rn(r1);
          lo[q] = __float2bfloat16_rn(r1 - __bfloat162float(md[q]));
        }
        hw[i] = pack_bf16(h[0], h[1]);
        mw[i] = pack_bf16(md[0], md[1]);
        lw[i] = pack_bf16(lo[0], lo[1]);
      }
      const size_t off = (size_t)(j / 8) * kTcRows * kRowBytes + sw128(tid, j % 8);
      *reinterpret_cast<uint4 *>(sA + off) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
      *reinterpret_cast<uint4 *>(sA + S::kTerm + off) = make_uint4(mw[0], mw[1], mw[2], mw[3]);
      *reinterpret_cast<uint4 *>(sA + 2 * S::kTerm + off) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
    // the tensor cores read shared memory through the async proxy
    fence_proxy_async();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
#pragma unroll 1
      for (int t = 0; t < 3; ++t)
#pragma unroll
        for (int kb = 0; kb < KB; ++kb) {
          const uint64_t ad = sw128_desc(sA + t * S::kTerm + (size_t)kb * kTcRows * kRowBytes);
          const uint64_t bd = sw128_desc(sB + (size_t)kb * NC * kRowBytes);
#pragma unroll
          for (int kk = 0; kk < kKBlock / 16; ++kk)  // 16 bfloat16 = 32 bytes per MMA
            umma_bf16(tmem, ad + 2 * kk, bd + 2 * kk, idesc, (t | kb | kk) != 0);
        }
      umma_commit(bar);
    }
    // lane (warp, lane) holds point p0 + 32 warp + lane, one TMEM column per channel
    const long p = p0 + 32 * warp + lane;
    float *cb = C + b * sCb + p;
    if (tile + (int)gridDim.x < ntiles) load_x(tile + gridDim.x);
    if constexpr (kPreC) {
      if (beta != 0.f)
#pragma unroll
        for (int m = 0; m < NC; ++m) cpre[m] = cb[m * sCm];
    }
    ok = mbar_wait_bounded(bar, (uint32_t)(it & 1));
    if (!__syncthreads_and(ok)) {
      // the MMAs never completed: record it, give them one more bounded wait
      if (tid == 0) atomicOr(flags, kErrTimeout);
      mbar_wait_bounded(bar, (uint32_t)(it & 1));
      ok = false;
      break;
    }
    tc_fence_after();
#pragma unroll
    for (int c0 = 0; c0 < NC; c0 += 16) {
      float v[16];
      tmem_ld16(tmem + ((uint32_t)(32 * warp) << 16) + (uint32_t)c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int m = c0 + i;
        float o = v[i];
        if (beta != 0.f) {
          if constexpr (kPreC) o = fmaf(beta, cpre[m], o);
          else o = fmaf(beta, cb[m * sCm], o);
        }
        if (bias) o += bias[m];
        cb[m * sCm] = o;
      }
    }
    // every lane is read before the next tile's MMAs overwrite the accumulator
    tc_fence_before();
    __syncthreads();
  }
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, NC);
  }
}

template <int NC, int KB>
cudaError_t launch_tc(const GemmR &g, cudaStream_t st) {
  auto kern = gemm_tc<NC, KB>;
  const size_t smem = TcSmem<NC, KB>::kBytes;
  static SmemGrant grant;
  cudaError_t e = grant(kern, smem);
  if (e != cudaSuccess) return e;
  static int occ = 0, sms = 0;
  if (!sms) {
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, 128, smem);
    if (e != cudaSuccess) return e;
    int dev = 0;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  }
  const int tpb = g.N / kTcRows, ntiles = tpb * g.batch;
  const int grid = std::max(1, std::min(ntiles, std::max(1, occ) * sms));
  kern<<<grid, 128, smem, st>>>(ntiles, tpb, static_cast<const __nv_bfloat16 *>(g.A), g.sAm, g.sAk, g.B, g.sBk,
                                g.sBb, g.C, g.sCm, g.sCb, g.beta, g.bias, g.flags);
  return cudaGetLastError();
}

// Weight gradients on the tensor cores: dW[m][n] = sum over samples and points
// of X[b](m, p) Y[b](n, p), m < M, n < N, both operands float32 with unit
// stride along p (the K dimension of the MMA), and the bias gradient db[m] =
// sum X[b](m, p) beside it (X is on its way through the registers anyway).
// Each operand is split into two bfloat16 terms (x = h + l, 16 significant
// bits), and the three products h h', h l', l h' are accumulated (the dropped
// l l' is below 2^-16 of the result).  The MMA tile is 128 rows of X (M <= MR =
// 64 or 128; the rows from M on stay zero) by NC = 16, 64 or 128 rows of Y (N <=
// NC, likewise); the terms of Y lie side by side, so that X's h term meets both
// in one MMA of 2 NC columns.  A CTA takes a run of 64-point blocks and leaves
// one partial sum: two CTAs per SM, and more of them once their runs would
// exceed kGradRun blocks (the accumulator truncates, so its error grows with the
// run); two operand buffers, the next block's values in registers while the
// tensor cores work.  Bound by the one read of both operands.
template <int MR, int NC> struct WgSmem {
  static constexpr size_t kA = (size_t)kTcRows * kRowBytes;  // one term of X
  static constexpr size_t kB = (size_t)NC * kRowBytes;       // one term of Y
  static constexpr size_t kStage = 2 * kA + 2 * kB;
  static constexpr size_t kBytes = 1024 + 2 * kStage + 64;
};

constexpr int kWgThreads = 256;
static_assert(kGradBlock == kKBlock, "a block of points is one K block");

template <int MR, int NC>
__global__ void __launch_bounds__(kWgThreads, 2) gemm_tc_wgrad(int M, int N, int nblk, int blocks_per_sample,
                                                            const float *__restrict__ X, long sXm, long sXb,
                                                            const float *__restrict__ Y, long sYn, long sYb, float *part,
                                                            long sPs, int with_bias, int *flags) {
  using S = WgSmem<MR, NC>;
  constexpr uint32_t kCols = 2 * NC < 32 ? 32 : 2 * NC;
  constexpr int CHX = MR * 8 / kWgThreads;  // 16-byte runs of X of one 64-point block per thread
  static_assert((MR + NC) * 8 % kWgThreads == 0 || NC == 16, "whole runs per thread");
  constexpr int CHT = ((MR + NC) * 8 + kWgThreads - 1) / kWgThreads;  // those of X and Y
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t *mma = reinterpret_cast<uint64_t *>(sm + 2 * S::kStage);
  uint32_t *slot = reinterpret_cast<uint32_t *>(mma + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b0 = (int)((long)blockIdx.x * nblk / gridDim.x), b1 = (int)((long)(blockIdx.x + 1) * nblk / gridDim.x);

  if (warp == 0) {
    tmem_alloc(slot, kCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&mma[0], 1);
    mbar_init(&mma[1], 1);
    mbar_fence_init();
  }
  // rows M..127 of both X terms and N..NC-1 of both Y terms stay zero
  for (int s = 0; s < 2; ++s) {
    unsigned char *sA = sm + s * S::kStage, *sB = sA + 2 * S::kA;
    for (int e = tid; e < (kTcRows - M) * 8; e += kWgThreads) {
      const int r = M + e / 8, c = e % 8;
      *reinterpret_cast<uint4 *>(sA + sw128(r, c)) = make_uint4(0, 0, 0, 0);
      *reinterpret_cast<uint4 *>(sA + S::kA + sw128(r, c)) = make_uint4(0, 0, 0, 0);
    }
    for (int e = tid; e < (NC - N) * 8; e += kWgThreads) {
      const int r = N + e / 8, c = e % 8;
      *reinterpret_cast<uint4 *>(sB + sw128(r, c)) = make_uint4(0, 0, 0, 0);
      *reinterpret_cast<uint4 *>(sB + S::kB + sw128(r, c)) = make_uint4(0, 0, 0, 0);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  // run q of a block: rows 0..MR-1 of X then rows of Y, 8 runs (64 points) per row
  float4 xr[CHT][2];
  float bsum[CHX];
#pragma unroll
  for (int q = 0; q < CHX; ++q) bsum[q] = 0.f;
  // valid rows only (the others keep their zeros)
  auto valid = [&](int r) { return r < MR ? r < M : r - MR < N; };
  auto load = [&](int blk) {
    const int b = blk / blocks_per_sample;
    const long k0 = (long)(blk - b * blocks_per_sample) * kKBlock;
    const float *xb = X + b * sXb + k0, *yb = Y + b * sYb + k0;
#pragma unroll
    for (int q = 0; q < CHT; ++q) {
      const int e = tid + q * kWgThreads, r = e / 8, c = e % 8;
      if (valid(r)) {
        const float *src = r < MR ? xb + r * sXm + 8 * c : yb + (r - MR) * sYn + 8 * c;
        xr[q][0] = *reinterpret_cast<const float4 *>(src);
        xr[q][1] = *reinterpret_cast<const float4 *>(src + 4);
      }
    }
  };
  bool ok = true;
  if (b0 < b1) load(b0);
  int i = 0;
  for (int blk = b0; blk < b1 && ok; ++blk, ++i) {
    const int s = i & 1;
    unsigned char *sA = sm + s * S::kStage, *sB = sA + 2 * S::kA;
    if (i >= 2) ok = mbar_wait_bounded(&mma[s], (uint32_t)(((i >> 1) - 1) & 1));
#pragma unroll
    for (int q = 0; q < CHT; ++q) {
      const int e = tid + q * kWgThreads, r = e / 8, c = e % 8;
      if (!valid(r)) continue;
      const float v[8] = {xr[q][0].x, xr[q][0].y, xr[q][0].z, xr[q][0].w,
                          xr[q][1].x, xr[q][1].y, xr[q][1].z, xr[q][1].w};
      if (q < CHX) bsum[q < CHX ? q : 0] += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
      uint32_t hw[4], lw[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        hw[j] = cvt_bf16x2(v[2 * j], v[2 * j + 1]);
        lw[j] = cvt_bf16x2(v[2 * j] - __uint_as_float(hw[j] << 16), v[2 * j + 1] - __uint_as_float(hw[j] & 0xffff0000u));
      }
      unsigned char *dst = r < MR ? sA + sw128(r, c) : sB + sw128(r - MR, c);
      const size_t term = r < MR ? S::kA : S::kB;
      *reinterpret_cast<uint4 *>(dst) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
      *reinterpret_cast<uint4 *>(dst + term) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
    if (blk + 1 < b1) load(blk + 1);
    fence_proxy_async();
    ok = __syncthreads_and(ok);
    if (tid == 0) {
      // (the commit follows in any case, so that every wait ends)
      tc_fence_after();
      const uint64_t ah = sw128_desc(sA), al = sw128_desc(sA + S::kA), bd = sw128_desc(sB);
      if (ok)
#pragma unroll
        for (int kk = 0; kk < kKBlock / 16; ++kk) {
          umma_bf16(tmem, ah + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, 2 * NC), (i | kk) != 0);
          umma_bf16(tmem, al + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, NC), 1);
        }
      umma_commit(&mma[s]);
    }
  }
  // every MMA issued is complete before the buffers go (and the barrier brings
  // the lanes together for the tensor-memory loads)
  if (i > 0) ok = mbar_wait_bounded(&mma[(i - 1) & 1], (uint32_t)(((i - 1) >> 1) & 1)) && ok;
  ok = __syncthreads_and(ok);
  if (!ok && tid == 0) atomicOr(flags, kErrTimeout);
  tc_fence_after();
  // rows 0..M-1 of the accumulator, columns n and NC + n: warps 0-3 and 4-7
  // hold the same lanes and take alternate groups of columns
  float *out = part + (long)blockIdx.x * sPs;
  if (ok && 32 * (warp & 3) < M) {
    const int m = 32 * (warp & 3) + lane;
#pragma unroll
    for (int c0 = 8 * (warp >> 2); c0 < NC; c0 += 16) {
      float v[8], u[8];
      tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
      tmem_ld8(tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(NC + c0), u);
      tmem_ld_wait();
      if (m < M)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (c0 + j < N) out[(long)m * N + c0 + j] = i > 0 ? v[j] + u[j] : 0.f;
    }
  }
  if (with_bias) {  // 8 lanes hold a row
#pragma unroll
    for (int q = 0; q < CHX; ++q) {
      float v = bsum[q];
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const int r = (tid + q * kWgThreads) / 8;
      if ((tid & 7) == 0 && r < M) out[(long)M * N + r] = v;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
}

template <int MR, int NC>
cudaError_t launch_wgrad(const WeightGrad &g, int grid, cudaStream_t st) {
  auto kern = gemm_tc_wgrad<MR, NC>;
  constexpr size_t smem = WgSmem<MR, NC>::kBytes;
  static SmemGrant grant;
  const cudaError_t e = grant(kern, smem);
  if (e != cudaSuccess) return e;
  const int bps = (int)(g.P / kKBlock);
  kern<<<grid, kWgThreads, smem, st>>>(g.M, g.N, g.batch * bps, bps, g.X, g.P, g.sXb, g.Y, g.P, g.sYb, g.part,
                                       (long)g.M * g.N + (g.bias ? g.M : 0), g.bias ? 1 : 0, g.flags);
  return cudaGetLastError();
}

}  // namespace

bool weight_grad_applies(const WeightGrad &g) {
  return g.M >= 1 && g.M <= 128 && g.N >= 1 && g.N <= 128 && g.P % kKBlock == 0 && g.sXb % 4 == 0 && g.sYb % 4 == 0 &&
         (reinterpret_cast<uintptr_t>(g.X) & 15) == 0 && (reinterpret_cast<uintptr_t>(g.Y) & 15) == 0;
}

cudaError_t weight_grad(const WeightGrad &g, int sms, cudaStream_t st) {
  const int grid = weight_grad_parts(g.batch, g.P, sms);
  cudaError_t e;
  if (g.M <= 64) {
    if (g.N <= 16) e = launch_wgrad<64, 16>(g, grid, st);
    else e = g.N <= 64 ? launch_wgrad<64, 64>(g, grid, st) : launch_wgrad<64, 128>(g, grid, st);
  } else {
    if (g.N <= 16) e = launch_wgrad<128, 16>(g, grid, st);
    else e = g.N <= 64 ? launch_wgrad<128, 64>(g, grid, st) : launch_wgrad<128, 128>(g, grid, st);
  }
  return e;
}

bool gemm_tc_applies(const GemmR &g) {
  return g.a_bf16 && g.flags && !g.partial && g.splits == 1 && g.alpha == 1.f && g.sAb == 0 && g.sBn == 1 &&
         g.sCn == 1 && (g.M == 64 || g.M == 128) && (g.K == 64 || g.K == 128) && g.N % kTcRows == 0 &&
         g.N >= kTcRows;
}

cudaError_t gemm_real_tc(const GemmR &g, cudaStream_t st) {
  if (!gemm_tc_applies(g)) return cudaErrorNotSupported;
  if (g.M == 64) return g.K == 64 ? launch_tc<64, 1>(g, st) : launch_tc<64, 2>(g, st);
  return g.K == 64 ? launch_tc<128, 1>(g, st) : launch_tc<128, 2>(g, st);
}

}  // namespace fno
}  // namespace spgpe
