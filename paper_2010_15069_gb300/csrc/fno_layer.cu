// The pointwise half of a spectral layer on the tensor cores (tcgen05), fused
// with the inverse transform along x and the activation:
//
//   u[b][c][y][x] = sum_c' W[c][c'] v[b][c'][y][x] + w[c]
//                 + sum_k T[x][k] G[b][c][y][k],     v_next = gelu(u)
//
// (k = 2 kx + part, T = cos, -sin; G from the inverse along y), and its
// transpose in the backward pass, dv = W^T du + T G, times gelu'(u of the
// layer before).  Run as separate products, a layer wrote u, read and wrote it
// again, and read and wrote it for the activation: five passes over the
// activations more than the read of v and the writes of u and v_next left
// here, which are what bounds the kernel.
//
// A tile is 128 points of one row y of one sample.  D[128 points][W channels]
// is summed in two parts: v (three bfloat16 terms per value, split_3) times the
// weights (bfloat16, exact), and T times G, both split in three with the
// leading products exact (split3_grid; G scaled per channel and row).  T stays
// in shared memory: a CTA keeps one x tile and walks (sample, y).  Two operand
// buffers and two sets of accumulators: a tile's results leave while the next
// one is in the tensor cores, and the values of the one after are in
// registers.
//
// Measured on GB300 at 256^2, batch 4, W = 64: 79 us forward for what
// took 61 + 153 + 33 us in three products and passes, 91 us backward for 61 +
// 153 + 68.
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

constexpr int kThreads = 512;
constexpr size_t kTermA = (size_t)kTcRows * kRowBytes;

enum LayerMode { kForward, kForwardLast, kBackward, kBackwardGelu };

struct LayerArgs {
  const float *v;             // [b][W][n][n] input
  const float *G;             // [b][W][n][2M]
  const unsigned char *tab;   // [x tiles][3 terms][128 rows][128 bytes], swizzled
  const __nv_bfloat16 *weights;
  long sOut, sIn;             // strides of the weights along output and input channels
  const float *bias;          // forward
  float *u;                   // forward: u, null to leave it out; backward: u of the layer before (read)
  float *out;                 // v_next or dv
  int n, M, xtiles, rows;     // rows = batch n
  float g0, g1;               // factors of G at kx = 0 and elsewhere
  int *flags;
};

template <int W> struct LayerSmem {
  static constexpr size_t kA2 = 3 * kTermA;                    // T
  static constexpr size_t kA1 = 2 * 3 * kTermA;                // v, two buffers
  static constexpr size_t kG = (size_t)3 * W * kRowBytes;      // G, one buffer
  static constexpr size_t kB1 = (size_t)W * kRowBytes;         // weights
  static constexpr size_t kBytes = 1024 + kA2 + kA1 + 2 * kG + kB1 + (3 * W + W) * sizeof(float) + 64;
};

template <int W, int MODE>
__global__ void __launch_bounds__(kThreads, 1) layer(const LayerArgs a) {
  using S = LayerSmem<W>;
  constexpr int RUNS = W / 32;     // runs of 8 channels per thread
  constexpr uint32_t kCols = 512;  // two tiles: W columns of W v, then 3 W of T G
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sT = sm, *sV = sT + S::kA2, *sG = sV + S::kA1, *sW = sG + 2 * S::kG;
  float *un = reinterpret_cast<float *>(sW + S::kB1);  // [tile % 3][channel] factor of the T G sum
  float *bias = un + 3 * W;
  uint64_t *mma = reinterpret_cast<uint64_t *>(bias + W), *full = mma + 2;
  uint32_t *slot = reinterpret_cast<uint32_t *>(full + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n, q2 = 2 * a.M;
  const int xt = blockIdx.x % a.xtiles, first = blockIdx.x / a.xtiles, stride = gridDim.x / a.xtiles;
  const int tiles = (a.rows - first + stride - 1) / stride;
  const int x0 = xt * kTcRows;
  const long plane = (long)n * n;

  if (warp == 0) {
    tmem_alloc(slot, kCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&mma[0], 1);
    mbar_init(&mma[1], 1);
    mbar_init(full, 1);
    mbar_fence_init();
    mbar_expect_tx(full, (uint32_t)S::kA2);
    bulk_g2s(sT, a.tab + (size_t)xt * S::kA2, (uint32_t)S::kA2, full);
  }
  for (int e = tid; e < W * (W / 8); e += kThreads) {  // weights: row c, run j holds inputs 8 j .. 8 j + 7
    const int c = e / (W / 8), j = e - c * (W / 8);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = pack_bf16(a.weights[c * a.sOut + (8 * j + 2 * i) * a.sIn], a.weights[c * a.sOut + (8 * j + 2 * i + 1) * a.sIn]);
    *reinterpret_cast<uint4 *>(sW + sw128(c, j)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if (tid < W) bias[tid] = (MODE == kForward || MODE == kForwardLast) ? a.bias[tid] : 0.f;

  // a thread's values of a tile: point tid & 127, channels 8 (tid >> 7) + 32 i
  // .. + 7; of G: channel tid >> 3, run tid & 7
  const int pt = tid & 127;
  const bool inside = x0 + pt < n;  // (a 64-point row fills half of its tile)
  float x[RUNS][8], gv[8];
  auto load = [&](int t) {
    const int row = first + t * stride, b = row / n, y = row - b * n;
    const float *p = a.v + (long)b * W * plane + (long)y * n + x0 + pt;
#pragma unroll
    for (int i = 0; i < RUNS; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) x[i][j] = inside ? p[((tid >> 7) * 8 + 32 * i + j) * plane] : 0.f;
    if (tid < 8 * W) {
      const float *q = a.G + (((long)b * W + (tid >> 3)) * n + y) * q2 + (tid & 7) * 8;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = (tid & 7) * 8 + 4 * h;
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < q2) r = *reinterpret_cast<const float4 *>(q + 4 * h);
        const float f = k == 0 ? a.g0 : a.g1;
        gv[4 * h] = r.x * f;
        gv[4 * h + 1] = r.y * f;
        gv[4 * h + 2] = r.z * a.g1;
        gv[4 * h + 3] = r.w * a.g1;
      }
    }
  };
  auto store = [&](int s, int slot3) {
    unsigned char *A = sV + s * 3 * kTermA;
#pragma unroll
    for (int i = 0; i < RUNS; ++i) {
      uint4 h, m, l;
      split3(x[i], h, m, l);
      const uint32_t off = sw128(pt, (tid >> 7) + 4 * i);
      *reinterpret_cast<uint4 *>(A + off) = h;
      *reinterpret_cast<uint4 *>(A + kTermA + off) = m;
      *reinterpret_cast<uint4 *>(A + 2 * kTermA + off) = l;
    }
    if (tid < 8 * W) {
      float vm = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) vm = fmaxf(vm, fabsf(gv[j]));
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) vm = fmaxf(vm, __shfl_xor_sync(0xffffffffu, vm, o));
      uint4 h, m, l;
      split3_grid(gv, grid_scale(vm), h, m, l);
      unsigned char *B = sG + s * S::kG;
      const uint32_t off = sw128(tid >> 3, tid & 7);
      *reinterpret_cast<uint4 *>(B + off) = h;
      *reinterpret_cast<uint4 *>(B + (size_t)W * kRowBytes + off) = m;
      *reinterpret_cast<uint4 *>(B + (size_t)2 * W * kRowBytes + off) = l;
      if ((tid & 7) == 0) un[slot3 * W + (tid >> 3)] = grid_unscale(vm);
    }
  };
  load(0);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  constexpr uint32_t idesc = idesc_bf16(kTcRows, W);
  const int xp = x0 + 32 * (warp & 3) + lane;  // the point of this thread's accumulator lane
  // results of tile t: warps of a group of four hold 32 points each, the four
  // groups take alternate runs of 8 channels
  auto epilogue = [&](int t, const float (&up)[RUNS][8]) {
    const int row = first + t * stride, b = row / n, y = row - b * n;
    const uint32_t base = tmem + 256 * (t & 1) + ((uint32_t)(32 * (warp & 3)) << 16);
    const float *f = un + (t % 3) * W;
    const long o0 = (long)b * W * plane + (long)y * n + xp;
#pragma unroll
    for (int i = 0; i < RUNS; ++i) {
      const int c0 = (warp >> 2) * 8 + 32 * i;
      float v[8], p[8], q[8], r[8];
      tmem_ld8(base + c0, v);
      tmem_ld8(base + W + c0, p);
      tmem_ld8(base + 2 * W + c0, q);
      tmem_ld8(base + 3 * W + c0, r);
      tmem_ld_wait();
      if (xp < n) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int c = c0 + j;
          const float d = fmaf(p[j] + (q[j] + r[j]), f[c], v[j]);
          const long o = o0 + c * plane;
          if constexpr (MODE == kForward) {
            const float u = d + bias[c];
            if (a.u) a.u[o] = u;
            a.out[o] = gelu_f(u);
          } else if constexpr (MODE == kForwardLast) {
            a.out[o] = d + bias[c];
          } else if constexpr (MODE == kBackwardGelu) {
            a.out[o] = d * gelu_d(up[i][j]);
          } else {
            a.out[o] = d;
          }
        }
      }
    }
    tc_fence_before();
  };
  // (backward) the activations whose derivative tile t is multiplied by
  auto load_u = [&](int t, float (&up)[RUNS][8]) {
    if constexpr (MODE == kBackwardGelu) {
      const int row = first + t * stride, b = row / n, y = row - b * n;
      const float *p = a.u + (long)b * W * plane + (long)y * n + xp;
#pragma unroll
      for (int i = 0; i < RUNS; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) up[i][j] = xp < n ? p[((warp >> 2) * 8 + 32 * i + j) * plane] : 0.f;
    }
  };

  bool ok = true, go = true;  // the thread's waits, and those of the whole block (what it leaves the loop by)
  float up[RUNS][8];
#pragma unroll 1
  for (int t = 0; t < tiles && go; ++t) {
    const int s = t & 1;
    if (t > 0) load_u(t - 1, up);
    if (t >= 2) ok = mbar_wait_bounded(&mma[s], (uint32_t)(((t >> 1) - 1) & 1)) && ok;
    store(s, t % 3);
    if (t + 1 < tiles) load(t + 1);
    fence_proxy_async();
    go = __syncthreads_and(ok);
    if (tid == 0) {
      // (the commit follows in any case, so that every wait ends)
      const bool landed = t > 0 || mbar_wait_bounded(full, 0);
      if (!landed || !go) atomicOr(a.flags, kErrTimeout);
      if (!landed) mbar_wait_bounded(full, 0);
      tc_fence_after();
      if (landed && go) {
        const uint32_t d = tmem + 256 * s;
        const uint64_t wd = sw128_desc(sW);
#pragma unroll 1
        for (int term = 0; term < 3; ++term) {
          const uint64_t vd = sw128_desc(sV + (s * 3 + term) * kTermA);
#pragma unroll
          for (int kk = 0; kk < W / 16; ++kk) umma_bf16(d, vd + 2 * kk, wd + 2 * kk, idesc, (term | kk) != 0);
        }
        umma_split33<W>(d + W, sT, kTermA, sG + s * S::kG, false);
      }
      umma_commit(&mma[s]);
    }
    if (t > 0) {
      // (the tensor-memory loads need a warp's lanes together)
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mma[s ^ 1], (uint32_t)(((t - 1) >> 1) & 1)) && ok);
      tc_fence_after();
      if (ok) epilogue(t - 1, up);
    }
    if (!go || t + 1 == tiles) {
      ok = __all_sync(0xffffffffu, mbar_wait_bounded(&mma[s], (uint32_t)((t >> 1) & 1)) && ok);
      tc_fence_after();
      if (ok && go) {
        load_u(t, up);
        epilogue(t, up);
      } else if (!ok) {
        atomicOr(a.flags, kErrTimeout);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
}

template <int W, int MODE> cudaError_t launch(const LayerArgs &a, int sms, cudaStream_t st) {
  auto kern = layer<W, MODE>;
  constexpr size_t smem = LayerSmem<W>::kBytes;
  static_assert(smem <= 227 * 1024, "operand buffers within a block's limit");
  static SmemGrant grant;
  const cudaError_t e = grant(kern, smem);
  if (e != cudaSuccess) return e;
  // every x tile has the same number of CTAs, at most one per row
  const int per = std::max(1, std::min(sms / a.xtiles, a.rows));
  kern<<<per * a.xtiles, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int MODE> cudaError_t launch_w(int width, const LayerArgs &a, int sms, cudaStream_t st) {
  return width == 64 ? launch<64, MODE>(a, sms, st) : launch<32, MODE>(a, sms, st);
}

}  // namespace

bool layer_applies(int n, int modes, int width) { return (width == 32 || width == 64) && dft_applies(n, modes, width); }

cudaError_t layer_forward(const float *v, const float2 *G, const void *table, const void *weights, const float *bias,
                          float *u, float *out, bool activate, int batch, int width, int n, int modes, int sms,
                          int *flags, cudaStream_t st) {
  const float w = (float)(1.0 / ((double)n * n));
  const LayerArgs a{v, reinterpret_cast<const float *>(G), static_cast<const unsigned char *>(table),
                    static_cast<const __nv_bfloat16 *>(weights), width, 1, bias, u, out, n, modes,
                    (n + kTcRows - 1) / kTcRows, batch * n, w, 2.f * w, flags};
  return activate ? launch_w<kForward>(width, a, sms, st) : launch_w<kForwardLast>(width, a, sms, st);
}

cudaError_t layer_backward(const float *du, const float2 *G, const void *table, const void *weights, const float *u_prev,
                           float *out, int batch, int width, int n, int modes, int sms, int *flags, cudaStream_t st) {
  const LayerArgs a{du, reinterpret_cast<const float *>(G), static_cast<const unsigned char *>(table),
                    static_cast<const __nv_bfloat16 *>(weights), 1, width, nullptr, const_cast<float *>(u_prev), out, n,
                    modes, (n + kTcRows - 1) / kTcRows, batch * n, 1.f, 1.f, flags};
  return u_prev ? launch_w<kBackwardGelu>(width, a, sms, st) : launch_w<kBackward>(width, a, sms, st);
}

}  // namespace fno
}  // namespace spgpe
