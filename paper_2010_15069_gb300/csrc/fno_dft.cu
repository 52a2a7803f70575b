// Truncated Fourier transforms of the neural operator's spectral layers on the
// tensor cores (tcgen05): along x, X1[row][q] = sum_x v[row][x] T[x][q] (q =
// 2 kx + part, real input); along y, vh[img][j][kx] = sum_y Ey[j][y] X1[img][y]
// [kx]; and the inverse along y, G[img][y][kx] = sum_j conj(Ey[j][y])
// oh[img][j][kx].
//
// Each is a product of a data operand (float32, from memory) with a constant
// twiddle matrix, D[128 data rows][N columns] in tensor memory.  Both operands
// are split into three bfloat16 terms, the first on a fixed grid (split3_grid:
// the data scaled by a power of two per row, from the row's largest value),
// so that the leading products add up exactly and the result keeps float32
// accuracy: 16 flop per byte of data become 100, still below the tensor
// cores' ratio, and the passes are bound by reading the data and by the
// threads that split it.  The twiddle matrices are split on the host and
// stored as the swizzled shared-memory image, fetched by bulk copies.
//
// Along y the kept wavenumbers are -M .. M - 1, so the complex product is taken
// as cosine and sine sums of the data rows (img, kx, part): 2 (M + 1) columns
// instead of the 4 M of the four real products, and lanes (kx, re), (kx, im)
// of a warp combine them: vh(+-k) = C -+ i S.
//
// The transform kernel: 512 threads hold a whole unit of 128 rows x 256 k in
// registers.  As a 64-wide block of it is split into one of two operand
// buffers, the same registers take the block of the next unit, so that up to
// 128 KB per SM are in flight; two sets of accumulators let a unit's results
// leave while the next unit's first block is in the tensor cores.
//
// Measured on GB300 (256 images = batch 4 x 64 channels, 32 modes) against the
// CUDA-core products they replace: at 256^2 along x 116 -> 32 us, along y 126
// -> 13 us, inverse along y 76 -> 14 us; at 512^2 442 -> 208, 126 -> 23 and 129
// -> 24 us.  With a plain three-term split (no grid) the accumulator's
// truncation showed: the weights after eight training steps were 6.5e-6 off
// the 64-bit result instead of 8e-7; with the grid they are 2 to 5e-7 off.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#include "async_copy.cuh"
#include "fno_internal.h"
#include "fno_umma.cuh"

namespace spgpe {
namespace fno {

namespace {

constexpr int kThreads = 512;   // transforms
constexpr int kThreadsI = 256;  // inverse along y
constexpr size_t kTermA = (size_t)kTcRows * kRowBytes;  // one term of 128 rows x 64 k

// columns of an accumulator: a multiple of 16
__host__ __device__ constexpr int pad16(int v) { return (v + 15) / 16 * 16; }

struct DftArgs {
  const float *src;
  const unsigned char *tab;  // [n / 64 blocks][3 terms][N rows][128 bytes], swizzled
  float *dst;
  int n, M, ntiles;
  float g0, g1;                // factors of the columns of kx = 0 and of the others (x transform)
  int *flags;
};

template <int N, int NB> struct DftSmem {
  static constexpr size_t kBlockB = (size_t)3 * N * kRowBytes;
  static constexpr size_t kA = 2 * 3 * kTermA;
  static constexpr size_t kBytes = 1024 + kA + NB * kBlockB + (2 * kTcRows + kThreads) * sizeof(float) + 64;
};

// ALONG_Y false: data rows are contiguous rows of n values (x transform);
// true: data row r = img 2M + q holds X1[img][y][q], y = 0..n-1.  A unit is a
// tile of 128 rows over a segment of NB blocks of 64 k: the whole row for grids
// up to 256.  Larger rows take several segments, each with its own scales,
// added up in memory by the thread that owns the value; a CTA runs all its
// tiles through one segment, whose part of the table stays in shared memory,
// before the next.
template <int N, int NB, bool ALONG_Y>
__global__ void __launch_bounds__(kThreads, 1) dft(const DftArgs a) {
  using S = DftSmem<N, NB>;
  constexpr uint32_t kCols = 512;  // two units' accumulators, 3 N columns from 0 and from 256
  static_assert(3 * N <= 256, "three accumulators within half of the tensor memory");
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int nseg = a.n / (NB * kKBlock);
  unsigned char *sB = sm + S::kA;
  float *rowmax = reinterpret_cast<float *>(sB + NB * S::kBlockB);        // [unit parity][row] largest value
  float *quarter = rowmax + 2 * kTcRows;                                  // [thread] maxima of quarter rows (along y)
  uint64_t *mma = reinterpret_cast<uint64_t *>(quarter + kThreads);       // [2] operand buffer's MMAs done
  uint64_t *full = mma + 2;                                               // the segment's table landed
  uint32_t *slot = reinterpret_cast<uint32_t *>(full + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q2 = 2 * a.M;
  const int mytiles = (a.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  const int units = mytiles * nseg;
  auto tile_of = [&](int u) { return (int)blockIdx.x + (u % mytiles) * (int)gridDim.x; };

  auto fetch_b = [&](int seg) {  // thread 0: a segment's part of the table
    mbar_expect_tx(full, (uint32_t)(NB * S::kBlockB));
    for (int k = 0; k < NB; ++k)
      bulk_g2s(sB + k * S::kBlockB, a.tab + (size_t)(seg * NB + k) * S::kBlockB, (uint32_t)S::kBlockB, full);
  };
  if (warp == 0) {
    tmem_alloc(slot, kCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) mbar_init(&mma[i], 1);
    mbar_init(full, 1);
    mbar_fence_init();
    fetch_b(0);
  }

  // The thread's part of a block: two runs of 8 k.  Along x: rows (tid >> 3) +
  // 64 i, run tid & 7, in the order of x_slot (4 of the block's first 32 k and 4
  // of the others, so that 8 lanes read whole 128-byte lines); along y: row tid & 127, runs (tid >> 7) + 4 i.
  float x[NB][16], c[2];
  auto load = [&](int u, int kc) {
    const int tile = tile_of(u), kb = (u / mytiles) * NB + kc;
    if constexpr (!ALONG_Y) {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 *p = reinterpret_cast<const float4 *>(
            a.src + (long)(tile * kTcRows + (tid >> 3) + 64 * i) * a.n + kb * kKBlock + (tid & 7) * 4);
        const float4 v = p[0], w = p[8];
        x[kc][8 * i] = v.x; x[kc][8 * i + 1] = v.y; x[kc][8 * i + 2] = v.z; x[kc][8 * i + 3] = v.w;
        x[kc][8 * i + 4] = w.x; x[kc][8 * i + 5] = w.y; x[kc][8 * i + 6] = w.z; x[kc][8 * i + 7] = w.w;
      }
    } else {
      const int r = tile * kTcRows + (tid & 127), img = r / q2, q = r - img * q2;
      const float *p = a.src + ((long)img * a.n + kb * kKBlock) * q2 + q;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) x[kc][8 * i + j] = p[(long)(((tid >> 7) + 4 * i) * 8 + j) * q2];
    }
  };
  // the scales of the unit in x, from its rows' largest magnitudes
  auto scale = [&](int parity) {
    float vm[2] = {0.f, 0.f};
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
      for (int j = 0; j < 16; ++j) vm[ALONG_Y ? 0 : j / 8] = fmaxf(vm[ALONG_Y ? 0 : j / 8], fabsf(x[k][j]));
    if constexpr (!ALONG_Y) {  // 8 lanes hold a row
      __syncthreads();         // the unit that had this slot of rowmax is out
#pragma unroll
      for (int i = 0; i < 2; ++i) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) vm[i] = fmaxf(vm[i], __shfl_xor_sync(0xffffffffu, vm[i], o));
        c[i] = grid_scale(vm[i]);
        if ((tid & 7) == 0) rowmax[parity * kTcRows + (tid >> 3) + 64 * i] = vm[i];
      }
    } else {  // four threads hold a row
      quarter[tid] = vm[0];
      __syncthreads();
      const int r = tid & 127;
      const float v = fmaxf(fmaxf(quarter[r], quarter[r + 128]), fmaxf(quarter[r + 256], quarter[r + 384]));
      c[0] = c[1] = grid_scale(v);
      if (tid < 128) rowmax[parity * kTcRows + tid] = v;
    }
  };
  auto store = [&](unsigned char *sA, int kc) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int row = ALONG_Y ? (tid & 127) : (tid >> 3) + 64 * i, ch = ALONG_Y ? (tid >> 7) + 4 * i : (tid & 7);
      const float v[8] = {x[kc][8 * i],     x[kc][8 * i + 1], x[kc][8 * i + 2], x[kc][8 * i + 3],
                          x[kc][8 * i + 4], x[kc][8 * i + 5], x[kc][8 * i + 6], x[kc][8 * i + 7]};
      uint4 h, m, l;
      split3_grid(v, c[i], h, m, l);
      const uint32_t off = sw128(row, ch);
      *reinterpret_cast<uint4 *>(sA + off) = h;
      *reinterpret_cast<uint4 *>(sA + kTermA + off) = m;
      *reinterpret_cast<uint4 *>(sA + 2 * kTermA + off) = l;
    }
  };
  for (int k = 0; k < NB; ++k) load(0, k);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  // results of a unit: lane 32 (warp & 3) + lane of the accumulators is the
  // data row; the four groups of four warps take alternate groups of 8 columns
  auto epilogue = [&](int u) {
    const int lr = 32 * (warp & 3) + lane, r = tile_of(u) * kTcRows + lr;
    const bool more = u >= mytiles;  // add to the segments before
    const uint32_t base = tmem + 256 * (u & 1) + ((uint32_t)(32 * (warp & 3)) << 16);
    const float un = grid_unscale(rowmax[(u & 1) * kTcRows + lr]);
#pragma unroll 1
    for (int g = warp >> 2; g < N / 8; g += 4) {
      float v[8], w[8], z[8];
      tmem_ld8(base + 8 * g, v);
      tmem_ld8(base + N + 8 * g, w);
      tmem_ld8(base + 2 * N + 8 * g, z);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = (v[i] + (w[i] + z[i])) * un;
      if constexpr (!ALONG_Y) {
        float *o = a.dst + (long)r * q2 + 8 * g;
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] *= g == 0 && i < 2 ? a.g0 : a.g1;
#pragma unroll
        for (int i = 0; i < 8; i += 4)
          if (8 * g + i < q2) {
            float4 s = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
            if (more) {
              const float4 p = *reinterpret_cast<const float4 *>(o + i);
              s = make_float4(p.x + s.x, p.y + s.y, p.z + s.z, p.w + s.w);
            }
            *reinterpret_cast<float4 *>(o + i) = s;
          }
      } else {
        const int img = r / q2, q = r - img * q2;
        float *o = a.dst + (long)img * q2 * q2 + q;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int k = 4 * g + i;  // columns 2k, 2k + 1: cosine and sine sums of wavenumber k
          const float sp = __shfl_xor_sync(0xffffffffu, v[2 * i + 1], 1);
          const float s = (q & 1) ? -sp : sp;
          if (k < a.M) {
            float *e = o + (long)k * q2;
            *e = more ? *e + (v[2 * i] + s) : v[2 * i] + s;
          }
          if (k >= 1 && k <= a.M) {
            float *e = o + (long)(q2 - k) * q2;
            *e = more ? *e + (v[2 * i] - s) : v[2 * i] - s;
          }
        }
      }
    }
    tc_fence_before();
  };

  bool ok = true;
  int g = 0;  // block counter: operand buffer g & 1, its MMAs' phase (g >> 1) & 1
#pragma unroll 1
  for (int u = 0; u < units && ok; ++u) {
    scale(u & 1);
    const int seg = u / mytiles;
    if (u > 0 && u % mytiles == 0) {  // the next segment's table, once nothing reads the one before
      ok = mbar_wait_bounded(&mma[(g - 1) & 1], (uint32_t)(((g - 1) >> 1) & 1));
      if (tid == 0 && ok) fetch_b(seg);
    }
#pragma unroll
    for (int kc = 0; kc < NB; ++kc, ++g) {
      const int s = g & 1;
      if (g >= 2) ok = mbar_wait_bounded(&mma[s], (uint32_t)(((g >> 1) - 1) & 1)) && ok;
      unsigned char *sA = sm + s * 3 * kTermA;
      store(sA, kc);
      if (u + 1 < units) load(u + 1, kc);
      fence_proxy_async();
      ok = __syncthreads_and(ok);
      if (tid == 0) {
        // (the commit follows in any case, so that every wait ends)
        const bool landed = mbar_wait_bounded(full, (uint32_t)(seg & 1));
        if (!landed || !ok) atomicOr(a.flags, kErrTimeout);
        if (!landed) mbar_wait_bounded(full, (uint32_t)(seg & 1));  // the copy may still land: once more before the buffer can go
        tc_fence_after();
        if (landed && ok)
          umma_split33<N>(tmem + 256 * (u & 1), sA, kTermA, sB + kc * S::kBlockB, kc > 0);
        umma_commit(&mma[s]);
      }
      // the unit before leaves while this unit's first block is in the tensor cores
      if (kc == 0 && u > 0) {
        ok = mbar_wait_bounded(&mma[s ^ 1], (uint32_t)(((g - 1) >> 1) & 1)) && ok;
        tc_fence_after();
        if (ok) epilogue(u - 1);
      }
    }
  }
  // everything issued is complete before the buffers go; then the last unit
  ok = mbar_wait_bounded(&mma[(g - 1) & 1], (uint32_t)(((g - 1) >> 1) & 1)) && ok;
  tc_fence_after();
  if (ok) epilogue(units - 1);
  else if (tid == 0) atomicOr(a.flags, kErrTimeout);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
}

// Inverse along y: data row r = img 2M + q of 128 and a tile of NY rows y per
// CTA.  K slots 2k, 2k + 1 (k = 0..31): P_k = o_k + o_-k with cos(k y) and
// Q_k = i (o_k - o_-k) with sin(k y); at M = 32 the slot of sin 0 carries
// cos(32 y) and the epilogue adds the one product left, sin(32 y) Q_32, in
// float32, so that K stays one block of 64.
struct IdftArgs {
  const float *src;           // oh [img][2M][M] complex
  const unsigned char *tab;   // [n / NY tiles][3 terms][NY rows][128 bytes], swizzled
  const float *sin32;         // [n] sin(2 pi 32 y / n), read at M = 32 only
  float *dst;                 // G [img][n][M] complex
  int n, M, ytiles;
  int *flags;
};

template <int NY> struct IdftSmem {
  static constexpr size_t kB = (size_t)3 * NY * kRowBytes;
  static constexpr size_t kBytes = 1024 + 3 * kTermA + kB + 2 * kTcRows * sizeof(float) + 64;
};

// The six products of one 64-wide block, the leading one into the accumulator
// at d, the others into that at d + NY.
template <int NY> __device__ __forceinline__ void issue_idft(uint32_t d, const unsigned char *a, const unsigned char *b) {
#pragma unroll 1
  for (int p = 0; p < 6; ++p) {
    // (A term, B term): (2,0) (0,2) (1,1) (1,0) (0,1), then (0,0)
    const int ta = p == 0 ? 2 : (p == 2 || p == 3) ? 1 : 0, tb = p == 1 ? 2 : (p == 2 || p == 4) ? 1 : 0;
    const uint64_t ad = sw128_desc(a + ta * kTermA), bd = sw128_desc(b + (size_t)tb * NY * kRowBytes);
#pragma unroll
    for (int kk = 0; kk < kKBlock / 16; ++kk)
      umma_bf16(p == 5 ? d : d + NY, ad + 2 * kk, bd + 2 * kk, idesc_bf16(kTcRows, NY), !((p == 0 || p == 5) && kk == 0));
  }
}

template <int NY>
__global__ void __launch_bounds__(kThreadsI, 2) idft_y(const IdftArgs a) {
  using S = IdftSmem<NY>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sB = sm + 3 * kTermA;
  float *half = reinterpret_cast<float *>(sB + S::kB);  // [thread] maxima of half rows
  uint64_t *mma = reinterpret_cast<uint64_t *>(half + 2 * kTcRows), *full = mma + 1;
  uint32_t *slot = reinterpret_cast<uint32_t *>(full + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int q2 = 2 * a.M, rt = blockIdx.x / a.ytiles, yt = blockIdx.x - rt * a.ytiles;
  if (warp == 0) {
    tmem_alloc(slot, 2 * NY);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(mma, 1);
    mbar_init(full, 1);
    mbar_fence_init();
    mbar_expect_tx(full, (uint32_t)S::kB);
    bulk_g2s(sB, a.tab + (size_t)yt * S::kB, (uint32_t)S::kB, full);
  }
  {
    const int row = tid & 127, r = rt * kTcRows + row, img = r / q2, q = r - img * q2;
    const float *o = a.src + (long)img * q2 * q2 + q;
    const float sg = (q & 1) ? 1.f : -1.f;
    float v[4][8], vm = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = (tid >> 7) + 2 * i;
      float op[4], om[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int k = 4 * c + j;
        op[j] = k < a.M ? o[(long)k * q2] : 0.f;
        om[j] = k >= 1 && k <= a.M ? o[(long)(q2 - k) * q2] : 0.f;
      }
      if (c == 0 && a.M == 32) om[0] = o[(long)32 * q2];  // wavenumber -32, for the slot of sin 0
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool first = 4 * c + j == 0;
        const float d = first ? 0.f : op[j] - om[j];
        v[i][2 * j] = first ? op[j] : op[j] + om[j];
        v[i][2 * j + 1] = sg * __shfl_xor_sync(0xffffffffu, d, 1);
        if (first && a.M == 32) v[i][1] = om[0];
        vm = fmaxf(vm, fmaxf(fabsf(v[i][2 * j]), fabsf(v[i][2 * j + 1])));
      }
    }
    half[tid] = vm;
    __syncthreads();
    const float c = grid_scale(fmaxf(half[row], half[row + 128]));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint4 h, m, l;
      split3_grid(v[i], c, h, m, l);
      const uint32_t off = sw128(row, (tid >> 7) + 2 * i);
      *reinterpret_cast<uint4 *>(sm + off) = h;
      *reinterpret_cast<uint4 *>(sm + kTermA + off) = m;
      *reinterpret_cast<uint4 *>(sm + 2 * kTermA + off) = l;
    }
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  if (tid == 0) {
    const bool landed = mbar_wait_bounded(full, 0);
    if (!landed) {
      atomicOr(a.flags, kErrTimeout);
      mbar_wait_bounded(full, 0);
    }
    if (landed)
      issue_idft<NY>(tmem, sm, sB);
    umma_commit(mma);
  }
  const int r = rt * kTcRows + 32 * (warp & 3) + lane, img = r / q2, q = r - img * q2;
  float q32 = 0.f;
  if (a.M == 32) {  // Q_32 = -i o_-32: re = im part of o, im = -(re part)
    const float other = a.src[((long)img * q2 + 32) * q2 + (q ^ 1)];
    q32 = (q & 1) ? -other : other;
  }
  const bool ok = mbar_wait_bounded(mma, 0);
  if (!ok) {
    atomicOr(a.flags, kErrTimeout);
    mbar_wait_bounded(mma, 0);
  }
  tc_fence_after();
  if (__syncthreads_and(ok)) {
    const uint32_t base = tmem + ((uint32_t)(32 * (warp & 3)) << 16);
    const int lr = 32 * (warp & 3) + lane;
    const float un = grid_unscale(fmaxf(half[lr], half[lr + 128]));
    for (int g = warp >> 2; g < NY / 16; g += 2) {
      float v[16], u[16];
      tmem_ld16(base + 16 * g, v);
      tmem_ld16(base + NY + 16 * g, u);
      tmem_ld_wait();
      const int y0 = yt * NY + 16 * g;
      float *o = a.dst + ((long)img * a.n + y0) * q2 + q;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        float w = (v[i] + u[i]) * un;
        if (a.M == 32) w = fmaf(__ldg(a.sin32 + y0 + i), q32, w);
        o[(long)i * q2] = w;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * NY);
  }
}

template <class K> cudaError_t grant(K kern, size_t smem, size_t &granted) {
  if (smem > granted) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    granted = smem;
  }
  return cudaSuccess;
}

template <int N, int NB, bool ALONG_Y> cudaError_t launch_dft_nb(DftArgs a, int sms, cudaStream_t st) {
  auto kern = dft<N, NB, ALONG_Y>;
  constexpr size_t smem = DftSmem<N, NB>::kBytes;
  static_assert(smem <= 227 * 1024, "operand buffers and a segment of the table within a block's limit");
  static size_t granted = 0;
  const cudaError_t e = grant(kern, smem, granted);
  if (e != cudaSuccess) return e;
  kern<<<std::max(1, std::min(a.ntiles, sms)), kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int N, bool ALONG_Y> cudaError_t launch_dft(const DftArgs &a, int sms, cudaStream_t st) {
  if (a.n == 64) return launch_dft_nb<N, 1, ALONG_Y>(a, sms, st);
  if (a.n == 128) return launch_dft_nb<N, 2, ALONG_Y>(a, sms, st);
  return launch_dft_nb<N, 4, ALONG_Y>(a, sms, st);
}

template <int NY> cudaError_t launch_idft(const IdftArgs &a, int rows, cudaStream_t st) {
  auto kern = idft_y<NY>;
  static size_t granted = 0;
  const cudaError_t e = grant(kern, IdftSmem<NY>::kBytes, granted);
  if (e != cudaSuccess) return e;
  kern<<<rows / kTcRows * a.ytiles, kThreadsI, IdftSmem<NY>::kBytes, st>>>(a);
  return cudaGetLastError();
}

// Host: entry k of row r, all three terms, of a swizzled [term][rows][64] block.
uint16_t bf16_bits(float v) {
  uint32_t u;
  std::memcpy(&u, &v, 4);
  return (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
}
float bf16_value(uint16_t b) {
  const uint32_t u = (uint32_t)b << 16;
  float v;
  std::memcpy(&v, &u, 4);
  return v;
}
// (the first term on the grid of 2^-7: split3_grid)
void put3(uint16_t *block, int rows, int r, int k, double v) {
  for (int t = 0; t < 3; ++t) {
    const uint16_t b = bf16_bits((float)(t == 0 ? std::nearbyint(v * 128.0) / 128.0 : v));
    block[((size_t)t * rows + r) * kKBlock + (((k >> 3) ^ (r & 7)) << 3) + (k & 7)] = b;
    v -= bf16_value(b);
  }
}

const double kTwoPi = 6.28318530717958647692528676655900577;

}  // namespace

bool dft_applies(int n, int modes, int width) {
  return n >= kKBlock && n % kKBlock == 0 && modes % 2 == 0 && modes <= 32 && 2 * modes <= n &&
         ((long)width * n) % kTcRows == 0 && ((long)width * 2 * modes) % kTcRows == 0;
}

// (The twiddles are the float32 ones of the general path, so that both paths
// compute the same transform.)
// Slot of x in its 64-wide block: run r = slot / 8 holds x = 4 r .. 4 r + 3 and
// 32 + 4 r .. 32 + 4 r + 3.
static int x_slot(int x) {
  const int k = x % kKBlock;
  return 8 * ((k % 32) / 4) + k % 4 + (k >= 32 ? 4 : 0);
}

std::vector<uint16_t> dft_table(DftTable which, int n, int M) {
  if (which == DftTable::X) {  // columns 2k, 2k + 1 = cos, -sin(2 pi k x / n), k < M
    const int N = pad16(2 * M);
    std::vector<uint16_t> t((size_t)(n / kKBlock) * 3 * N * kKBlock, 0);
    for (int x = 0; x < n; ++x)
      for (int k = 0; k < M; ++k) {
        const double th = kTwoPi * (double)((long)k * x % n) / n;
        uint16_t *b = t.data() + (size_t)(x / kKBlock) * 3 * N * kKBlock;
        put3(b, N, 2 * k, x_slot(x), (float)std::cos(th));
        put3(b, N, 2 * k + 1, x_slot(x), (float)-std::sin(th));
      }
    return t;
  }
  if (which == DftTable::Y) {  // columns 2k, 2k + 1 = cos, sin(2 pi k y / n), k = 0..M
    const int N = pad16(2 * (M + 1));
    std::vector<uint16_t> t((size_t)(n / kKBlock) * 3 * N * kKBlock, 0);
    for (int y = 0; y < n; ++y)
      for (int k = 0; k <= M; ++k) {
        const double th = kTwoPi * (double)((long)k * y % n) / n;
        uint16_t *b = t.data() + (size_t)(y / kKBlock) * 3 * N * kKBlock;
        put3(b, N, 2 * k, y % kKBlock, (float)std::cos(th));
        put3(b, N, 2 * k + 1, y % kKBlock, (float)std::sin(th));
      }
    return t;
  }
  if (which == DftTable::LayerX) {  // row x, slots 2k, 2k + 1 = cos, -sin(2 pi k x / n), k < M; tiles of 128 rows
    std::vector<uint16_t> t((size_t)((n + kTcRows - 1) / kTcRows) * 3 * kTcRows * kKBlock, 0);
    for (int x = 0; x < n; ++x)
      for (int k = 0; k < M; ++k) {
        const double th = kTwoPi * (double)((long)k * x % n) / n;
        uint16_t *b = t.data() + (size_t)(x / kTcRows) * 3 * kTcRows * kKBlock;
        put3(b, kTcRows, x % kTcRows, 2 * k, (float)std::cos(th));
        put3(b, kTcRows, x % kTcRows, 2 * k + 1, (float)-std::sin(th));
      }
    return t;
  }
  // inverse along y: row y, slots 2k, 2k + 1 = cos, sin(2 pi k y / n); slot 1 = cos(32 ...) at M = 32
  const int NY = std::min(n, 128);
  std::vector<uint16_t> t((size_t)n * 3 * kKBlock, 0);
  for (int y = 0; y < n; ++y) {
    uint16_t *b = t.data() + (size_t)(y / NY) * 3 * NY * kKBlock;
    for (int k = 0; k <= std::min(M, 31); ++k) {
      const double th = kTwoPi * (double)((long)k * y % n) / n;
      put3(b, NY, y % NY, 2 * k, (float)std::cos(th));
      if (k > 0) put3(b, NY, y % NY, 2 * k + 1, (float)std::sin(th));
    }
    if (M == 32) put3(b, NY, y % NY, 1, (float)std::cos(kTwoPi * (double)(32l * y % n) / n));
  }
  return t;
}

cudaError_t dft_x(const float *v, const void *table, bool adjoint, float *X1, int images, int n, int modes, int sms,
                  int *flags, cudaStream_t st) {
  const float w = adjoint ? (float)(1.0 / ((double)n * n)) : 1.f;
  const DftArgs a{v, static_cast<const unsigned char *>(table), X1, n, modes, (int)((long)images * n / kTcRows),
                  w, adjoint ? 2.f * w : w, flags};
  switch (pad16(2 * modes)) {
    case 16: return launch_dft<16, false>(a, sms, st);
    case 32: return launch_dft<32, false>(a, sms, st);
    case 48: return launch_dft<48, false>(a, sms, st);
    case 64: return launch_dft<64, false>(a, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t dft_y(const float *X1, const void *table, float2 *vh, int images, int n, int modes, int sms, int *flags,
                  cudaStream_t st) {
  const DftArgs a{X1, static_cast<const unsigned char *>(table), reinterpret_cast<float *>(vh), n, modes,
                  (int)((long)images * 2 * modes / kTcRows), 1.f, 1.f, flags};
  switch (pad16(2 * (modes + 1))) {
    case 16: return launch_dft<16, true>(a, sms, st);
    case 32: return launch_dft<32, true>(a, sms, st);
    case 48: return launch_dft<48, true>(a, sms, st);
    case 64: return launch_dft<64, true>(a, sms, st);
    case 80: return launch_dft<80, true>(a, sms, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t idft_y(const float2 *oh, const void *table, const float *sin32, float2 *G, int images, int n, int modes,
                   int *flags, cudaStream_t st) {
  const int NY = std::min(n, 128), rows = images * 2 * modes;
  const IdftArgs a{reinterpret_cast<const float *>(oh), static_cast<const unsigned char *>(table), sin32,
                   reinterpret_cast<float *>(G), n, modes, n / NY, flags};
  return NY == 128 ? launch_idft<128>(a, rows, st) : launch_idft<64>(a, rows, st);
}

}  // namespace fno
}  // namespace spgpe
