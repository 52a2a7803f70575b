// Truncated Fourier transforms of the neural operator's spectral layers: along
// x, X1[row][q] = sum_x v[row][x] E[x][q] (q = 2 kx + part, real input); along
// y, vh[img][j][kx] = sum_y Ey[j][y] X1[img][y][kx]; and the inverse along y,
// G[img][y][kx] = sum_j conj(Ey[j][y]) oh[img][j][kx].
//
// The forward transforms feed the spectral weights' gradients, where what is
// left of a smooth field at high wavenumbers is as small as the transform's
// own rounding; they are float32 sums in ascending order, one fma per term
// (the order of the general products they replace, bit for bit), on the CUDA
// cores, which 16 flop per byte keep busy: two packed fma per complex term or
// pair of columns, operands from shared memory in wide reads, copied in
// asynchronously one block ahead.
//
// The inverse along y runs on the tensor cores (tcgen05): D[128 data rows][N
// columns] in tensor memory, data and twiddles split into three bfloat16
// terms, the first on a fixed grid (split3_grid: the data scaled by a power of
// two per row, from the row's largest value), so that the leading products add
// up exactly and the result keeps float32 accuracy.  The kept wavenumbers are
// -M .. M - 1, so the complex product is taken with cosines and sines of 0 .. M
// only.  The twiddle matrix is split on the host and stored as the swizzled
// shared-memory image, fetched by bulk copies.
//
// Measured on GB300 (256 images = batch 4 x 64 channels, 32 modes) against the
// general products: at 256^2 along x 116 -> 53 us, along y 126 -> 42 us, inverse
// along y 76 -> 14 us; at 512^2 442 -> 170, 126 -> 80 and 129 -> 24 us.  (On the
// tensor cores, split like the inverse, the forward transforms took 32 and 13
// us at 256^2 and came out nearer to the 64-bit result; weights trained for a
// few steps then differ from those of the general path by that path's own
// rounding error, up to 8e-4 of their size.)
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
#include "internal.h"
#include "smem_grant.h"

namespace spgpe {
namespace fno {

namespace {

constexpr int kThreadsI = 256;  // inverse along y
constexpr size_t kTermA = (size_t)kTcRows * kRowBytes;  // one term of 128 rows x 64 k

// 16 bytes global -> shared, asynchronous (both addresses 16-byte aligned).
__device__ __forceinline__ void cp16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int LEFT> __device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(LEFT) : "memory");
}

// Along x: 128 rows x 8 CT columns per block, 8 rows x CT columns per thread,
// blocks of 32 x.  A warp's reads hit every bank once: rows ty + 16 i (36 floats
// apart, 4 x at a time) and columns in runs of 4 (or 2) per thread, 128 bytes a
// read: 16 reads for the 128 packed fma of 4 x.
constexpr int kXRows = 128, kXBlock = 32, kXStride = kXBlock + 4;

// First column of a thread's pair j: pairs come in runs of 4 columns over all
// of the warp's 8 column threads, a last run of 2 when CT is not a multiple of 4.
template <int CT> __host__ __device__ constexpr int x_col(int tx, int j) {
  return (j / 2) * 32 + (4 * (j / 2) + 4 <= CT ? 4 * tx + 2 * (j % 2) : 2 * tx);
}

template <int CT>
__global__ void __launch_bounds__(128, 3) dft_rows(const float *__restrict__ v, const float *__restrict__ E, int n, int q2,
                                                   float g0, float g1, float *__restrict__ out) {
  constexpr int N = 8 * CT, P = CT / 2, R = 8;  // columns (padded), packed pairs and rows per thread
  extern __shared__ __align__(16) float smem_f[];
  float *sv = smem_f, *se = smem_f + 2 * kXRows * kXStride;  // [2][row][kXStride], [2][x][N]
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  const long row0 = (long)blockIdx.x * kXRows;
  const int blocks = n / kXBlock;
  auto fetch = [&](int b) {
    float *dv = sv + (b & 1) * kXRows * kXStride, *de = se + (b & 1) * kXBlock * N;
#pragma unroll
    for (int i = 0; i < kXRows * kXBlock / 4 / 128; ++i) {
      const int e = tid + 128 * i, r = e >> 3, c = e & 7;
      cp16(dv + r * kXStride + 4 * c, v + (row0 + r) * n + b * kXBlock + 4 * c);
    }
    for (int e = tid; e < kXBlock * q2 / 4; e += 128) {
      const int x = 4 * e / q2, c = 4 * e - x * q2;
      cp16(de + x * N + c, E + (long)(b * kXBlock + x) * q2 + c);
    }
    cp_commit();
  };
  for (int e = tid; e < 2 * kXBlock * N; e += 128)
    if (e % N >= q2) se[e] = 0.f;  // the columns of the padding
  float2 acc[R][P];
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < P; ++j) acc[i][j] = make_float2(0.f, 0.f);
  fetch(0);
#pragma unroll 1
  for (int b = 0; b < blocks; ++b) {
    if (b + 1 < blocks) {
      fetch(b + 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const float *pv = sv + (b & 1) * kXRows * kXStride + ty * kXStride, *pe = se + (b & 1) * kXBlock * N;
#pragma unroll 2
    for (int k = 0; k < kXBlock; k += 4) {
      float a[R][4];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const float4 t = *reinterpret_cast<const float4 *>(pv + 16 * i * kXStride + k);
        a[i][0] = t.x; a[i][1] = t.y; a[i][2] = t.z; a[i][3] = t.w;
      }
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float2 w[P];
#pragma unroll
        for (int j = 0; j < P; ++j) {
          if (j % 2 == 0 && j + 1 < P) {
            const float4 t = *reinterpret_cast<const float4 *>(pe + (k + kk) * N + x_col<CT>(tx, j));
            w[j] = make_float2(t.x, t.y);
            w[j + 1 < P ? j + 1 : j] = make_float2(t.z, t.w);
          } else if (j % 2 == 0) {
            w[j] = *reinterpret_cast<const float2 *>(pe + (k + kk) * N + x_col<CT>(tx, j));
          }
        }
#pragma unroll
        for (int i = 0; i < R; ++i)
#pragma unroll
          for (int j = 0; j < P; ++j) acc[i][j] = __ffma2_rn(w[j], make_float2(a[i][kk], a[i][kk]), acc[i][j]);
      }
    }
    __syncthreads();  // the block's buffers are read: the block after next may go there
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    float *o = out + (row0 + ty + 16 * i) * q2;
#pragma unroll
    for (int j = 0; j < P; ++j) {
      const int c = x_col<CT>(tx, j);
      const float g = c == 0 ? g0 : g1;
      if (c < q2) *reinterpret_cast<float2 *>(o + c) = make_float2(acc[i][j].x * g, acc[i][j].y * g);
    }
  }
}

// Along y: one image per 256 threads (or several small ones), 4 wavenumbers j x
// 2 kx per thread, blocks of 32 y, the next y's operands in registers.  The
// complex term a b is two packed fma, (-a.y, a.y) (b.y, b.x), then (a.x, a.x)
// (b.x, b.y); the table holds the pairs (a.x, a.x, -a.y, a.y) ready, so that the
// 16 packed fma of a y need no register shuffling but b's swap (44 -> 42 us at
// 256^2, 84 -> 80 us at 512^2).
constexpr int kYBlock = 32, kYThreads = 256;

__global__ void __launch_bounds__(kYThreads, 2) dft_cols(const float2 *__restrict__ X1, const float4 *__restrict__ Et, int n,
                                                      int M, int images, int per_block, float2 *__restrict__ out) {
  extern __shared__ __align__(16) float4 smem_c[];
  const int J = 2 * M, jt = (J + 3) / 4, kt = M / 2, Jp = 4 * jt;  // (M is even) wavenumbers padded to whole thread tiles
  float4 *se = smem_c;                                             // [2][y][Jp]
  float2 *sx = reinterpret_cast<float2 *>(smem_c + 2 * kYBlock * Jp);  // [2][image][y][M]
  const int tid = threadIdx.x, per = jt * kt;
  const int im = min(tid / per, per_block - 1), loc = tid % per, tj = loc / kt, tk = loc - tj * kt;
  const int img0 = blockIdx.x * per_block;
  const bool mine = tid < per * per_block && img0 + im < images;
  const int blocks = n / kYBlock;
  for (int e = tid; e < 2 * kYBlock * Jp; e += kYThreads)
    if (e % Jp >= J) se[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto fetch = [&](int b) {
    float4 *de = se + (b & 1) * kYBlock * Jp;
    float2 *dx = sx + (b & 1) * per_block * kYBlock * M;
    for (int e = tid; e < kYBlock * J; e += kYThreads) {
      const int y = e / J, c = e - y * J;
      cp16(de + y * Jp + c, Et + (long)(b * kYBlock + y) * J + c);
    }
    const int h = kYBlock * M / 2;  // 16-byte pieces of an image's block, which is contiguous
    for (int e = tid; e < per_block * h; e += kYThreads) {
      const int i = e / h, r = e - i * h;
      if (img0 + i < images) cp16(dx + i * kYBlock * M + 2 * r, X1 + ((long)(img0 + i) * n + b * kYBlock) * M + 2 * r);
    }
    cp_commit();
  };
  float2 acc[4][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
  fetch(0);
#pragma unroll 1
  for (int b = 0; b < blocks; ++b) {
    if (b + 1 < blocks) {
      fetch(b + 1);
      cp_wait<1>();
    } else {
      cp_wait<0>();
    }
    __syncthreads();
    const float4 *pe = se + (b & 1) * kYBlock * Jp + 4 * tj;
    const float2 *px = sx + ((b & 1) * per_block + im) * kYBlock * M + 2 * tk;
    float4 en[4], xn = *reinterpret_cast<const float4 *>(px);
#pragma unroll
    for (int j = 0; j < 4; ++j) en[j] = pe[j];
#pragma unroll 8
    for (int y = 0; y < kYBlock; ++y) {
      float4 a[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = en[j];
      const float4 x = xn;
      if (y + 1 < kYBlock) {
#pragma unroll
        for (int j = 0; j < 4; ++j) en[j] = pe[(y + 1) * Jp + j];
        xn = *reinterpret_cast<const float4 *>(px + (y + 1) * M);
      }
      const float2 x0 = make_float2(x.x, x.y), x1 = make_float2(x.z, x.w), s0 = make_float2(x.y, x.x),
                   s1 = make_float2(x.w, x.z);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[j][0] = __ffma2_rn(make_float2(a[j].z, a[j].w), s0, acc[j][0]);
        acc[j][1] = __ffma2_rn(make_float2(a[j].z, a[j].w), s1, acc[j][1]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        acc[j][0] = __ffma2_rn(make_float2(a[j].x, a[j].y), x0, acc[j][0]);
        acc[j][1] = __ffma2_rn(make_float2(a[j].x, a[j].y), x1, acc[j][1]);
      }
    }
    __syncthreads();  // the block's buffers are read: the block after next may go there
  }
  if (!mine) return;
  float2 *o = out + (long)(img0 + im) * J * M;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int jj = 4 * tj + j;
    if (jj < J)
      *reinterpret_cast<float4 *>(o + (long)jj * M + 2 * tk) = make_float4(acc[j][0].x, acc[j][0].y, acc[j][1].x, acc[j][1].y);
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

template <int CT>
cudaError_t launch_rows(const float *v, const float *E, int n, int q2, float g0, float g1, float *out, long rows,
                        cudaStream_t st) {
  auto kern = dft_rows<CT>;
  constexpr size_t smem = (size_t)2 * (kXRows * kXStride + kXBlock * 8 * CT) * sizeof(float);
  static SmemGrant grant;
  const cudaError_t e = grant(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<(unsigned)(rows / kXRows), 128, smem, st>>>(v, E, n, q2, g0, g1, out);
  return cudaGetLastError();
}

template <int NY> cudaError_t launch_idft(const IdftArgs &a, int rows, cudaStream_t st) {
  auto kern = idft_y<NY>;
  static SmemGrant grant;
  const cudaError_t e = grant(kern, IdftSmem<NY>::kBytes);
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
std::vector<uint16_t> dft_table(DftTable which, int n, int M) {
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

cudaError_t dft_x(const float *v, const float *E, bool adjoint, float *X1, int images, int n, int modes, cudaStream_t st) {
  const float w = adjoint ? (float)(1.0 / ((double)n * n)) : 1.f, g1 = adjoint ? 2.f * w : w;  // powers of two: exact
  const long rows = (long)images * n;
  const int q2 = 2 * modes;
  switch ((q2 + 15) / 16) {
    case 1: return launch_rows<2>(v, E, n, q2, w, g1, X1, rows, st);
    case 2: return launch_rows<4>(v, E, n, q2, w, g1, X1, rows, st);
    case 3: return launch_rows<6>(v, E, n, q2, w, g1, X1, rows, st);
    case 4: return launch_rows<8>(v, E, n, q2, w, g1, X1, rows, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t dft_y(const float *X1, const float4 *Et, float2 *vh, int images, int n, int modes, cudaStream_t st) {
  // as many images as the threads cover and two buffers of kYBlock rows hold (two
  // modes: 223 of 256, 232064 bytes; more modes are bounded by the threads)
  const int jt = (2 * modes + 3) / 4;
  const size_t table = 4 * jt * sizeof(float4), row = modes * sizeof(float2);  // of one y
  const int fit = (int)((kMaxSmemPerBlock / (2 * kYBlock) - table) / row);
  const int per_block = std::min(std::max(1, kYThreads / (jt * (modes / 2))), fit);
  const size_t smem = 2 * kYBlock * (table + per_block * row);
  static SmemGrant grant;
  const cudaError_t e = grant(dft_cols, smem);
  if (e != cudaSuccess) return e;
  dft_cols<<<(unsigned)((images + per_block - 1) / per_block), kYThreads, smem, st>>>(reinterpret_cast<const float2 *>(X1), Et, n,
                                                                               modes, images, per_block, vh);
  return cudaGetLastError();
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
