// Per-mode channel mixing of the Fourier neural operator's spectral layers and
// the optimiser step of its spectral weights, as streaming kernels over the
// weights R[mode][o][c] (bfloat16 pairs for the products, float32 masters and
// moments for Adam).
//
// What bounds them is the weights' traffic: a mode's W x W complex matrix is
// used for `batch` matrix-vector products only (4 flop per byte at batch 4).
// So one warp takes one mode, reads its matrix once straight from global
// memory into registers, and keeps the batch's spectra of the block's modes
// in shared memory, where every lane reads the same value (a broadcast); the
// spectra's [sample][channel][mode] layout is read and written in runs of
// kModes modes.  Measured on GB300 at W = 64, 32 x 64 modes, batch 4 (33.5 MB
// of bfloat16 weights per layer) against the batched 64 x 64-tile products
// they replace (whose 2048 blocks filled 4 of 64 tile columns: 129 us forward,
// 132 us transposed, 74 us for the gradient, then 475 us of Adam over the
// whole parameter vector and a cleared gradient): a training step of the
// full-size network at 256^2 8.8 -> 7.7 ms, its inference at 512^2 8.1 -> 7.7
// ms.  The gradient with its Adam step moves 436 MB (64 us at the copy rate):
// 140 us with one block for all rows of four modes, 117 us with four rows'
// loads ahead of their use, 92 us with 16 rows per block.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "fno_internal.h"

namespace spgpe {
namespace fno {

namespace {

constexpr int kModes = 8;  // modes per block, one per warp (64-byte runs of the spectra)

struct c2f {
  float x, y;
};
__device__ __forceinline__ c2f unpack_c(uint32_t w) {  // bfloat16 pair -> float32 pair, exact
  return {__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)};
}

// NC adjacent complex columns as one access.
template <int NC> struct alignas(8 * NC) Cols {
  float2 e[NC];
};
template <int NC> struct alignas(4 * NC) ColsB {
  __nv_bfloat162 e[NC];
};

// Shared-memory elements (float2) of one mode's spectra: BG samples x W
// channels, plus two that move the next mode's rows to other banks.
__host__ __device__ constexpr int mode_stride(int w, int bg) { return w * bg + 2; }

// The spectra of modes m0 .. m0 + 7 of samples b0 .. b0 + BG - 1 (zero beyond
// the batch) into s[mode][sample][channel]; src is [sample][channel][mode].
template <int W, int BG>
__device__ __forceinline__ void load_modes(float2 *s, const float2 *__restrict__ src, long modes, long m0, int b0,
                                           int batch) {
  for (int e = threadIdx.x; e < BG * W * kModes; e += blockDim.x) {
    const int i = e & (kModes - 1), bc = e / kModes, b = bc / W;
    float2 v = make_float2(0.f, 0.f);
    if (b0 + b < batch) v = src[((long)b0 * W + bc) * modes + m0 + i];
    s[i * mode_stride(W, BG) + bc] = v;
  }
}

// out[b][o][m] = sum_c R[m][o][c] in[b][c][m]  (TRANS: out[b][c][m] =
// sum_o conj(R[m][o][c]) in[b][o][m]); BG samples per block, gridDim.y groups.
// Forward: a lane owns rows o = lane + 32 i and reads them 4 channels (16
// bytes) at a time.  Transposed: a lane owns adjacent columns c and reads
// each row with its neighbours.
template <int W, int BG, bool TRANS>
__global__ void __launch_bounds__(32 * kModes) mix(const __nv_bfloat162 *__restrict__ R, const float2 *__restrict__ in,
                                                   float2 *out, long modes, int batch) {
  constexpr int NO = W / 32;  // outputs per lane
  __shared__ __align__(16) float2 s[kModes * mode_stride(W, BG)];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long m0 = (long)blockIdx.x * kModes;
  const int b0 = blockIdx.y * BG;
  load_modes<W, BG>(s, in, modes, m0, b0, batch);
  __syncthreads();
  float2 *sm = s + w * mode_stride(W, BG);
  const uint32_t *Rm = reinterpret_cast<const uint32_t *>(R) + (m0 + w) * W * W;
  float2 acc[NO][BG];
#pragma unroll
  for (int i = 0; i < NO; ++i)
#pragma unroll
    for (int b = 0; b < BG; ++b) acc[i][b] = make_float2(0.f, 0.f);
  if constexpr (!TRANS) {
#pragma unroll 4
    for (int c = 0; c < W; c += 4) {
      uint4 r[NO];
#pragma unroll
      for (int i = 0; i < NO; ++i)
        r[i] = __ldg(reinterpret_cast<const uint4 *>(Rm + (long)(lane + 32 * i) * W + c));
#pragma unroll
      for (int b = 0; b < BG; ++b) {
        const float4 v0 = *reinterpret_cast<const float4 *>(&sm[b * W + c]);
        const float4 v1 = *reinterpret_cast<const float4 *>(&sm[b * W + c + 2]);
        const float2 v[4] = {{v0.x, v0.y}, {v0.z, v0.w}, {v1.x, v1.y}, {v1.z, v1.w}};
#pragma unroll
        for (int i = 0; i < NO; ++i) {
          const uint32_t rw[4] = {r[i].x, r[i].y, r[i].z, r[i].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const c2f q = unpack_c(rw[k]);
            acc[i][b].x = fmaf(q.x, v[k].x, fmaf(-q.y, v[k].y, acc[i][b].x));
            acc[i][b].y = fmaf(q.x, v[k].y, fmaf(q.y, v[k].x, acc[i][b].y));
          }
        }
      }
    }
  } else {
#pragma unroll 8
    for (int o = 0; o < W; ++o) {
      uint32_t rw[NO];
      if constexpr (NO == 2) {
        const uint2 r = __ldg(reinterpret_cast<const uint2 *>(Rm + (long)o * W + 2 * lane));
        rw[0] = r.x;
        rw[NO - 1] = r.y;
      } else {
        rw[0] = __ldg(Rm + (long)o * W + lane);
      }
#pragma unroll
      for (int b = 0; b < BG; ++b) {
        const float2 v = sm[b * W + o];
#pragma unroll
        for (int i = 0; i < NO; ++i) {
          const c2f q = unpack_c(rw[i]);
          acc[i][b].x = fmaf(q.x, v.x, fmaf(q.y, v.y, acc[i][b].x));
          acc[i][b].y = fmaf(q.x, v.y, fmaf(-q.y, v.x, acc[i][b].y));
        }
      }
    }
  }
  __syncwarp();  // the mode's input is read: its area takes the result
#pragma unroll
  for (int i = 0; i < NO; ++i)
#pragma unroll
    for (int b = 0; b < BG; ++b) sm[b * W + (TRANS ? NO * lane + i : lane + 32 * i)] = acc[i][b];
  __syncthreads();
  for (int e = threadIdx.x; e < BG * W * kModes; e += blockDim.x) {
    const int i = e & (kModes - 1), bc = e / kModes;
    if (b0 + bc / W < batch) out[((long)b0 * W + bc) * modes + m0 + i] = s[i * mode_stride(W, BG) + bc];
  }
}

// Gradient of a layer's spectral weights, dR[m][o][c] = sum_b d[b][o][m]
// conj(v[b][c][m]) over at most BG samples, written to g (float2 [m][o][c]);
// or (g null) applied at once as the weights' Adam step, so that the
// gradient never goes through memory: w, m, v read and written, the bfloat16
// weights written, 26 bytes per parameter.  One warp per mode, four modes per
// block and kGradRows of the rows o (so that a layer has many more blocks
// than there is room for at once); a lane owns adjacent columns c and walks the
// rows, four at a time.
constexpr int kGradModes = 4, kGradRows = 16;

template <int W, int BG, bool ADAM>
__global__ void __launch_bounds__(32 * kGradModes) mix_grad(const float2 *__restrict__ d, const float2 *__restrict__ v,
                                                            long modes, int batch, float2 *__restrict__ g,
                                                            float2 *__restrict__ w, float2 *__restrict__ mo,
                                                            float2 *__restrict__ ve, __nv_bfloat162 *__restrict__ wb,
                                                            AdamRates ar) {
  constexpr int NC = W / 32;
  constexpr int ST = W * BG + 2;
  __shared__ __align__(16) float2 s[kGradModes * ST];
  const int row0 = blockIdx.y * kGradRows, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const long m0 = (long)blockIdx.x * kGradModes, m = m0 + wp;
  // [sample][nc channels from c0]
  auto load = [&](const float2 *__restrict__ src, int c0, int nc) {
    for (int e = threadIdx.x; e < BG * nc * kGradModes; e += blockDim.x) {
      const int i = e & (kGradModes - 1), bc = e / kGradModes, b = bc / nc;
      s[i * ST + bc] = b < batch ? src[((long)b * W + c0 + bc - b * nc) * modes + m0 + i] : make_float2(0.f, 0.f);
    }
  };
  load(v, 0, W);
  __syncthreads();
  const float2 *sm = s + wp * ST;
  float2 vc[NC][BG];  // the lane's columns of v
#pragma unroll
  for (int i = 0; i < NC; ++i)
#pragma unroll
    for (int b = 0; b < BG; ++b) vc[i][b] = sm[b * W + NC * lane + i];
  __syncthreads();
  load(d, row0, kGradRows);
  __syncthreads();
  // four rows' weights and moments are on their way before the first is needed
  constexpr int G = ADAM ? 4 : 1;
  using V = Cols<NC>;
#pragma unroll 1
  for (int o0 = 0; o0 < kGradRows; o0 += G) {
    const long p0 = (m * W + row0 + o0) * W + NC * lane;
    V wv[G], mv[G], vv[G];
    if constexpr (ADAM) {
#pragma unroll
      for (int q = 0; q < G; ++q) {
        wv[q] = *reinterpret_cast<const V *>(w + p0 + q * W);
        mv[q] = *reinterpret_cast<const V *>(mo + p0 + q * W);
        vv[q] = *reinterpret_cast<const V *>(ve + p0 + q * W);
      }
    }
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const long p = p0 + q * W;
      V gr;
#pragma unroll
      for (int i = 0; i < NC; ++i) gr.e[i] = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < BG; ++b) {
        const float2 dv = sm[b * kGradRows + o0 + q];
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          gr.e[i].x = fmaf(dv.x, vc[i][b].x, fmaf(dv.y, vc[i][b].y, gr.e[i].x));
          gr.e[i].y = fmaf(dv.y, vc[i][b].x, fmaf(-dv.x, vc[i][b].y, gr.e[i].y));
        }
      }
      if constexpr (ADAM) {
        ColsB<NC> r;
#pragma unroll
        for (int i = 0; i < NC; ++i) {
          adam_one(wv[q].e[i].x, mv[q].e[i].x, vv[q].e[i].x, gr.e[i].x, ar);
          adam_one(wv[q].e[i].y, mv[q].e[i].y, vv[q].e[i].y, gr.e[i].y, ar);
          r.e[i] = __floats2bfloat162_rn(wv[q].e[i].x, wv[q].e[i].y);
        }
        *reinterpret_cast<V *>(w + p) = wv[q];
        *reinterpret_cast<V *>(mo + p) = mv[q];
        *reinterpret_cast<V *>(ve + p) = vv[q];
        *reinterpret_cast<ColsB<NC> *>(wb + p) = r;
      } else {
        *reinterpret_cast<V *>(g + p) = gr;
      }
    }
  }
}

template <int W, bool TRANS>
cudaError_t mix_w(const void *R, const float2 *in, float2 *out, long modes, int batch, cudaStream_t st) {
  const int bg = batch == 1 ? 1 : batch == 2 ? 2 : batch <= 4 ? 4 : 8;
  const dim3 grid((unsigned)(modes / kModes), (unsigned)((batch + bg - 1) / bg));
  const __nv_bfloat162 *r = static_cast<const __nv_bfloat162 *>(R);
  switch (bg) {
    case 1: mix<W, 1, TRANS><<<grid, 32 * kModes, 0, st>>>(r, in, out, modes, batch); break;
    case 2: mix<W, 2, TRANS><<<grid, 32 * kModes, 0, st>>>(r, in, out, modes, batch); break;
    case 4: mix<W, 4, TRANS><<<grid, 32 * kModes, 0, st>>>(r, in, out, modes, batch); break;
    default: mix<W, 8, TRANS><<<grid, 32 * kModes, 0, st>>>(r, in, out, modes, batch); break;
  }
  return cudaGetLastError();
}

template <int W, bool ADAM>
cudaError_t grad_w(const float2 *d, const float2 *v, long modes, int batch, float *g, float *w, float *m, float *ve,
                   void *wb, const AdamRates &ar, cudaStream_t st) {
  const dim3 grid((unsigned)(modes / kGradModes), W / kGradRows);
  auto go = [&](auto kern) {
    kern<<<grid, 32 * kGradModes, 0, st>>>(d, v, modes, batch, reinterpret_cast<float2 *>(g),
                                           reinterpret_cast<float2 *>(w), reinterpret_cast<float2 *>(m),
                                           reinterpret_cast<float2 *>(ve), static_cast<__nv_bfloat162 *>(wb), ar);
    return cudaGetLastError();
  };
  if (batch == 1) return go(mix_grad<W, 1, ADAM>);
  if (batch == 2) return go(mix_grad<W, 2, ADAM>);
  if (batch <= 4) return go(mix_grad<W, 4, ADAM>);
  return go(mix_grad<W, 8, ADAM>);
}

}  // namespace

bool mix_applies(int width, int modes) { return (width == 32 || width == 64) && (2L * modes * modes) % kModes == 0; }

cudaError_t mix_modes(const void *R, const float2 *in, float2 *out, int width, int modes, int batch, bool transposed,
                      cudaStream_t st) {
  const long n = 2L * modes * modes;
  if (width == 64)
    return transposed ? mix_w<64, true>(R, in, out, n, batch, st) : mix_w<64, false>(R, in, out, n, batch, st);
  return transposed ? mix_w<32, true>(R, in, out, n, batch, st) : mix_w<32, false>(R, in, out, n, batch, st);
}

cudaError_t mix_gradient(const float2 *d, const float2 *v, int width, int modes, int batch, float *g, cudaStream_t st) {
  const AdamRates ar{};
  const long n = 2L * modes * modes;
  return width == 64 ? grad_w<64, false>(d, v, n, batch, g, nullptr, nullptr, nullptr, nullptr, ar, st)
                     : grad_w<32, false>(d, v, n, batch, g, nullptr, nullptr, nullptr, nullptr, ar, st);
}

cudaError_t mix_adam(const float2 *d, const float2 *v, int width, int modes, int batch, float *w, float *m, float *ve,
                     void *wb, float lr, int t, cudaStream_t st) {
  const AdamRates ar = adam_rates(lr, t);
  const long n = 2L * modes * modes;
  return width == 64 ? grad_w<64, true>(d, v, n, batch, nullptr, w, m, ve, wb, ar, st)
                     : grad_w<32, true>(d, v, n, batch, nullptr, w, m, ve, wb, ar, st);
}

}  // namespace fno
}  // namespace spgpe
