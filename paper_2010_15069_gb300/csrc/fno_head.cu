// The network's lift and projection: pointwise maps with their activation,
// second map, gradients and bias sums fused around one pass over the points.
//
// Projection, forward: hp = Q1 v + q1 on the tensor cores (tcgen05, v split
// into three bfloat16 terms, weights exact in bfloat16), then out = Q2
// gelu(hp) + q2 from the accumulators; hp is written for the backward pass
// only, gelu(hp) never.  Backward: one pass over hp forms dhp = (Q2^T dout)
// gelu'(hp) and sums dQ2 = dout gelu(hp)^T, dq2 and dq1 beside it; then dv =
// Q1^T dhp on the tensor cores.  All are bound by the one read or write of the
// hidden activations.
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

constexpr size_t kTermA = (size_t)kTcRows * kRowBytes;
constexpr int kOut = 4;  // output channels the fused projection holds per point

struct MapArgs {
  const float *x;  // [b][K][P]
  const __nv_bfloat16 *weights;
  long sOut, sIn;  // strides of the weights along output and input channels
  float *y;        // [b][N][P], or null (projection: not kept)
  const float *bias, *q2w, *q2b;  // projection: q1, Q2 [cout][N], q2
  float *out;                     // projection: [b][cout][P]
  int cout, ntiles, tiles_per_sample;
  long P;
  int *flags;
};

constexpr int kThreads = 512;

template <int K, int N> struct MapSmem {
  static constexpr int KB = K > 64 ? K / 64 : 1;
  static constexpr size_t kA = (size_t)2 * 3 * KB * kTermA;
  static constexpr size_t kB = (size_t)KB * N * kRowBytes;
  static constexpr size_t kBytes = 1024 + kA + kB + ((size_t)N * (kOut + 1) + 4 * kOut * kTcRows) * sizeof(float) + 64;
};

// y[b][m][p] = sum_k A(m, k) x[b][k][p] (+ bias, activation and second map with
// PROJECT).  Tiles of 128 points; two operand buffers and two accumulators: a
// tile's results leave while the next one is in the tensor cores, and the
// values of the one after are in registers.
template <int K, int N, bool PROJECT>
__global__ void __launch_bounds__(kThreads, 1) map_points(const MapArgs a) {
  using S = MapSmem<K, N>;
  constexpr int KB = S::KB, RUNS = K / 32;
  constexpr uint32_t kCols = 2 * N;
  static_assert(kCols >= 32 && kCols <= 512, "two accumulators in tensor memory");
  extern __shared__ unsigned char smem_raw[];
  unsigned char *sm =
      reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char *sX = sm, *sW = sX + S::kA;
  float *bias = reinterpret_cast<float *>(sW + S::kB), *q2 = bias + N;  // q2[channel][kOut]
  float *part = q2 + N * kOut;                                          // [group][output][point]
  uint64_t *mma = reinterpret_cast<uint64_t *>(part + 4 * kOut * kTcRows);
  uint32_t *slot = reinterpret_cast<uint32_t *>(mma + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    tmem_alloc(slot, kCols);
    tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&mma[0], 1);
    mbar_init(&mma[1], 1);
    mbar_fence_init();
  }
  for (int e = tid; e < N * (K / 8); e += kThreads) {
    const int c = e / (K / 8), j = e - c * (K / 8);
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = pack_bf16(a.weights[c * a.sOut + (8 * j + 2 * i) * a.sIn], a.weights[c * a.sOut + (8 * j + 2 * i + 1) * a.sIn]);
    *reinterpret_cast<uint4 *>(sW + (size_t)(j / 8) * N * kRowBytes + sw128(c, j % 8)) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  if constexpr (PROJECT) {
    for (int e = tid; e < N; e += kThreads) {
      bias[e] = a.bias[e];
      for (int o = 0; o < kOut; ++o) q2[e * kOut + o] = o < a.cout ? a.q2w[(long)o * N + e] : 0.f;
    }
  }
  const int pt = tid & 127;
  float x[RUNS][8];
  auto load = [&](int tile) {
    const int b = tile / a.tiles_per_sample;
    const float *p = a.x + (long)b * K * a.P + (long)(tile - b * a.tiles_per_sample) * kTcRows + pt;
#pragma unroll
    for (int i = 0; i < RUNS; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) x[i][j] = p[((tid >> 7) * 8 + 32 * i + j) * a.P];
  };
  auto store = [&](int s) {
    unsigned char *A = sX + (size_t)s * 3 * KB * kTermA;
#pragma unroll
    for (int i = 0; i < RUNS; ++i) {
      uint4 h, m, l;
      split3(x[i], h, m, l);
      const int run = (tid >> 7) + 4 * i;
      const size_t off = (size_t)(run / 8) * kTermA + sw128(pt, run % 8);
      *reinterpret_cast<uint4 *>(A + off) = h;
      *reinterpret_cast<uint4 *>(A + KB * kTermA + off) = m;
      *reinterpret_cast<uint4 *>(A + 2 * KB * kTermA + off) = l;
    }
  };
  const int tiles = (a.ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  load(blockIdx.x);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *slot;
  constexpr uint32_t idesc = idesc_bf16(kTcRows, N);
  // results of tile t: warps of a group of four hold 32 points each, the four
  // groups take alternate runs of 8 channels
  auto epilogue = [&](int t) {
    const int tile = blockIdx.x + t * gridDim.x, b = tile / a.tiles_per_sample;
    const long p0 = (long)(tile - b * a.tiles_per_sample) * kTcRows;
    const uint32_t base = tmem + N * (t & 1) + ((uint32_t)(32 * (warp & 3)) << 16);
    const int lp = 32 * (warp & 3) + lane;
    float *y = a.y ? a.y + (long)b * N * a.P + p0 + lp : nullptr;
    float acc[kOut] = {};
#pragma unroll
    for (int c0 = (warp >> 2) * 8, i = 0; i < N / 32; ++i, c0 += 32) {
      float v[8];
      tmem_ld8(base + c0, v);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int c = c0 + j;
        if constexpr (PROJECT) {
          const float u = v[j] + bias[c];
          if (y) y[c * a.P] = u;
          const float g = gelu_f(u);
          const float4 q = *reinterpret_cast<const float4 *>(q2 + c * kOut);
          acc[0] = fmaf(q.x, g, acc[0]);
          acc[1] = fmaf(q.y, g, acc[1]);
          acc[2] = fmaf(q.z, g, acc[2]);
          acc[3] = fmaf(q.w, g, acc[3]);
        } else {
          y[c * a.P] = v[j];
        }
      }
    }
    tc_fence_before();
    if constexpr (PROJECT) {
#pragma unroll
      for (int o = 0; o < kOut; ++o) part[((warp >> 2) * kOut + o) * kTcRows + lp] = acc[o];
      __syncthreads();
      const int o = tid >> 7;  // kThreads = kOut x 128
      if (o < a.cout) {
        const float s = (part[o * kTcRows + pt] + part[(kOut + o) * kTcRows + pt]) +
                        (part[(2 * kOut + o) * kTcRows + pt] + part[(3 * kOut + o) * kTcRows + pt]);
        a.out[((long)b * a.cout + o) * a.P + p0 + pt] = s + a.q2b[o];
      }
    }
  };
  bool ok = true;
#pragma unroll 1
  for (int t = 0; t < tiles && ok; ++t) {
    const int s = t & 1;
    if (t >= 2) ok = mbar_wait_bounded(&mma[s], (uint32_t)(((t >> 1) - 1) & 1));
    store(s);
    if (t + 1 < tiles) load(blockIdx.x + (t + 1) * gridDim.x);
    fence_proxy_async();
    ok = __syncthreads_and(ok);
    if (tid == 0) {
      // (the commit follows in any case, so that every wait ends)
      if (!ok) atomicOr(a.flags, kErrTimeout);
      tc_fence_after();
      if (ok)
#pragma unroll 1
        for (int term = 0; term < 3; ++term)
#pragma unroll
          for (int kb = 0; kb < KB; ++kb) {
            const uint64_t ad = sw128_desc(sX + (size_t)((s * 3 + term) * KB + kb) * kTermA);
            const uint64_t bd = sw128_desc(sW + (size_t)kb * N * kRowBytes);
#pragma unroll
            for (int kk = 0; kk < (K < 64 ? K : 64) / 16; ++kk)
              umma_bf16(tmem + N * s, ad + 2 * kk, bd + 2 * kk, idesc, (term | kb | kk) != 0);
          }
      umma_commit(&mma[s]);
    }
    // (every wait on the MMAs is followed by a barrier: the tensor-memory loads
    // of a warp need its lanes together)
    if (t > 0) {
      ok = __syncthreads_and(mbar_wait_bounded(&mma[s ^ 1], (uint32_t)(((t - 1) >> 1) & 1)) && ok);
      tc_fence_after();
      if (ok) epilogue(t - 1);
    }
    if (!ok || t + 1 == tiles) {
      ok = __syncthreads_and(mbar_wait_bounded(&mma[s], (uint32_t)((t >> 1) & 1)) && ok);
      tc_fence_after();
      if (ok) epilogue(t);
      else if (tid == 0) atomicOr(a.flags, kErrTimeout);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
}

// Projection, backward.  A warp owns H / 16 hidden channels, a lane 4 points of
// a tile of 128: dhp[b][c][p] = (sum_o Q2[o][c] dout[b][o][p]) gelu'(hp), in
// place of hp or beside it; the sums dQ2[o][c] = sum dout[o] gelu(hp[c]),
// dq1[c] = sum dhp[c] and dq2[o] = sum dout[o] stay in registers over the CTA's
// tiles (one CTA per SM; more once they would exceed kHeadRun tiles each, which
// keeps the float32 chains short) and leave as partials [CTA][cout H + H + cout].
constexpr int kBackThreads = 512;
static_assert(kHeadTile == kTcRows, "tiles of the projection");

template <int H>
__global__ void __launch_bounds__(kBackThreads, 1) project_backward(const float *__restrict__ dout,
                                                                const float *__restrict__ hp,
                                                                const float *__restrict__ q2w, int cout, int ntiles,
                                                                int tiles_per_sample, long P, float *__restrict__ dhp,
                                                                float *__restrict__ part) {
  constexpr int C = H / 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c0 = warp * C;
  float w[C][kOut], s[C][kOut], sb[C], so[kOut];
#pragma unroll
  for (int i = 0; i < C; ++i) {
    sb[i] = 0.f;
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      w[i][o] = o < cout ? q2w[(long)o * H + c0 + i] : 0.f;
      s[i][o] = 0.f;
    }
  }
#pragma unroll
  for (int o = 0; o < kOut; ++o) so[o] = 0.f;
#pragma unroll 1
  for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int b = tile / tiles_per_sample;
    const long p0 = (long)(tile - b * tiles_per_sample) * kTcRows + 4 * lane;
    float4 d[kOut];
#pragma unroll
    for (int o = 0; o < kOut; ++o)
      d[o] = o < cout ? *reinterpret_cast<const float4 *>(dout + ((long)b * cout + o) * P + p0) : make_float4(0, 0, 0, 0);
    const float *h0 = hp + ((long)b * H + c0) * P + p0;
    float *g0 = dhp + ((long)b * H + c0) * P + p0;
    float4 u[C];
#pragma unroll
    for (int i = 0; i < C; ++i) u[i] = *reinterpret_cast<const float4 *>(h0 + i * P);
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const float uv[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
      float r[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float dj[kOut] = {j == 0 ? d[0].x : j == 1 ? d[0].y : j == 2 ? d[0].z : d[0].w,
                                j == 0 ? d[1].x : j == 1 ? d[1].y : j == 2 ? d[1].z : d[1].w,
                                j == 0 ? d[2].x : j == 1 ? d[2].y : j == 2 ? d[2].z : d[2].w,
                                j == 0 ? d[3].x : j == 1 ? d[3].y : j == 2 ? d[3].z : d[3].w};
        float g, dg;
        gelu_both(uv[j], g, dg);
        float t = 0.f;
#pragma unroll
        for (int o = 0; o < kOut; ++o) {
          t = fmaf(w[i][o], dj[o], t);
          s[i][o] = fmaf(dj[o], g, s[i][o]);
        }
        r[j] = t * dg;
      }
      sb[i] += (r[0] + r[1]) + (r[2] + r[3]);
      *reinterpret_cast<float4 *>(g0 + i * P) = make_float4(r[0], r[1], r[2], r[3]);
    }
#pragma unroll
    for (int o = 0; o < kOut; ++o) so[o] += (d[o].x + d[o].y) + (d[o].z + d[o].w);
  }
  auto lanes = [](float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  };
  float *out = part + (long)blockIdx.x * (cout * H + H + cout);
#pragma unroll
  for (int i = 0; i < C; ++i) {
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      const float v = lanes(s[i][o]);
      if (lane == 0 && o < cout) out[o * H + c0 + i] = v;
    }
    const float v = lanes(sb[i]);
    if (lane == 0) out[cout * H + c0 + i] = v;
  }
  if (warp == 0)
#pragma unroll
    for (int o = 0; o < kOut; ++o) {
      const float v = lanes(so[o]);
      if (lane == 0 && o < cout) out[cout * H + H + o] = v;
    }
}

// Lift: v[b][c][p] = sum_i A[c][i] a[b][i][p] + bias[c].  A thread holds four
// points' inputs and writes kLiftOut channels of them; bound by the write of v.
constexpr int kLiftIn = 8, kLiftOut = 16;

template <int CIN>
__global__ void __launch_bounds__(256) lift_points(const float *__restrict__ in, const float *__restrict__ A,
                                                   const float *__restrict__ bias, int cin, int W, long P, float *v) {
  __shared__ float sw[kLiftOut][kLiftIn + 1];
  const int c0 = blockIdx.y * kLiftOut, b = blockIdx.z;
  for (int e = threadIdx.x; e < kLiftOut * (kLiftIn + 1); e += blockDim.x) {
    const int c = e / (kLiftIn + 1), i = e - c * (kLiftIn + 1);
    sw[c][i] = i == kLiftIn ? bias[c0 + c] : i < cin ? A[(long)(c0 + c) * cin + i] : 0.f;
  }
  __syncthreads();
  const long p = ((long)blockIdx.x * blockDim.x + threadIdx.x) * 4;
  if (p >= P) return;
  float4 x[CIN];
#pragma unroll
  for (int i = 0; i < CIN; ++i) x[i] = *reinterpret_cast<const float4 *>(in + ((long)b * cin + i) * P + p);
  float *o = v + ((long)b * W + c0) * P + p;
#pragma unroll
  for (int c = 0; c < kLiftOut; ++c) {
    float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int i = 0; i < CIN; ++i) {
      const float w = sw[c][i];
      r.x = fmaf(w, x[i].x, r.x);
      r.y = fmaf(w, x[i].y, r.y);
      r.z = fmaf(w, x[i].z, r.z);
      r.w = fmaf(w, x[i].w, r.w);
    }
    const float q = sw[c][kLiftIn];
    *reinterpret_cast<float4 *>(o + c * P) = make_float4(r.x + q, r.y + q, r.z + q, r.w + q);
  }
}

template <int K, int N, bool PROJECT> cudaError_t launch_map(const MapArgs &a, int sms, cudaStream_t st) {
  auto kern = map_points<K, N, PROJECT>;
  constexpr size_t smem = MapSmem<K, N>::kBytes;
  static_assert(smem <= 227 * 1024, "operand buffers within a block's limit");
  static SmemGrant grant;
  const cudaError_t e = grant(kern, smem);
  if (e != cudaSuccess) return e;
  kern<<<std::max(1, std::min(a.ntiles, sms)), kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

bool head_applies(int width, int hidden, int cout, long P) {
  return (width == 32 || width == 64) && hidden == 2 * width && cout <= kOut && P % kTcRows == 0;
}

cudaError_t project_forward(const float *v, const void *q1w, const float *q1b, const float *q2w, const float *q2b,
                            float *hp, float *out, int batch, int width, int cout, long P, int sms, int *flags,
                            cudaStream_t st) {
  const int tpb = (int)(P / kTcRows);
  const MapArgs a{v, static_cast<const __nv_bfloat16 *>(q1w), width, 1, hp, q1b, q2w, q2b, out, cout, batch * tpb, tpb, P, flags};
  return width == 64 ? launch_map<64, 128, true>(a, sms, st) : launch_map<32, 64, true>(a, sms, st);
}

cudaError_t project_transpose(const float *dhp, const void *q1w, float *dv, int batch, int width, long P, int sms,
                              int *flags, cudaStream_t st) {
  const int tpb = (int)(P / kTcRows);
  const MapArgs a{dhp, static_cast<const __nv_bfloat16 *>(q1w), 1, width, dv, nullptr, nullptr, nullptr, nullptr, 0,
                  batch * tpb, tpb, P, flags};
  return width == 64 ? launch_map<128, 64, false>(a, sms, st) : launch_map<64, 32, false>(a, sms, st);
}

cudaError_t project_gradient(const float *dout, const float *hp, const float *q2w, float *dhp, float *part, int batch,
                             int hidden, int cout, long P, int sms, cudaStream_t st) {
  const int tpb = (int)(P / kTcRows), nt = batch * tpb, grid = project_parts(batch, P, sms);
  if (hidden == 128)
    project_backward<128><<<grid, kBackThreads, 0, st>>>(dout, hp, q2w, cout, nt, tpb, P, dhp, part);
  else
    project_backward<64><<<grid, kBackThreads, 0, st>>>(dout, hp, q2w, cout, nt, tpb, P, dhp, part);
  return cudaGetLastError();
}

bool lift_applies(const float *in, int width, int cin, long P) {
  return width % kLiftOut == 0 && cin <= kLiftIn && P % 4 == 0 && (reinterpret_cast<uintptr_t>(in) & 15) == 0;
}

cudaError_t lift_forward(const float *in, const float *w, const float *bias, float *v, int batch, int width, int cin,
                         long P, cudaStream_t st) {
  const dim3 grid((unsigned)((P / 4 + 255) / 256), (unsigned)(width / kLiftOut), (unsigned)batch);
  switch (cin) {
    case 1: lift_points<1><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 2: lift_points<2><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 3: lift_points<3><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 4: lift_points<4><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 5: lift_points<5><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 6: lift_points<6><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 7: lift_points<7><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    case 8: lift_points<8><<<grid, 256, 0, st>>>(in, w, bias, cin, width, P, v); break;
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace fno
}  // namespace spgpe
