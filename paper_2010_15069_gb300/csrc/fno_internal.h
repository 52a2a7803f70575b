// Launchers of the Fourier-neural-operator kernels, used by the C ABI in fno.cu:
// general products and reductions (fno_kernels.cu), tensor-core channel maps and
// weight gradients (fno_tc.cu), transforms (fno_dft.cu), layers (fno_layer.cu),
// mode mixing (fno_mix.cu), lift and projection (fno_head.cu).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace spgpe {
namespace fno {

// C(m, n) = alpha sum_k A(m, k) B(k, n) + beta C(m, n) + bias[m] per batch
// entry; element (m, k) of A at A + b sAb + m sAm + k sAk (likewise B, C).
// partial: split-K over `splits` ranges of k, the partial product of split s
// of batch entry b to C + (b splits + s) sCs (alpha 1, beta and bias
// ignored) for sum_splits.
struct GemmR {
  int M, N, K, batch = 1, splits = 1;
  bool partial = false;
  float alpha = 1.f, beta = 0.f;
  const void *A;
  bool a_bf16 = false;
  long sAm, sAk, sAb = 0;
  const float *B;
  long sBk, sBn, sBb = 0;
  float *C;
  long sCm, sCn, sCb = 0, sCs = 0;
  const float *bias = nullptr;
  // device error flags of the model; non-null also admits the tensor-core
  // path (gemm_real_tc), which records a wait that ran out there
  int *flags = nullptr;
};

// Complex C(m, n) = sum_k op(A)(m, k) op(B)(k, n), strides in complex elements; op conjugates when conj_a / conj_b (not both); A may be
// bfloat16 pairs (a_bf16; then not conjugated).
struct GemmC {
  int M, N, K, batch = 1;
  const void *A;
  bool a_bf16 = false, conj_a = false, conj_b = false;
  long sAm, sAk, sAb = 0;
  const float2 *B;
  long sBk, sBn, sBb = 0;
  float2 *C;
  long sCm, sCn, sCb = 0;
};

cudaError_t gemm_real(const GemmR &g, cudaStream_t st);
// The same product on the tensor cores (fno_tc.cu) for the pointwise channel
// maps: bfloat16 weights A (sAb = 0; M = 64 or 128 rows, K = 64 or 128), a
// float32 B with unit stride along N (N a multiple of 128), C with unit
// stride along N, no split-K, alpha = 1, flags set; cudaErrorNotSupported
// for any other shape.
bool gemm_tc_applies(const GemmR &g);
cudaError_t gemm_real_tc(const GemmR &g, cudaStream_t st);
// Weight and bias gradients on the tensor cores (fno_tc.cu): per CTA (of
// weight_grad_parts), a partial dW [M][N] = sum over its points of X[b](m, p)
// Y[b](n, p) and, with bias, db [M] = sum X[b](m, p), (M N + M) or M N floats
// each in part, for sum_parts.  X [b][M][P], Y [b][N][P] with sample strides
// sXb, sYb; M, N <= 128, P a multiple of 64, 16-byte aligned.
struct WeightGrad {
  int M, N, batch;
  long P;
  const float *X;
  long sXb;
  const float *Y;
  long sYb;
  float *part;
  bool bias;
  int *flags;
};
// A CTA sums at most kGradRun blocks: the accumulator truncates, so its errors
// have one sign and grow with the run (1024^2, batch 8: 5e-4 of a gradient in
// runs of 431 blocks).
constexpr long kGradBlock = 64;  // points per block of the MMA's K
constexpr long kGradRun = 16;
bool weight_grad_applies(const WeightGrad &g);
inline int weight_grad_parts(int batch, long P, int sms) {
  const long blocks = batch * (P / kGradBlock);
  return (int)std::max<long>(1, std::min(blocks, std::max(2L * sms, (blocks + kGradRun - 1) / kGradRun)));
}
cudaError_t weight_grad(const WeightGrad &g, int sms, cudaStream_t st);
cudaError_t sum_splits(const float *part, long n, int splits, float *out, cudaStream_t st);
cudaError_t gemm_complex(const GemmC &g, cudaStream_t st);
// Truncated Fourier transforms (fno_dft.cu) of `images` n x n fields with the
// kept modes kx < M, ky = -M .. M - 1 (M even, at most 32; n a multiple of 64;
// `width` channels per sample, whose rows fill whole tiles of 128): along x
// (E[x][2 k + part] = cos, -sin; adjoint: times g_k / n^2, g_0 = 1, g_k = 2) and
// along y (Et[y][j] = (a.x, a.x, -a.y, a.y), a = exp(-2 pi i ky_j y / n)) in float32, the inverse along y
// on the tensor cores (table: dft_table(InverseY) as it is; sin32[y] = sin(2 pi
// 32 y / n)); flags receives a wait that ran out.
enum class DftTable { InverseY, LayerX };
bool dft_applies(int n, int modes, int width);
std::vector<uint16_t> dft_table(DftTable which, int n, int modes);
cudaError_t dft_x(const float *v, const float *E, bool adjoint, float *X1, int images, int n, int modes, cudaStream_t st);
cudaError_t dft_y(const float *X1, const float4 *Et, float2 *vh, int images, int n, int modes, cudaStream_t st);
cudaError_t idft_y(const float2 *oh, const void *table, const float *sin32, float2 *G, int images, int n, int modes,
                   int *flags, cudaStream_t st);
// The rest of a spectral layer in one pass (fno_layer.cu; W = 32 or 64 where
// dft_applies): forward, u = W v + w + the real inverse of G along x, written
// to u (null: not kept) with out = gelu(u), or (activate false) out = u;
// backward, out = (W^T du + the adjoint of the transform along x of G) times
// gelu'(u_prev) (null: without).  table: dft_table(LayerX).
bool layer_applies(int n, int modes, int width);
cudaError_t layer_forward(const float *v, const float2 *G, const void *table, const void *weights, const float *bias,
                          float *u, float *out, bool activate, int batch, int width, int n, int modes, int sms,
                          int *flags, cudaStream_t st);
cudaError_t layer_backward(const float *du, const float2 *G, const void *table, const void *weights, const float *u_prev,
                           float *out, int batch, int width, int n, int modes, int sms, int *flags, cudaStream_t st);
// Lift and projection (fno_head.cu).  head_applies: W = 32 or 64 channels, 2 W
// hidden ones, at most 4 outputs, P a multiple of 128.  project_forward: out =
// Q2 gelu(Q1 v + q1) + q2, Q1 v + q1 to hp unless null.  project_gradient: dhp =
// (Q2^T dout) gelu'(hp) and, per CTA (project_parts() of them), the sums dQ2
// [cout][H], dq1 [H], dq2 [cout] in project_partials() floats.  project_transpose: dv =
// Q1^T dhp.  lift_forward: v = A a + bias.
bool head_applies(int width, int hidden, int cout, long P);
cudaError_t project_forward(const float *v, const void *q1w, const float *q1b, const float *q2w, const float *q2b,
                            float *hp, float *out, int batch, int width, int cout, long P, int sms, int *flags,
                            cudaStream_t st);
constexpr long kHeadTile = 128;  // points per tile
constexpr long kHeadRun = 16;    // tiles whose float32 sums a CTA adds up at most
inline long project_partials(int hidden, int cout) { return (long)cout * hidden + hidden + cout; }
inline int project_parts(int batch, long P, int sms) {
  const long tiles = batch * (P / kHeadTile);
  return (int)std::max<long>(1, std::min(tiles, std::max<long>(sms, (tiles + kHeadRun - 1) / kHeadRun)));
}
cudaError_t project_gradient(const float *dout, const float *hp, const float *q2w, float *dhp, float *part, int batch,
                             int hidden, int cout, long P, int sms, cudaStream_t st);
cudaError_t project_transpose(const float *dhp, const void *q1w, float *dv, int batch, int width, long P, int sms,
                              int *flags, cudaStream_t st);
bool lift_applies(const float *in, int width, int cin, long P);
cudaError_t lift_forward(const float *in, const float *w, const float *bias, float *v, int batch, int width, int cin,
                         long P, cudaStream_t st);
// Floats that the partial sums of a network's weight gradients take, the largest
// of: every product of weight and bias (M outputs, N inputs), per CTA on the
// tensor cores or per split of `splits` in the general path, and the
// projection's sums.
inline int general_splits(long P) { return (int)std::max<long>(1, P / 1024); }
inline size_t partial_floats(int cin, int cout, int width, int hidden, int batch, long P, int sms) {
  const int shapes[4][2] = {{width, cin}, {width, width}, {hidden, width}, {cout, hidden}};
  size_t most = (size_t)project_parts(batch, P, sms) * project_partials(hidden, cout);
  for (const auto &q : shapes) {
    const size_t mn = (size_t)q[0] * q[1];
    most = std::max(most, (size_t)weight_grad_parts(batch, P, sms) * (mn + q[0]));
    most = std::max(most, (size_t)batch * general_splits(P) * mn);
  }
  return most;
}
// out[i] = sum of part[k][i] over k < parts, in a fixed order; stride floats
// from one part to the next.
cudaError_t sum_parts(const float *part, long stride, int parts, long n, float *out, cudaStream_t st);
cudaError_t gelu_forward(const float *u, float *v, long n, cudaStream_t st);
cudaError_t gelu_backward(const float *u, float *d, long n, cudaStream_t st);
// grad[c] = sum over the batch and the points of x[b][c][p]; scratch holds
// 64 C doubles.
cudaError_t bias_gradient(const float *x, int B, int C, long P, float *grad, double *scratch, cudaStream_t st);
// sums[2 b], sums[2 b + 1] = sum (out - t)^2, sum t^2 of sample b; sums holds
// 130 B doubles (the rest is scratch); dout (nullable) = 2 (out - t) / den_b / B.
cudaError_t loss_terms(const float *out, const float *t, long n, int B, double *sums, float *dout, cudaStream_t st);
// Adam (Kingma & Ba 2015) with bias correction: the rates of step t (from 1),
// and one parameter's update.
struct AdamRates {
  float lr = 0.f, c1 = 1.f, c2 = 1.f;
};
inline AdamRates adam_rates(float lr, int t) {
  return {lr, (float)(1.0 - std::pow(0.9, t)), (float)(1.0 - std::pow(0.999, t))};
}
__device__ __forceinline__ void adam_one(float &w, float &m, float &v, float g, const AdamRates &r) {
  m = fmaf(0.9f, m, 0.1f * g);
  v = fmaf(0.999f, v, 0.001f * g * g);
  w -= r.lr * (m / r.c1) / (sqrtf(v / r.c2) + 1e-8f);
}
// The exact GELU x Phi(x) and its derivative.
__device__ __forceinline__ float gelu_f(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_d(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}
// Both of them (one erf).
__device__ __forceinline__ void gelu_both(float x, float &g, float &d) {
  const float phi = 0.5f * (1.f + erff(x * 0.70710678118654752f));
  g = x * phi;
  d = phi + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}
// Up to kRanges [begin, end) ranges of the parameter vector.
constexpr int kRanges = 16;
struct Ranges {
  int n = 0;
  long begin[kRanges], end[kRanges];
};
// Adam on the FP32 masters w of the ranges; wb (bfloat16) and wr (FP32)
// receive the rounded weights.
cudaError_t adam_update(float *w, void *wb, float *wr, const float *g, float *m, float *v, const Ranges &rg, float lr,
                        int t, cudaStream_t st);
// The spectral layers' channel mixing per mode (fno_mix.cu; W = 32 or 64
// channels, a multiple of 8 modes, bfloat16 pairs R[mode][o][c], spectra
// [sample][channel][mode]): out[b][o][m] = sum_c R[m][o][c] in[b][c][m], or
// transposed out[b][c][m] = sum_o conj(R[m][o][c]) in[b][o][m]; the weights'
// gradient dR[m][o][c] = sum_b d[b][o][m] conj(v[b][c][m]) for at most
// kMixGradBatch samples, written to g or applied as their Adam step.
constexpr int kMixGradBatch = 8;
bool mix_applies(int width, int modes);
cudaError_t mix_modes(const void *R, const float2 *in, float2 *out, int width, int modes, int batch, bool transposed,
                      cudaStream_t st);
cudaError_t mix_gradient(const float2 *d, const float2 *v, int width, int modes, int batch, float *g, cudaStream_t st);
cudaError_t mix_adam(const float2 *d, const float2 *v, int width, int modes, int batch, float *w, float *m, float *ve,
                     void *wb, float lr, int t, cudaStream_t st);
cudaError_t round_weights(const float *w, void *wb, float *wr, long n, cudaStream_t st);

}  // namespace fno
}  // namespace spgpe
