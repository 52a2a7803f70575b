// Observables of the spin-Hall ground states (Sec. 6) and the annealing noise
// of the ground-state protocol, both precisions.
//
//  * sums_and_hist: FP64 sums rho_up rho_dn, rho_up^2, rho_dn^2 and rho_up +
//    rho_dn per instance (the phase-separation parameter of Eq. 14 and the
//    total), and the atom number in radial bins of width h about the trap
//    centre (the contour of Eq. 15 encloses 99 % of it), in one read of psi.
//  * winding: phase steps of psi_j (bilinearly interpolated) around the circle
//    of radius R99, summed in FP64 (Eq. 15 winding numbers).
//  * add_noise: psi += sigma xi, xi complex standard normal from a
//    counter-based SplitMix64 stream (Sec. 6 annealing).
#include <cuda_runtime.h>

#include <algorithm>

#include "fft_core.cuh"
#include "internal.h"
#include "smem_grant.h"

namespace spgpe {

namespace {

// Block sum of v, valid in thread 0; red: K x 32 doubles of shared memory.
template <int K> __device__ __forceinline__ void obs_block_sum(double (&v)[K], double (*red)[32]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0)
#pragma unroll
    for (int k = 0; k < K; ++k) red[k][w] = v[k];
  __syncthreads();
  if (w == 0) {
    const int nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) v[k] = (l < nw) ? red[k][l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < K; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
  }
  __syncthreads();
}

// One block per (row group, instance): the FP64 sums of its rows into
// partials[inst][block][4], and a shared-memory histogram of nb bins merged into
// hist[inst][nb] (zeroed by the caller).  What bounds it is the FP64 units, so
// a bin costs no FP64 root and division but where it must: the radius over h is
// taken in float32, and only within nb 2^-21 of a whole number (twice its
// rounding) does each point's FP64 value decide; the bins are those of FP64
// throughout.  A thread takes a point with its mirror images (columns c and nx -
// c, rows r and ny - r; those without one, 0 and n / 2, go together) and adds the
// four densities, which lie at one radius, as one; a warp adds up its runs of
// equal bins before their first lane touches the histogram (FP64 additions in
// shared memory are compare-and-swap loops).  Measured on GB300, 16 instances
// of 512^2 in complex64: 294 us with an addition per point and FP64 radii, 251 us
// with FP64 within 1/128 of an edge, 207 us as it is.
template <class T>
__global__ void __launch_bounds__(256) sums_and_hist(const cx<T> *__restrict__ psi, ObsGeom g, int rows_per_block,
                                                     double *partials, double *hist) {
  extern __shared__ double sh[];
  const int inst = blockIdx.y;
  for (int b = threadIdx.x; b < g.nb; b += blockDim.x) sh[b] = 0.0;
  __syncthreads();
  const long plane = (long)g.nx * g.ny;
  const cx<T> *u = psi + (long)inst * 2 * plane, *d = u + plane;
  const int hx = g.nx / 2, hy = g.ny / 2, lx = __ffs(hx) - 1;  // nx is a power of two
  const int r0 = blockIdx.x * rows_per_block, r1 = min(hy, r0 + rows_per_block);
  const float dxf = (float)(g.dx / g.h), dyf = (float)(g.dy / g.h), edge = 0x1p-21f * g.nb;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  const int lane = threadIdx.x & 31, end = r1 << lx;
  for (int base = r0 << lx; base < end; base += blockDim.x) {  // whole warps stay together
    const int i = base + (int)threadIdx.x;
    int bin = -1 - lane;  // equal to no neighbour's
    double sum = 0.0;
    if (i < end) {
      const int row = i >> lx, col = i & (hx - 1);
      const int iy[2] = {row, row == 0 ? hy : g.ny - row}, ix[2] = {col, col == 0 ? hx : g.nx - col};
      cx<T> a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long p = (long)iy[q >> 1] * g.nx + ix[q & 1];
        a[q] = u[p];
        b[q] = d[p];
      }
      double r[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const double ar = widen(a[q].re), ai = widen(a[q].im), br = widen(b[q].re), bi = widen(b[q].im);
        const double ru = fma(ar, ar, ai * ai), rd = fma(br, br, bi * bi);
        r[q] = ru + rd;
        s[0] = fma(ru, rd, s[0]);
        s[1] = fma(ru, ru, s[1]);
        s[2] = fma(rd, rd, s[2]);
      }
      sum = (r[0] + r[1]) + (r[2] + r[3]);
      s[3] += sum;
      // -xmax + ix dx = (ix - nx / 2) dx
      const float xf = (float)(col - hx) * dxf, yf = (float)(row - hy) * dyf;
      const float rf = sqrtf(fmaf(xf, xf, yf * yf)), off = fabsf(rf - rintf(rf));
      if (row != 0 && col != 0 && off >= edge) {
        bin = min(g.nb - 1, (int)rf);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const double x = -g.xmax + ix[q & 1] * g.dx, y = -g.ymax + iy[q >> 1] * g.dy;
          if (r[q] != 0.0) atomicAdd(&sh[min(g.nb - 1, (int)(sqrt(x * x + y * y) / g.h))], r[q]);
        }
      }
    }
    const int before = __shfl_up_sync(0xffffffffu, bin, 1);
    const bool first = lane == 0 || bin != before;
    const unsigned heads = __ballot_sync(0xffffffffu, first), later = lane == 31 ? 0u : heads >> (lane + 1);
    const int stop = later ? lane + __ffs(later) : 32;  // one past the lane's run
    for (int k = 1; __any_sync(0xffffffffu, lane + k < stop); k <<= 1) {
      const double t = __shfl_down_sync(0xffffffffu, sum, k);
      if (lane + k < stop) sum += t;
    }
    if (first && bin >= 0 && sum != 0.0) atomicAdd(&sh[bin], sum);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < g.nb; b += blockDim.x)
    if (sh[b] != 0.0) atomicAdd(&hist[(long)inst * g.nb + b], sh[b]);
  __syncthreads();  // the histogram is merged: its memory takes the sums
  obs_block_sum<4>(s, reinterpret_cast<double(*)[32]>(sh));
  if (threadIdx.x == 0)
    for (int k = 0; k < 4; ++k) partials[((long)inst * gridDim.x + blockIdx.x) * 4 + k] = s[k];
}

template <class T> __device__ __forceinline__ double phase_at(const cx<T> *f, const ObsGeom &g, double x, double y) {
  const double uu = (x + g.xmax) / g.dx, vv = (y + g.ymax) / g.dy;
  const double fu0 = floor(uu), fv0 = floor(vv);
  const double fu = uu - fu0, fv = vv - fv0;
  const int i0 = (((int)fu0) % g.nx + g.nx) % g.nx, j0 = (((int)fv0) % g.ny + g.ny) % g.ny;
  const int i1 = (i0 + 1) % g.nx, j1 = (j0 + 1) % g.ny;
  const cx<T> a = f[(long)j0 * g.nx + i0], b = f[(long)j0 * g.nx + i1];
  const cx<T> c = f[(long)j1 * g.nx + i0], e = f[(long)j1 * g.nx + i1];
  const double w00 = (1 - fu) * (1 - fv), w10 = fu * (1 - fv), w01 = (1 - fu) * fv, w11 = fu * fv;
  const double re = w00 * a.re + w10 * b.re + w01 * c.re + w11 * e.re;
  const double im = w00 * a.im + w10 * b.im + w01 * c.im + w11 * e.im;
  return atan2(im, re);
}

// Sum of the wrapped phase steps around the circle of radius R[inst] with npts
// points, over the block's share of them (one of kWindBlocks per component and
// instance): out[inst][comp][block], for the host to add and round.  Each
// point's phase is taken once and its neighbour's read from shared memory (a
// phase is about a hundred FP64 instructions); with one block per component and
// every phase taken twice, 16 instances of 512^2 took 144 us on 32 SMs.
constexpr int kWindThreads = 256;
template <class T>
__global__ void __launch_bounds__(kWindThreads) winding(const cx<T> *__restrict__ psi, ObsGeom g, const double *R,
                                                        int npts, double *out) {
  __shared__ double ph[kWindThreads + 1], red[1][32];
  const int comp = blockIdx.y, inst = blockIdx.z;
  const long plane = (long)g.nx * g.ny;
  const cx<T> *f = psi + ((long)inst * 2 + comp) * plane;
  const double r = R[inst];
  const double pi = 3.14159265358979323846;
  const int per = (npts + gridDim.x - 1) / gridDim.x, k1 = min(npts, (int)(blockIdx.x + 1) * per);
  double s[1] = {0.0};
  for (int k0 = blockIdx.x * per; k0 < k1; k0 += kWindThreads) {
    const int n = min(kWindThreads, k1 - k0);  // steps k0 .. k0 + n - 1, phases k0 .. k0 + n
    for (int j = threadIdx.x; j <= n; j += kWindThreads) {
      double sn, cs;
      sincospi(2.0 * ((k0 + j) % npts) / npts, &sn, &cs);
      ph[j] = phase_at(f, g, r * cs, r * sn);
    }
    __syncthreads();
    if ((int)threadIdx.x < n) {
      double dph = ph[threadIdx.x + 1] - ph[threadIdx.x];
      while (dph > pi) dph -= 2.0 * pi;
      while (dph <= -pi) dph += 2.0 * pi;
      s[0] += dph;
    }
    __syncthreads();
  }
  obs_block_sum<1>(s, red);
  if (threadIdx.x == 0) out[((long)inst * 2 + comp) * gridDim.x + blockIdx.x] = s[0];
}

// SplitMix64 (Steele, Lea & Flood, OOPSLA 2014) as a counter-based generator:
// draw c of stream `seed` is the output function applied to
// seed + (c + 1) * 0x9E3779B97F4A7C15.
__device__ __forceinline__ unsigned long long mix64(unsigned long long seed, unsigned long long c) {
  unsigned long long z = seed + (c + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// psi += sigma xi: element e of instance i (global index inst0 + i) takes the
// draws 2E and 2E + 1, E = (inst0 + i) * n2 + e, as uniforms u = (draw >> 11)
// 2^-53, and xi = sqrt(-ln(1 - u1)) e^{2 pi i u2}.
template <class T>
__global__ void __launch_bounds__(256) add_noise(cx<T> *psi, long n2, int ninst, long inst0, double sigma,
                                                 unsigned long long seed) {
  const long total = n2 * ninst;
  for (long j = (long)blockIdx.x * blockDim.x + threadIdx.x; j < total; j += (long)gridDim.x * blockDim.x) {
    const unsigned long long E = (unsigned long long)(inst0 * n2 + j);
    const double u1 = (double)(mix64(seed, 2 * E) >> 11) * 0x1.0p-53;
    const double u2 = (double)(mix64(seed, 2 * E + 1) >> 11) * 0x1.0p-53;
    const double r = sigma * sqrt(-log(1.0 - u1));
    double sn, cs;
    sincospi(2.0 * u2, &sn, &cs);
    cx<T> v = psi[j];
    v.re = T(double(v.re) + r * cs);
    v.im = T(double(v.im) + r * sn);
    psi[j] = v;
  }
}

template <class T> cudaError_t obs_launch(const void *psi, const ObsGeom &g, int ninst, double *partials,
                                          int sum_blocks, double *hist, const double *R, int npts, double *wind,
                                          int phase, cudaStream_t st) {
  const cx<T> *p = reinterpret_cast<const cx<T> *>(psi);
  if (phase == 0) {
    const int rpb = (g.ny / 2 + sum_blocks - 1) / sum_blocks;  // pairs of mirrored rows
    // the histogram, or the sums after it; no other shared memory, so that up to
    // 48 KB need no grant and kMaxSmemPerBlock bins of 8 bytes are the limit
    const size_t sm = std::max((size_t)g.nb, (size_t)4 * 32) * sizeof(double);
    static SmemGrant grant;
    const cudaError_t e = sm > 48 * 1024 ? grant(sums_and_hist<T>, sm) : cudaSuccess;
    if (e != cudaSuccess) return e;
    sums_and_hist<T><<<dim3(sum_blocks, ninst), 256, sm, st>>>(p, g, rpb, partials, hist);
  } else {
    winding<T><<<dim3(kWindBlocks, 2, ninst), kWindThreads, 0, st>>>(p, g, R, npts, wind);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_observables(int es, const void *psi, const ObsGeom &g, int ninst, double *partials,
                               int sum_blocks, double *hist, const double *R, int npts, double *wind, int phase,
                               cudaStream_t st) {
  return es == 8 ? obs_launch<float>(psi, g, ninst, partials, sum_blocks, hist, R, npts, wind, phase, st)
                 : obs_launch<double>(psi, g, ninst, partials, sum_blocks, hist, R, npts, wind, phase, st);
}

cudaError_t launch_add_noise(int es, void *psi, long n2, int ninst, long inst0, double sigma, unsigned long long seed,
                             int sms, cudaStream_t st) {
  const long want = (n2 * ninst + 255) / 256;
  const int grid = (int)(want < 8L * sms ? want : 8L * sms);
  if (grid < 1) return cudaSuccess;
  if (es == 8)
    add_noise<float><<<grid, 256, 0, st>>>(reinterpret_cast<cx<float> *>(psi), n2, ninst, inst0, sigma, seed);
  else
    add_noise<double><<<grid, 256, 0, st>>>(reinterpret_cast<cx<double> *>(psi), n2, ninst, inst0, sigma, seed);
  return cudaGetLastError();
}

}  // namespace spgpe
