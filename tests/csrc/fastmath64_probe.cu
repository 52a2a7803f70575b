// Test probe of the double-precision series of the pointwise operators
// (paper_2010_15069_gb300/csrc/fastmath.cuh).  Built by
// tests/test_fp64_ranges_gpu.py; not part of the library.
#include <cuda_runtime.h>

#include "fastmath.cuh"

namespace {

// fn: 0 expm1_32nd -> (e); 1 expm1_small -> (e); 2 shear_consts_2h_tiny -> (t, s);
// 3 shear_consts_2h_small -> (t, s).  out holds 2 doubles per argument.
__global__ void probe(int fn, const double *__restrict__ x, int n, double *__restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double h = x[i];
  double a = 0.0, b = 0.0;
  switch (fn) {
    case 0: a = spgpe::expm1_32nd(h); break;
    case 1: a = spgpe::expm1_small(h); break;
    case 2: spgpe::shear_consts_2h_tiny(h, a, b); break;
    default: spgpe::shear_consts_2h_small(h, a, b); break;
  }
  out[2 * i] = a;
  out[2 * i + 1] = b;
}

}  // namespace

// x and out are device pointers (n doubles in, 2 n doubles out); returns the
// CUDA status of the launch and of the synchronisation after it.
extern "C" int fastmath64_probe(int fn, const double *x, int n, double *out) {
  if (n <= 0) return 0;
  probe<<<(n + 255) / 256, 256>>>(fn, x, n, out);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaDeviceSynchronize();
  return (int)e;
}
