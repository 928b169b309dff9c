// The FP64 functions of csrc/nswe_fp64.cuh and CUDA's own on arrays (for
// test_gpu_fp64.py). Build: nvcc -shared, with the library's flags.
#include "../paper_2505_10857_gb300/csrc/nswe_fp64.cuh"

namespace {

__device__ double apply(int op, double a, double b) {
  switch (op) {
  case 0: return nswe::fast_rcp(a);
  case 1: return nswe::fast_sqrt(a);
  case 2: return nswe::fast_rsqrt(a);
  case 3: return nswe::fast_div(a, b, nswe::fast_rcp(b));
  case 4: return 1.0 / a;
  case 5: return sqrt(a);
  case 6: return rsqrt(a);
  default: return a / b;
  }
}

__global__ void k_apply(int op, long n, const double *a, const double *b, double *out) {
  const long i = blockIdx.x * (long)blockDim.x + threadIdx.x;
  if (i < n) out[i] = apply(op, a[i], b[i]);
}

}  // namespace

// Device arrays of n values.
extern "C" int fp64_apply(int op, long n, const double *a, const double *b, double *out) {
  k_apply<<<(unsigned)((n + 255) / 256), 256>>>(op, n, a, b, out);
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
}
