// The residual's reciprocal against CUDA's correctly rounded one, for tests/test_gpu_reciprocal.py.
#include "k_nl_lines.cuh"

__global__ void reciprocal_kernel(const double* x, double* r, double* ref, long long n) {
  const long long st = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += st) {
    r[i] = ridg::nl::reciprocal(x[i]);
    ref[i] = __drcp_rn(x[i]);
  }
}

// device arrays of n doubles, the legacy default stream; 0 on success
extern "C" int reciprocal_check(const double* x, double* r, double* ref, long long n) {
  reciprocal_kernel<<<512, 256>>>(x, r, ref, n);
  if (cudaGetLastError() != cudaSuccess) return 1;
  return cudaDeviceSynchronize() == cudaSuccess ? 0 : 2;
}
