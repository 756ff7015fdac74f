// Device functions of the solvers, one launch each, for test_gpu_arithmetic.py.
#include "../paper_2602_12105_gb300/csrc/ig_device.cuh"

namespace ig {
namespace {

__global__ void quotient_kernel(const double* a, const double* b, double* q, double* d, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    q[i] = quotient(a[i], b[i]);
    d[i] = a[i] / b[i];
  }
}
__global__ void widen_kernel(const float* a, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = f32_to_f64_exact(a[i]);
}
// One warp per set of 32 J addends.
template <int J>
__global__ void sum_kernel(const double* v, double* out, int sets) {
  const int set = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (set >= sets) return;  // whole warps
  double x[J];
#pragma unroll
  for (int j = 0; j < J; ++j) x[j] = v[(size_t)set * 32 * J + 32 * j + lane];
  const double s = warp_sum_fixed<J>(x);
  out[(size_t)set * 32 + lane] = s;
}

}  // namespace
}  // namespace ig

extern "C" {
int df_quotient(const double* a, const double* b, double* q, double* d, int n) {
  ig::quotient_kernel<<<(n + 255) / 256, 256>>>(a, b, q, d, n);
  return (int)cudaDeviceSynchronize();
}
int df_widen(const float* a, double* out, int n) {
  ig::widen_kernel<<<(n + 255) / 256, 256>>>(a, out, n);
  return (int)cudaDeviceSynchronize();
}
int df_sum(const double* v, double* out, int sets, int per_lane) {
  const int blocks = (sets * 32 + 255) / 256;
  if (per_lane == 1) ig::sum_kernel<1><<<blocks, 256>>>(v, out, sets);
  else if (per_lane == 5) ig::sum_kernel<5><<<blocks, 256>>>(v, out, sets);
  else return -1;
  return (int)cudaDeviceSynchronize();
}
}
