// The device's scalar routines over arrays, for tests/test_gpu_scalars.py.
#include "rlbm_device.cuh"
#include "rlbm_dfloat.cuh"

using namespace rlbm;

namespace {
__global__ void k_f64(int n, const double* b, double* rcp, double* div, double* rsq, float* cut, double* wide) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = rcp64(b[i]);
  div[i] = 1.0 / b[i];
  rsq[i] = rsqrt64(fabs(b[i]));
  cut[i] = cut_f32(b[i]);
  wide[i] = widen_f64((float)b[i]);
}
__global__ void k_df(int n, const float* hi, const float* lo, double* got, double* want) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  got[i] = df_to_f64(df_make(hi[i], lo[i]));
  want[i] = (double)hi[i] + (double)lo[i];
}
}  // namespace

extern "C" int scalars_f64(int n, const double* b, double* rcp, double* div, double* rsq, float* cut, double* wide) {
  k_f64<<<(n + 255) / 256, 256>>>(n, b, rcp, div, rsq, cut, wide);
  return (int)cudaDeviceSynchronize();
}
extern "C" int scalars_df(int n, const float* hi, const float* lo, double* got, double* want) {
  k_df<<<(n + 255) / 256, 256>>>(n, hi, lo, got, want);
  return (int)cudaDeviceSynchronize();
}
