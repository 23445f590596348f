// The kernels' own arithmetic on arrays, for tests/test_gpu_arith.py.
#include <cstdint>

#include "cgks_internal.h"
#include "cgks_physics.cuh"
#include "cgks_vec.cuh"

namespace {
__global__ void k_recip(int n, const double *x, double *rcp, double *rsq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rcp[i] = cgks::dev::d_rcp(x[i]);
  rsq[i] = cgks::dev::d_rsqrt3(x[i]);
}
__global__ void k_half(int n, const double *U, const double *th, double *out) {   // out [n][6]: sl, isp, (m0, m1) x 2
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double *o = out + 6 * static_cast<size_t>(i);
  cgks::dev::sqrt_lambda(th[i], o[0], o[1]);
  cgks::dev::half01(U[i], o[0], o[1], +1, o[2], o[3]);
  cgks::dev::half01(U[i], o[0], o[1], -1, o[4], o[5]);
}
// every FP32 pattern, alone and in a run of five with an ordinary, a zero, a
// subnormal, and an infinite companion
__global__ void k_widen_all(unsigned long long *bad) {
  const unsigned companion[4] = { 0x3f9d70a4u, 0u, 0x00000123u, 0x7f800000u };
  unsigned long long mine = 0;
  for (uint64_t b = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; b < (1ull << 32);
       b += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
    const float x = __uint_as_float(static_cast<unsigned>(b));
    const float one[1] = { x };
    double y[1];
    cgks::widen<1>(one, y);
    const long long want = __double_as_longlong(static_cast<double>(x));
    mine += __double_as_longlong(y[0]) != want;
    float run[5] = { 1.5f, -2.25f, x, 3e-30f, __uint_as_float(companion[b >> 30]) };
    double z[5];
    cgks::widen<5>(run, z);
#pragma unroll
    for (int k = 0; k < 5; ++k) mine += __double_as_longlong(z[k]) != __double_as_longlong(static_cast<double>(run[k]));
  }
  if (mine) atomicAdd(bad, mine);
}
// every high word of an FP64 pattern with low words about the ties and ends
__global__ void k_narrow_all(unsigned long long *bad) {
  const unsigned low[10] = { 0u, 1u, 0x0fffffffu, 0x10000000u, 0x10000001u, 0x1fffffffu, 0x20000000u, 0x30000000u,
                             0xf0000000u, 0xffffffffu };
  unsigned long long mine = 0;
  for (uint64_t h = blockIdx.x * static_cast<uint64_t>(blockDim.x) + threadIdx.x; h < (1ull << 32);
       h += static_cast<uint64_t>(gridDim.x) * blockDim.x) {
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const double x = __hiloint2double(static_cast<int>(static_cast<unsigned>(h)), static_cast<int>(low[k]));
      mine += __float_as_uint(cgks::narrow<float>(x)) != __float_as_uint(static_cast<float>(x));
    }
  }
  if (mine) atomicAdd(bad, mine);
}
}  // namespace

extern "C" {
// device pointers; each call returns the CUDA status after its kernel
int arith_recip(int n, const double *x, double *rcp, double *rsq) {
  k_recip<<<(n + 127) / 128, 128>>>(n, x, rcp, rsq);
  return cudaDeviceSynchronize();
}
int arith_half(int n, const double *U, const double *th, double *out) {
  k_half<<<(n + 127) / 128, 128>>>(n, U, th, out);
  return cudaDeviceSynchronize();
}
int arith_conversions(unsigned long long *bad) {   // [2]: widen, narrow; zeroed by the caller
  k_widen_all<<<1216, 256>>>(bad);
  k_narrow_all<<<1216, 256>>>(bad + 1);
  return cudaDeviceSynchronize();
}
}
