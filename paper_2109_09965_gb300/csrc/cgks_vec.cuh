// Aligned vector loads and stores of runs of a cell's or face's values
// (float4 in FP32, double2 in FP64): a neighbour's data arrives in one or two
// cache sectors.  Also the exact widening of FP32 runs to FP64.
#pragma once

#include <cuda_runtime.h>

namespace cgks {

template <typename T> struct VecOf;
template <> struct VecOf<float> { using V = float4; static constexpr int W = 4; };
template <> struct VecOf<double> { using V = double2; static constexpr int W = 2; };

// N values from a 16-byte aligned address (N a multiple of the vector
// width); CG: through L2, for values other blocks of the launch wrote
template <typename T, int N, bool CG = false>
__device__ __forceinline__ void vload(const T *p, T out[N]) {
  using V = typename VecOf<T>::V;
  constexpr int W = VecOf<T>::W;
  static_assert(N % W == 0, "whole vectors");
#pragma unroll
  for (int k = 0; k < N / W; ++k) {
    const V x = CG ? __ldcg(reinterpret_cast<const V *>(p) + k) : reinterpret_cast<const V *>(p)[k];
    const T *e = reinterpret_cast<const T *>(&x);
#pragma unroll
    for (int c = 0; c < W; ++c) out[k * W + c] = e[c];
  }
}
template <bool CG, typename T>
__device__ __forceinline__ T ld(const T *p) { return CG ? __ldcg(p) : *p; }

template <typename T, int N>
__device__ __forceinline__ void vstore(T *__restrict__ p, const T in[N]) {
  using V = typename VecOf<T>::V;
  constexpr int W = VecOf<T>::W;
  static_assert(N % W == 0, "whole vectors");
#pragma unroll
  for (int k = 0; k < N / W; ++k) {
    V x;
    T *e = reinterpret_cast<T *>(&x);
#pragma unroll
    for (int c = 0; c < W; ++c) e[c] = in[k * W + c];
    reinterpret_cast<V *>(p)[k] = x;
  }
}

// FP32 -> FP64, exact.  The conversion instruction runs on the FP64 pipe (a
// warp's takes as long as a multiply-add, 64 clocks of a sub-core), so a run
// of normal numbers is widened with integer instructions: the exponent
// rebiased by 1023 - 127, the fraction moved.  A run holding a zero, a
// subnormal, an infinity or a NaN takes the instruction.
template <int N>
__device__ __forceinline__ void widen(const float x[N], double y[N]) {
  unsigned low = 0xffffffffu;   // 2 * bits + 2^24 wraps below 2^25 for exponents 0 and 255
#pragma unroll
  for (int k = 0; k < N; ++k) low = min(low, (__float_as_uint(x[k]) << 1) + 0x01000000u);
  if (low >= 0x02000000u) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const unsigned b = __float_as_uint(x[k]);
      y[k] = __hiloint2double(static_cast<int>((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)),
                              static_cast<int>(b << 29));
    }
  } else {
#pragma unroll
    for (int k = 0; k < N; ++k) y[k] = static_cast<double>(x[k]);
  }
}
template <int N>
__device__ __forceinline__ void widen(const double x[N], double y[N]) {
#pragma unroll
  for (int k = 0; k < N; ++k) y[k] = x[k];
}

}  // namespace cgks
