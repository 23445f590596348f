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

// FP64 -> TF, rounded to nearest even as the conversion instruction does; to
// FP32 with integer instructions for the same reason (values whose FP32 form is
// normal, and zeros; the rest by the instruction).
template <typename TF> __device__ __forceinline__ TF narrow(double x);
template <> __device__ __forceinline__ double narrow<double>(double x) { return x; }
template <> __device__ __forceinline__ float narrow<float>(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x)), lo = static_cast<unsigned>(__double2loint(x));
  const unsigned sign = hi & 0x80000000u, mag = hi & 0x7fffffffu;
  if (mag - 0x38100000u < 0x0fd00000u) {   // FP32 exponents 1 to 253: rounding cannot overflow
    unsigned b = ((mag - 0x38000000u) << 3) | (lo >> 29);
    const unsigned rest = lo & 0x1fffffffu;
    b += rest > 0x10000000u - (b & 1u);    // above half, or half and odd
    return __uint_as_float(sign | b);
  }
  if ((mag | lo) == 0u) return __uint_as_float(sign);
  return static_cast<float>(x);
}

}  // namespace cgks
