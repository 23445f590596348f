// Kernels of the 3-D hot path (included by cgks_device3.cu only).
//
// One solve; cells colour-major with reverse Cuthill-McKee order inside a
// colour, faces sorted by their lower cell; structure-of-arrays
// [component][n].  Flux kernels are templated on the flux type TF (double,
// or float in the mixed path, where W, W_x, U and every accumulation into
// them stay double).
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "cgks_internal.h"
#include "cgks_physics3.cuh"
#include "cgks_pdl.cuh"
#include "cgks_shapes.h"
#include "cgks_vec.cuh"

namespace cgks {
namespace kern3 {

namespace D3 = cgks::dev3;
namespace dev = cgks::dev;
constexpr int NV = 5;
// as in 2-D; 64 would make the residual's sums of a large mesh longer than it
// saves (512,000 cells: final sum 10.2 us with 256, 12.2 with 128, 18.0 with 64;
// V-cycle 3546, 3529, 3528)
constexpr int kCellBlock = 128;
constexpr int kFO = 4 * NV;                        // face outputs of the high level: F0, F1, Wc, Wt
constexpr int kBadState = 1;

template <typename T>
__host__ __device__ constexpr bool is_f32() { return std::is_same<T, float>::value; }

template <typename T>
struct ParamsT {
  T gamma, K, cfl_hi, icfl_lo, mu;   // icfl_lo = 1 / CFL of the low-order level
  D3::KC<T> kc;
  const int *bc_kind;          // [16]
  const T *bc_uw;              // [16][3] wall velocity (global)
  const T *bc_rho, *bc_u, *bc_p;  // [16], [16][3], [16] free stream (global)
  int flux_lo;                    // low-level flux: CGKS_FLUX_KFVS or CGKS_FLUX_LF
  T tau_c1, tau_c2;               // numerical collision time constants of the full flux
  T weno_eps, weno_g0;            // compact WENO epsilon (0: linear weights), linear weight of P2
  int lo_viscous;                 // 1: the low-order residual carries a first-order viscous flux
};

template <typename T>
struct MeshT {
  int nc, nf;
  const T *vol, *ivol, *ih, *hdt, *m2, *op;       // m2 [6][nc], op [27*9][nc]
  const T *fe, *fS, *fjump, *fw, *fxi;            // fe [9][nf] (n, t1, t2), fw [4][nf], fxi [24][nf]
  const T *fidl;                                  // 1/delta: centre distance along n (boundary: twice to the face)
  const T *sn, *shs;                              // [6*3][nc] outward normal per slot (FP64: times S/2), [6][nc] S/2
  const int *fng, *cface, *cnbr, *fc0, *fc1;
};

struct Ctl {
  double dt_fixed;
  int res_ctr, pad_;
};

__device__ __forceinline__ double dt_of(const Ctl *ctl, const unsigned long long *dt_bits, double cfl) {
  if (ctl->dt_fixed > 0.0) return ctl->dt_fixed;
  return cfl * __longlong_as_double(static_cast<long long>(*dt_bits));
}
// positive and finite, by the bits (a comparison takes the FP64 pipe)
__device__ __forceinline__ bool positive_finite(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x));
  return hi < 0x7ff00000u && (hi | static_cast<unsigned>(__double2loint(x))) != 0u;
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
// density and pressure positive, everything finite (see the 2-D one)
__device__ __forceinline__ bool state_ok(const double w[NV]) {
  const double q = w[4] * w[0] - 0.5 * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]);
  return positive_finite(w[0]) && positive_finite(q) && finite_bits(w[1]) && finite_bits(w[2]) &&
         finite_bits(w[3]) && finite_bits(w[4]);
}

__device__ __forceinline__ void block_sum2(double a, double b, double *out2) {
  __shared__ double sa[32], sb[32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sa[warp] = a; sb[warp] = b; }
  __syncthreads();
  if (warp == 0) {
    const int nw = blockDim.x >> 5;
    a = lane < nw ? sa[lane] : 0.0;
    b = lane < nw ? sb[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { out2[0] = a; out2[1] = b; }
  }
}

template <typename T>
__device__ __forceinline__ D3::Frame<T> frame_of(const MeshT<T> &m, int f) {
  D3::Frame<T> F;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int d = 0; d < 3; ++d) F.e[a][d] = m.fe[(3 * a + d) * m.nf + f];
  return F;
}

// ------------------------------------------------------------------
__global__ void k_reset_dt(Ctl *ctl, unsigned long long *dt_bits, double dt_fixed) {
  pdl_enter();
  if (threadIdx.x == 0) { *dt_bits = 0x7ff0000000000000ull; ctl->dt_fixed = dt_fixed; }
  pdl_exit();
}

// explicit step: min over cells of h / (|U| + c + 2 nu / h), h = 3|Omega| / sum S
__global__ void __launch_bounds__(kCellBlock) k_dt(MeshT<double> m, ParamsT<double> P, const double *W,
                                                   unsigned long long *dt_bits) {
  pdl_enter();
  // the minimum on the bits, positive doubles sort like integers (a NaN sorts
  // last): comparisons of doubles take the FP64 pipe
  __shared__ unsigned long long wmin[kCellBlock / 32];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double d = INFINITY;
  if (i < m.nc) {
    const int n = m.nc;
    const double rho = W[i], ir = dev::d_rcp(rho);
    const double u = W[n + i] * ir, v = W[2 * n + i] * ir, w = W[3 * n + i] * ir, q2 = u * u + v * v + w * w;
    const double p = (P.gamma - 1.0) * (W[4 * n + i] - 0.5 * rho * q2);
    const double hh = m.hdt[i];
    const double speed = dev::sqrt_fast(q2) + dev::sqrt_fast(P.gamma * p * ir);
    d = hh * hh * dev::d_rcp(fma(hh, speed, 2.0 * (P.mu * ir)));   // hh / (speed + 2 nu / hh)
  }
  unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
  for (int o = 16; o > 0; o >>= 1) b = min(b, __shfl_down_sync(0xffffffffu, b, o));
  if ((threadIdx.x & 31) == 0) wmin[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kCellBlock / 32; ++w) b = min(b, wmin[w]);
    constexpr unsigned long long kInf = 0x7ff0000000000000ull;
    if (b < kInf) atomicMin(dt_bits, b);
  }
  pdl_exit();
}

// FP32: wall ghost of a state and its gradient (global), through the face frame
template <typename T>
__device__ __forceinline__ void wall_ghost(const ParamsT<T> &P, int tag, const D3::Frame<T> &F, const T w[NV],
                                           const T g[3][NV], T wg[NV], T gg[3][NV]) {
  T wl[NV], dl[3][NV], wgl[NV], dgl[3][NV];
  D3::rot_in(F, w, wl);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    T t[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) t[v] = F.e[k][0] * g[0][v] + F.e[k][1] * g[1][v] + F.e[k][2] * g[2][v];
    D3::rot_in(F, t, dl[k]);
  }
  if (P.bc_kind[tag] == CGKS_BC_SLIP) {
    D3::ghost_slip(wl, dl, wgl, dgl);
  } else {
    T uw[3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      uw[a] = F.e[a][0] * P.bc_uw[3 * tag] + F.e[a][1] * P.bc_uw[3 * tag + 1] + F.e[a][2] * P.bc_uw[3 * tag + 2];
    D3::ghost_noslip(P.gamma, uw, wl, dl, wgl, dgl);
  }
  D3::rot_out(F, wgl, wg);
  T gk[3][NV];
#pragma unroll
  for (int k = 0; k < 3; ++k) D3::rot_out(F, dgl[k], gk[k]);
  // global gradient: grad_d = sum_k e_k[d] (derivative along e_k)
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int v = 0; v < NV; ++v) gg[d][v] = F.e[0][d] * gk[0][v] + F.e[1][d] * gk[1][v] + F.e[2][d] * gk[2][v];
}

template <typename T>
__device__ __forceinline__ void farfield_ghost(const ParamsT<T> &P, int tag, const D3::Frame<T> &F, const T wl[NV],
                                               T wg[NV]) {
  T ue[3];
#pragma unroll
  for (int a = 0; a < 3; ++a)
    ue[a] = F.e[a][0] * P.bc_u[3 * tag] + F.e[a][1] * P.bc_u[3 * tag + 1] + F.e[a][2] * P.bc_u[3 * tag + 2];
  D3::ghost_farfield(P.kc, P.gamma, P.bc_rho[tag], ue, P.bc_p[tag], wl, wg);
}

// Compact WENO (conservative variables), 3-D form of the 2-D weno_combine:
// candidates P2 (c) and the nk linear polynomials h g.(xi, eta, zeta) of the
// mean gradients of the cell and its face neighbours (lin[k][d][v]).  beta:
// cell mean of the squared first derivatives (centroid value squared plus
// the quadratic form of the cell's second moments M = m2) plus the squared
// second derivatives, each multi-index once.  w ~ gamma / (beta + eps)^2,
// gamma_0 = g0, the rest (1 - g0)/nk; result
// (w_0 / gamma_0)(P2 - sum gamma_k P1_k) + sum w_k P1_k.
// Candidate 0 is the cell's own; candidate 1 + s, of face slot s, counts where
// bit 1 + s of on is set (slots by a constant index: no local memory).
__device__ __forceinline__ float quot(float a, float b) { return a / b; }
__device__ __forceinline__ double quot(double a, double b) { return a * dev::d_rcp(b); }
template <typename T, int NC>
__device__ __forceinline__ void weno_combine3(const ParamsT<T> &P, const T M[6], unsigned on, const T (&lin)[7][3][NC],
                                              T (&c)[kNM3][NC]) {
  const int nk = __popc(on);
  const T g0 = P.weno_g0, eps = P.weno_eps;
  const T gk = quot(T(1) - g0, T(nk));
  // symmetric M: xx xy xz yy yz zz
  const T Mx[3][3] = { { M[0], M[1], M[2] }, { M[1], M[3], M[4] }, { M[2], M[4], M[5] } };
#pragma unroll
  for (int v = 0; v < NC; ++v) {
    const T q[kNM3] = { c[0][v], c[1][v], c[2][v], c[3][v], c[4][v], c[5][v], c[6][v], c[7][v], c[8][v] };
    const T G[3][3] = { { T(2) * q[3], q[4], q[5] }, { q[4], T(2) * q[6], q[7] }, { q[5], q[7], T(2) * q[8] } };
    T b0 = q[0] * q[0] + q[1] * q[1] + q[2] * q[2];
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int e = 0; e < 3; ++e) b0 += G[d][a] * Mx[a][e] * G[d][e];
    b0 += T(4) * q[3] * q[3] + q[4] * q[4] + q[5] * q[5] + T(4) * q[6] * q[6] + q[7] * q[7] + T(4) * q[8] * q[8];
    const T w0 = quot(g0, (b0 + eps) * (b0 + eps));
    T ws = w0, wk[7];
    T l[3] = { T(0), T(0), T(0) };
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      if (!(on >> k & 1)) continue;
      const T b = lin[k][0][v] * lin[k][0][v] + lin[k][1][v] * lin[k][1][v] + lin[k][2][v] * lin[k][2][v];
      wk[k] = quot(gk, (b + eps) * (b + eps));
      ws += wk[k];
#pragma unroll
      for (int d = 0; d < 3; ++d) l[d] += gk * lin[k][d][v];
    }
    const T iws = quot(T(1), ws);
    const T f0 = quot(w0 * iws, g0);
    T sel[3] = { T(0), T(0), T(0) };
#pragma unroll
    for (int k = 0; k < 7; ++k) {
      if (!(on >> k & 1)) continue;
#pragma unroll
      for (int d = 0; d < 3; ++d) sel[d] += wk[k] * iws * lin[k][d][v];
    }
#pragma unroll
    for (int d = 0; d < 3; ++d) c[d][v] = f0 * (q[d] - l[d]) + sel[d];
#pragma unroll
    for (int r = 3; r < kNM3; ++r) c[r][v] = f0 * q[r];
  }
}

// K1: compact quadratic per cell: coef[(q*5 + v)][n], 9 monomials.  FP64: one
// thread per cell and variable, FP32: per cell (as in 2-D).  us per launch,
// FP64, before / now (with the wall mirrors as linear maps): 9,177 hexahedra
// 120.5 / 48.4, a sphere of 128,000 cells 318.9 / 280.5.
template <typename T> __host__ __device__ constexpr int recon_vars() { return is_f32<T>() ? NV : 1; }
// f(cell, variable) over the items of a launch, a warp per variable of 32 cells
template <typename T, typename F>
__device__ __forceinline__ void for_recon(const int n, F &&f) {
  constexpr int G = NV / recon_vars<T>();
  for_items((n + 31) / 32 * 32 * G, [&](int t) {
    const int i = G == 1 ? t : t / (32 * G) * 32 + t % 32;
    if (i < n) f(i, t / 32 % G);
  });
}
template <typename T, bool WENO, int NC>
__device__ __forceinline__ void recon_at(const MeshT<T> &m, const ParamsT<T> &P, const T *W,
                                         const T *Wx, T *__restrict__ coef,
                                         const unsigned char *__restrict__ wenok, const int i, const int comp) {
  const int n = m.nc, vo = NC == NV ? 0 : comp;
  T wi[NC], gi[3][NC];
#pragma unroll
  for (int v = 0; v < NC; ++v) {
    wi[v] = W[(vo + v) * n + i];
#pragma unroll
    for (int d = 0; d < 3; ++d) gi[d][v] = Wx[(d * NV + vo + v) * n + i];
  }
  T c[kNM3][NC];
#pragma unroll
  for (int q = 0; q < kNM3; ++q) {
    const T o0 = m.op[((4 * kMaxFace3) * kNM3 + q) * n + i];
    const T o1 = m.op[((4 * kMaxFace3 + 1) * kNM3 + q) * n + i];
    const T o2 = m.op[((4 * kMaxFace3 + 2) * kNM3 + q) * n + i];
#pragma unroll
    for (int v = 0; v < NC; ++v) c[q][v] = o0 * gi[0][v] + o1 * gi[1][v] + o2 * gi[2][v];
  }
  T lin[WENO ? 7 : 1][3][NC];
  unsigned on = 1;
  if constexpr (WENO) {
    const T h = quot(T(1), m.ih[i]);
#pragma unroll
    for (int v = 0; v < NC; ++v)
#pragma unroll
      for (int d = 0; d < 3; ++d) lin[0][d][v] = h * gi[d][v];
  }
#pragma unroll (WENO || NC == 1 ? kMaxFace3 : 2)   // 2: loads of two slots in flight, 162 -> 151 us (512,000 cells)
  for (int s = 0; s < kMaxFace3; ++s) {
    const int fs = m.cface[s * n + i];
    if (fs == kNoFace) continue;
    const int j = m.cnbr[s * n + i];
    T b0[NC], b[3][NC];
    if (j >= 0) {
#pragma unroll
      for (int v = 0; v < NC; ++v) {
        b0[v] = W[(vo + v) * n + j] - wi[v];
#pragma unroll
        for (int d = 0; d < 3; ++d) b[d][v] = Wx[(d * NV + vo + v) * n + j];
      }
      if constexpr (WENO) {
        const T h = quot(T(1), m.ih[i]);
#pragma unroll
        for (int v = 0; v < NC; ++v)
#pragma unroll
          for (int d = 0; d < 3; ++d) lin[1 + s][d][v] = h * b[d][v];
        on |= 2u << s;
      }
    } else {
      const int f = fs >= 0 ? fs : ~fs;
      const int tag = -1 - m.fc1[f];
      if (P.bc_kind[tag] == CGKS_BC_FARFIELD) continue;
      if constexpr (NC == NV) {
        const D3::Frame<T> F = frame_of(m, f);
        T wg[NV];
        wall_ghost(P, tag, F, wi, gi, wg, b);
#pragma unroll
        for (int v = 0; v < NV; ++v) b0[v] = wg[v] - wi[v];
      } else {   // the mirror image mixes the variables
        const double nn[3] = { m.fe[f], m.fe[m.nf + f], m.fe[2 * m.nf + f] };
        double g[3];
        dev::WallMap<3>(P.bc_kind[tag], P.bc_uw + 3 * tag, nn).one(comp, W + i, Wx + i, n, b0[0], g);
#pragma unroll
        for (int d = 0; d < 3; ++d) b[d][0] = g[d];
      }
    }
#pragma unroll
    for (int q = 0; q < kNM3; ++q) {
      const T o0 = m.op[((4 * s) * kNM3 + q) * n + i], o1 = m.op[((4 * s + 1) * kNM3 + q) * n + i];
      const T o2 = m.op[((4 * s + 2) * kNM3 + q) * n + i], o3 = m.op[((4 * s + 3) * kNM3 + q) * n + i];
#pragma unroll
      for (int v = 0; v < NC; ++v) c[q][v] += o0 * b0[v] + o1 * b[0][v] + o2 * b[1][v] + o3 * b[2][v];
    }
  }
  if constexpr (WENO) {
    if (wenok[i]) {
      const T M[6] = { m.m2[i], m.m2[n + i], m.m2[2 * n + i], m.m2[3 * n + i], m.m2[4 * n + i], m.m2[5 * n + i] };
      weno_combine3(P, M, on, lin, c);
    }
  }
#pragma unroll
  for (int q = 0; q < kNM3; ++q)
#pragma unroll
    for (int v = 0; v < NC; ++v) coef[(q * NV + vo + v) * n + i] = c[q][v];
}
template <typename T>
__global__ void __launch_bounds__(kMaxShapeBlock)
    k_recon(MeshT<T> m, ParamsT<T> P, const T *W, const T *Wx, T *coef) {
  pdl_enter();
  for_recon<T>(m.nc, [&](int i, int comp) { recon_at<T, false, recon_vars<T>()>(m, P, W, Wx, coef, nullptr, i, comp); });
  pdl_exit();
}
// with the compact WENO step; wenok[i] = 1 where the stencil gave a quadratic
template <typename T>
__global__ void __launch_bounds__(kMaxShapeBlock)
    k_recon_weno(MeshT<T> m, ParamsT<T> P, const T *W, const T *Wx, T *coef,
                 const unsigned char *wenok) {
  pdl_enter();
  for_recon<T>(m.nc, [&](int i, int comp) { recon_at<T, true, recon_vars<T>()>(m, P, W, Wx, coef, wenok, i, comp); });
  pdl_exit();
}

// value and gradient of cell i's quadratic at scaled offset x; the gradient
// is left in the cell's scaled coordinates (times 1/h = ih for the physical one)
__device__ __forceinline__ void recon_scaled(const MeshT<double> &m, const double *W, const double *coef,
                                             int i, const double x[3], double val[NV], double g[3][NV]) {
  const int n = m.nc;
  const double a = x[0], b = x[1], e = x[2];
  const double a2 = a + a, b2 = b + b, e2 = e + e;
  const double p[6] = { a * a - m.m2[i], a * b - m.m2[n + i], a * e - m.m2[2 * n + i], b * b - m.m2[3 * n + i],
                   b * e - m.m2[4 * n + i], e * e - m.m2[5 * n + i] };
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    double c[kNM3];
#pragma unroll
    for (int q = 0; q < kNM3; ++q) c[q] = coef[(q * NV + v) * n + i];
    val[v] = W[v * n + i] + c[0] * a + c[1] * b + c[2] * e + c[3] * p[0] + c[4] * p[1] + c[5] * p[2] + c[6] * p[3] +
             c[7] * p[4] + c[8] * p[5];
    g[0][v] = c[0] + c[3] * a2 + c[4] * b + c[5] * e;
    g[1][v] = c[1] + c[4] * a + c[6] * b2 + c[7] * e;
    g[2][v] = c[2] + c[5] * a + c[7] * b + c[8] * e2;
  }
}

// value and gradient of cell i's quadratic at scaled offset x
template <typename T>
__device__ __forceinline__ void recon_point(const MeshT<T> &m, const T *W, const T *coef,
                                            int i, const T x[3], T val[NV], T g[3][NV]) {
  const int n = m.nc;
  const T ih = m.ih[i];
  const T a = x[0], b = x[1], e = x[2];
  const T p[6] = { a * a - m.m2[i], a * b - m.m2[n + i], a * e - m.m2[2 * n + i], b * b - m.m2[3 * n + i],
                   b * e - m.m2[4 * n + i], e * e - m.m2[5 * n + i] };
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T c[kNM3];
#pragma unroll
    for (int q = 0; q < kNM3; ++q) c[q] = coef[(q * NV + v) * n + i];
    val[v] = W[v * n + i] + c[0] * a + c[1] * b + c[2] * e + c[3] * p[0] + c[4] * p[1] + c[5] * p[2] + c[6] * p[3] +
             c[7] * p[4] + c[8] * p[5];
    g[0][v] = (c[0] + T(2) * c[3] * a + c[4] * b + c[5] * e) * ih;
    g[1][v] = (c[1] + c[4] * a + T(2) * c[6] * b + c[7] * e) * ih;
    g[2][v] = (c[2] + c[5] * a + c[7] * b + T(2) * c[8] * e) * ih;
  }
}

// K2: smooth GKS flux and interface state at the Gauss points of every face:
// out[f][k*5 + v], k = 0 F0, 1 F1, 2 Wc, 3 Wt, weighted sums, global frame:
// one run of kFO values per face (AoS), so that the cells gathering a face
// read it in one piece.
// Two forms, as in 2-D: face_raw_at (raw moments in the face frame: the FP32
// of the mixed path) and face_points_at (FP64).
template <typename T, bool FULL>
__device__ __forceinline__ void face_raw_at(const MeshT<T> &m, const ParamsT<T> &P, const T *W,
                                        const T *coef, T *__restrict__ out, const Ctl *ctl,
                                        const unsigned long long *dt_bits, const int f) {
  const int nf = m.nf;
  T dt = T(0);
  if constexpr (FULL) dt = static_cast<T>(dt_of(ctl, dt_bits, static_cast<double>(P.cfl_hi)));
  const int c0 = m.fc0[f], c1 = m.fc1[f], ng = m.fng[f];
  const T ajump = m.fjump[f];
  const D3::Frame<T> F = frame_of(m, f);
  T acc[4][NV];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[k][v] = T(0);
  int tag = 0;
  bool farfield = false;
  T wff[NV];
  if (c1 < 0) {
    tag = -1 - c1;
    farfield = P.bc_kind[tag] == CGKS_BC_FARFIELD;
    if (farfield) {
      T wm[NV], wl[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) wm[v] = W[v * m.nc + c0];
      D3::rot_in(F, wm, wl);
      farfield_ghost(P, tag, F, wl, wff);
    }
  }
  for (int k = 0; k < ng; ++k) {
    T x0[3], wL[NV], gL[3][NV];
#pragma unroll
    for (int d = 0; d < 3; ++d) x0[d] = m.fxi[(3 * k + d) * nf + f];
    recon_point(m, W, coef, c0, x0, wL, gL);
    T wl[NV], dl[3][NV];
    D3::rot_in(F, wL, wl);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      T t[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) t[v] = F.e[a][0] * gL[0][v] + F.e[a][1] * gL[1][v] + F.e[a][2] * gL[2][v];
      D3::rot_in(F, t, dl[a]);
    }
    T wr[NV], dr[3][NV];
    if (c1 >= 0) {
      T x1[3], wR[NV], gR[3][NV];
#pragma unroll
      for (int d = 0; d < 3; ++d) x1[d] = m.fxi[(12 + 3 * k + d) * nf + f];
      recon_point(m, W, coef, c1, x1, wR, gR);
      D3::rot_in(F, wR, wr);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        T t[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) t[v] = F.e[a][0] * gR[0][v] + F.e[a][1] * gR[1][v] + F.e[a][2] * gR[2][v];
        D3::rot_in(F, t, dr[a]);
      }
    } else if (farfield) {
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        wr[v] = wff[v];
        dr[0][v] = dr[1][v] = dr[2][v] = T(0);
      }
    } else if (P.bc_kind[tag] == CGKS_BC_SLIP) {
      D3::ghost_slip(wl, dl, wr, dr);
    } else {
      T uw[3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
        uw[a] = F.e[a][0] * P.bc_uw[3 * tag] + F.e[a][1] * P.bc_uw[3 * tag + 1] + F.e[a][2] * P.bc_uw[3 * tag + 2];
      D3::ghost_noslip(P.gamma, uw, wl, dl, wr, dr);
    }
    T F0[NV], F1[NV], Wc[NV], Wt[NV];
    if constexpr (FULL)
      D3::gks_full_point_local(P.kc, P.mu, ajump, dt, P.tau_c1, P.tau_c2, wl, wr, dl, dr, F0, F1, Wc, Wt);
    else
      D3::gks_point_local(P.kc, P.mu, ajump, wl, wr, dl, dr, F0, F1, Wc, Wt);
    const T wk = m.fw[k * nf + f];
    T gq[NV];
    D3::rot_out(F, F0, gq);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[0][v] += wk * gq[v];
    D3::rot_out(F, F1, gq);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[1][v] += wk * gq[v];
    D3::rot_out(F, Wc, gq);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[2][v] += wk * gq[v];
    D3::rot_out(F, Wt, gq);
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[3][v] += wk * gq[v];
  }
  T o[kFO];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int v = 0; v < NV; ++v) o[k * NV + v] = acc[k][v];
  vstore<T, kFO>(out + static_cast<size_t>(f) * kFO, o);
}
// The FP64 flux by the 2-D face_point_at's scheme.  LANES threads share a
// face's 3 or 4 Gauss points.
template <bool FULL, int LANES>
__device__ __forceinline__ void face_points_at(const MeshT<double> &m, const ParamsT<double> &P,
                                               const double *W, const double *coef,
                                               double *__restrict__ out, const Ctl *ctl,
                                               const unsigned long long *dt_bits, const int f, const int lane) {
  using T = double;
  const int nf = m.nf;
  const int c0 = m.fc0[f], c1 = m.fc1[f], ng = m.fng[f];
  const T ajump = m.fjump[f];
  const D3::Frame<T> F = frame_of(m, f);
  T acc[4][NV];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int v = 0; v < NV; ++v) acc[k][v] = T(0);
  const int tag = c1 < 0 ? -1 - c1 : 0;
  const bool farfield = c1 < 0 && P.bc_kind[tag] == CGKS_BC_FARFIELD;
  const T ihL = m.ih[c0], ihR = c1 >= 0 ? m.ih[c1] : ihL;
  T wff[NV];   // the far-field state, one for the face
  if (farfield) {
    T wm[NV], wi[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) wm[v] = W[v * m.nc + c0];
    D3::rot_in(F, wm, wi);
    farfield_ghost(P, tag, F, wi, wff);
  }
#pragma unroll 1
  for (int k = lane; k < ng; k += LANES) {
    T x0[3], wL[NV], gL[3][NV], wR[NV], gR[3][NV];
#pragma unroll
    for (int d = 0; d < 3; ++d) x0[d] = m.fxi[(3 * k + d) * nf + f];
    recon_scaled(m, W, coef, c0, x0, wL, gL);
    T wl[NV], wr[NV];
    D3::rot_in(F, wL, wl);
    if (c1 >= 0) {
      T x1[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) x1[d] = m.fxi[(12 + 3 * k + d) * nf + f];
      recon_scaled(m, W, coef, c1, x1, wR, gR);
      D3::rot_in(F, wR, wr);
    } else if (farfield) {
#pragma unroll
      for (int v = 0; v < NV; ++v) wr[v] = wff[v];
      D3::rot_out(F, wr, wR);
#pragma unroll
      for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int v = 0; v < NV; ++v) gR[d][v] = T(0);
    } else {
      const dev::WallMap<3> mirror(P.bc_kind[tag], P.bc_uw + 3 * tag, F.e[0]);
      mirror.apply(wL, wR);
      mirror.apply_gradient(gL, gR);
      D3::rot_in(F, wR, wr);
    }
    // slopes of the equilibrium at W^c: the mean of the sides plus, along
    // n, alpha / delta times the jump
    T Wc[NV], G[3][NV], F0[NV], F1[NV], Wt[NV];
    const T hl = T(0.5) * ihL, hr = T(0.5) * ihR;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T aj = ajump * F.e[0][d];
#pragma unroll
      for (int v = 0; v < NV; ++v) G[d][v] = hl * gL[d][v] + hr * gR[d][v] + aj * (wR[v] - wL[v]);
    }
    if constexpr (FULL) {
      // each side's derivatives along the face axes, in the face frame
      T dl[3][NV], dr[3][NV];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        T t[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v)
          t[v] = ihL * (F.e[a][0] * gL[0][v] + F.e[a][1] * gL[1][v] + F.e[a][2] * gL[2][v]);
        D3::rot_in(F, t, dl[a]);
#pragma unroll
        for (int v = 0; v < NV; ++v)
          t[v] = ihR * (F.e[a][0] * gR[0][v] + F.e[a][1] * gR[1][v] + F.e[a][2] * gR[2][v]);
        D3::rot_in(F, t, dr[a]);
      }
      const T dt = dt_of(ctl, dt_bits, P.cfl_hi);   // the full flux integrates over the step
      D3::gks_full(P.kc, P.mu, dt, P.tau_c1, P.tau_c2, F, wl, wr, dl, dr, G, F0, F1, Wc, Wt);
    } else {
      // W^c from the two half ranges
      T wc[NV];
      D3::half_state<T, false>(P.kc, wl, +1, wc);
      D3::half_state<T, true>(P.kc, wr, -1, wc);
      D3::rot_out(F, wc, Wc);
      D3::gks_smooth(P.kc, P.mu, F.e[0], Wc, G, F0, F1, Wt);
    }
    const T wk = m.fw[k * nf + f];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      acc[0][v] += wk * F0[v];
      acc[1][v] += wk * F1[v];
      acc[2][v] += wk * Wc[v];
      acc[3][v] += wk * Wt[v];
    }
  }
  T *o = out + static_cast<size_t>(f) * kFO;
  if constexpr (LANES == 1) {
    T r[kFO];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int v = 0; v < NV; ++v) r[k * NV + v] = acc[k][v];
    vstore<T, kFO>(o, r);
  } else {
    // lane l collects and stores output l: halves exchanged, then quarters
    static_assert(LANES == 4, "one lane per output");
    const unsigned quad = 0xfu << (threadIdx.x & 28);
    const bool b1 = lane & 2, b0 = lane & 1;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T p = (b1 ? acc[2][v] : acc[0][v]) + __shfl_xor_sync(quad, b1 ? acc[0][v] : acc[2][v], 2);
      const T q = (b1 ? acc[3][v] : acc[1][v]) + __shfl_xor_sync(quad, b1 ? acc[1][v] : acc[3][v], 2);
      o[lane * NV + v] = (b0 ? q : p) + __shfl_xor_sync(quad, b0 ? p : q, 1);
    }
  }
}
// Threads per face, FP64.  A launch takes as long as the warps of one sub-core
// (608 of them) issue one after another: per 32 faces one warp of 3 or 4 points
// with one thread, 4 warps of a point with four.  Four lose nothing where there
// are quadrilaterals (a warp with one among its faces takes 4 points either way)
// and are the finer quantum, one is a little shorter on large meshes; on
// triangles alone the fourth lane idles, and one thread is shorter from two
// warps of the four-lane form a sub-core on (9,728 faces).  us per launch, smooth
// flux, one / four: hexahedra 13,056 faces 86 / 76, 61,236 319 / 287, 92,256
// 409 / 420, 196,800 851 / 856; prisms 41,600 248 / 199, 112,896 483 / 507;
// sphere shells (prisms and tetrahedra) 51,520 261 / 238, 70,720 306 / 321, 98,560
// 477 / 446, 142,080 590 / 630; tetrahedra 9,234 68 / 53, 12,600 69 / 76, 50,688
// 195 / 242, 113,778 372 / 516.  (Raw moments in one thread took 358 us on 28,850
// faces of hexahedra and 2809 us on 282,880 of a shell; now 145 and 1074.)
constexpr int64_t kFaceLanes4 = 100000, kFaceLanes4Tri = 9728;
inline int face_lanes(int64_t n_faces, bool quads) { return n_faces < (quads ? kFaceLanes4 : kFaceLanes4Tri) ? 4 : 1; }
// FP32: one thread per face.  Bound by latency at two warps a scheduler (255
// registers); the smooth flux is shorter with 128 and four warps, in spite of
// some spills: 512,000 cells 411 -> 377 us a launch (112: 390, 144: 427); the
// full flux is not (128,000 cells 241; 128 registers 252, 168: 248).
template <typename T, bool FULL>
__global__ void __maxnreg__(FULL ? 255 : 128)
    k_face(MeshT<T> m, ParamsT<T> P, const T *W, const T *coef, T *out,
           const Ctl *ctl, const unsigned long long *dt_bits) {
  pdl_enter();
  for_items(m.nf, [&](int f) { face_raw_at<T, FULL>(m, P, W, coef, out, ctl, dt_bits, f); });
  pdl_exit();
}
// FP64
template <bool FULL, int LANES>
__global__ void __launch_bounds__(kMaxShapeBlock)
    k_face_points(MeshT<double> m, ParamsT<double> P, const double *W, const double *coef,
                  double *out, const Ctl *ctl, const unsigned long long *dt_bits) {
  pdl_enter();
  for_items(LANES * m.nf,
            [&](int i) { face_points_at<FULL, LANES>(m, P, W, coef, out, ctl, dt_bits, i / LANES, i % LANES); });
  pdl_exit();
}

enum UpdMode { kS1O2 = 0, kS2O4Stage = 1, kS2O4Final = 2, kResidual = 3 };

// K3: per cell gather of the face sums in FP64 (see the 2-D k_update):
//   R = -sum sgn S (a0 F0A + a1 F1(A, B));  W_out = W_base + dt/|Omega| R;
//   Wx_out = 1/|Omega| sum sgn S n (WcA + b1 Wt)
// In the mixed path the runs are widened and the mirrors rounded with integer
// instructions (the FP64 pipe bounds the kernel): 223 -> 119 us a launch on
// 512,000 cells.
// The mode is a template argument so that each variant holds only the runs
// it reads: the residual reads F0 and F1 of one buffer, the stages one
// whole run, the final S2O4 stage two.
template <typename TF, int mode>
__global__ void __launch_bounds__(kCellBlock) k_update(MeshT<double> m, ParamsT<double> P,
                                                       const double *Wbase, const TF *FA,
                                                       const TF *FB, const Ctl *ctl,
                                                       const unsigned long long *dt_bits, int *status,
                                                       double *Wout, double *Wxout,
                                                       double *partial, double *Rout,
                                                       TF *Wout_m, TF *Wxout_m) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = m.nc;
  double num = 0.0, den = 0.0;
  // mesh data first (nothing in a cycle writes it), then wait for the predecessor
  int fsl[kMaxFace3];
  if (i < n)
#pragma unroll
    for (int s = 0; s < kMaxFace3; ++s) fsl[s] = m.cface[s * n + i];
  pdl_enter();
  if (i < n) {
    const double dt = dt_of(ctl, dt_bits, P.cfl_hi);
    const double a1 = mode == kS2O4Stage ? 0.125 * dt : mode == kS2O4Final ? dt / 6.0 : 0.5 * dt;
    const double b1 = mode == kS2O4Stage ? 0.5 * dt : dt;
    double R[NV] = { 0, 0, 0, 0, 0 }, g[3][NV] = { { 0 } };
#pragma unroll
    for (int s = 0; s < kMaxFace3; ++s) {
      const int fs = fsl[s];
      if (fs == kNoFace) continue;
      const size_t at = static_cast<size_t>(fs >= 0 ? fs : ~fs) * kFO;
      // half the slot's area and sgn S n_f from the per-cell slot arrays (coalesced)
      const double h = m.shs[s * n + i], S = fs >= 0 ? h : -h;
      // the face's run of F0, F1, Wc, Wt (and the second stage's, when used);
      // the residual reads the leading F0, F1 part only
      constexpr int kRes = (2 * NV + VecOf<TF>::W - 1) / VecOf<TF>::W * VecOf<TF>::W;
      constexpr int NA = mode == kResidual ? kRes : kFO;
      TF fa[NA];
      double a[NA], b[mode == kS2O4Final ? kFO : 1];
      vload<TF, NA>(FA + at, fa);
      widen<mode == kResidual ? 2 * NV : NA>(fa, a);
      if constexpr (mode == kS2O4Final) {
        TF fb[kFO];
        vload<TF, kFO>(FB + at, fb);
        widen<NV>(fb + NV, b + NV);
        widen<NV>(fb + 3 * NV, b + 3 * NV);
      }
      double nn[3] = { 0.0, 0.0, 0.0 };
      if constexpr (mode != kResidual)
#pragma unroll
        for (int d = 0; d < 3; ++d) nn[d] = m.sn[(3 * s + d) * n + i];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        double f1 = a[NV + v];
        if constexpr (mode == kS2O4Final) f1 += 2.0 * b[NV + v];
        const double f0 = mode == kS2O4Stage ? 0.5 * a[v] : a[v];
        R[v] -= S * (f0 + a1 * f1);
        if constexpr (mode != kResidual) {
          double wt;
          if constexpr (mode == kS2O4Final) wt = b[3 * NV + v];
          else wt = a[3 * NV + v];
          const double wp = a[2 * NV + v] + b1 * wt;
#pragma unroll
          for (int d = 0; d < 3; ++d) g[d][v] += nn[d] * wp;
        }
      }
    }
    if (Rout)
#pragma unroll
      for (int v = 0; v < NV; ++v) Rout[v * n + i] = 2.0 * R[v];
    if constexpr (mode != kResidual) {
      const double iv2 = 2.0 * m.ivol[i], k = dt * iv2;
      const double old = Wbase[i];   // Wout may be Wbase (explicit steps update in place)
      double w[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        w[v] = Wbase[v * n + i] + k * R[v];
        Wout[v * n + i] = w[v];
        if (Wout_m) Wout_m[v * n + i] = narrow<TF>(w[v]);
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const double x = g[d][v] * iv2;
          Wxout[(d * NV + v) * n + i] = x;
          if (Wxout_m) Wxout_m[(d * NV + v) * n + i] = narrow<TF>(x);
        }
      }
      if (!state_ok(w)) atomicOr(status, kBadState);
      num = fabs(w[0] - old);
      den = old;
    }
  }
  if (partial) block_sum2(num, den, &partial[2 * blockIdx.x]);
  pdl_exit();
}

__global__ void k_res_final(const double *partial, int nblocks, Ctl *ctl, double *hist, int cap,
                            double *last) {
  pdl_enter();
  double a = 0.0, b = 0.0;
  for (int k = threadIdx.x; k < nblocks; k += blockDim.x) { a += partial[2 * k]; b += partial[2 * k + 1]; }
  __shared__ double tot[2];
  block_sum2(a, b, tot);
  __syncthreads();
  if (threadIdx.x == 0) {
    const double r = tot[0] / tot[1];
    last[0] = r; last[1] = tot[0]; last[2] = tot[1];
    const int c = ctl->res_ctr;
    if (hist && c < cap) hist[c] = r;
    ctl->res_ctr = c + 1;
  }
  pdl_exit();
}

// ---------------------------- low-order level ----------------------------
// Records of the low level, as in 2-D (cgks_kernels.cuh):
//   base  [kBase] per cell, the part a sweep reads first: in FP64 rho, u, v,
//         w, H = rho E + p; p, 1/(2 lambda), sqrt(lambda), 1/sqrt(pi lambda),
//         c, rho u, rho v, rho w, rho E, 0, 0; in FP32 U (5), u, v, w; p,
//         1/(2 lambda), sqrt(lambda), 1/sqrt(pi lambda), c, 0, 0, 0;
//   delta [del_run] per cell: dU; in FP64 then du, dv, dw, dp, the changes of
//         velocity and pressure it makes; 0;
//   Flo   [lo_run] per face: the flux, lambda_p, padding.
constexpr int kBase = 16;
template <typename T> __host__ __device__ constexpr int del_run() { return is_f32<T>() ? 8 : 10; }
template <typename T> __host__ __device__ constexpr int lo_run() { return is_f32<T>() ? 8 : 6; }

// positions in a base record
template <typename T>
struct BaseAt {
  static constexpr bool f = is_f32<T>();
  static constexpr int u = f ? 5 : 1, H = 4, p = f ? 8 : 5, i2l = f ? 9 : 6, sl = f ? 10 : 7, isp = f ? 11 : 8,
                       c = f ? 12 : 9, m = f ? 1 : 10, E = f ? 4 : 13;
};
template <typename T>
__device__ __forceinline__ D3::Prim<T> base_prim(const T r[kBase]) {
  using A = BaseAt<T>;
  D3::Prim<T> q;
  q.rho = r[0]; q.u = r[A::u]; q.v = r[A::u + 1]; q.w = r[A::u + 2];
  q.p = r[A::p]; q.i2l = r[A::i2l]; q.sl = r[A::sl]; q.isp = r[A::isp]; q.c = r[A::c];
  return q;
}
// base record of the FP64 state u
template <typename TF>
__device__ __forceinline__ void base_record(const ParamsT<TF> &P, const double u[NV], TF r[kBase]) {
  using A = BaseAt<TF>;
  TF w[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) w[v] = narrow<TF>(u[v]);
  const D3::Prim<TF> q = D3::prim_of(w, P.gamma, P.kc);
#pragma unroll
  for (int v = 13; v < kBase; ++v) r[v] = TF(0);
  if constexpr (!is_f32<TF>()) r[A::H] = w[4] + q.p;
  r[0] = w[0];
  r[A::u] = q.u; r[A::u + 1] = q.v; r[A::u + 2] = q.w;
  r[A::p] = q.p; r[A::i2l] = q.i2l; r[A::sl] = q.sl; r[A::isp] = q.isp; r[A::c] = q.c;
  r[A::m] = w[1]; r[A::m + 1] = w[2]; r[A::m + 2] = w[3]; r[A::E] = w[4];
}
template <typename TF>
__device__ __forceinline__ void store_base(const ParamsT<TF> &P, const double u[NV], TF *base, int i) {
  TF r[kBase];
  base_record(P, u, r);
  vstore<TF, kBase>(base + static_cast<size_t>(i) * kBase, r);
}
// the delta record of an increment d on a cell with base b = (rho, u, v, w),
// see the 2-D store_delta
__device__ __forceinline__ void delta_record(double gamma, const double b[4], const double d[NV], double r[10]) {
  const double ir = dev::d_rcp(b[0] + d[0]);
  double du[3], a = 0.0, e = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    du[k] = (d[1 + k] - b[1 + k] * d[0]) * ir;
    a += d[1 + k] * (b[1 + k] + du[k]);
    e += b[1 + k] * du[k];
  }
  const double g1 = gamma - 1.0;
#pragma unroll
  for (int v = 0; v < NV; ++v) r[v] = d[v];
  r[5] = du[0]; r[6] = du[1]; r[7] = du[2];
  r[8] = g1 * d[4] - 0.5 * g1 * (a + b[0] * e);
  r[9] = 0.0;
}
__device__ __forceinline__ void delta_record(float, const float *, const float d[NV], float r[8]) {
#pragma unroll
  for (int v = 0; v < NV; ++v) r[v] = d[v];
  r[5] = r[6] = r[7] = 0.0f;
}
template <typename T>
__device__ __forceinline__ void store_delta(T gamma, const T b[4], const T d[NV], T *delta, int i) {
  T r[del_run<T>()];
  delta_record(gamma, b, d, r);
  vstore<T, del_run<T>()>(delta + static_cast<size_t>(i) * del_run<T>(), r);
}

// U^{k+1} = U^k + dU (FP64), base record of U^{k+1}; first: U = W_p0
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_lo_cell(int n, ParamsT<TF> P, int first, const double *Wp0,
                                                        double *U, const TF *delta,
                                                        TF *base) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  TF d[del_run<TF>()];
  if (!first) vload<TF, del_run<TF>()>(delta + static_cast<size_t>(i) * del_run<TF>(), d);
  double u[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    u[v] = first ? Wp0[v * n + i] : U[v * n + i] + static_cast<double>(d[v]);
    U[v * n + i] = u[v];
  }
  store_base(P, u, base, i);
  pdl_exit();
}

// ghost of a cell-mean state (zero gradients), global
template <typename T>
__device__ __forceinline__ void lo_ghost(const ParamsT<T> &P, int tag, const D3::Frame<T> &F, const T w[NV],
                                         T wg[NV]) {
  const int kind = P.bc_kind[tag];
  if constexpr (!is_f32<T>())
    if (kind != CGKS_BC_FARFIELD) {
      dev::WallMap<3>(kind, P.bc_uw + 3 * tag, F.e[0]).apply(w, wg);
      return;
    }
  T wl[NV], wgl[NV];
  D3::rot_in(F, w, wl);
  if (kind == CGKS_BC_FARFIELD) {
    farfield_ghost(P, tag, F, wl, wgl);
  } else {
    T z[3][NV], dz[3][NV];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int v = 0; v < NV; ++v) z[k][v] = T(0);
    if (kind == CGKS_BC_SLIP) {
      D3::ghost_slip(wl, z, wgl, dz);
    } else {
      T uw[3];
#pragma unroll
      for (int a = 0; a < 3; ++a)
        uw[a] = F.e[a][0] * P.bc_uw[3 * tag] + F.e[a][1] * P.bc_uw[3 * tag + 1] + F.e[a][2] * P.bc_uw[3 * tag + 2];
      D3::ghost_noslip(P.gamma, uw, wl, z, wgl, dz);
    }
  }
  D3::rot_out(F, wgl, wg);
}

// KFVS (or Lax-Friedrichs) flux, lambda_p = max of both sides
__device__ __forceinline__ float third(float x) { return x / 3.0f; }
__device__ __forceinline__ double third(double x) { return x * (1.0 / 3.0); }
template <typename T>
__device__ __forceinline__ void lo_face_at(const MeshT<T> &m, const ParamsT<T> &P, const T *base,
                                           T *__restrict__ Flo, const int f) {
  const int c0 = m.fc0[f], c1 = m.fc1[f];
  // FP32 and boundary faces take the whole frame, an inner FP64 face its normal
  D3::Frame<T> F;
  if (is_f32<T>() || c1 < 0) F = frame_of(m, f);
  else
#pragma unroll
    for (int d = 0; d < 3; ++d) F.e[0][d] = m.fe[d * m.nf + f];
  T ra[kBase], rb[kBase];
  vload<T, kBase>(base + static_cast<size_t>(c0) * kBase, ra);
  const D3::Prim<T> a = base_prim(ra);
  D3::Prim<T> b;
  using A = BaseAt<T>;
  const T wa[NV] = { ra[0], ra[A::m], ra[A::m + 1], ra[A::m + 2], ra[A::E] };
  T wb[NV];
  if (c1 >= 0) {
    vload<T, kBase>(base + static_cast<size_t>(c1) * kBase, rb);
    b = base_prim(rb);
    wb[0] = rb[0]; wb[1] = rb[A::m]; wb[2] = rb[A::m + 1]; wb[3] = rb[A::m + 2]; wb[4] = rb[A::E];
  } else {
    lo_ghost(P, -1 - c1, F, wa, wb);
    b = D3::prim_of(wb, P.gamma, P.kc);
  }
  T la3[3], lb3[3];
#pragma unroll
  for (int k = 0; k < (is_f32<T>() ? 3 : 1); ++k) {
    la3[k] = a.u * F.e[k][0] + a.v * F.e[k][1] + a.w * F.e[k][2];
    lb3[k] = b.u * F.e[k][0] + b.v * F.e[k][1] + b.w * F.e[k][2];
  }
  T la = fabs(la3[0]) + a.c, lb = fabs(lb3[0]) + b.c, ira = T(0), irb = T(0);
  if (P.mu != T(0)) {
    const T S = m.fS[f];
    ira = dev::d_rcp(a.rho);
    irb = dev::d_rcp(b.rho);
    la += T(2) * (P.mu * ira) * S * m.ivol[c0];
    lb += T(2) * (P.mu * irb) * S * m.ivol[c1 >= 0 ? c1 : c0];
  }
  const T lmax = la > lb ? la : lb;
  const T nx = F.e[0][0], ny = F.e[0][1], nz = F.e[0][2];
  T Fg[NV];
  if (P.flux_lo == CGKS_FLUX_LF) {
    // Lax-Friedrichs alternative of Section 3 with the implicit operator's
    // lambda_p: (F_n(U_l) + F_n(U_r)) / 2 - lambda_p (U_r - U_l) / 2
    const T una = la3[0], unb = lb3[0];
    const T Fa[NV] = { a.rho * una, wa[1] * una + a.p * nx, wa[2] * una + a.p * ny, wa[3] * una + a.p * nz,
                       (wa[4] + a.p) * una };
    const T Fb[NV] = { b.rho * unb, wb[1] * unb + b.p * nx, wb[2] * unb + b.p * ny, wb[3] * unb + b.p * nz,
                       (wb[4] + b.p) * unb };
#pragma unroll
    for (int v = 0; v < NV; ++v) Fg[v] = T(0.5) * (Fa[v] + Fb[v]) - T(0.5) * lmax * (wb[v] - wa[v]);
  } else if constexpr (!is_f32<T>()) {
    // KFVS without the face frame, as in 2-D
    const T una = la3[0], unb = lb3[0];
    T m0a, m1a, m0b, m1b;
    dev::half01(una, a.sl, a.isp, +1, m0a, m1a);
    dev::half01(unb, b.sl, b.isp, -1, m0b, m1b);
    const T ja = a.rho * m1a, jb = b.rho * m1b, pa = a.p * m0a, pb = b.p * m0b, pn = pa + pb;
    Fg[0] = ja + jb;
    Fg[1] = ja * a.u + jb * b.u + pn * nx;
    Fg[2] = ja * a.v + jb * b.v + pn * ny;
    Fg[3] = ja * a.w + jb * b.w + pn * nz;
    Fg[4] = m1a * (wa[4] + T(0.5) * a.p) + m1b * (wb[4] + T(0.5) * b.p) + T(0.5) * (pa * una + pb * unb);
  } else {
    T Fl[NV];
    D3::kfvs(P.K, a.rho, la3[0], la3[1], la3[2], a.i2l, a.sl, a.isp, b.rho, lb3[0], lb3[1], lb3[2], b.i2l, b.sl,
             b.isp, Fl);
    D3::rot_out(F, Fl, Fg);
  }
  if (P.lo_viscous && P.mu > T(0)) {
    // first-order viscous flux: normal gradients from the two cell states
    // over the centre distance delta, Stokes' hypothesis, Pr = 1 heat flux
    //   tau.n = mu / delta (du + (n.du) n / 3),  q.n = -kappa (T_r - T_l) / delta
    const T md = P.mu * m.fidl[f];
    const T du[3] = { b.u - a.u, b.v - a.v, b.w - a.w };
    const T nn[3] = { nx, ny, nz };
    const T dn = third(du[0] * nx + du[1] * ny + du[2] * nz);
    const T um[3] = { T(0.5) * (a.u + b.u), T(0.5) * (a.v + b.v), T(0.5) * (a.w + b.w) };
    T work = T(0);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const T tau = md * (du[d] + dn * nn[d]);
      Fg[1 + d] -= tau;
      work += tau * um[d];
    }
    T qn;   // gamma / (gamma - 1) = N / 2 + 1
    if constexpr (is_f32<T>()) qn = -md * P.gamma / (P.gamma - T(1)) * (b.p * irb - a.p * ira);
    else qn = -md * (P.kc.hN + T(1)) * (b.p * irb - a.p * ira);
    Fg[4] -= work - qn;
  }
  // one run per face (AoS): the flux and lambda_p, read together by the
  // right-hand side of each cell
  constexpr int N = lo_run<T>();
  T o[N];
#pragma unroll
  for (int v = 0; v < NV; ++v) o[v] = Fg[v];
  o[NV] = lmax;
#pragma unroll
  for (int v = NV + 1; v < N; ++v) o[v] = T(0);
  vstore<T, N>(Flo + static_cast<size_t>(f) * N, o);
}
template <typename T>
__global__ void __launch_bounds__(kMaxShapeBlock)
    k_lo_face(MeshT<T> m, ParamsT<T> P, const T *base, T *Flo) {
  pdl_enter();
  for_items(m.nf, [&](int f) { lo_face_at(m, P, base, Flo, f); });
  pdl_exit();
}

// right-hand side R^k = R_lo + S (FP64 sums), 1/D_i (FP64), lambda per slot (in
// FP64 times S/2), first colour pass (dU = R / D on colour 0, zero elsewhere)
// The FP64 pipe bounds it in both precisions (a cell's fluxes are summed in
// FP64): FP32 fluxes are widened with integer instructions and only colour 0
// forms R / D.  512,000 cells mixed: 107 -> 78.4 us a launch.
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_lo_rhs(MeshT<double> m, ParamsT<double> P, TF gamma, int first,
                                                       int colour0_end, const TF *base,
                                                       const TF *Flo,
                                                       const double *Rp0, double *Src,
                                                       TF *Rk, TF *invD,
                                                       TF *delta, TF *lamS) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.nc) { pdl_enter(); return; }
  const int n = m.nc;
  // mesh data first (nothing in a cycle writes it), then wait for the predecessor
  int fsl[kMaxFace3];
  double Sh[kMaxFace3];
#pragma unroll
  for (int s = 0; s < kMaxFace3; ++s) {
    fsl[s] = m.cface[s * n + i];
    Sh[s] = m.shs[s * n + i];
  }
  pdl_enter();
  constexpr int N = lo_run<TF>();
  double R[NV] = { 0, 0, 0, 0, 0 }, sum = 0.0;
  TF fl[kMaxFace3][N];
#pragma unroll
  for (int s = 0; s < kMaxFace3; ++s) {
    const int fs = fsl[s];
    if (fs == kNoFace) continue;
    vload<TF, N>(Flo + static_cast<size_t>(fs >= 0 ? fs : ~fs) * N, fl[s]);   // flux and lambda_p
  }
#pragma unroll
  for (int s = 0; s < kMaxFace3; ++s) {
    const int fs = fsl[s];
    if (fs == kNoFace) { lamS[s * n + i] = TF(0); continue; }
    const double h = Sh[s], hg = fs >= 0 ? -h : h;
    double x[NV + 1];
    widen<NV + 1>(fl[s], x);
#pragma unroll
    for (int v = 0; v < NV; ++v) R[v] += hg * x[v];
    if constexpr (is_f32<TF>()) lamS[s * n + i] = fl[s][NV];
    else lamS[s * n + i] = fl[s][NV] * h;
    sum += x[NV] * h;
  }
  // sums of S/2 times the values: R / 2 and sum / 2
  const double id = dev::d_rcp(sum * (2.0 * P.icfl_lo + 1.0));
  invD[i] = narrow<TF>(id);
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    // (twice the sum, exactly: one rounding as if the areas were whole)
    double src;
    if (first) { src = fma(-2.0, R[v], Rp0[v * n + i]); Src[v * n + i] = src; }
    else src = Src[v * n + i];
    R[v] = fma(2.0, R[v], src);
    Rk[v * n + i] = narrow<TF>(R[v]);
  }
  if (i < colour0_end) {
    TF b[4], d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) d[v] = narrow<TF>(R[v] * id);
    vload<TF, 4>(base + static_cast<size_t>(i) * kBase, b);
    store_delta(gamma, b, d, delta, i);
  } else {
    TF z[del_run<TF>()];
#pragma unroll
    for (int v = 0; v < del_run<TF>(); ++v) z[v] = TF(0);
    vstore<TF, del_run<TF>()>(delta + static_cast<size_t>(i) * del_run<TF>(), z);
  }
  pdl_exit();
}

// point relaxation of the cells [begin, begin + count) of one colour, Eq.
// (implicit-local), as the 2-D k_sweep: FP64 in the increment form of the
// bracket from the neighbours' base and delta records, 22 FP64 instructions
// per neighbour and 33 per cell (before: about 55 per face slot, one IEEE
// division each); FP32 with the expressions and the order of sums that fix
// its rounding.
// LANES: one thread per cell, or eight (one per face slot, six used) where a
// colour has too few cells to fill the device (sweep_lanes).
// LAST: the cell's last relaxation of the implicit step, from cell adv on (the
// others are relaxed once more), also advances U and writes the next step's
// base record (second buffer).
template <typename T>
struct SlotData {
  static constexpr int NB = is_f32<T>() ? 8 : 5;   // part of a base record a sweep reads
  T b[NB], q[del_run<T>()], ls, nn[3], hS;
};
template <typename T>
__device__ __forceinline__ void slot_load(const MeshT<T> &m, int i, int s, int j, const T *base, const T *lamS,
                                          const T *delta, SlotData<T> &x) {
  const int n = m.nc;
  if constexpr (is_f32<T>()) {
    vload<T, 8>(base + static_cast<size_t>(j) * kBase, x.b);
    x.hS = m.shs[s * n + i];
  } else {
    vload<T, 4>(base + static_cast<size_t>(j) * kBase, x.b);
    x.b[4] = base[static_cast<size_t>(j) * kBase + 4];
  }
  vload<T, del_run<T>()>(delta + static_cast<size_t>(j) * del_run<T>(), x.q);
  x.ls = lamS[s * n + i];
#pragma unroll
  for (int k = 0; k < 3; ++k) x.nn[k] = m.sn[(3 * s + k) * n + i];
}
__device__ __forceinline__ void slot_bracket(float gamma, const SlotData<float> &x, float c[NV]) {
  const float *uj = x.b, *du = x.q;
  // pressure of U_j, the expression of its primitives
  const float pj = (gamma - 1.0f) * (uj[4] - 0.5f * uj[0] * (uj[5] * uj[5] + uj[6] * uj[6] + uj[7] * uj[7]));
  float dF[NV];
  D3::euler_flux_delta(gamma, uj, uj[5], uj[6], uj[7], pj, du, x.nn, dF);
#pragma unroll
  for (int v = 0; v < NV; ++v) c[v] = __fmul_rn(x.hS, dF[v] - x.ls * du[v]);
}
// r minus the slot's bracket
__device__ __forceinline__ void slot_subtract(const SlotData<double> &x, double r[NV]) {
  const double *b = x.b, *q = x.q, *nn = x.nn;
  const double dun = q[5] * nn[0] + q[6] * nn[1] + q[7] * nn[2], dp = q[8];
  const double un1 = dun + b[1] * nn[0] + b[2] * nn[1] + b[3] * nn[2];
  const double w = un1 - x.ls, t = b[0] * dun;
  r[0] = r[0] - q[0] * w - t;
#pragma unroll
  for (int k = 0; k < 3; ++k) r[1 + k] = r[1 + k] - q[1 + k] * w - b[1 + k] * t - dp * nn[k];
  r[4] = r[4] - q[4] * w - dp * un1 - b[4] * dun;
}
constexpr int kSweepLanes = 8;
// FP64: a launch takes as long as the warps of one sub-core (608 of them) issue
// one after another: about 70 instructions for each 4 cells with eight lanes,
// 150 for each 32 with one, so eight are shorter up to two warps a sub-core,
// 4,864 cells.  Event-timed, us per launch, eight / one: colours of 3,960 cells
// 11.7 / 13.3; 15,360 25.0 / 14.6; 25,000 to 51,463 42.6 / 18.8 (before: 41.4).
// FP32 is bound by the latency of its gathers and then by their number: 3,960
// 6.5 / 7.7; 12,779 7.2 / 7.7; 15,360 8.3 / 8.0; 211,181 17.0 / 15.9
// (one thread with the loads of all six slots in flight; less now).
constexpr int kOneLane64 = 4864, kOneLane32 = 14000;
template <typename T> int sweep_lanes(int cnt) { return cnt >= (is_f32<T>() ? kOneLane32 : kOneLane64) ? 1 : kSweepLanes; }
template <typename T, bool LAST, int LANES>
__global__ void __launch_bounds__(kMaxShapeBlock)
    k_sweep(MeshT<T> m, ParamsT<T> P, int begin, int count, int adv, const T *base, const T *Rk, const T *invD,
            const T *lamS, T *delta, double *U, T *base_next) {
  const int n = m.nc;
  constexpr int ND = del_run<T>();
  const int g = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x) / LANES;
  const int i = g < count ? begin + g : -1;
  if constexpr (LANES == 1) {
    // slots whose loads are in flight together: all six took 137 registers in
    // FP32, six warps an SM (V-cycle's sweeps, 512,000 cells mixed: 1412 us with
    // six, 1313 with three, 1273 with two, 1300 with one; FP64, 128,000: 1305
    // with three, 1297 with two)
    constexpr int CH = 2;
    if (i < 0) { pdl_enter(); return; }   // waits too: this grid ends after its predecessor
    // the neighbours (mesh data) before the wait for the predecessor
    int nb[kMaxFace3];
#pragma unroll
    for (int s = 0; s < kMaxFace3; ++s) nb[s] = m.cnbr[s * n + i];
    pdl_enter();
    T r[NV], bi[4] = { T(0), T(0), T(0), T(0) }, d[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) r[v] = Rk[v * n + i];
    if constexpr (!is_f32<T>()) vload<T, 4>(base + static_cast<size_t>(i) * kBase, bi);
    const T iD = invD[i];
    T c[is_f32<T>() ? kMaxFace3 : 1][NV];
#pragma unroll
    for (int s0 = 0; s0 < kMaxFace3; s0 += CH) {
      SlotData<T> x[CH];
#pragma unroll
      for (int s = 0; s < CH; ++s)
        if (nb[s0 + s] >= 0) slot_load(m, i, s0 + s, nb[s0 + s], base, lamS, delta, x[s]);
#pragma unroll
      for (int s = 0; s < CH; ++s) {
        if constexpr (is_f32<T>()) {
#pragma unroll
          for (int v = 0; v < NV; ++v) c[s0 + s][v] = T(0);
          if (nb[s0 + s] >= 0) slot_bracket(P.gamma, x[s], c[s0 + s]);
        } else {
          if (nb[s0 + s] >= 0) slot_subtract(x[s], r);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if constexpr (is_f32<T>()) {
        const T lo = __fadd_rn(__fadd_rn(c[0][v], c[1][v]), __fadd_rn(c[2][v], c[3][v]));
        d[v] = (r[v] - __fadd_rn(lo, __fadd_rn(c[4][v], c[5][v]))) * iD;
      } else {
        d[v] = r[v] * iD;
      }
    }
    store_delta(P.gamma, bi, d, delta, i);
    if (LAST && i >= adv) {
      double u[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        u[v] = U[v * n + i] + static_cast<double>(d[v]);
        U[v * n + i] = u[v];
      }
      store_base(P, u, base_next, i);
    }
  } else {
    const int s = threadIdx.x & (LANES - 1);
    const int j = (i >= 0 && s < kMaxFace3) ? m.cnbr[s * n + i] : -1;
    pdl_enter();
    T bi[4] = { T(0), T(0), T(0), T(0) }, r = T(0), iD = T(0);
    double us = 0.0;
    if (i >= 0 && s < NV) {
      r = Rk[s * n + i];
      iD = invD[i];
      if (LAST) us = U[s * n + i];
    }
    if constexpr (!is_f32<T>())
      if (i >= 0) vload<T, 4>(base + static_cast<size_t>(i) * kBase, bi);
    T c[NV] = { T(0), T(0), T(0), T(0), T(0) };
    if (j >= 0) {
      SlotData<T> x;
      slot_load(m, i, s, j, base, lamS, delta, x);
      if constexpr (is_f32<T>()) slot_bracket(P.gamma, x, c);
      else slot_subtract(x, c);   // minus the bracket
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      c[v] += __shfl_xor_sync(0xffffffffu, c[v], 1);
      c[v] += __shfl_xor_sync(0xffffffffu, c[v], 2);
      c[v] += __shfl_xor_sync(0xffffffffu, c[v], 4);
    }
    const T mine = s == 0 ? c[0] : s == 1 ? c[1] : s == 2 ? c[2] : s == 3 ? c[3] : c[4];
    const T ds = (is_f32<T>() ? r - mine : r + mine) * iD;
    if constexpr (is_f32<T>()) {
      if (i >= 0) delta[static_cast<size_t>(i) * ND + s] = s < NV ? ds : T(0);
    } else {
      T d[NV], rec[ND];
#pragma unroll
      for (int v = 0; v < NV; ++v) d[v] = __shfl_sync(0xffffffffu, ds, v, LANES);
      delta_record(P.gamma, bi, d, rec);
#pragma unroll
      for (int v = 0; v < ND / 2; ++v)
        if (i >= 0 && s == v) {
          const T two[2] = { rec[2 * v], rec[2 * v + 1] };
          vstore<T, 2>(delta + static_cast<size_t>(i) * ND + 2 * v, two);
        }
    }
    if constexpr (LAST) {
      us += static_cast<double>(ds);
      if (i >= adv && s < NV) U[s * n + i] = us;
      double u[NV];
#pragma unroll
      for (int v = 0; v < NV; ++v) u[v] = __shfl_sync(0xffffffffu, us, v, LANES);
      T rec[kBase];
      base_record(P, u, rec);
#pragma unroll
      for (int v = 0; v < LANES; ++v)
        if (i >= adv && s == v) {
          const T two[2] = { rec[2 * v], rec[2 * v + 1] };
          T *o = base_next + static_cast<size_t>(i) * kBase + 2 * v;
          o[0] = two[0];
          o[1] = two[1];
        }
    }
  }
  pdl_exit();
}

// W = W_p0 + (U - W_p0), density residual partials, state check
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_prolong(MeshT<double> m, ParamsT<double> P, double *W,
                                                        const double *Wp0, const double *U,
                                                        int *status, double *partial,
                                                        TF *Wm) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = m.nc;
  double num = 0.0, den = 0.0;
  if (i < n) {
    double w[NV];
    const double old = W[i];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double wp = Wp0[v * n + i];
      w[v] = wp + (U[v * n + i] - wp);
      W[v * n + i] = w[v];
      if (Wm) Wm[v * n + i] = narrow<TF>(w[v]);
    }
    if (!state_ok(w)) atomicOr(status, kBadState);
    num = fabs(w[0] - old);
    den = old;
  }
  block_sum2(num, den, &partial[2 * blockIdx.x]);
  pdl_exit();
}

// caller AoS <-> internal SoA
__global__ void k_gather_state(int n, const int *__restrict__ perm, const double *__restrict__ Wa,
                               const double *__restrict__ Wxa, double *__restrict__ W, double *__restrict__ Wx,
                               float *__restrict__ W32, float *__restrict__ Wx32) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = perm[i];
  for (int v = 0; v < NV; ++v) {
    const double w = Wa[NV * c + v];
    W[v * n + i] = w;
    if (W32) W32[v * n + i] = static_cast<float>(w);
  }
  for (int q = 0; q < 3 * NV; ++q) {
    const double g = Wxa ? Wxa[3 * NV * c + q] : 0.0;
    Wx[q * n + i] = g;
    if (Wx32) Wx32[q * n + i] = static_cast<float>(g);
  }
}
__global__ void k_scatter_state(int n, const int *__restrict__ perm, const double *__restrict__ W,
                                const double *__restrict__ Wx, double *__restrict__ Wa, double *__restrict__ Wxa) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = perm[i];
  if (Wa) for (int v = 0; v < NV; ++v) Wa[NV * c + v] = W[v * n + i];
  if (Wxa) for (int q = 0; q < 3 * NV; ++q) Wxa[3 * NV * c + q] = Wx[q * n + i];
}

}  // namespace kern3
}  // namespace cgks
