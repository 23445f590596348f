// Kernels of the batched hot path (included by cgks_device.cu only).
//
// Index space: a batch holds one or more solves in slots.  Each solve owns
// a contiguous range of cells (padded to a multiple of kCellBlock with
// inert cells, csid = -1) and a contiguous range of faces; space no solve
// holds is inert too (csid / fsid = -1).  Within a solve, cells are
// colour-major with reverse Cuthill-McKee order inside a colour.  Boundary
// faces store -1 - (16 * slot + tag) in fc1, so one table holds every
// solve's boundary conditions.  Per-solve values (viscosity, time step,
// status, residual) are indexed by the slot.  Arrays are strided by the
// batch capacity (m.nc cells, m.nf faces).
//
// Precision: kernels that evaluate fluxes are templated on the flux type
// TF.  FP64 mode runs everything in double.  Mixed mode keeps the
// conservative variables (W, W_x, U) and every accumulation into them, the
// residuals and the diagonal inversion in double, and runs reconstruction,
// face fluxes and relaxation sweeps in float on float mirrors of the state.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "cgks_internal.h"
#include "cgks_physics.cuh"
#include "cgks_pdl.cuh"
#include "cgks_shapes.h"
#include "cgks_vec.cuh"

namespace cgks {
namespace kern {

namespace D = cgks::dev;

// Threads of the kernels with one thread per cell, the unit of a solve's padding
// and of the residual's partial sums.  Bound by the FP64 pipe or by latency,
// they want their warps spread over the SMs: with 64 instead of 256 a V-cycle
// takes, event-timed, 600 instead of 619 us (57,344 cells mixed), 592 / 603
// (2,048 FP64); six served solves 0.36 / 0.42 ms.
constexpr int kCellBlock = 64;
constexpr int kTagsPerSolve = CGKS_MAX_BC;
constexpr int kBadState = 1;   // bit of a solve's status word
constexpr int kFO = 16;        // face outputs of the high level: F0, F1, Wc, Wt

template <typename T>
__host__ __device__ constexpr bool is_f32() { return std::is_same<T, float>::value; }

// Shared model constants and pointers to per-solve / per-tag tables.
template <typename T>
struct ParamsT {
  T gamma, K, cfl_hi, icfl_lo;   // icfl_lo = 1 / CFL of the low-order level
  D::KC<T> kc;
  const T *mu;                   // [S] dynamic viscosity per solve
  const int *bc_kind;            // [16 S] boundary kind per global tag
  const T *bc_uw;                // [16 S][2] wall velocity
  const T *bc_rho, *bc_u, *bc_p; // [16 S], [16 S][2], [16 S] far-field free stream
  int flux_lo;                   // low-level flux: CGKS_FLUX_KFVS or CGKS_FLUX_LF
  int flux_hi;                   // high-level flux: CGKS_FLUX_SMOOTH or CGKS_FLUX_FULL
  T tau_c1, tau_c2;              // numerical collision time constants of the full flux
  T weno_eps, weno_g0;           // compact WENO epsilon (0: linear weights), linear weight of P2
  int weno_vars;                 // CGKS_WENO_CONSERVATIVE (per cell) or CGKS_WENO_CHARACTERISTIC (per face side)
  // [S] per solve: 1 = limited (full flux + compact WENO), 0 = smooth flux,
  // linear weights; null when every solve of the batch takes the batch-wide
  // flux.  With it each instantiation of k_recon / k_face treats only the
  // solves of its own class.
  const int *slim;
  int lo_viscous;                // 1: the low-order residual carries a first-order viscous flux
};

template <typename T>
struct MeshT {
  int nc, nf;                                // padded cells, faces
  const T *vol, *ivol, *per, *ih, *m2;       // ih = 1/h; m2: [3][nc]
  const T *op;                               // [kNCol*kNM][nc]
  const T *fn, *fS, *fjump, *fxi;            // fn [2][nf], fjump = alpha/delta, fxi [8][nf]
  const T *fidl;                             // 1/delta: the centre distance along n (boundary: twice to the face)
  const T *snx, *sny, *shs;                  // [4][nc] per face slot: outward normal of the cell (FP64: times S/2), S/2 (FP64: S)
  const int *cface, *cnbr;                   // [4][nc]
  const int *fc0, *fc1;
  const int *csid, *fsid;                    // solve of each cell (-1: padding) and face
  const unsigned char *ccol;                 // colour of each cell (255: padding)
  const unsigned char *wenok;                // 1: least-squares quadratic (WENO may limit it)
};

// per-batch control words on the device
struct Ctl {
  double dt_fixed;   // > 0: prescribed step for every solve
  int res_ctr;       // next slot of solve 0's residual history
  int pad_;
};

__device__ __forceinline__ double dt_of(const Ctl *ctl, const unsigned long long *dt_bits, int sid, double cfl) {
  if (ctl->dt_fixed > 0.0) return ctl->dt_fixed;
  return cfl * __longlong_as_double(static_cast<long long>(dt_bits[sid]));
}

// positive and finite, by the bits (a comparison takes the FP64 pipe)
__device__ __forceinline__ bool positive_finite(double x) {
  const unsigned hi = static_cast<unsigned>(__double2hiint(x));
  return hi < 0x7ff00000u && (hi | static_cast<unsigned>(__double2loint(x))) != 0u;
}
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
// density and pressure positive, everything finite; rho p / (gamma - 1) has
// the sign of p and needs no division
__device__ __forceinline__ bool state_ok(const double w[4]) {
  const double q = w[3] * w[0] - 0.5 * (w[1] * w[1] + w[2] * w[2]);
  return positive_finite(w[0]) && positive_finite(q) && finite_bits(w[1]) && finite_bits(w[2]) && finite_bits(w[3]);
}

// Block reduction of two doubles in a fixed order; thread 0 writes them.
__device__ __forceinline__ void block_sum2(double a, double b, double *out2) {
  __shared__ double sa[32], sb[32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) { sa[warp] = a; sb[warp] = b; }
  __syncthreads();
  if (warp == 0) {
    int nw = blockDim.x >> 5;
    a = lane < nw ? sa[lane] : 0.0;
    b = lane < nw ? sb[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { out2[0] = a; out2[1] = b; }
  }
}

// ------------------------------------------------------------------
// K0: reset the per-solve time steps
__global__ void k_reset_dt(Ctl *ctl, unsigned long long *dt_bits, int S, double dt_fixed) {
  pdl_enter();
  for (int s = threadIdx.x; s < S; s += blockDim.x) dt_bits[s] = 0x7ff0000000000000ull;  // +inf
  if (threadIdx.x == 0) ctl->dt_fixed = dt_fixed;
  pdl_exit();
}

// K4: local explicit step per cell, per-solve min by atomicMin on the bits
// (min is order independent).  h = 2|Omega|/perimeter, speed |U| + c + 2 nu / h.
// Solves are padded to whole blocks, so a block never spans two solves and
// its first cell is a real one: one atomic per block.  Bound by the FP64 pipe:
// with the library's division and square root and minima of doubles it took
// 28.3 us with the reset launch on 57,344 cells, now 17.7.
__global__ void __launch_bounds__(kCellBlock) k_dt(MeshT<double> m, ParamsT<double> P, const double *W,
                                                   unsigned long long *dt_bits) {
  pdl_enter();
  // the minimum on the bits, positive doubles sort like integers (a NaN sorts
  // last): comparisons of doubles take the FP64 pipe
  __shared__ unsigned long long wmin[kCellBlock / 32];
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  double d = INFINITY;
  int sid = i < m.nc ? m.csid[i] : -1;
  if (sid >= 0) {
    int n = m.nc;
    const double rho = W[i], ir = D::d_rcp(rho);
    const double u = W[n + i] * ir, v = W[2 * n + i] * ir, q2 = u * u + v * v;
    const double p = (P.gamma - 1.0) * (W[3 * n + i] - 0.5 * rho * q2);
    const double speed = D::sqrt_fast(q2) + D::sqrt_fast(P.gamma * p * ir) + P.mu[sid] * ir * (m.per[i] * m.ivol[i]);
    d = 2.0 * m.vol[i] * D::d_rcp(m.per[i] * speed);
  }
  unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
  for (int o = 16; o > 0; o >>= 1) b = min(b, __shfl_down_sync(0xffffffffu, b, o));
  if ((threadIdx.x & 31) == 0) wmin[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kCellBlock / 32; ++w) b = min(b, wmin[w]);
    constexpr unsigned long long kInf = 0x7ff0000000000000ull;
    const int s0 = blockIdx.x * blockDim.x < m.nc ? m.csid[blockIdx.x * blockDim.x] : -1;
    if (s0 >= 0 && b < kInf) atomicMin(&dt_bits[s0], b);
  }
  pdl_exit();
}

// FP32: wall ghost of a state and its gradient (global frame), through the face frame.
template <typename T>
__device__ __forceinline__ void wall_ghost_global(const ParamsT<T> &P, int tag, T nx, T ny, const T w[4],
                                                  const T gx[4], const T gy[4], T wg[4], T ggx[4], T ggy[4]) {
  T wl[4], dn[4], dt[4], tn[4], tt[4];
  D::rot_in(nx, ny, w, wl);
  for (int v = 0; v < 4; ++v) { tn[v] = nx * gx[v] + ny * gy[v]; tt[v] = -ny * gx[v] + nx * gy[v]; }
  D::rot_in(nx, ny, tn, dn);
  D::rot_in(nx, ny, tt, dt);
  T wgl[4], dng[4], dtg[4];
  if (P.bc_kind[tag] == CGKS_BC_SLIP) {
    D::ghost_slip(wl, dn, dt, wgl, dng, dtg);
  } else {
    T wn = P.bc_uw[2 * tag] * nx + P.bc_uw[2 * tag + 1] * ny;
    T wt = -P.bc_uw[2 * tag] * ny + P.bc_uw[2 * tag + 1] * nx;
    D::ghost_noslip(P.gamma, wn, wt, wl, dn, dt, wgl, dng, dtg);
  }
  T gn[4], gt[4];
  D::rot_out(nx, ny, wgl, wg);
  D::rot_out(nx, ny, dng, gn);
  D::rot_out(nx, ny, dtg, gt);
  for (int v = 0; v < 4; ++v) { ggx[v] = nx * gn[v] - ny * gt[v]; ggy[v] = ny * gn[v] + nx * gt[v]; }
}

template <typename T>
__device__ __forceinline__ void farfield_ghost(const ParamsT<T> &P, int tag, T nx, T ny, const T wl[4], T wg[4]) {
  T une = D::dot2(P.bc_u[2 * tag], nx, P.bc_u[2 * tag + 1], ny);
  T ute = D::dot2(-P.bc_u[2 * tag], ny, P.bc_u[2 * tag + 1], nx);
  D::ghost_farfield(P.kc, P.gamma, P.bc_rho[tag], une, ute, P.bc_p[tag], wl, wg);
}

// prescribed state of a Dirichlet boundary in the face frame
template <typename T>
__device__ __forceinline__ void dirichlet_ghost(const ParamsT<T> &P, int tag, T nx, T ny, T wg[4]) {
  const T r = P.bc_rho[tag], p = P.bc_p[tag];
  const T un = D::dot2(P.bc_u[2 * tag], nx, P.bc_u[2 * tag + 1], ny);
  const T ut = D::dot2(-P.bc_u[2 * tag], ny, P.bc_u[2 * tag + 1], nx);
  wg[0] = r; wg[1] = r * un; wg[2] = r * ut;
  wg[3] = D::mad(T(0.5) * r, D::dot2(un, un, ut, ut), p / (P.gamma - T(1)));
}

__host__ __device__ __forceinline__ bool is_wall_kind(int k) { return k == CGKS_BC_SLIP || k == CGKS_BC_NOSLIP; }

// Compact WENO with nonlinear weights (Section 4, transonic and supersonic
// cases; the scheme is the cited one, read as follows).  Candidates: the
// compact quadratic P2 (scaled coefficients c[q][v]) and the m linear
// polynomials W_i + h g.(xi, eta), g the cell-mean gradient of the cell
// itself and of each face neighbour (h g given in lin[k][0..1][v]).
// Smoothness: the cell mean of (h D P)^2 over first and second derivative
// multi-indices; with the centroid at the origin and the cell's second
// moments M = (xi^2, xi eta, eta^2) means m2 this is, for
// P_xi = c0 + 2 c2 xi + c3 eta, P_eta = c1 + c3 xi + 2 c4 eta,
//   c0^2 + c1^2 + (4 c2^2 + c3^2) M_xx + (c3^2 + 4 c4^2) M_yy
//   + (4 c2 c3 + 4 c3 c4) M_xy + 4 c2^2 + c3^2 + 4 c4^2.
// Weights w_k ~ gamma_k / (beta_k + eps)^2 (gamma_0 = g0, the rest
// (1 - g0) / m); result (w_0/gamma_0)(P2 - sum gamma_k P1_k) + sum w_k P1_k.
// Candidate 0 is the cell's own; candidate 1 + s, of face slot s, counts where
// bit 1 + s of on is set (slots by a constant index: no local memory).
__device__ __forceinline__ float quot(float a, float b) { return a / b; }
__device__ __forceinline__ double quot(double a, double b) { return a * D::d_rcp(b); }
template <typename T, int NC>
__device__ __forceinline__ void weno_combine(const ParamsT<T> &P, T mxx, T mxy, T myy, unsigned on,
                                             const T (&lin)[5][2][NC], T (&c)[kNM][NC]) {
  const int nk = __popc(on);
  const T g0 = P.weno_g0, eps = P.weno_eps;
  const T gk = quot(T(1) - g0, T(nk));
#pragma unroll
  for (int v = 0; v < NC; ++v) {
    const T c0 = c[0][v], c1 = c[1][v], c2 = c[2][v], c3 = c[3][v], c4 = c[4][v];
    const T b0 = c0 * c0 + c1 * c1 + (T(4) * c2 * c2 + c3 * c3) * mxx + (c3 * c3 + T(4) * c4 * c4) * myy +
                 (T(4) * c2 * c3 + T(4) * c3 * c4) * mxy + T(4) * c2 * c2 + c3 * c3 + T(4) * c4 * c4;
    T w0 = quot(g0, (b0 + eps) * (b0 + eps));
    T wk[5], ws = w0;
    T lin0 = T(0), lin1 = T(0);
#pragma unroll
    for (int k = 0; k < 5; ++k) {
      if (on >> k & 1) {
        const T a0 = lin[k][0][v], a1 = lin[k][1][v];
        const T b = a0 * a0 + a1 * a1;
        wk[k] = quot(gk, (b + eps) * (b + eps));
        ws += wk[k];
        lin0 += gk * a0;
        lin1 += gk * a1;
      }
    }
    const T iws = quot(T(1), ws);
    const T f0 = quot(w0 * iws, g0);
    T sel0 = T(0), sel1 = T(0);
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (on >> k & 1) {
        const T w = is_f32<T>() ? wk[k] * iws : wk[k];
        sel0 += w * lin[k][0][v];
        sel1 += w * lin[k][1][v];
      }
    if constexpr (!is_f32<T>()) { sel0 *= iws; sel1 *= iws; }
    c[0][v] = f0 * (c0 - lin0) + sel0;
    c[1][v] = f0 * (c1 - lin1) + sel1;
    c[2][v] = f0 * c2;
    c[3][v] = f0 * c3;
    c[4][v] = f0 * c4;
  }
}

// K1: compact least-squares quadratic of every cell.
//   coef[(q*4 + v)*nc + i], q over (xi, eta, xi^2, xi eta, eta^2).
// NC: conserved variables per thread.  FP64: one, the warps of a block on the
// same 32 cells each taking another, because an FP64 launch takes as long as
// the warps of one sub-core (608 of them) issue one after another, and one
// thread per cell left most sub-cores idle below 20,000 cells; the operator
// is then read from the cache by three of the four.  FP32: all four, the reads
// of the operator bound it.  us per launch, FP64, before / now (with the wall
// mirrors as linear maps): 128 cells 32.8 / 15.3, 2,048 31.1 / 14.4, 6,354 with
// nonlinear weights 38.2 / 20.7, 57,344 46.9 / 45.8.
template <typename T> __host__ __device__ constexpr int recon_vars() { return is_f32<T>() ? 4 : 1; }
// threads of a launch over n cells with a warp per variable of 32 cells
template <int VARS> __host__ __device__ constexpr int64_t var_items(int64_t n) { return (n + 31) / 32 * 32 * VARS; }
template <typename T, bool WENO, int NC>
__device__ __forceinline__ void recon_at(const MeshT<T> &m, const ParamsT<T> &P, const T *W,
                                         const T *Wx, T *__restrict__ coef, const int i,
                                         const int comp) {
  const int n = m.nc, vo = NC == 4 ? 0 : comp;
  T wi[NC], gxi[NC], gyi[NC];
#pragma unroll
  for (int v = 0; v < NC; ++v) {
    wi[v] = W[(vo + v) * n + i];
    gxi[v] = Wx[(vo + v) * n + i];
    gyi[v] = Wx[(4 + vo + v) * n + i];
  }
  T c[kNM][NC];
#pragma unroll
  for (int q = 0; q < kNM; ++q) {
    T o0 = m.op[((kNCol - 2) * kNM + q) * n + i], o1 = m.op[((kNCol - 1) * kNM + q) * n + i];
#pragma unroll
    for (int v = 0; v < NC; ++v) c[q][v] = o0 * gxi[v] + o1 * gyi[v];
  }
  // linear WENO candidates: h times the cell-mean gradients of the cell and its face neighbours
  T lin[WENO ? 5 : 1][2][NC];
  unsigned on = 1;
  if constexpr (WENO) {
    const T hi = quot(T(1), m.ih[i]);
#pragma unroll
    for (int v = 0; v < NC; ++v) { lin[0][0][v] = hi * gxi[v]; lin[0][1][v] = hi * gyi[v]; }
  }
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
    int fs = m.cface[s * n + i];
    if (fs == kNoFace) continue;
    int j = m.cnbr[s * n + i];
    T b0[NC], b1[NC], b2[NC];
    if (j >= 0) {
#pragma unroll
      for (int v = 0; v < NC; ++v) {
        b0[v] = W[(vo + v) * n + j] - wi[v];
        b1[v] = Wx[(vo + v) * n + j];
        b2[v] = Wx[(4 + vo + v) * n + j];
      }
      if constexpr (WENO) {
        const T hi = quot(T(1), m.ih[i]);
#pragma unroll
        for (int v = 0; v < NC; ++v) { lin[1 + s][0][v] = hi * b1[v]; lin[1 + s][1][v] = hi * b2[v]; }
        on |= 2u << s;
      }
    } else {
      int f = fs >= 0 ? fs : ~fs;
      int tag = -1 - m.fc1[f];
      if (!is_wall_kind(P.bc_kind[tag])) continue;
      if constexpr (NC == 4) {
        T wg[4];
        wall_ghost_global(P, tag, m.fn[f], m.fn[m.nf + f], wi, gxi, gyi, wg, b1, b2);
#pragma unroll
        for (int v = 0; v < 4; ++v) b0[v] = wg[v] - wi[v];
      } else {   // the mirror image mixes the variables
        const double nn[2] = { m.fn[f], m.fn[m.nf + f] };
        double b[2];
        D::WallMap<2>(P.bc_kind[tag], P.bc_uw + 2 * tag, nn).one(comp, W + i, Wx + i, n, b0[0], b);
        b1[0] = b[0];
        b2[0] = b[1];
      }
    }
#pragma unroll
    for (int q = 0; q < kNM; ++q) {
      T o0 = m.op[((3 * s) * kNM + q) * n + i];
      T o1 = m.op[((3 * s + 1) * kNM + q) * n + i];
      T o2 = m.op[((3 * s + 2) * kNM + q) * n + i];
#pragma unroll
      for (int v = 0; v < NC; ++v) c[q][v] += o0 * b0[v] + o1 * b1[v] + o2 * b2[v];
    }
  }
  // cells whose stencil fell back to the linear polynomial of their own
  // gradient (too few neighbours, rank deficiency) carry no quadratic terms
  // in the operator and keep it; the others may be limited
  if constexpr (WENO)
    if (m.wenok[i]) weno_combine(P, m.m2[i], m.m2[n + i], m.m2[2 * n + i], on, lin, c);
#pragma unroll
  for (int q = 0; q < kNM; ++q)
#pragma unroll
    for (int v = 0; v < NC; ++v) coef[(q * 4 + vo + v) * n + i] = c[q][v];
}
template <typename T, bool WENO>
__global__ void __launch_bounds__(kMaxShapeBlock) k_recon(MeshT<T> m, ParamsT<T> P,
                                                                        const T *W,
                                                                        const T *Wx,
                                                                        T *coef) {
  pdl_enter();
  constexpr int NC = recon_vars<T>(), G = 4 / NC;   // threads per cell
  for_items(static_cast<int>(var_items<G>(m.nc)), [&](int t) {
    const int i = G == 1 ? t : t / (32 * G) * 32 + t % 32, comp = t / 32 % G;
    if (i >= m.nc) return;
    if (P.slim) {
      const int sid = m.csid[i];
      if (sid >= 0 && (P.slim[sid] != 0) != WENO) return;
    }
    recon_at<T, WENO, NC>(m, P, W, Wx, coef, i, comp);
  });
  pdl_exit();
}

// value and gradient of the quadratic of cell i at scaled offset (x, y)
template <typename T>
__device__ __forceinline__ void recon_point(const MeshT<T> &m, const T *W, const T *coef,
                                            int i, T x, T y, T val[4], T gx[4], T gy[4]) {
  const int n = m.nc;
  T ih = m.ih[i];
  T p2 = x * x - m.m2[i], p3 = x * y - m.m2[n + i], p4 = y * y - m.m2[2 * n + i];
  for (int v = 0; v < 4; ++v) {
    T c0 = coef[(0 * 4 + v) * n + i], c1 = coef[(1 * 4 + v) * n + i], c2 = coef[(2 * 4 + v) * n + i];
    T c3 = coef[(3 * 4 + v) * n + i], c4 = coef[(4 * 4 + v) * n + i];
    val[v] = W[v * n + i] + c0 * x + c1 * y + c2 * p2 + c3 * p3 + c4 * p4;
    gx[v] = (c0 + T(2) * c2 * x + c3 * y) * ih;
    gy[v] = (c1 + c3 * x + T(2) * c4 * y) * ih;
  }
}

// value and gradient at scaled offset (x, y) of a polynomial of cell i with
// the given coefficients c[q][v]
template <typename T>
__device__ __forceinline__ void poly_point(const MeshT<T> &m, const T *W, const T c[kNM][4], int i, T x,
                                           T y, T val[4], T gx[4], T gy[4]) {
  const int n = m.nc;
  T ih = m.ih[i];
  T p2 = x * x - m.m2[i], p3 = x * y - m.m2[n + i], p4 = y * y - m.m2[2 * n + i];
  for (int v = 0; v < 4; ++v) {
    val[v] = W[v * n + i] + c[0][v] * x + c[1][v] * y + c[2][v] * p2 + c[3][v] * p3 + c[4][v] * p4;
    gx[v] = (c[0][v] + T(2) * c[2][v] * x + c[3][v] * y) * ih;
    gy[v] = (c[1][v] + c[3][v] * x + T(2) * c[4][v] * y) * ih;
  }
}

// the same from given coefficients, the gradient left in the cell's scaled
// coordinates (to be multiplied by 1/h)
__device__ __forceinline__ void side_scaled(const MeshT<double> &m, const double *W,
                                            const double c[kNM][4], int i, double x, double y, double val[4],
                                            double gx[4], double gy[4]) {
  const int n = m.nc;
  const double p2 = x * x - m.m2[i], p3 = x * y - m.m2[n + i], p4 = y * y - m.m2[2 * n + i];
  const double x2 = x + x, y2 = y + y;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    val[v] = W[v * n + i] + c[0][v] * x + c[1][v] * y + c[2][v] * p2 + c[3][v] * p3 + c[4][v] * p4;
    gx[v] = c[0][v] + c[2][v] * x2 + c[3][v] * y;
    gy[v] = c[1][v] + c[3][v] * x + c[4][v] * y2;
  }
}
__device__ __forceinline__ void load_coef(int n, const double *coef, int i, double c[kNM][4]) {
#pragma unroll
  for (int q = 0; q < kNM; ++q)
#pragma unroll
    for (int v = 0; v < 4; ++v) c[q][v] = coef[(q * 4 + v) * n + i];
}

// Compact WENO on characteristic variables (Section 4, shock reflection),
// for the side of a face held by cell i: the candidates of cell i (its
// linear-weight quadratic from coef, h times the mean gradients of the cell
// and its face neighbours) are projected on the left eigenvectors of the
// Euler flux Jacobian along the face normal n at the state wref (the mean
// of the two cell averages; the cell's own on a boundary face), combined by
// weno_combine per characteristic field and projected back.  Right
// eigenvectors (columns): u_n - c, entropy, shear, u_n + c; the left ones
// in closed form with b1 = (gamma - 1)/c^2, b2 = b1 |u|^2 / 2.
// The fields of a conservative vector and back, FP64: the eigenvectors' products
// with what they share taken once (12 and 13 instructions, as matrices 16), no
// division: face flux of a 3,600-cell shock reflection 84.5 -> 80.0 us.
struct CharFrame {
  double u, v, q2h, H, c, un, ut, nx, ny;              // q2h = |u|^2 / 2
  double b1, b1u, b1v, b2, cn, cnx, cny;               // of the left ones; cn = un / (2 c), ...
  __device__ __forceinline__ CharFrame(double gamma, const double w[4], double nx_, double ny_) : nx(nx_), ny(ny_) {
    const double ir = D::d_rcp(w[0]);
    u = w[1] * ir;
    v = w[2] * ir;
    const double q2 = u * u + v * v, p = (gamma - 1.0) * (w[3] - 0.5 * w[0] * q2), c2 = gamma * p * ir;
    const double ic = D::d_rsqrt3(c2);
    c = c2 * ic;
    q2h = 0.5 * q2;
    H = (w[3] + p) * ir;
    un = u * nx + v * ny;
    ut = v * nx - u * ny;
    b1 = (gamma - 1.0) * ic * ic;
    b1u = b1 * u;
    b1v = b1 * v;
    b2 = b1 * q2h;
    const double h = 0.5 * ic;
    cn = un * h;
    cnx = nx * h;
    cny = ny * h;
  }
  // the left eigenvectors times s
  __device__ __forceinline__ CharFrame scaled(double s) const {
    CharFrame f(*this);
    f.b1 *= s; f.b1u *= s; f.b1v *= s; f.b2 *= s; f.cn *= s; f.cnx *= s; f.cny *= s;
    f.ut *= s; f.nx *= s; f.ny *= s;
    return f;
  }
  __device__ __forceinline__ void fields(double one, const double x[4], double a[4]) const {
    const double s = b2 * x[0] - b1u * x[1] - b1v * x[2] + b1 * x[3];
    const double d = cnx * x[1] + cny * x[2] - cn * x[0];
    a[0] = 0.5 * s - d;
    a[1] = one * x[0] - s;
    a[2] = nx * x[2] - ny * x[1] - ut * x[0];
    a[3] = 0.5 * s + d;
  }
  __device__ __forceinline__ void conservative(const double a[4], double x[4]) const {
    const double s = a[0] + a[3], d = c * (a[3] - a[0]);
    x[0] = s + a[1];
    x[1] = u * x[0] + nx * d - ny * a[2];
    x[2] = v * x[0] + ny * d + nx * a[2];
    x[3] = H * s + q2h * a[1] + un * d + ut * a[2];
  }
};
__device__ __forceinline__ void char_side(const MeshT<double> &m, const ParamsT<double> &P, const double *W,
                                          const double *Wx, const double *coef, int i, const double wref[4],
                                          double nx, double ny, double out[kNM][4]) {
  const int n = m.nc;
  const CharFrame f(P.gamma, wref, nx, ny);
  const double h = quot(1.0, m.ih[i]);
  double lin[5][2][4];
  unsigned on = 1;
  {
    const CharFrame g = f.scaled(h);
    auto add = [&](int k, int j) {
      double x[4], a[4];
#pragma unroll
      for (int d = 0; d < 2; ++d) {
#pragma unroll
        for (int b = 0; b < 4; ++b) x[b] = Wx[(4 * d + b) * n + j];
        g.fields(h, x, a);
#pragma unroll
        for (int b = 0; b < 4; ++b) lin[k][d][b] = a[b];
      }
    };
    add(0, i);
#pragma unroll
    for (int s = 0; s < kMaxFace; ++s) {
      const int j = m.cnbr[s * n + i];
      if (m.cface[s * n + i] != kNoFace && j >= 0) {
        add(1 + s, j);
        on |= 2u << s;
      }
    }
  }
  double cq[kNM][4];
#pragma unroll
  for (int q = 0; q < kNM; ++q) {
    double x[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) x[b] = coef[(q * 4 + b) * n + i];
    f.fields(1.0, x, cq[q]);
  }
  weno_combine(P, m.m2[i], m.m2[n + i], m.m2[2 * n + i], on, lin, cq);
#pragma unroll
  for (int q = 0; q < kNM; ++q) f.conservative(cq[q], out[q]);
}
template <typename T>
__device__ void char_side(const MeshT<T> &m, const ParamsT<T> &P, const T *W, const T *Wx,
                          const T *coef, int i, const T wref[4], T nx, T ny, T out[kNM][4]) {
  const int n = m.nc;
  const T g = P.gamma;
  const T ir = T(1) / wref[0];
  const T u = wref[1] * ir, v = wref[2] * ir;
  const T q2 = u * u + v * v;
  const T p = (g - T(1)) * (wref[3] - T(0.5) * wref[0] * q2);
  const T c = D::d_sqrt(g * p * ir), ic = T(1) / c;
  const T H = (wref[3] + p) * ir;
  const T un = u * nx + v * ny, ut = -u * ny + v * nx;
  const T b1 = (g - T(1)) * ic * ic, b2 = T(0.5) * b1 * q2;
  const T R[4][4] = { { T(1), T(1), T(0), T(1) },
                      { u - c * nx, u, -ny, u + c * nx },
                      { v - c * ny, v, nx, v + c * ny },
                      { H - c * un, T(0.5) * q2, ut, H + c * un } };
  const T L[4][4] = { { T(0.5) * (b2 + un * ic), T(0.5) * (-b1 * u - nx * ic), T(0.5) * (-b1 * v - ny * ic),
                        T(0.5) * b1 },
                      { T(1) - b2, b1 * u, b1 * v, -b1 },
                      { -ut, -ny, nx, T(0) },
                      { T(0.5) * (b2 - un * ic), T(0.5) * (-b1 * u + nx * ic), T(0.5) * (-b1 * v + ny * ic),
                        T(0.5) * b1 } };
  const T h = T(1) / m.ih[i];
  T lin[5][2][4];
  unsigned on = 1;
  auto add = [&](int k, int j) {
    T gx[4], gy[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) { gx[a] = Wx[a * n + j]; gy[a] = Wx[(4 + a) * n + j]; }
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      T sx = T(0), sy = T(0);
#pragma unroll
      for (int b = 0; b < 4; ++b) { sx += L[a][b] * gx[b]; sy += L[a][b] * gy[b]; }
      lin[k][0][a] = h * sx;
      lin[k][1][a] = h * sy;
    }
  };
  add(0, i);
#pragma unroll
  for (int sl = 0; sl < kMaxFace; ++sl) {
    const int j = m.cnbr[sl * n + i];
    if (m.cface[sl * n + i] != kNoFace && j >= 0) {
      add(1 + sl, j);
      on |= 2u << sl;
    }
  }
  T cq[kNM][4];
  for (int q = 0; q < kNM; ++q) {
    T cv[4];
    for (int b = 0; b < 4; ++b) cv[b] = coef[(q * 4 + b) * n + i];
    for (int a = 0; a < 4; ++a) {
      T acc = T(0);
      for (int b = 0; b < 4; ++b) acc += L[a][b] * cv[b];
      cq[q][a] = acc;
    }
  }
  weno_combine(P, m.m2[i], m.m2[n + i], m.m2[2 * n + i], on, lin, cq);
  for (int q = 0; q < kNM; ++q)
    for (int b = 0; b < 4; ++b) {
      T acc = T(0);
      for (int a = 0; a < 4; ++a) acc += R[b][a] * cq[q][a];
      out[q][b] = acc;
    }
}

// ghost of a cell-mean state (zero gradients)
template <typename T>
__device__ __forceinline__ void lo_ghost(const ParamsT<T> &P, int tag, T nx, T ny, const T w[4], T wg[4]) {
  T wl[4], z[4] = { T(0), T(0), T(0), T(0) }, wgl[4], a[4], b[4];
  int kind = P.bc_kind[tag];
  if constexpr (!is_f32<T>())
    if (is_wall_kind(kind)) {
      const double nn[2] = { nx, ny };
      D::WallMap<2>(kind, P.bc_uw + 2 * tag, nn).apply(w, wg);
      return;
    }
  D::rot_in(nx, ny, w, wl);
  if (kind == CGKS_BC_FARFIELD) {
    farfield_ghost(P, tag, nx, ny, wl, wgl);
  } else if (kind == CGKS_BC_DIRICHLET) {
    dirichlet_ghost(P, tag, nx, ny, wgl);
  } else if (kind == CGKS_BC_OUTFLOW) {
    for (int v = 0; v < 4; ++v) wgl[v] = wl[v];
  } else if (kind == CGKS_BC_SLIP) {
    D::ghost_slip(wl, z, z, wgl, a, b);
  } else {
    T wn = P.bc_uw[2 * tag] * nx + P.bc_uw[2 * tag + 1] * ny;
    T wt = -P.bc_uw[2 * tag] * ny + P.bc_uw[2 * tag + 1] * nx;
    D::ghost_noslip(P.gamma, wn, wt, wl, z, z, wgl, a, b);
  }
  D::rot_out(nx, ny, wgl, wg);
}

// K2: gas-kinetic flux and interface state at the two Gauss points of every
// face; writes the weighted sums F0, F1, Wc, Wt (global frame) per face:
//   out[f*kFO + k*4 + v], k = 0 F0, 1 F1, 2 Wc, 3 Wt,
// one run per face, so that a cell gathers a face in whole sectors.
// Two forms.  face_raw_at: both Gauss points of a face in one thread, raw
// moments in the face frame: the FP32 of the mixed path (whose rounding it
// fixes: the implicit solves of a V-cycle carry a changed FP32 rounding into
// every cell, and the mixed results are to stay what they are).  face_point_at:
// FP64.
template <typename T, bool FULL, bool CHAR>
__device__ __forceinline__ void face_raw_at(const MeshT<T> &m, const ParamsT<T> &P, const T *W,
                                        const T *Wx, const T *coef, T *__restrict__ out,
                                        const Ctl *ctl, const unsigned long long *dt_bits, const int f) {
  const int sid = m.fsid[f];
  if (sid < 0) return;   // free face space of a batch
  if (P.slim && (P.slim[sid] != 0) != FULL) return;   // the other flux class's launch
  const int nf = m.nf;
  const int c0 = m.fc0[f], c1 = m.fc1[f];
  const T nx = m.fn[f], ny = m.fn[nf + f], ajump = m.fjump[f];
  const T mu = P.mu[sid];
  // the full flux integrates over the step: it needs the step's dt
  T dt = T(0);
  if constexpr (FULL) dt = static_cast<T>(dt_of(ctl, dt_bits, sid, static_cast<double>(P.cfl_hi)));
  T acc[4][4];
  for (int k = 0; k < 4; ++k) for (int v = 0; v < 4; ++v) acc[k][v] = T(0);
  T wff[4];
  bool farfield = false;
  int tag = 0, kind = -1;
  if (c1 < 0) {
    tag = -1 - c1;
    kind = P.bc_kind[tag];
    farfield = kind == CGKS_BC_FARFIELD || kind == CGKS_BC_DIRICHLET;
    if (kind == CGKS_BC_FARFIELD) {
      // Riemann-invariant state from the cell mean and the free stream
      T wm[4], wl[4];
      for (int v = 0; v < 4; ++v) wm[v] = W[v * m.nc + c0];
      D::rot_in(nx, ny, wm, wl);
      farfield_ghost(P, tag, nx, ny, wl, wff);
    } else if (kind == CGKS_BC_DIRICHLET) {
      dirichlet_ghost(P, tag, nx, ny, wff);
    }
  }
  // characteristic WENO: the two sides' polynomials limited for this face
  T cs0[CHAR ? kNM : 1][4], cs1[CHAR ? kNM : 1][4];
  bool lim0 = false, lim1 = false;
  if constexpr (CHAR) {
    T wref[4];
    for (int v = 0; v < 4; ++v)
      wref[v] = c1 >= 0 ? T(0.5) * (W[v * m.nc + c0] + W[v * m.nc + c1]) : W[v * m.nc + c0];
    lim0 = m.wenok[c0] != 0;
    if (lim0) char_side(m, P, W, Wx, coef, c0, wref, nx, ny, cs0);
    lim1 = c1 >= 0 && m.wenok[c1] != 0;
    if (lim1) char_side(m, P, W, Wx, coef, c1, wref, nx, ny, cs1);
  }
  for (int k = 0; k < 2; ++k) {
    T wL[4], gxL[4], gyL[4];
    if (CHAR && lim0)
      poly_point(m, W, cs0, c0, m.fxi[(2 * k) * nf + f], m.fxi[(2 * k + 1) * nf + f], wL, gxL, gyL);
    else
      recon_point(m, W, coef, c0, m.fxi[(2 * k) * nf + f], m.fxi[(2 * k + 1) * nf + f], wL, gxL, gyL);
    T wl[4], dnl[4], dtl[4], t0[4], t1[4];
    D::rot_in(nx, ny, wL, wl);
    for (int v = 0; v < 4; ++v) { t0[v] = nx * gxL[v] + ny * gyL[v]; t1[v] = -ny * gxL[v] + nx * gyL[v]; }
    D::rot_in(nx, ny, t0, dnl);
    D::rot_in(nx, ny, t1, dtl);
    T wr[4], dnr[4], dtr[4];
    if (c1 >= 0) {
      T wR[4], gxR[4], gyR[4];
      if (CHAR && lim1)
        poly_point(m, W, cs1, c1, m.fxi[(4 + 2 * k) * nf + f], m.fxi[(5 + 2 * k) * nf + f], wR, gxR, gyR);
      else
        recon_point(m, W, coef, c1, m.fxi[(4 + 2 * k) * nf + f], m.fxi[(5 + 2 * k) * nf + f], wR, gxR, gyR);
      D::rot_in(nx, ny, wR, wr);
      for (int v = 0; v < 4; ++v) { t0[v] = nx * gxR[v] + ny * gyR[v]; t1[v] = -ny * gxR[v] + nx * gyR[v]; }
      D::rot_in(nx, ny, t0, dnr);
      D::rot_in(nx, ny, t1, dtr);
    } else if (farfield) {
      for (int v = 0; v < 4; ++v) { wr[v] = wff[v]; dnr[v] = T(0); dtr[v] = T(0); }
    } else if (kind == CGKS_BC_OUTFLOW) {
      for (int v = 0; v < 4; ++v) { wr[v] = wl[v]; dnr[v] = dnl[v]; dtr[v] = dtl[v]; }
    } else if (kind == CGKS_BC_SLIP) {
      D::ghost_slip(wl, dnl, dtl, wr, dnr, dtr);
    } else {
      T wn = P.bc_uw[2 * tag] * nx + P.bc_uw[2 * tag + 1] * ny;
      T wt = -P.bc_uw[2 * tag] * ny + P.bc_uw[2 * tag + 1] * nx;
      D::ghost_noslip(P.gamma, wn, wt, wl, dnl, dtl, wr, dnr, dtr);
    }
    T F0[4], F1[4], Wc[4], Wt[4];
    if constexpr (FULL)
      D::gks_full_point_local(P.kc, mu, ajump, dt, P.tau_c1, P.tau_c2, wl, wr, dnl, dtl, dnr, dtr, F0, F1, Wc, Wt);
    else
      D::gks_point_local(P.kc, mu, ajump, wl, wr, dnl, dtl, dnr, dtr, F0, F1, Wc, Wt);
    T g[4];
    D::rot_out(nx, ny, F0, g); for (int v = 0; v < 4; ++v) acc[0][v] += T(0.5) * g[v];
    D::rot_out(nx, ny, F1, g); for (int v = 0; v < 4; ++v) acc[1][v] += T(0.5) * g[v];
    D::rot_out(nx, ny, Wc, g); for (int v = 0; v < 4; ++v) acc[2][v] += T(0.5) * g[v];
    D::rot_out(nx, ny, Wt, g); for (int v = 0; v < 4; ++v) acc[3][v] += T(0.5) * g[v];
  }
  T o[kFO];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int v = 0; v < 4; ++v) o[k * 4 + v] = acc[k][v];
  vstore<T, kFO>(out + static_cast<size_t>(f) * kFO, o);
}
// The FP64 flux.  One thread evaluates Gauss point k of face f; in the
// pair of lanes of a face lane 0 collects and stores F0 and F1, lane 1 Wc and
// Wt.  GB300's FP64 units take 64 clocks of a sub-core per warp instruction
// whatever the number of active lanes, so the FP64 instructions of a thread
// are what the kernel costs: the gradients of the two sides are averaged in
// the global frame before the moments need them, the moments close about the
// mean velocity (gks_smooth), erf and exp share one argument (half01), and
// one point per thread halves the serial chain of a small mesh.  Bound by the
// FP64 pipe.  Smooth flux, before (face_raw_at) and now: 319 -> 140 us on
// 90,368 faces, 66 -> 23 us on 208; full flux (gks_full): 167 -> 75 us on 10,088
// faces; with characteristic WENO, each lane limiting one side, 217 -> 85 us on
// 7,350.
__device__ __forceinline__ void pair_sum_store(const double F0[4], const double F1[4], const double Wc[4],
                                               const double Wt[4], int k, unsigned pair, double *__restrict__ out,
                                               int f) {
  double a[8];
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double s0 = k ? F0[v] : Wc[v], s1 = k ? F1[v] : Wt[v];
    a[v] = (k ? Wc[v] : F0[v]) + __shfl_xor_sync(pair, s0, 1);
    a[4 + v] = (k ? Wt[v] : F1[v]) + __shfl_xor_sync(pair, s1, 1);
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) a[q] *= 0.5;
  vstore<double, 8>(out + static_cast<size_t>(f) * kFO + 8 * k, a);
}
template <bool FULL, bool CHAR>
__device__ __forceinline__ void face_point_at(const MeshT<double> &m, const ParamsT<double> &P,
                                              const double *W, const double *Wx,
                                              const double *coef, double *__restrict__ out,
                                              const Ctl *ctl, const unsigned long long *dt_bits, const int f,
                                              const int k) {
  const int sid = m.fsid[f];
  if (sid < 0) return;   // free face space of a batch
  if (P.slim && (P.slim[sid] != 0) != FULL) return;   // the other flux class's launch
  const unsigned pair = 3u << (threadIdx.x & 30);      // the lanes of this face
  const int nf = m.nf;
  const int c0 = m.fc0[f], c1 = m.fc1[f];
  const double nx = m.fn[f], ny = m.fn[nf + f], ajump = m.fjump[f];
  // the two sides' polynomials.  Characteristic WENO limits them for this
  // face: lane k that of side k, exchanged within the pair
  double cL[kNM][4], cR[kNM][4];
  if constexpr (CHAR) {
    double wref[4];
    for (int v = 0; v < 4; ++v) wref[v] = c1 >= 0 ? 0.5 * (W[v * m.nc + c0] + W[v * m.nc + c1]) : W[v * m.nc + c0];
    const int ci = k && c1 >= 0 ? c1 : c0;
    double own[kNM][4];
    if (m.wenok[ci]) char_side(m, P, W, Wx, coef, ci, wref, nx, ny, own);
    else load_coef(m.nc, coef, ci, own);
#pragma unroll
    for (int q = 0; q < kNM; ++q)
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const double other = __shfl_xor_sync(pair, own[q][v], 1);
        cL[q][v] = k ? other : own[q][v];
        cR[q][v] = k ? own[q][v] : other;
      }
  } else {
    load_coef(m.nc, coef, c0, cL);
    if (c1 >= 0) load_coef(m.nc, coef, c1, cR);
  }
  // value and scaled gradient, global frame
  double wL[4], gL[2][4], wR[4], gR[2][4], wl[4], wr[4];
  side_scaled(m, W, cL, c0, m.fxi[(2 * k) * nf + f], m.fxi[(2 * k + 1) * nf + f], wL, gL[0], gL[1]);
  D::rot_in(nx, ny, wL, wl);
  const double ihL = m.ih[c0];
  double ihR = ihL;
  if (c1 >= 0) {
    side_scaled(m, W, cR, c1, m.fxi[(4 + 2 * k) * nf + f], m.fxi[(5 + 2 * k) * nf + f], wR, gR[0], gR[1]);
    D::rot_in(nx, ny, wR, wr);
    ihR = m.ih[c1];
  } else {
    const int tag = -1 - c1, kind = P.bc_kind[tag];
    if (kind == CGKS_BC_FARFIELD || kind == CGKS_BC_DIRICHLET) {
      if (kind == CGKS_BC_FARFIELD) {
        // Riemann-invariant state from the cell mean and the free stream
        double wm[4], wi[4];
        for (int v = 0; v < 4; ++v) wm[v] = W[v * m.nc + c0];
        D::rot_in(nx, ny, wm, wi);
        farfield_ghost(P, tag, nx, ny, wi, wr);
      } else {
        dirichlet_ghost(P, tag, nx, ny, wr);
      }
      D::rot_out(nx, ny, wr, wR);
      for (int v = 0; v < 4; ++v) gR[0][v] = gR[1][v] = 0.0;
    } else if (kind == CGKS_BC_OUTFLOW) {
      for (int v = 0; v < 4; ++v) { wR[v] = wL[v]; wr[v] = wl[v]; gR[0][v] = gL[0][v]; gR[1][v] = gL[1][v]; }
    } else {
      const double nn[2] = { nx, ny };
      const D::WallMap<2> mirror(kind, P.bc_uw + 2 * tag, nn);
      mirror.apply(wL, wR);
      mirror.apply_gradient(gL, gR);
      D::rot_in(nx, ny, wR, wr);
    }
  }
  // slopes of the equilibrium at W^c: the mean of the sides plus, along n,
  // alpha / delta times the jump
  double Wc[4], G[2][4], F0[4], F1[4], Wt[4];
  const double hl = 0.5 * ihL, hr = 0.5 * ihR, ax = ajump * nx, ay = ajump * ny;
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const double d = wR[v] - wL[v];
    G[0][v] = hl * gL[0][v] + hr * gR[0][v] + ax * d;
    G[1][v] = hl * gL[1][v] + hr * gR[1][v] + ay * d;
  }
  if constexpr (FULL) {
    // each side's derivatives along n and t in the face frame
    double dnl[4], dtl[4], dnr[4], dtr[4], t0[4], t1[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      t0[v] = ihL * (nx * gL[0][v] + ny * gL[1][v]);
      t1[v] = ihL * (nx * gL[1][v] - ny * gL[0][v]);
    }
    D::rot_in(nx, ny, t0, dnl);
    D::rot_in(nx, ny, t1, dtl);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      t0[v] = ihR * (nx * gR[0][v] + ny * gR[1][v]);
      t1[v] = ihR * (nx * gR[1][v] - ny * gR[0][v]);
    }
    D::rot_in(nx, ny, t0, dnr);
    D::rot_in(nx, ny, t1, dtr);
    const double dt = dt_of(ctl, dt_bits, sid, P.cfl_hi);   // the full flux integrates over the step
    D::gks_full(P.kc, P.mu[sid], dt, P.tau_c1, P.tau_c2, nx, ny, wl, wr, dnl, dtl, dnr, dtr, G, F0, F1, Wc, Wt);
  } else {
    // W^c from the two half ranges
    double wc[4];
    D::half_state<double, false>(P.kc, wl, +1, wc);
    D::half_state<double, true>(P.kc, wr, -1, wc);
    D::rot_out(nx, ny, wc, Wc);
    D::gks_smooth(P.kc, P.mu[sid], nx, ny, Wc, G, F0, F1, Wt);
  }
  pair_sum_store(F0, F1, Wc, Wt, k, pair, out, f);
}
// threads a face takes
template <typename T> __host__ __device__ constexpr int face_threads() { return is_f32<T>() ? 1 : 2; }
template <typename T, bool FULL, bool CHAR>
__global__ void __launch_bounds__(kMaxShapeBlock) k_face(MeshT<T> m, ParamsT<T> P, const T *W,
                                                         const T *Wx, const T *coef,
                                                         T *out, const Ctl *ctl,
                                                         const unsigned long long *dt_bits) {
  pdl_enter();
  if constexpr (!is_f32<T>())
    for_items(2 * m.nf, [&](int i) {
      face_point_at<FULL, CHAR>(m, P, W, Wx, coef, out, ctl, dt_bits, i >> 1, i & 1);
    });
  else
    for_items(m.nf, [&](int f) { face_raw_at<T, FULL, CHAR>(m, P, W, Wx, coef, out, ctl, dt_bits, f); });
  pdl_exit();
}

// K3 modes
enum UpdMode { kS1O2 = 0, kS2O4Stage = 1, kS2O4Final = 2, kResidual = 3 };

// K3: gather the face sums of each cell (accumulated in FP64).
//   net flux   R  = -sum_p sgn S_p (a0 F0A + a1 F1A + a2 F1B)
//   W_out = W_base + dt/|Omega| R   (not in kResidual mode)
//   Wx_out = 1/|Omega| sum_p sgn S_p n_p (WcA + b1 WtX)
// optional outputs: R itself, float mirrors of W_out / Wx_out, the
// per-block density-residual partial sums; plus the state check.
// In the mixed path bound by the FP64 pipe as well (every FP32 face value is
// accumulated in FP64): runs are widened and mirrors rounded with integer
// instructions, areas and normals come from the cell's slots (coalesced), the
// mode is a template argument so that only the values it needs are read.
// us per launch, before and now: 57,344 cells mixed 30.2 -> 16.6, FP64 22.7 -> 16.9.
template <typename TF, int mode>
__global__ void __launch_bounds__(kCellBlock) k_update(MeshT<double> m, ParamsT<double> P, const double *Wbase,
                                                       const TF *FA, const TF *FB, const Ctl *ctl,
                                                       const unsigned long long *dt_bits, int *status, double *Wout,
                                                       double *Wxout, double *partial, double *Rout, TF *Wout_m,
                                                       TF *Wxout_m) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = m.nc;
  double num = 0.0, den = 0.0;
  const int sid = i < n ? m.csid[i] : -1;
  // mesh data first (nothing in a cycle writes it), then wait for the predecessor
  int fsl[kMaxFace];
  double Ss[kMaxFace];
  if (sid >= 0)
#pragma unroll
    for (int s = 0; s < kMaxFace; ++s) {
      fsl[s] = m.cface[s * n + i];
      Ss[s] = m.shs[s * n + i];
    }
  pdl_enter();
  if (sid >= 0) {
    const double dt = dt_of(ctl, dt_bits, sid, P.cfl_hi);
    const double a1 = mode == kS2O4Stage ? 0.125 * dt : mode == kS2O4Final ? dt / 6.0 : 0.5 * dt;
    const double b1 = mode == kS2O4Stage ? 0.5 * dt : dt;
    double R[4] = { 0, 0, 0, 0 }, gx[4] = { 0, 0, 0, 0 }, gy[4] = { 0, 0, 0, 0 };
#pragma unroll
    for (int s = 0; s < kMaxFace; ++s) {
      const int fs = fsl[s];
      if (fs == kNoFace) continue;
      const size_t at = static_cast<size_t>(fs >= 0 ? fs : ~fs) * kFO;
      const double S = fs >= 0 ? Ss[s] : -Ss[s];
      constexpr int NA = mode == kResidual ? 8 : kFO;   // the residual reads F0, F1 only
      TF fa[NA];
      double a[NA];
      vload<TF, NA>(FA + at, fa);
      widen<NA>(fa, a);
      double b[mode == kS2O4Final ? 8 : 1];             // F1, Wt of the second stage
      if constexpr (mode == kS2O4Final) {
        TF fb[8];
        vload<TF, 4>(FB + at + 4, fb);
        vload<TF, 4>(FB + at + 12, fb + 4);
        widen<8>(fb, b);
      }
      double nx = 0.0, ny = 0.0;
      if constexpr (mode != kResidual) {
        nx = m.snx[s * n + i];   // sgn S n / 2
        ny = m.sny[s * n + i];
      }
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        double f1 = a[4 + v];
        if constexpr (mode == kS2O4Final) f1 += 2.0 * b[v];
        const double f0 = mode == kS2O4Stage ? 0.5 * a[v] : a[v];
        // (the product rounded by itself: a last bit of R_p0 becomes one of the
        // mixed path's FP32 right-hand side, and the implicit solves spread it)
        R[v] -= __dmul_rn(S, f0 + a1 * f1);
        if constexpr (mode != kResidual) {
          double wt;
          if constexpr (mode == kS2O4Final) wt = b[4 + v];
          else wt = a[12 + v];
          const double wp = a[8 + v] + b1 * wt;
          gx[v] += nx * wp;
          gy[v] += ny * wp;
        }
      }
    }
    if (Rout)
#pragma unroll
      for (int v = 0; v < 4; ++v) Rout[v * n + i] = R[v];
    if constexpr (mode != kResidual) {
      const double iv = m.ivol[i], k = dt * iv, iv2 = 2.0 * iv;
      const double old = Wbase[i];   // Wout may be Wbase (explicit steps update in place)
      double w[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        w[v] = Wbase[v * n + i] + k * R[v];
        gx[v] *= iv2;
        gy[v] *= iv2;
        Wout[v * n + i] = w[v];
        Wxout[v * n + i] = gx[v];
        Wxout[(4 + v) * n + i] = gy[v];
        if (Wout_m) {
          Wout_m[v * n + i] = narrow<TF>(w[v]);
          Wxout_m[v * n + i] = narrow<TF>(gx[v]);
          Wxout_m[(4 + v) * n + i] = narrow<TF>(gy[v]);
        }
      }
      if (!state_ok(w)) atomicOr(&status[sid], kBadState);
      num = fabs(w[0] - old);
      den = old;
    }
  }
  if (partial) block_sum2(num, den, &partial[2 * blockIdx.x]);
  pdl_exit();
}

// Sum each solve's block partials in a fixed order (one block per solve
// slot; blk[2s], blk[2s+1] its cell blocks): Res_s = num / den.  Slot 0
// also appends to the residual history.
__global__ void k_res_final(const double *partial, const int *__restrict__ blk, Ctl *ctl,
                            double *res, double *hist, int cap, double *last) {
  pdl_enter();
  const int s = blockIdx.x;
  double a = 0.0, b = 0.0;
  for (int k = blk[2 * s] + threadIdx.x; k < blk[2 * s + 1]; k += blockDim.x) {
    a += partial[2 * k];
    b += partial[2 * k + 1];
  }
  __shared__ double tot[2];
  block_sum2(a, b, tot);
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = tot[0] / tot[1];
    res[s] = r;
    if (s == 0) {
      last[0] = r; last[1] = tot[0]; last[2] = tot[1];
      int c = ctl->res_ctr;
      if (hist && c < cap) hist[c] = r;
      ctl->res_ctr = c + 1;
    }
  }
  pdl_exit();
}

// ---------------------------- low-order level ----------------------------
// Records of the low level, one run of values per cell or face, so that a
// neighbour's data costs whole sectors:
//   base  [kBase] per cell, the state U at the start of an implicit step, the
//         part a sweep reads first: in FP64 rho, u, v, H = rho E + p; p,
//         1/(2 lambda), sqrt(lambda), 1/sqrt(pi lambda), c, rho u, rho v, rho E;
//         in FP32 rho, rho u, rho v, rho E, u, v, p, 0; 1/(2 lambda),
//         sqrt(lambda), 1/sqrt(pi lambda), c;
//   delta [del_run] per cell, its increment dU; in FP64 then du, dv and dp,
//         the exact changes of velocity and pressure it makes, 0;
//   Flo   [lo_run] per face: the flux, lambda_p, padding.
// The device functions serve the per-phase kernels and the persistent
// launch; CG reads what other blocks of a launch wrote through L2.
constexpr int kBase = 12;
template <typename T> __host__ __device__ constexpr int del_run() { return is_f32<T>() ? 4 : 8; }
template <typename T> __host__ __device__ constexpr int lo_run() { return is_f32<T>() ? 8 : 6; }

__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }

// positions in a base record
template <typename T>
struct BaseAt {
  static constexpr bool f = is_f32<T>();
  static constexpr int m = f ? 1 : 9, E = f ? 3 : 11, u = f ? 4 : 1, p = f ? 6 : 4, i2l = f ? 8 : 5, sl = f ? 9 : 6,
                       isp = f ? 10 : 7, c = f ? 11 : 8;
};
template <typename T>
__device__ __forceinline__ D::Prim<T> base_prim(const T r[kBase]) {
  using A = BaseAt<T>;
  D::Prim<T> q;
  q.rho = r[0]; q.u = r[A::u]; q.v = r[A::u + 1]; q.p = r[A::p];
  q.i2l = r[A::i2l]; q.sl = r[A::sl]; q.isp = r[A::isp]; q.c = r[A::c];
  return q;
}
// base record of the FP64 state u
template <typename TF>
__device__ __forceinline__ void base_record(const ParamsT<TF> &P, const double u[4], TF r[kBase]) {
  using A = BaseAt<TF>;
  const TF w[4] = { narrow<TF>(u[0]), narrow<TF>(u[1]), narrow<TF>(u[2]), narrow<TF>(u[3]) };
  const D::Prim<TF> q = D::prim_of(w, P.gamma, P.kc);
  if constexpr (is_f32<TF>()) r[7] = TF(0);
  else r[3] = w[3] + q.p;
  r[0] = w[0];
  r[A::m] = w[1]; r[A::m + 1] = w[2]; r[A::E] = w[3];
  r[A::u] = q.u; r[A::u + 1] = q.v; r[A::p] = q.p;
  r[A::i2l] = q.i2l; r[A::sl] = q.sl; r[A::isp] = q.isp; r[A::c] = q.c;
}
// The delta record of an increment d on a cell with base (rho, u, v, H).  FP64:
//   du = (dm - u d rho) / (rho + d rho),
//   dp = (gamma - 1)(dE - d(|m|^2 / 2 rho)), d(m.u) = dm.(u + du) + rho u.du,
// every term proportional to the increment (no cancellation between two
// nearly equal states), with one reciprocal per relaxed cell.
// (Fused multiply-adds are written out: the sweep's two forms below must round
// alike.)
__device__ __forceinline__ void delta_record(double gamma, const double b[4], const double d[4], double r[8]) {
  const double ir = D::d_rcp(b[0] + d[0]);
  const double du = fma(-b[1], d[0], d[1]) * ir, dv = fma(-b[2], d[0], d[2]) * ir;
  const double k1 = fma(d[2], b[2] + dv, __dmul_rn(d[1], b[1] + du));
  const double dk = fma(b[0], fma(b[2], dv, __dmul_rn(b[1], du)), k1);
  const double g1 = gamma - 1.0;
  r[0] = d[0]; r[1] = d[1]; r[2] = d[2]; r[3] = d[3];
  r[4] = du; r[5] = dv; r[6] = fma(g1, d[3], __dmul_rn(-0.5 * g1, dk)); r[7] = 0.0;
}
__device__ __forceinline__ void store_delta(double gamma, const double b[4], const double d[4], double *delta, int i) {
  double r[8];
  delta_record(gamma, b, d, r);
  vstore<double, 8>(delta + static_cast<size_t>(i) * 8, r);
}
__device__ __forceinline__ void store_delta(float, const float *, const float d[4], float *delta, int i) {
  vstore<float, 4>(delta + static_cast<size_t>(i) * 4, d);
}

// K5a: per-cell start of an implicit step: U = W_p0 (first step) or
// U += dU (Algorithm 1's update, in FP64), then the base record of U.
template <typename TF, bool CG>
__device__ __forceinline__ void lo_cell_at(int n, const ParamsT<TF> &P, int first, const double *Wp0,
                                           double *U, const TF *delta, TF *base, int i) {
  double u[4];   // (all loads before the first store, which they might alias)
  if (first) {
#pragma unroll
    for (int v = 0; v < 4; ++v) u[v] = Wp0[v * n + i];
  } else {
    TF d[4];
    vload<TF, 4, CG>(delta + static_cast<size_t>(i) * del_run<TF>(), d);
#pragma unroll
    for (int v = 0; v < 4; ++v) u[v] = ld<CG>(&U[v * n + i]) + static_cast<double>(d[v]);
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) U[v * n + i] = u[v];
  TF r[kBase];
  base_record(P, u, r);
  vstore<TF, kBase>(base + static_cast<size_t>(i) * kBase, r);
}
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_lo_cell(int n, ParamsT<TF> P, int first, const double *Wp0,
                                                        double *U, const TF *delta,
                                                        TF *base) {
  pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  lo_cell_at<TF, false>(n, P, first, Wp0, U, delta, base, i);
  pdl_exit();
}

// K5b: first-order KFVS (or Lax-Friedrichs) flux and the spectral radius
// lambda_p = max of both sides.  FP64 is bound by its pipe, so it has no face
// frame, no division and no pow.  us per launch, FP64, before and now: 57,344
// cells 68 -> 28.4, a 128,000-cell sphere (3-D) 220 -> 93.5.
template <typename T>
struct LoFaceGeo {
  int sid, c0, c1;
  T nx, ny, S, mu, iva, ivb;
};
// mesh and per-solve data of face f (nothing in a cycle writes them)
template <typename T>
__device__ __forceinline__ LoFaceGeo<T> lo_face_geo(const MeshT<T> &m, const ParamsT<T> &P, const int f) {
  LoFaceGeo<T> g;
  g.sid = m.fsid[f];
  g.c0 = g.c1 = 0;
  g.nx = g.ny = g.S = g.mu = g.iva = g.ivb = T(0);
  if (g.sid < 0) return g;
  const int nf = m.nf;
  g.c0 = m.fc0[f];
  g.c1 = m.fc1[f];
  g.nx = m.fn[f];
  g.ny = m.fn[nf + f];
  g.mu = P.mu[g.sid];
  if (g.mu != T(0)) {   // the viscous part of lambda_p
    g.S = m.fS[f];
    g.iva = m.ivol[g.c0];
    g.ivb = g.c1 >= 0 ? m.ivol[g.c1] : g.iva;
  }
  return g;
}
__device__ __forceinline__ float third(float x) { return x / 3.0f; }
__device__ __forceinline__ double third(double x) { return x * (1.0 / 3.0); }
// the flux (out of c0) and, in o[4], lambda_p
template <typename T, bool CG>
__device__ __forceinline__ void lo_flux_at(const MeshT<T> &m, const ParamsT<T> &P, const LoFaceGeo<T> &g,
                                           const T *base, const int f, T o[lo_run<T>()]) {
  const int c1 = g.c1;
  const T nx = g.nx, ny = g.ny, mu = g.mu;
  T ra[kBase], rb[kBase];
  vload<T, kBase, CG>(base + static_cast<size_t>(g.c0) * kBase, ra);
  const D::Prim<T> a = base_prim(ra);
  D::Prim<T> b;
  using A = BaseAt<T>;
  const T wa[4] = { ra[0], ra[A::m], ra[A::m + 1], ra[A::E] };   // states of the two sides (global frame)
  T wb[4];                                                       // the ghost on a boundary
  if (c1 >= 0) {
    vload<T, kBase, CG>(base + static_cast<size_t>(c1) * kBase, rb);
    b = base_prim(rb);
    wb[0] = rb[0]; wb[1] = rb[A::m]; wb[2] = rb[A::m + 1]; wb[3] = rb[A::E];
  } else {
    lo_ghost(P, -1 - c1, nx, ny, wa, wb);
    b = D::prim_of(wb, P.gamma, P.kc);
  }
  const T una = D::dot2(a.u, nx, a.v, ny), unb = D::dot2(b.u, nx, b.v, ny);
  T la = fabs(una) + a.c, lb = fabs(unb) + b.c, ira = T(0), irb = T(0);
  if (mu != T(0)) {
    ira = D::d_rcp(a.rho);
    irb = D::d_rcp(b.rho);
    la = D::mad(T(2) * (mu * ira) * g.S, g.iva, la);
    lb = D::mad(T(2) * (mu * irb) * g.S, g.ivb, lb);
  }
  const T lmax = la > lb ? la : lb;
  T F[4];
  if (P.flux_lo == CGKS_FLUX_LF) {
    // Lax-Friedrichs alternative of Section 3 with the implicit operator's
    // lambda_p: (F_n(U_l) + F_n(U_r)) / 2 - lambda_p (U_r - U_l) / 2
    // (products rounded by themselves: the mixed path's FP32 results stay what they are)
    const T Fa[4] = { mul_rn(a.rho, una), D::dot2(wa[1], una, a.p, nx), D::dot2(wa[2], una, a.p, ny),
                      mul_rn(wa[3] + a.p, una) };
    const T Fb[4] = { mul_rn(b.rho, unb), D::dot2(wb[1], unb, b.p, nx), D::dot2(wb[2], unb, b.p, ny),
                      mul_rn(wb[3] + b.p, unb) };
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      if constexpr (is_f32<T>()) F[v] = T(0.5) * (Fa[v] + Fb[v]) - T(0.5) * lmax * (wb[v] - wa[v]);
      else F[v] = D::dot2(T(0.5), Fa[v] + Fb[v], -(T(0.5) * lmax), wb[v] - wa[v]);
    }
  } else if constexpr (is_f32<T>()) {
    const T uta = -a.u * ny + a.v * nx, utb = -b.u * ny + b.v * nx;
    T Fl[4];
    D::kfvs_prims(P.K, a.rho, una, uta, a.i2l, a.sl, a.isp, b.rho, unb, utb, b.i2l, b.sl, b.isp, Fl);
    D::rot_out(nx, ny, Fl, F);
  } else {
    // KFVS without the face frame: with m0, m1 the half moments 1 and <u>,
    // a side's flux is rho m1 (1, u, v) + p m0 (0, n) and
    // m1 (H - p / 2) + p m0 u_n / 2 for the energy
    T m0a, m1a, m0b, m1b;
    D::half01(una, a.sl, a.isp, +1, m0a, m1a);
    D::half01(unb, b.sl, b.isp, -1, m0b, m1b);
    const T ja = D::prod(a.rho, m1a), jb = D::prod(b.rho, m1b), pa = D::prod(a.p, m0a), pb = D::prod(b.p, m0b);
    const T pn = pa + pb;
    F[0] = ja + jb;
    F[1] = fma(pn, nx, D::dot2(ja, a.u, jb, b.u));
    F[2] = fma(pn, ny, D::dot2(ja, a.v, jb, b.v));
    F[3] = fma(T(0.5), D::dot2(pa, una, pb, unb),
               D::dot2(m1a, fma(T(0.5), a.p, wa[3]), m1b, fma(T(0.5), b.p, wb[3])));
  }
  if (P.lo_viscous && mu > T(0)) {
    // first-order viscous flux: normal gradients from the two cell states
    // over the centre distance delta, Stokes' hypothesis, Pr = 1 heat flux
    //   tau.n = mu / delta (du + (n.du) n / 3),  q.n = -kappa (T_r - T_l) / delta
    const T md = mu * m.fidl[f];
    const T dux = b.u - a.u, duy = b.v - a.v;
    const T dn = third(D::dot2(dux, nx, duy, ny));
    const T tx = D::prod(md, D::mad(dn, nx, dux)), ty = D::prod(md, D::mad(dn, ny, duy));
    T qn;   // gamma / (gamma - 1) = N / 2 + 1
    if constexpr (is_f32<T>()) qn = -md * P.gamma / (P.gamma - T(1)) * (b.p * irb - a.p * ira);
    else qn = D::prod(-md * (P.kc.hN + T(1)), D::dot2(b.p, irb, -a.p, ira));
    F[1] -= tx;
    F[2] -= ty;
    F[3] -= D::dot2(tx, T(0.5) * (a.u + b.u), ty, T(0.5) * (a.v + b.v)) - qn;
  }
#pragma unroll
  for (int v = 0; v < 4; ++v) o[v] = F[v];
  o[4] = lmax;
#pragma unroll
  for (int v = 5; v < lo_run<T>(); ++v) o[v] = T(0);
}
template <typename T, bool CG>
__device__ __forceinline__ void lo_face_at(const MeshT<T> &m, const ParamsT<T> &P, const LoFaceGeo<T> &g,
                                           const T *base, T *__restrict__ Flo, const int f) {
  if (g.sid < 0) return;   // free face space of a batch
  T o[lo_run<T>()];
  lo_flux_at<T, CG>(m, P, g, base, f, o);
  vstore<T, lo_run<T>()>(Flo + static_cast<size_t>(f) * lo_run<T>(), o);
}
template <typename T>
__global__ void __launch_bounds__(kMaxShapeBlock) k_lo_face(MeshT<T> m, ParamsT<T> P, const T *base, T *Flo) {
  for_items_pdl(m.nf, [&](int f) { return lo_face_geo(m, P, f); },
                [&](int f, const LoFaceGeo<T> &g) { lo_face_at<T, false>(m, P, g, base, Flo, f); });
  pdl_exit();
}

// K6: low-order right-hand side R^k = R_lo(U^k) + S (FP64 sums), 1/D_i
// (FP64), each slot's lambda for the sweeps (in FP64 times S/2), and the first colour pass
// of the relaxation: with dU = 0 everywhere the update of a colour-0 cell
// reduces to R_i / D_i; all other cells start at 0.  first: also forms the
// forcing S = R_p0 - R_lo(W_p0) (Section 3, step 3).
struct RhsGeo {
  int fs[kMaxFace];
  double S[kMaxFace];
  bool c0;
};
__device__ __forceinline__ RhsGeo rhs_geo(const MeshT<double> &m, int i, int colour0) {
  RhsGeo g;
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
    g.fs[s] = m.cface[s * m.nc + i];
    g.S[s] = m.shs[s * m.nc + i];
  }
  g.c0 = colour0 && m.ccol[i] == 0;
  return g;
}
template <typename TF, bool CG>
__device__ __forceinline__ void lo_rhs_at(const MeshT<double> &m, const ParamsT<double> &P, TF gamma, const RhsGeo &g,
                                          int first, const TF *base, const TF *Flo, const double *Rp0,
                                          double *Src, TF *Rk, TF *invD, TF *delta, TF *lamS, int i) {
  const int n = m.nc;
  constexpr int N = lo_run<TF>();
  double R[4] = { 0, 0, 0, 0 }, sum = 0.0;
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
    const int fs = g.fs[s];
    if (fs == kNoFace) { lamS[s * n + i] = TF(0); continue; }
    const double S = g.S[s], Sg = fs >= 0 ? -S : S;
    TF fl[N];
    double x[N];
    vload<TF, N, CG>(Flo + static_cast<size_t>(fs >= 0 ? fs : ~fs) * N, fl);
    widen<5>(fl, x);
#pragma unroll
    for (int v = 0; v < 4; ++v) R[v] = D::mad(Sg, x[v], R[v]);
    sum = D::mad(x[4], S, sum);
    if constexpr (is_f32<TF>()) lamS[s * n + i] = fl[4];
    else lamS[s * n + i] = fl[4] * (0.5 * S);
  }
  // dt_i = CFL_lo |Omega| / sum;  D_i = |Omega| / dt_i + sum / 2 (padding cells: 0)
  const double id = sum > 0.0 ? D::d_rcp(sum * (P.icfl_lo + 0.5)) : 0.0;
  double src[4];
#pragma unroll
  for (int v = 0; v < 4; ++v) src[v] = first ? Rp0[v * n + i] - R[v] : ld<CG>(&Src[v * n + i]);
  invD[i] = narrow<TF>(id);
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    if (first) Src[v * n + i] = src[v];
    R[v] += src[v];
    Rk[v * n + i] = narrow<TF>(R[v]);
  }
  if (g.c0) {
    TF b[4], d[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) d[v] = narrow<TF>(__dmul_rn(R[v], id));
    vload<TF, 4, CG>(base + static_cast<size_t>(i) * kBase, b);
    store_delta(gamma, b, d, delta, i);
  } else {
    TF z[del_run<TF>()];
#pragma unroll
    for (int v = 0; v < del_run<TF>(); ++v) z[v] = TF(0);
    vstore<TF, del_run<TF>()>(delta + static_cast<size_t>(i) * del_run<TF>(), z);
  }
}
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_lo_rhs(MeshT<double> m, ParamsT<double> P, TF gamma, int first,
                                                       int colour0, const TF *base,
                                                       const TF *Flo, const double *Rp0,
                                                       double *Src, TF *Rk,
                                                       TF *invD, TF *delta,
                                                       TF *lamS) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m.nc) { pdl_enter(); return; }
  // mesh data first (nothing in a cycle writes it), then wait for the predecessor
  const RhsGeo g = rhs_geo(m, i, colour0);
  pdl_enter();
  lo_rhs_at<TF, false>(m, P, gamma, g, first, base, Flo, Rp0, Src, Rk, invD, delta, lamS, i);
  pdl_exit();
}

// K5b and K6 in one launch, four lanes per cell, one per face slot: the lane
// forms its slot's flux, then the sums of one variable.  Every face is
// evaluated twice, with the same bits, but a launch and its wait are saved and
// the chain of FP64 instructions that a small launch waits for shrinks (the
// sums of one variable, 20 instructions, where one thread took 60).
// us per V-cycle, two launches / one: mixed 2,048 cells 183 / 169, FP64 321 / 302.
template <typename TF>
__global__ void __launch_bounds__(kMaxShapeBlock) k_lo_flux_rhs(MeshT<TF> fm, ParamsT<TF> fP, MeshT<double> m,
                                                                ParamsT<double> P, int first, int colour0,
                                                                const TF *base, const double *Rp0, double *Src,
                                                                TF *Rk, TF *invD, TF *delta, TF *lamS) {
  const int t = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  const int i = t / kMaxFace, s = t % kMaxFace, n = m.nc;
  const bool in = i < n;
  // mesh data first (nothing in a cycle writes it), then wait for the predecessor
  const int fs = in ? m.cface[s * n + i] : kNoFace, f = fs >= 0 ? fs : ~fs;
  const double S = in ? m.shs[s * n + i] : 0.0;
  const bool c0 = in && colour0 && m.ccol[i] == 0, there = fs != kNoFace;
  LoFaceGeo<TF> g;
  if (there) g = lo_face_geo(fm, fP, f);
  pdl_enter();
  double x[5] = { 0.0, 0.0, 0.0, 0.0, 0.0 };
  TF lam = TF(0);
  if (there) {
    TF o[lo_run<TF>()];
    lo_flux_at<TF, false>(fm, fP, g, base, f, o);
    widen<5>(o, x);
    if constexpr (is_f32<TF>()) lam = o[4];
    else lam = o[4] * (0.5 * S);
  }
  // lane s sums variable s, in the order of the slots
  double R = 0.0, sum = 0.0;
#pragma unroll
  for (int q = 0; q < kMaxFace; ++q) {
    double y[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) y[v] = __shfl_sync(0xffffffffu, x[v], q, kMaxFace);
    const double Sq = __shfl_sync(0xffffffffu, S, q, kMaxFace);
    const int fq = __shfl_sync(0xffffffffu, fs, q, kMaxFace);
    const double xv = s == 0 ? y[0] : s == 1 ? y[1] : s == 2 ? y[2] : y[3];
    if (fq != kNoFace) {
      R = D::mad(fq >= 0 ? -Sq : Sq, xv, R);
      sum = D::mad(y[4], Sq, sum);
    }
  }
  const double id = sum > 0.0 ? D::d_rcp(sum * (P.icfl_lo + 0.5)) : 0.0;
  if (in) {
    double src;
    if (first) { src = Rp0[s * n + i] - R; Src[s * n + i] = src; }
    else src = Src[s * n + i];
    R += src;
    Rk[s * n + i] = narrow<TF>(R);
    lamS[s * n + i] = lam;
    if (s == 0) invD[i] = narrow<TF>(id);
  }
  const TF ds = c0 ? narrow<TF>(__dmul_rn(R, id)) : TF(0);
  if constexpr (is_f32<TF>()) {
    if (in) delta[static_cast<size_t>(i) * 4 + s] = ds;
  } else {
    TF d[4], rec[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) rec[v] = TF(0);
#pragma unroll
    for (int v = 0; v < 4; ++v) d[v] = __shfl_sync(0xffffffffu, ds, v, 4);
    if (c0) {
      TF b[4];
      vload<TF, 4>(base + static_cast<size_t>(i) * kBase, b);
      delta_record(fP.gamma, b, d, rec);
    }
    const TF lo = s == 0 ? rec[0] : s == 1 ? rec[2] : s == 2 ? rec[4] : rec[6];
    const TF hi = s == 0 ? rec[1] : s == 1 ? rec[3] : s == 2 ? rec[5] : rec[7];
    const TF two[2] = { lo, hi };
    if (in) vstore<TF, 2>(delta + static_cast<size_t>(i) * 8 + 2 * s, two);
  }
  pdl_exit();
}
// Cells up to which the merged launch is the shorter one: in FP64 while its
// four lanes per cell give a sub-core (608) one or two warps (4,864 to 9,728
// cells), in FP32 until evaluating every face twice costs more than a launch;
// the lines lie in the ranges where both sides take the same.  us per V-cycle,
// split / merged (cavities): FP64 4,608 cells 310 / 298, 5,832 315 / 316, 6,498
// 319 / 319, 7,200 326 / 329, 8,192 333 / 346; mixed 20,000 199 / 192, 26,450
// 201 / 198, 29,768 213 / 211, 33,800 214 / 216, 41,472 230 / 240.
template <typename T> __host__ __device__ constexpr int64_t merge_cells() { return is_f32<T>() ? 30000 : 6656; }

// The cells of one colour form one contiguous range per solve.  A sweep
// launch covers up to kMaxRanges ranges, carried in the kernel parameters
// (constant bank) so no dependent global load precedes the cell's own
// loads: block b works on range r with blk[r] <= b < blk[r+1].
constexpr int kMaxRanges = 64;
struct Ranges {
  int n;
  int blk[kMaxRanges + 1];
  int begin[kMaxRanges], end[kMaxRanges];
};

// cell of local index cl (cells per block: cpb) in the block's range, or -1
__device__ __forceinline__ int range_cell(const Ranges &R, int cl, int cpb) {
  int r = 0;
  if (R.n > 1) {
    int lo = 0, hi = R.n - 1;   // largest r with blk[r] <= blockIdx.x
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (R.blk[mid] <= static_cast<int>(blockIdx.x)) lo = mid; else hi = mid - 1;
    }
    r = lo;
  }
  const int i = R.begin[r] + (static_cast<int>(blockIdx.x) - R.blk[r]) * cpb + cl;
  return i < R.end[r] ? i : -1;
}

// K7: point relaxation of the cells of one colour (ranges or a list
// spanning every solve of the batch), Eq. (implicit-local):
//   dU_i = (R_i - sum_p S_p [F^-(U_ip + dU_ip) - F^-(U_ip)]) / D_i,
//   F^-(U) = (F_n(U) - lambda_p U) / 2, ghost increments zero.
// FP64: the bracket in increment form, Q = (rho, rho u, rho v, rho E + p),
//   F_n(U + dU) - F_n(U) = dQ u_n' + Q du_n + dp (0, n, 0),  u_n' = u_n + du_n,
// from the neighbour's base and delta records, with n S/2 and lambda S/2 per
// slot.  The velocity and pressure changes of an increment are formed once,
// by the cell that makes it (store_delta), not by each of its neighbours: 17
// FP64 instructions per neighbour and 21 per cell, no division, where each
// face slot took about 45 with an IEEE division.  FP32 (the mixed path) keeps
// its expressions and the order of its sums (euler_flux_delta; pairs of
// slots), which fix its rounding.
// Two forms with the same roundings (the four slots' brackets are summed in
// pairs).  One thread per cell: an FP64 instruction costs a warp the same
// however many lanes are active, so no lane is spent on absent slots, sums or
// the cell's own part; for FP64 launches with more cells than fill the FP64
// units (sweep_lanes).  Four lanes per cell, one per slot: for fewer cells,
// where the chain of FP64 instructions of one warp is what a launch waits for
// (about 42 instead of 90), and for FP32, where it is the chain of loads.
// Cells of one colour never neighbour each other, so the deltas read here are
// not written by this launch.

// static (mesh) data of slot s of cell i; read before the kernel waits on its
// predecessor, since no kernel of a cycle writes it
template <typename T>
struct SlotGeo {
  int j;
  T nx, ny, hS;
};
template <typename T>
__device__ __forceinline__ SlotGeo<T> slot_geo(const MeshT<T> &m, const int i, const int s) {
  SlotGeo<T> g;
  g.j = i >= 0 ? m.cnbr[s * m.nc + i] : -1;
  if (g.j >= 0) {
    g.nx = m.snx[s * m.nc + i];
    g.ny = m.sny[s * m.nc + i];
    if constexpr (is_f32<T>()) g.hS = m.shs[s * m.nc + i];
  }
  return g;
}
// what a sweep reads of a neighbour, and of slot s
template <typename T>
struct SlotData {
  static constexpr int NB = is_f32<T>() ? 8 : 4;
  T b[NB], q[del_run<T>()], ls;
};
template <typename T, bool CG, bool CGD>
__device__ __forceinline__ void slot_load(const MeshT<T> &m, int i, int s, int j, const T *base, const T *lamS,
                                          const T *del, SlotData<T> &x) {
  vload<T, SlotData<T>::NB, CG>(base + static_cast<size_t>(j) * kBase, x.b);
  vload<T, del_run<T>(), CGD>(del + static_cast<size_t>(j) * del_run<T>(), x.q);
  x.ls = ld<CG>(&lamS[s * m.nc + i]);
}
// the slot's bracket times S / 2
__device__ __forceinline__ void slot_bracket(float gamma, const SlotGeo<float> &g, const SlotData<float> &x,
                                             float c[4]) {
  float dF[4];
  D::euler_flux_delta(gamma, x.b, x.b[4], x.b[5], x.b[6], x.q, g.nx, g.ny, dF);
#pragma unroll
  for (int v = 0; v < 4; ++v) c[v] = __fmul_rn(g.hS, dF[v] - x.ls * x.q[v]);
}
__device__ __forceinline__ void slot_bracket(double, const SlotGeo<double> &g, const SlotData<double> &x,
                                             double c[4]) {
  const double *b = x.b, *q = x.q;
  const double dun = fma(q[5], g.ny, __dmul_rn(q[4], g.nx));
  const double un1 = fma(b[2], g.ny, fma(b[1], g.nx, dun));
  const double w = un1 - x.ls, t = __dmul_rn(b[0], dun);
  c[0] = fma(q[0], w, t);
  c[1] = fma(q[6], g.nx, fma(b[1], t, __dmul_rn(q[1], w)));
  c[2] = fma(q[6], g.ny, fma(b[2], t, __dmul_rn(q[2], w)));
  c[3] = fma(b[3], dun, fma(q[6], un1, __dmul_rn(q[3], w)));
}
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

// One thread per cell: the new increment of cell i in d, its delta record
// written to out.  The neighbours' delta records are read from del_of(j)
// (through L2 when CGD is set).
template <typename T, bool CGD, typename DelOf>
__device__ __forceinline__ void sweep_cell(const MeshT<T> &m, T gamma, const SlotGeo<T> g[kMaxFace], const int i,
                                           const T *base, const T *Rk, const T *invD, const T *lamS, DelOf &&del_of,
                                           T *out, T d[4]) {
  const int n = m.nc;
  T r[4], bi[4] = { T(0), T(0), T(0), T(0) };
#pragma unroll
  for (int v = 0; v < 4; ++v) r[v] = Rk[v * n + i];
  if constexpr (!is_f32<T>()) vload<T, 4>(base + static_cast<size_t>(i) * kBase, bi);
  const T iD = invD[i];
  // every neighbour's loads are in flight before the first is used
  SlotData<T> x[kMaxFace];
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s)
    if (g[s].j >= 0) slot_load<T, false, CGD>(m, i, s, g[s].j, base, lamS, del_of(g[s].j), x[s]);
  T c[kMaxFace][4];
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
#pragma unroll
    for (int v = 0; v < 4; ++v) c[s][v] = T(0);
    if (g[s].j >= 0) slot_bracket(gamma, g[s], x[s], c[s]);
  }
  const bool four = g[3].j >= 0;   // (adding an absent slot's 0 changes nothing)
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    const T hi = four ? add_rn(c[2][v], c[3][v]) : c[2][v];
    d[v] = (r[v] - add_rn(add_rn(c[0][v], c[1][v]), hi)) * iD;
  }
  store_delta(gamma, bi, d, out, i);
}
// Four lanes per cell (i < 0: none), lane s one slot: the new increment's
// component s is returned, the delta record written to out; CG and CGD as for
// slot_load.  Whole warps call it.
template <typename T, bool CG, bool CGD, typename DelOf>
__device__ __forceinline__ T sweep_quad(const MeshT<T> &m, T gamma, const SlotGeo<T> &geo, const int i, const int s,
                                        const T *base, const T *Rk, const T *invD, const T *lamS, DelOf &&del_of,
                                        T *out) {
  const int n = m.nc;
  T bi[4] = { T(0), T(0), T(0), T(0) }, r = T(0), iD = T(0);
  if (i >= 0) {
    r = ld<CG>(&Rk[s * n + i]);
    iD = ld<CG>(&invD[i]);
    if constexpr (!is_f32<T>()) vload<T, 4, CG>(base + static_cast<size_t>(i) * kBase, bi);
  }
  T c[4] = { T(0), T(0), T(0), T(0) };
  if (geo.j >= 0) {
    SlotData<T> x;
    slot_load<T, CG, CGD>(m, i, s, geo.j, base, lamS, del_of(geo.j), x);
    slot_bracket(gamma, geo, x, c);
  }
  // lane s needs component s summed over the group: a transposing
  // reduction (3 additions per lane instead of an all-reduce of 4 values);
  // every lane stays to the shuffles, absent cells and slots add 0
  const bool b0 = s & 1, b1 = s & 2;
  const T k0 = add_rn(b0 ? c[1] : c[0], __shfl_xor_sync(0xffffffffu, b0 ? c[0] : c[1], 1));   // component b0
  const T k1 = add_rn(b0 ? c[3] : c[2], __shfl_xor_sync(0xffffffffu, b0 ? c[2] : c[3], 1));   // component b0 + 2
  const T mine = add_rn(b1 ? k1 : k0, __shfl_xor_sync(0xffffffffu, b1 ? k0 : k1, 2));
  const T ds = (r - mine) * iD;
  if constexpr (is_f32<T>()) {
    if (i >= 0) out[static_cast<size_t>(i) * 4 + s] = ds;
  } else {
    T d[4], rec[8];
#pragma unroll
    for (int v = 0; v < 4; ++v) d[v] = __shfl_sync(0xffffffffu, ds, v, 4);
    delta_record(gamma, bi, d, rec);
    if (i >= 0) {
      const T lo = s == 0 ? rec[0] : s == 1 ? rec[2] : s == 2 ? rec[4] : rec[6];
      const T hi = s == 0 ? rec[1] : s == 1 ? rec[3] : s == 2 ? rec[5] : rec[7];
      const T two[2] = { lo, hi };
      vstore<T, 2>(out + static_cast<size_t>(i) * 8 + 2 * s, two);
    }
  }
  return ds;
}
// Lanes per cell of a sweep over cnt cells.  An FP64 launch takes as long as
// the warps of one sub-core (608 of them) issue one after another: about 43
// instructions for each 8 cells with four lanes, 91 for each 32 with one, so
// four are shorter up to two warps a sub-core, 9,728 cells.  Event-timed, us
// per launch, four / one: colours of 1,000 cells 8.0 / 10.6, 2,900 8.2 / 11.1,
// 28,480 15.1 / 13.0 (before: 14.5).
constexpr int kSweepOneLane = 9728;
template <typename T> int sweep_lanes(int cnt) { return !is_f32<T>() && cnt >= kSweepOneLane ? 1 : 4; }
// The cells of one colour form one contiguous range per solve; a block works
// on blockDim / LANES cells of a range.
// LAST: the cell's last relaxation of the implicit step.  It then also
// advances its state, U += dU (FP64), and writes the base record of the next
// implicit step (to a second buffer: later colours of this step still read
// the present one), which takes the place of a pass over all cells.
template <typename T, bool LAST, int LANES>
__global__ void __launch_bounds__(kMaxShapeBlock) k_sweep(MeshT<T> m, ParamsT<T> P,
                                                          const __grid_constant__ Ranges R,
                                                          const int *__restrict__ list, int count, const T *base,
                                                          const T *Rk, const T *invD, const T *lamS, T *delta,
                                                          double *U, T *base_next) {
  const int n = m.nc, cpb = blockDim.x / LANES, cl = static_cast<int>(threadIdx.x) / LANES;
  int i;
  if (list) {
    const int g = static_cast<int>(blockIdx.x) * cpb + cl;
    i = g < count ? list[g] : -1;
  } else {
    i = range_cell(R, cl, cpb);
  }
  if constexpr (LANES == 1) {
    if (i < 0) { pdl_enter(); return; }   // waits too: this grid ends after its predecessor
    SlotGeo<T> geo[kMaxFace];
#pragma unroll
    for (int s = 0; s < kMaxFace; ++s) geo[s] = slot_geo(m, i, s);
    pdl_enter();
    T d[4];
    sweep_cell<T, false>(m, P.gamma, geo, i, base, Rk, invD, lamS, [&](int) -> const T * { return delta; },
                                delta, d);
    if constexpr (LAST) {
      double u[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        u[v] = U[v * n + i] + static_cast<double>(d[v]);
        U[v * n + i] = u[v];
      }
      T rec[kBase];
      base_record(P, u, rec);
      vstore<T, kBase>(base_next + static_cast<size_t>(i) * kBase, rec);
    }
  } else {
    static_assert(LANES == kMaxFace, "a lane per slot");
    const int s = threadIdx.x & (kMaxFace - 1);
    const SlotGeo<T> geo = slot_geo(m, i, s);
    pdl_enter();
    const double us0 = LAST && i >= 0 ? U[s * n + i] : 0.0;
    const T ds = sweep_quad<T, false, false>(m, P.gamma, geo, i, s, base, Rk, invD, lamS,
                                             [&](int) -> const T * { return delta; }, delta);
    if constexpr (LAST) {
      const double us = us0 + static_cast<double>(ds);
      if (i >= 0) U[s * n + i] = us;
      double u[4];
#pragma unroll
      for (int v = 0; v < 4; ++v) u[v] = __shfl_sync(0xffffffffu, us, v, 4);
      T rec[kBase];
      base_record(P, u, rec);
      if (i >= 0 && s < 3) {
        T part[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) part[v] = s == 0 ? rec[v] : s == 1 ? rec[4 + v] : rec[8 + v];
        vstore<T, 4>(base_next + static_cast<size_t>(i) * kBase + 4 * s, part);
      }
    }
  }
  pdl_exit();
}

// ---- the partitioned sweep (CGKS_SWEEP_PARTITIONED) ----
// One launch is one sweep of Algorithm 1 -- a forward pass over the
// colours, then a backward pass -- over every partition at once.  A
// thread-block cluster owns one partition: its CTAs share out each
// colour's cells of the partition, and a cluster barrier (release /
// acquire at cluster scope) separates consecutive colours, so a cell sees
// the increments its partition's earlier colours just wrote to delta_out
// (read through L2).  Neighbours in other partitions, and cells of this
// partition not yet relaxed in this sweep, are read from delta_in, the
// increments at the start of the sweep: partitions exchange once per
// sweep, lagged, like the paper's threads.  Every cell of every partition
// is written to delta_out.  The colour C-1 ending the forward pass is not
// relaxed again at the start of the backward pass: with its inputs
// unchanged it would recompute the same values.
constexpr int kPartBlock = 256;        // threads per CTA: one cell per thread and pass
constexpr int kPartCluster = 8;        // CTAs per partition (portable cluster size)
constexpr int kMaxPartColours = 16;
// Lanes per cell, from the longest run of cells that one colour has in a
// partition.  A cluster takes 2,048 cells a pass with one lane and 512 with
// four, which need half the registers (twice the clusters at once) and half
// the chain; past two to three such passes one lane is the shorter.  us per
// V-cycle, one / four lanes: FP64 runs of 127 cells 5504 / 1921, 1,020
// 1714 / 1306, 1,365 738 / 779, 2,000 1290 / 1406 (8,192 cells for the third,
// else 57,344); mixed 1415 / 487, 424 / 357, 319 / 297, 330 / 344 (18,432 for
// the last).
template <typename T> int part_lanes(int run) { return run <= (is_f32<T>() ? 1536 : 1280) ? 4 : 1; }

__device__ __forceinline__ unsigned cluster_ctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_nctarank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// every thread of every CTA of the cluster; orders the global writes before
// it (release) before the reads after it (acquire), cluster scope
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// ptab [Q][C][2]: first and end cell (internal index) of colour c in
// partition q; C colours
template <typename T, int LANES>
__global__ void __launch_bounds__(kPartBlock) k_sweep_part(MeshT<T> m, ParamsT<T> P, const int *__restrict__ ptab,
                                                           int C, const T *base,
                                                           const T *Rk, const T *invD,
                                                           const T *lamS,
                                                           const T *delta_in, T *delta_out) {
  __shared__ int sb[kMaxPartColours], se[kMaxPartColours];
  const unsigned K = cluster_nctarank(), rank = cluster_ctarank();
  const int q = static_cast<int>(blockIdx.x / K);
  if (static_cast<int>(threadIdx.x) < C) {
    sb[threadIdx.x] = ptab[2 * (q * C + threadIdx.x)];
    se[threadIdx.x] = ptab[2 * (q * C + threadIdx.x) + 1];
  }
  __syncthreads();
  pdl_enter();
  const int steps = 2 * C - 1;
  for (int step = 0; step < steps; ++step) {
    const bool fwd = step < C;
    const int c = fwd ? step : 2 * C - 2 - step;
    const int b = sb[c], e = se[c];
    // the increments of j: this sweep's where its colour is done, else those at its start
    auto del_of = [&](int j) -> const T * {
      const int cj = m.ccol[j];
      const bool fresh = cj < C && j >= sb[cj] && j < se[cj] && (!fwd || cj < c);
      return fresh ? delta_out : delta_in;
    };
    constexpr int kCells = kPartBlock / LANES;   // of a CTA's pass
    // (LANES == 4: the 8 cells of a warp iterate together)
    const int lead = static_cast<int>(LANES == 1 ? threadIdx.x : threadIdx.x / 32 * 8);
    for (int i0 = b + static_cast<int>(rank) * kCells + lead; i0 < e; i0 += static_cast<int>(K) * kCells) {
      if constexpr (LANES == 1) {
        SlotGeo<T> g[kMaxFace];
#pragma unroll
        for (int k = 0; k < kMaxFace; ++k) g[k] = slot_geo(m, i0, k);
        T d[4];
        sweep_cell<T, true>(m, P.gamma, g, i0, base, Rk, invD, lamS, del_of, delta_out, d);
      } else {
        const int at = i0 + static_cast<int>(threadIdx.x % 32 / 4), i = at < e ? at : -1, k = threadIdx.x % 4;
        sweep_quad<T, false, true>(m, P.gamma, slot_geo(m, i, k), i, k, base, Rk, invD, lamS, del_of, delta_out);
      }
    }
    if (step + 1 < steps) cluster_sync();
  }
  pdl_exit();
}

// K9: prolongation W = W_p0 + (U - W_p0) (Section 3, step 5), density
// residual against the state at the start of the cycle, state check.
template <typename TF>
__global__ void __launch_bounds__(kCellBlock) k_prolong(MeshT<double> m, ParamsT<double> P, double *W,
                                                        const double *Wp0, const double *U,
                                                        int *status, double *partial,
                                                        TF *Wm) {
  pdl_enter();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = m.nc;
  double num = 0.0, den = 0.0;
  const int sid = i < n ? m.csid[i] : -1;
  if (i < n) {
    double w[4];
    double old_rho = W[i];
    for (int v = 0; v < 4; ++v) {
      double wp = Wp0[v * n + i];
      w[v] = wp + (U[v * n + i] - wp);
      W[v * n + i] = w[v];
      if (Wm) Wm[v * n + i] = narrow<TF>(w[v]);
    }
    if (sid >= 0) {
      if (!state_ok(w)) atomicOr(&status[sid], kBadState);
      num = fabs(w[0] - old_rho);
      den = old_rho;
    }
  }
  block_sum2(num, den, &partial[2 * blockIdx.x]);
  pdl_exit();
}

// Caller AoS order <-> internal SoA order for the n cells of one solve
// starting at internal offset off (perm: internal within solve -> caller).
__global__ void k_gather_state(int ns, int off, int N, const int *__restrict__ perm, const double *__restrict__ Wa,
                               const double *__restrict__ Wxa, double *__restrict__ W, double *__restrict__ Wx,
                               float *__restrict__ W32, float *__restrict__ Wx32) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= ns) return;
  int c = perm[k], i = off + k;
  for (int v = 0; v < 4; ++v) {
    double w = Wa[4 * c + v];
    W[v * N + i] = w;
    if (W32) W32[v * N + i] = static_cast<float>(w);
  }
  for (int q = 0; q < 8; ++q) {
    double g = Wxa ? Wxa[8 * c + q] : 0.0;
    Wx[q * N + i] = g;
    if (Wx32) Wx32[q * N + i] = static_cast<float>(g);
  }
}
__global__ void k_scatter_state(int ns, int off, int N, const int *__restrict__ perm, const double *__restrict__ W,
                                const double *__restrict__ Wx, double *__restrict__ Wa, double *__restrict__ Wxa) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= ns) return;
  int c = perm[k], i = off + k;
  if (Wa) for (int v = 0; v < 4; ++v) Wa[4 * c + v] = W[v * N + i];
  if (Wxa) for (int q = 0; q < 8; ++q) Wxa[8 * c + q] = Wx[q * N + i];
}
// The momentum fluxes (F0) of the listed faces: [n][2] in a row.  Copying every
// face's run of 16 values to the host instead took most of a call: ms for a wall
// of a 500,000-cell cavity, FP64 10.9 -> 2.6, mixed 3.2 -> 0.7.
template <typename T>
__global__ void k_pack_traction(int n, int off, const int *list, const T *FA, T *out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const T *F0 = FA + static_cast<size_t>(off + list[k]) * kFO;
  out[2 * k] = F0[1];
  out[2 * k + 1] = F0[2];
}
// Inert cells (padding, free space of a batch): no faces, no neighbours,
// no solve, no colour, and a valid uniform state so that the arithmetic the
// cell kernels still do for them stays finite.
__global__ void k_clear_cells(int c0, int c1, int N, int *__restrict__ csid, unsigned char *__restrict__ ccol,
                              int *__restrict__ cface, int *__restrict__ cnbr, double *__restrict__ W,
                              double *__restrict__ Wx, double *__restrict__ Wn, double *__restrict__ Ws,
                              double *__restrict__ Wxs, float *__restrict__ W32, float *__restrict__ Wx32,
                              float *__restrict__ Wn32, float *__restrict__ Ws32, float *__restrict__ Wxs32) {
  const int i = c0 + blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= c1) return;
  csid[i] = -1;
  ccol[i] = 255;
  for (int s = 0; s < kMaxFace; ++s) { cface[s * N + i] = kNoFace; cnbr[s * N + i] = -1; }
  const double w[4] = { 1.0, 0.0, 0.0, 2.5 };
  for (int v = 0; v < 4; ++v) {
    W[v * N + i] = w[v]; Wn[v * N + i] = w[v]; Ws[v * N + i] = w[v];
    if (W32) { W32[v * N + i] = static_cast<float>(w[v]); Wn32[v * N + i] = static_cast<float>(w[v]);
               Ws32[v * N + i] = static_cast<float>(w[v]); }
  }
  for (int q = 0; q < 8; ++q) {
    Wx[q * N + i] = 0.0; Wxs[q * N + i] = 0.0;
    if (Wx32) { Wx32[q * N + i] = 0.0f; Wxs32[q * N + i] = 0.0f; }
  }
}

}  // namespace kern
}  // namespace cgks
