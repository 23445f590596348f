// Device-side gas-kinetic physics of the compact GKS, 2-D (Sections 2.2-2.3
// and 3 of Ji, Shyy & Xu, arXiv:2109.09965).
//
// All routines work in the local face frame (normal n, tangent t = (-ny, nx))
// on conservative variables (rho, rho*u_n, rho*u_t, rho*E) and their
// derivatives along n and t.  Moments of the Maxwellian are normalised by
// rho: <u^a> by the standard recurrence, <xi^2> = K/(2 lambda),
// <xi^4> = K(K+2)/(4 lambda^2).  The micro-slope solve <a psi> = b uses its
// closed form.  Templated on the arithmetic type so the same code serves
// the FP64 path and the FP32 flux of the mixed path.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace cgks {
namespace dev {

constexpr int NV = 4;

// the library's, in the FP32 forms (the FP64 ones have their own arithmetic below)
__device__ __forceinline__ float d_erfc(float x) { return erfcf(x); }
__device__ __forceinline__ float d_exp(float x) { return expf(x); }
__device__ __forceinline__ float d_expm1(float x) { return expm1f(x); }
__device__ __forceinline__ float d_sqrt(float x) { return sqrtf(x); }
__device__ __forceinline__ float d_rsqrt(float x) { return rsqrtf(x); }

// a b and a b + c d with the roundings spelled out in FP64, so that code
// compiled into two kernels gives the same bits in both.  In FP32 they are what
// the compiler makes of them (the mixed path's results keep those roundings):
// that it fuses the low-level flux alike in the two kernels that hold it is
// checked, not ensured (test_merged_and_separate_right_hand_sides_round_alike).
__device__ __forceinline__ float prod(float a, float b) { return a * b; }
__device__ __forceinline__ double prod(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float dot2(float a, float b, float c, float d) { return a * b + c * d; }
__device__ __forceinline__ double dot2(double a, double b, double c, double d) { return fma(c, d, __dmul_rn(a, b)); }
// a b + c, one rounding
__device__ __forceinline__ float mad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double mad(double a, double b, double c) { return __fma_rn(a, b, c); }

// Rotate a conservative vector between global and face frames.
template <typename T>
__device__ __forceinline__ void rot_in(T nx, T ny, const T g[NV], T l[NV]) {
  l[0] = g[0];
  l[1] = dot2(g[1], nx, g[2], ny);
  l[2] = dot2(-g[1], ny, g[2], nx);
  l[3] = g[3];
}
template <typename T>
__device__ __forceinline__ void rot_out(T nx, T ny, const T l[NV], T g[NV]) {
  g[0] = l[0];
  g[1] = dot2(l[1], nx, -l[2], ny);
  g[2] = dot2(l[1], ny, l[2], nx);
  g[3] = l[3];
}

// Constants of the kinetic model with K internal degrees of freedom,
// computed once on the host: c2K = 2/(K+2), c4K = 4/(K+2), hN = (K+2)/2,
// sq2g = sqrt(2 gamma), iN = K+2 = 2/(gamma-1) where it is a whole number up to
// 64, else 0.
template <typename T>
struct KC {
  T K, c2K, c4K, hN, sq2g;
  int iN;
};
constexpr double kInvSqrtPi = 0.56418958354775628694807945156;

// Maxwellian of local-frame conservative W: rho, 1/rho, U, V, lambda and
// 1/(2 lambda).  Two divisions; everything downstream multiplies.
template <typename T>
struct Maxw {
  T rho, ir, U, V, lam, i2l;
};
template <typename T>
__device__ __forceinline__ Maxw<T> maxw(const T W[NV], T c2K) {
  // lambda = (K+2) rho / (4 (rho E - rho |U|^2 / 2)),  c2K = 2 / (K+2)
  Maxw<T> g;
  g.rho = W[0];
  g.ir = T(1) / W[0];
  g.U = W[1] * g.ir;
  g.V = W[2] * g.ir;
  T eps = W[3] - T(0.5) * g.rho * (g.U * g.U + g.V * g.V);
  g.i2l = c2K * eps * g.ir;
  g.lam = T(0.5) / g.i2l;
  return g;
}

// Reciprocal and reciprocal square root.  GB300 issues two FP64 lanes per
// clock per SM, so the number of FP64 instructions is what an FP64 kernel
// costs: the FP64 forms take the hardware's estimate (20 mantissa bits; e below is
// at most 2^-19.9 for 1/x and 2^-19.0 for 1/sqrt(x), measured) and one third-order
// step of Newton's family (Householder's iteration), which leaves e^3 = 2^-59.8 and
// 5/16 e^3 = 2^-58.7: with the roundings, relative errors below 1.1 and 2 units
// (2^-53), where the IEEE quotient is correctly rounded.
//   1/x:        e = 1 - x r,    r <- r + r (e + e^2)             3 FP64
//   1/sqrt(x):  e = 1 - x r^2,  r <- r + r e (1/2 + 3/8 e)       5 FP64
// against 8-9 for the IEEE quotient and the library's rsqrt.  Normal
// arguments; zero, infinity and NaN give NaN or infinity (the state check
// marks them as it did).  FP32 keeps the library's.
__device__ __forceinline__ float d_rcp(float x) { return 1.0f / x; }
__device__ __forceinline__ double d_rcp(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}
__device__ __forceinline__ double d_rsqrt3(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

// sqrt(lambda) and 1/sqrt(pi lambda) of a Maxwellian with 1/(2 lambda) = i2l
__device__ __forceinline__ void sqrt_lambda(float i2l, float &sl, float &isp) {
  const float lam = 0.5f / i2l;
  sl = sqrtf(lam);
  isp = rsqrtf(lam) * static_cast<float>(kInvSqrtPi);
}
__device__ __forceinline__ void sqrt_lambda(double i2l, double &sl, double &isp) {
  const double t = 2.0 * i2l;
  sl = d_rsqrt3(t);
  isp = t * sl * kInvSqrtPi;
}

// The first two half-range moments, <1> = (1 + sgn erf(z)) / 2 and <u>, over
// u > 0 (sgn = +1) or u < 0 (-1), z = sl U.  In FP64, for |z| < 1 (normal Mach
// number below 1.19), erf(z) / (2 z) and exp(-z^2) come from polynomials in
// t = z^2, the interpolants at the Chebyshev nodes of [0, 1] (degrees 11 and
// 12; with the coefficients rounded to double relative errors 4e-17 and 1e-16,
// before the roundings of the evaluation): 24 FP64 instructions in place of about
// 90 of the library pair; beyond, and for NaN, the library's functions.  <1> is
// then 0.5 plus a product, exact to a few units of 2^-53 absolutely; where it is
// small (0.08 at |z| = 1) that is several units relative to itself, but the other
// side's share of the same sum is near 1.  FP32 keeps the library's: its
// arithmetic is not what the mixed path waits for.
__device__ __forceinline__ void half01(double U, double sl, double isp, int sgn, double &m0, double &m1) {
  const double z = sl * U, t = z * z;
  double ex;
  if (static_cast<unsigned>(__double2hiint(t)) < 0x3ff00000u) {
    double p = -3.8979494135010711208e-10, q = 1.2719039650810422692e-09;
    p = fma(p, t, 6.8600322733888428021e-09);  q = fma(q, t, -2.2905624278899245573e-08);
    p = fma(p, t, -8.1042419009358529508e-08); q = fma(q, t, 2.7213633679812669228e-07);
    p = fma(p, t, 8.2237123516586812051e-07);  q = fma(q, t, -2.7521178006932174539e-06);
    p = fma(p, t, -7.4623684537098301688e-06); q = fma(q, t, 2.4798998659720724886e-05);
    p = fma(p, t, 6.0276474524198539583e-05);  q = fma(q, t, -1.9841141919339012344e-04);
    p = fma(p, t, -4.2741629876948460403e-04); q = fma(q, t, 1.3888884549085944042e-03);
    p = fma(p, t, 2.6119888035582113661e-03);  q = fma(q, t, -8.3333332344813161057e-03);
    p = fma(p, t, -1.343308532161888518e-02);  q = fma(q, t, 4.1666666652193343912e-02);
    p = fma(p, t, 5.6418958354725031328e-02);  q = fma(q, t, -1.6666666666540416823e-01);
    p = fma(p, t, -1.8806319451591770219e-01); q = fma(q, t, 4.999999999999427302e-01);
    p = fma(p, t, 5.6418958354775628327e-01);  q = fma(q, t, -9.9999999999999897845e-01);
    ex = fma(q, t, 9.9999999999999999698e-01);
    m0 = fma(sgn > 0 ? z : -z, p, 0.5);
  } else {
    m0 = 0.5 * erfc(sgn > 0 ? -z : z);
    ex = exp(-t);
  }
  const double e = 0.5 * (ex * isp);
  m1 = fma(U, m0, sgn > 0 ? e : -e);
}

// Half-range moments <u^k>, k = 0..KMAX, over u > 0 (sgn = +1) or u < 0
// (-1), of the Maxwellian with mean U, 1/(2 lambda) = i2l, sqrt(lambda) = sl
// and 1/sqrt(pi lambda) = isp.
template <typename T, int KMAX>
__device__ __forceinline__ void half_moments(T U, T i2l, T sl, T isp, int sgn, T mu[KMAX + 1]) {
  if constexpr (std::is_same<T, double>::value) {
    half01(U, sl, isp, sgn, mu[0], mu[1]);
  } else {
    T z = sl * U;
    T e = d_exp(-z * z) * isp;
    if (sgn > 0) {
      mu[0] = T(0.5) * d_erfc(-z);
      mu[1] = U * mu[0] + T(0.5) * e;
    } else {
      mu[0] = T(0.5) * d_erfc(z);
      mu[1] = U * mu[0] - T(0.5) * e;
    }
  }
#pragma unroll
  for (int k = 2; k <= KMAX; ++k) mu[k] = U * mu[k - 1] + T(k - 1) * i2l * mu[k - 2];
}

// Full-range moment tables of the equilibrium used by the flux.
template <typename T>
struct Mom {
  T mu[7], mv[7], x2, x4;   // <u^k>, <v^k>, <xi^2>, <xi^4>
};
template <typename T>
__device__ __forceinline__ void full_moments(const Maxw<T> &g, T K, Mom<T> &m) {
  const T i2l = g.i2l;
  m.mu[0] = T(1); m.mu[1] = g.U;
  m.mv[0] = T(1); m.mv[1] = g.V;
#pragma unroll
  for (int k = 2; k < 7; ++k) {
    m.mu[k] = g.U * m.mu[k - 1] + T(k - 1) * i2l * m.mu[k - 2];
    m.mv[k] = g.V * m.mv[k - 1] + T(k - 1) * i2l * m.mv[k - 2];
  }
  m.x2 = K * i2l;
  m.x4 = K * (K + T(2)) * i2l * i2l;
}

// <u^a v^b xi^(2d) * s>, slope s = s0 + s1 u + s2 v + s3 (u^2+v^2+xi^2)/2
template <typename T>
__device__ __forceinline__ T mslope(const Mom<T> &m, int a, int b, int d, const T s[NV]) {
  const T xd = d == 0 ? T(1) : (d == 1 ? m.x2 : m.x4);
  const T xd1 = d == 0 ? m.x2 : m.x4;
  T r = s[0] * m.mu[a] * m.mv[b] * xd + s[1] * m.mu[a + 1] * m.mv[b] * xd + s[2] * m.mu[a] * m.mv[b + 1] * xd;
  r += T(0.5) * s[3] * (m.mu[a + 2] * m.mv[b] * xd + m.mu[a] * m.mv[b + 2] * xd + m.mu[a] * m.mv[b] * xd1);
  return r;
}
// vector <u^a v^b s psi>
template <typename T>
__device__ __forceinline__ void gpsi(const Mom<T> &m, int a, int b, const T s[NV], T out[NV]) {
  out[0] = mslope(m, a, b, 0, s);
  out[1] = mslope(m, a + 1, b, 0, s);
  out[2] = mslope(m, a, b + 1, 0, s);
  out[3] = T(0.5) * (mslope(m, a + 2, b, 0, s) + mslope(m, a, b + 2, 0, s) + mslope(m, a, b, 1, s));
}

// Closed-form solution of <s psi> = b (b already divided by rho), 2-D,
// K internal degrees of freedom.  q = U^2 + V^2 + (K+2)/(2 lambda),
// tl = 2 lambda, l2 = 4 lambda^2 / (K+2): shared by the three solves.
template <typename T>
struct SlopeSolver {
  T U, V, q, tl, l2;
};
template <typename T>
__device__ __forceinline__ SlopeSolver<T> slope_solver(const Maxw<T> &g, const KC<T> &kc) {
  SlopeSolver<T> S;
  S.U = g.U; S.V = g.V;
  S.q = g.U * g.U + g.V * g.V + (kc.K + T(2)) * g.i2l;
  S.tl = T(2) * g.lam;
  S.l2 = kc.c4K * g.lam * g.lam;
  return S;
}
template <typename T>
__device__ __forceinline__ void micro_slope(const SlopeSolver<T> &S, const T b[NV], T s[NV]) {
  T R4 = T(2) * b[3] - S.q * b[0];
  T R3 = b[2] - S.V * b[0];
  T R2 = b[1] - S.U * b[0];
  s[3] = S.l2 * (R4 - T(2) * S.U * R2 - T(2) * S.V * R3);
  s[2] = S.tl * R3 - S.V * s[3];
  s[1] = S.tl * R2 - S.U * s[3];
  s[0] = b[0] - S.U * s[1] - S.V * s[2] - T(0.5) * s[3] * S.q;
}

// Smooth gas-kinetic flux at one Gauss point, Eq. (2nd-smooth-flux), by raw
// moments in the face frame: the FP32 form of the 2-D mixed path, whose
// results it keeps (a flux rounded differently moves the FP32 gradients by as
// much as their own error); the FP64 form is gks_smooth.
//   f = g^c - tau (a_n u + a_t v + A) g^c + A g^c t,   tau = mu / p^c
// with W^c from the half-range moments of g^l (u>0) and g^r (u<0), the
// equilibrium slopes from the mean of the side derivatives plus, along n,
// ajump * (W^r - W^l) with ajump = alpha / delta.  Inputs and outputs in
// the local frame: F0 + t F1 = flux, Wc + t Wt = interface state.
template <typename T>
__device__ __forceinline__ void gks_point_local(const KC<T> &kc, T mu_visc, T ajump,
                                                const T Wl[NV], const T Wr[NV],
                                                const T dnl[NV], const T dtl[NV],
                                                const T dnr[NV], const T dtr[NV],
                                                T F0[NV], T F1[NV], T Wc[NV], T Wt[NV]) {
  const T K = kc.K, c2K = kc.c2K;
  Maxw<T> gl = maxw(Wl, c2K), gr = maxw(Wr, c2K);
  T ml[3], mr[3];
  half_moments<T, 2>(gl.U, gl.i2l, d_sqrt(gl.lam), d_rsqrt(gl.lam) * T(kInvSqrtPi), +1, ml);
  half_moments<T, 2>(gr.U, gr.i2l, d_sqrt(gr.lam), d_rsqrt(gr.lam) * T(kInvSqrtPi), -1, mr);
  T el = gl.V * gl.V + (K + T(1)) * gl.i2l;
  T er = gr.V * gr.V + (K + T(1)) * gr.i2l;
  Wc[0] = gl.rho * ml[0] + gr.rho * mr[0];
  Wc[1] = gl.rho * ml[1] + gr.rho * mr[1];
  Wc[2] = gl.rho * ml[0] * gl.V + gr.rho * mr[0] * gr.V;
  Wc[3] = gl.rho * T(0.5) * (ml[2] + ml[0] * el) + gr.rho * T(0.5) * (mr[2] + mr[0] * er);
  Maxw<T> gc = maxw(Wc, c2K);
  Mom<T> m;
  full_moments(gc, K, m);
  SlopeSolver<T> SS = slope_solver(gc, kc);
  T bn[NV], bt[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    T dn = T(0.5) * (dnl[v] + dnr[v]) + ajump * (Wr[v] - Wl[v]);
    bn[v] = dn * gc.ir;
    bt[v] = T(0.5) * (dtl[v] + dtr[v]) * gc.ir;
  }
  T an[NV], at[NV], A[NV], bA[NV], g1[NV], g2[NV];
  micro_slope(SS, bn, an);
  micro_slope(SS, bt, at);
  gpsi(m, 1, 0, an, g1);
  gpsi(m, 0, 1, at, g2);
#pragma unroll
  for (int v = 0; v < NV; ++v) bA[v] = -(g1[v] + g2[v]);
  micro_slope(SS, bA, A);
  T tau = mu_visc * SS.tl * gc.ir;          // mu / p^c, p^c = rho / (2 lambda)
  T gAu[NV], gA[NV], gn2[NV], gtuv[NV];
  gpsi(m, 1, 0, A, gAu);
  gpsi(m, 0, 0, A, gA);
  gpsi(m, 2, 0, an, gn2);
  gpsi(m, 1, 1, at, gtuv);
  T feq[NV] = { m.mu[1], m.mu[2], m.mu[1] * gc.V,
                T(0.5) * (m.mu[3] + m.mu[1] * m.mv[2] + m.mu[1] * m.x2) };
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    F0[v] = gc.rho * (feq[v] - tau * (gn2[v] + gtuv[v] + gAu[v]));
    F1[v] = gc.rho * gAu[v];
    Wt[v] = gc.rho * gA[v];
  }
}

// One side of a Gauss point in the face frame: its share of W^c (the
// half-range moments <psi> of its Maxwellian over u > 0 for sgn = +1, u < 0
// for -1), added to or stored in Wc.
template <typename T, bool ADD>
__device__ __forceinline__ void half_state(const KC<T> &kc, const T W[NV], int sgn, T Wc[NV]) {
  const T ir = d_rcp(W[0]);
  const T U = W[1] * ir, V = W[2] * ir;
  const T th = kc.c2K * ((W[3] - T(0.5) * (W[1] * U + W[2] * V)) * ir);   // 1 / (2 lambda)
  T sl, isp, m[2];
  sqrt_lambda(th, sl, isp);
  half_moments<T, 1>(U, th, sl, isp, sgn, m);
  const T a = W[0] * m[0], b = W[0] * m[1];
  const T E = T(0.5) * (b * U + a * (V * V + (kc.K + T(2)) * th));
  if (ADD) { Wc[0] += a; Wc[1] += b; Wc[2] += a * V; Wc[3] += E; }
  else { Wc[0] = a; Wc[1] = b; Wc[2] = a * V; Wc[3] = E; }
}

// Smooth gas-kinetic flux at one Gauss point, Eq. (2nd-smooth-flux):
//   f = g^c - tau (a_n u + a_t v + A) g^c + A g^c t,   tau = mu / p^c,
// for the interface state W^c = Wc and its spatial derivatives G[j] along
// x and y, in the global frame (n the face normal).  F0 + t F1 = flux,
// Wc + t Wt = interface state.
// The moments are taken about the mean velocity, where they close: with
// theta = 1/(2 lambda) and N = K + 2 degrees of freedom the micro-slope of a
// direction is the one of (rho, U, theta),
//   a = d rho / rho + c.dU / theta + ((c^2 + xi^2) / theta - N) d theta / (2 theta),
// the condition <A + a.u> = 0 gives A as the same expression of the Euler
// time derivatives
//   d_t rho = -rho (U.grad rho / rho + div U), d_t U = -U.grad U - grad p / rho,
//   d_t theta = -U.grad theta - (2/N) theta div U,
// so that <A psi> and <u A psi> are the time derivatives of the conservative
// variables and of the Euler flux, and -tau <u (a.u + A) psi> is the viscous
// traction mu (dU/dn + grad U_n - (2/N) div U n) with the heat flux
// mu (N/2 + 1) d theta / dn.  About 110 FP64 instructions where the tables
// of raw moments took about 650.
//
// gks_centre: Fe the Euler flux of Wc, F1 = <u A psi> and Wt = <A psi> (times
// rho), Hv the viscous part per unit viscosity.
__device__ __forceinline__ void gks_centre(const KC<double> &kc, double nx, double ny, const double Wc[NV],
                                           const double G[2][NV], bool visc, double Fe[NV], double F1[NV],
                                           double Wt[NV], double Hv[NV], double &p) {
  using T = double;
  const T c2 = kc.c2K, hN = kc.hN;
  const T rho = Wc[0], ir = d_rcp(rho);
  const T u = Wc[1] * ir, v = Wc[2] * ir, E = Wc[3] * ir;
  const T th = c2 * (E - T(0.5) * (u * u + v * v)), H = E + th;
  T r[2], ux[2], vx[2], Tx[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    r[j] = G[j][0] * ir;
    ux[j] = G[j][1] * ir - u * r[j];
    vx[j] = G[j][2] * ir - v * r[j];
    Tx[j] = c2 * (G[j][3] * ir - E * r[j] - u * ux[j] - v * vx[j]);
  }
  const T div = ux[0] + vx[1];
  const T rt = -(u * r[0] + v * r[1] + div);
  const T ut = -(u * ux[0] + v * ux[1] + th * r[0] + Tx[0]);
  const T vt = -(u * vx[0] + v * vx[1] + th * r[1] + Tx[1]);
  const T Tt = -(u * Tx[0] + v * Tx[1] + c2 * th * div);
  const T un = u * nx + v * ny, mn = rho * un;
  p = rho * th;
  const T a0 = rho * rt, ek = u * ut + v * vt, ei = ek + hN * Tt;
  Wt[0] = a0;
  Wt[1] = u * a0 + rho * ut;
  Wt[2] = v * a0 + rho * vt;
  Wt[3] = E * a0 + rho * ei;
  const T mt = Wt[1] * nx + Wt[2] * ny, pt = th * a0 + rho * Tt;
  F1[0] = mt;
  F1[1] = u * mt + mn * ut + nx * pt;
  F1[2] = v * mt + mn * vt + ny * pt;
  F1[3] = H * mt + mn * (ei + Tt);
  Fe[0] = mn;
  Fe[1] = mn * u + p * nx;
  Fe[2] = mn * v + p * ny;
  Fe[3] = mn * H;
  if (visc) {
    const T s = ux[1] + vx[0], d = c2 * div;
    Hv[0] = T(0);
    Hv[1] = (T(2) * ux[0] - d) * nx + s * ny;
    Hv[2] = s * nx + (T(2) * vx[1] - d) * ny;
    Hv[3] = u * Hv[1] + v * Hv[2] + (hN + T(1)) * (Tx[0] * nx + Tx[1] * ny);
  }
}
__device__ __forceinline__ void gks_smooth(const KC<double> &kc, double mu_visc, double nx, double ny,
                                           const double Wc[NV], const double G[2][NV], double F0[NV], double F1[NV],
                                           double Wt[NV]) {
  double Hv[NV], p;
  gks_centre(kc, nx, ny, Wc, G, mu_visc != 0.0, F0, F1, Wt, Hv, p);
  if (mu_visc != 0.0)
#pragma unroll
    for (int v = 1; v < NV; ++v) F0[v] -= mu_visc * Hv[v];
}

// ---------------- full flux, Eq. (2nd-flux) ----------------
// Moment table of one Maxwellian whose u-moments are taken over a half
// range (sgn = +1: u > 0, -1: u < 0); v and xi moments full.
template <typename T>
__device__ __forceinline__ void half_table(const Maxw<T> &g, T K, int sgn, Mom<T> &m) {
  half_moments<T, 6>(g.U, g.i2l, d_sqrt(g.lam), d_rsqrt(g.lam) * T(kInvSqrtPi), sgn, m.mu);
  m.mv[0] = T(1); m.mv[1] = g.V;
#pragma unroll
  for (int k = 2; k < 7; ++k) m.mv[k] = g.V * m.mv[k - 1] + T(k - 1) * g.i2l * m.mv[k - 2];
  m.x2 = K * g.i2l;
  m.x4 = K * (K + T(2)) * g.i2l * g.i2l;
}

// Spatial micro-slopes of a Maxwellian from its normal / tangential
// derivatives (dn, dt), and the temporal one from <A + a_n u + a_t v> = 0.
template <typename T>
__device__ __forceinline__ void maxw_slopes(const Maxw<T> &g, const Mom<T> &mf, const KC<T> &kc, const T dn[NV],
                                            const T dt[NV], T an[NV], T at[NV], T A[NV]) {
  SlopeSolver<T> SS = slope_solver(g, kc);
  T b[NV], g1[NV], g2[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) b[v] = dn[v] * g.ir;
  micro_slope(SS, b, an);
#pragma unroll
  for (int v = 0; v < NV; ++v) b[v] = dt[v] * g.ir;
  micro_slope(SS, b, at);
  gpsi(mf, 1, 0, an, g1);
  gpsi(mf, 0, 1, at, g2);
#pragma unroll
  for (int v = 0; v < NV; ++v) b[v] = -(g1[v] + g2[v]);
  micro_slope(SS, b, A);
}

// rho-weighted moments of one piece of the distribution: flux moments
// Q = (<u psi>, <u (a_n u + a_t v) psi>, <u A psi>) and state moments
// P = (<psi>, <(a_n u + a_t v) psi>, <A psi>).
template <typename T>
__device__ __forceinline__ void piece(T rho, const Mom<T> &m, const T an[NV], const T at[NV], const T A[NV],
                                      T Q[3][NV], T P[3][NV]) {
  const T one[NV] = { T(1), T(0), T(0), T(0) };
  T a[NV], b[NV];
  gpsi(m, 1, 0, one, a);
#pragma unroll
  for (int v = 0; v < NV; ++v) Q[0][v] = rho * a[v];
  gpsi(m, 2, 0, an, a);
  gpsi(m, 1, 1, at, b);
#pragma unroll
  for (int v = 0; v < NV; ++v) Q[1][v] = rho * (a[v] + b[v]);
  gpsi(m, 1, 0, A, a);
#pragma unroll
  for (int v = 0; v < NV; ++v) Q[2][v] = rho * a[v];
  gpsi(m, 0, 0, one, a);
#pragma unroll
  for (int v = 0; v < NV; ++v) P[0][v] = rho * a[v];
  gpsi(m, 1, 0, an, a);
  gpsi(m, 0, 1, at, b);
#pragma unroll
  for (int v = 0; v < NV; ++v) P[1][v] = rho * (a[v] + b[v]);
  gpsi(m, 0, 0, A, a);
#pragma unroll
  for (int v = 0; v < NV; ++v) P[2][v] = rho * a[v];
}

// Eq. (2nd-flux) with time coefficients (c1, c2, c3, e, te) applied to the
// equilibrium (X0), left (XL) and right (XR) pieces.
template <typename T>
__device__ __forceinline__ void full_sum(T c1, T c2, T c3, T e, T te, T tau, const T X0[3][NV], const T XL[3][NV],
                                         const T XR[3][NV], T out[NV]) {
#pragma unroll
  for (int v = 0; v < NV; ++v)
    out[v] = c1 * X0[0][v] + c2 * X0[1][v] + c3 * X0[2][v] +
             e * ((XL[0][v] + XR[0][v]) - tau * (XL[1][v] + XR[1][v]) - tau * (XL[2][v] + XR[2][v])) -
             te * (XL[1][v] + XR[1][v]);
}

// Full gas-kinetic flux at one Gauss point, Eq. (2nd-flux):
//   f = (1 - e) g^c + [(t + tau) e - tau] a^c.u g^c + (t - tau + tau e) A^c g^c
//     + e g^l [1 - (tau + t) a^l.u - tau A^l] H(u) + e g^r [...] (1 - H(u)),
// e = exp(-t / tau_n), tau = mu / p^c,
// tau_n = tau + c1 dt + c2 dt |p_l - p_r| / (p_l + p_r).
// Brought to the linear-in-time form of the time schemes through the time
// integrals over [0, dt] and [0, dt/2]: F0 dt + F1 dt^2/2 = Fhat(dt),
// F0 dt/2 + F1 dt^2/8 = Fhat(dt/2); the interface state W_p(t) = <psi f(t)>
// by the line Wc + t Wt through its values at dt/2 and dt.  Same frame and
// arguments as gks_point_local, plus dt and the two tau_n constants.
template <typename T>
__device__ void gks_full_point_local(const KC<T> &kc, T mu_visc, T ajump, T dt, T tc1, T tc2, const T Wl[NV],
                                     const T Wr[NV], const T dnl[NV], const T dtl[NV], const T dnr[NV],
                                     const T dtr[NV], T F0[NV], T F1[NV], T Wc[NV], T Wt[NV]) {
  const T K = kc.K, c2K = kc.c2K;
  Maxw<T> gl = maxw(Wl, c2K), gr = maxw(Wr, c2K);
  T Q0[3][NV], P0[3][NV], QL[3][NV], PL[3][NV], QR[3][NV], PR[3][NV];
  T anl[NV], atl[NV], Al[NV], anr[NV], atr[NV], Ar[NV];
  {
    Mom<T> mf;
    full_moments(gl, K, mf);
    maxw_slopes(gl, mf, kc, dnl, dtl, anl, atl, Al);
    full_moments(gr, K, mf);
    maxw_slopes(gr, mf, kc, dnr, dtr, anr, atr, Ar);
  }
  T W0[NV];
  {
    Mom<T> mh;
    half_table(gl, K, +1, mh);
    piece(gl.rho, mh, anl, atl, Al, QL, PL);
    half_table(gr, K, -1, mh);
    piece(gr.rho, mh, anr, atr, Ar, QR, PR);
  }
  // W^c: the collision of the particles of g^l moving right and g^r moving left
#pragma unroll
  for (int v = 0; v < NV; ++v) W0[v] = PL[0][v] + PR[0][v];
  Maxw<T> gc = maxw(W0, c2K);
  T an[NV], at[NV], A[NV];
  {
    Mom<T> m;
    full_moments(gc, K, m);
    T dn[NV], dtg[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      dn[v] = T(0.5) * (dnl[v] + dnr[v]) + ajump * (Wr[v] - Wl[v]);
      dtg[v] = T(0.5) * (dtl[v] + dtr[v]);
    }
    maxw_slopes(gc, m, kc, dn, dtg, an, at, A);
    piece(gc.rho, m, an, at, A, Q0, P0);
  }
  const T tau = mu_visc * T(2) * gc.lam * gc.ir;          // mu / p^c
  const T pl = gl.rho * gl.i2l, pr = gr.rho * gr.i2l;
  const T taun = tau + tc1 * dt + tc2 * dt * fabs(pl - pr) / (pl + pr);
  T Fd[NV], Fh[NV], Wd[NV], Wh[NV];
#pragma unroll 1
  for (int k = 0; k < 2; ++k) {
    const T t = k == 0 ? dt : T(0.5) * dt;
    // coefficient functions at t and their integrals over [0, t]
    const T e = taun > T(0) ? d_exp(-t / taun) : T(0);
    const T om = taun > T(0) ? -d_expm1(-t / taun) : T(1);
    const T ie = taun * om, ite = taun * taun * om - taun * t * e;
    full_sum(t - ie, ite + tau * ie - tau * t, T(0.5) * t * t - tau * t + tau * ie, ie, ite, tau, Q0, QL, QR,
             k == 0 ? Fd : Fh);
    full_sum(T(1) - e, (t + tau) * e - tau, t - tau + tau * e, e, t * e, tau, P0, PL, PR, k == 0 ? Wd : Wh);
  }
  const T idt = T(1) / dt;
#pragma unroll
  for (int v = 0; v < NV; ++v) {
    F0[v] = (T(4) * Fh[v] - Fd[v]) * idt;
    F1[v] = T(4) * (Fd[v] - T(2) * Fh[v]) * idt * idt;
    Wc[v] = T(2) * Wh[v] - Wd[v];
    Wt[v] = T(2) * (Wd[v] - Wh[v]) * idt;
  }
}

// ---- full flux, FP64 ----
// Eq. (2nd-flux) from moments taken about the mean velocity in the tangential
// and internal directions and over the half range of the normal one.  A
// micro-slope along direction j is
//   a_j = d_j rho / rho + c.d_j U / theta + ((c^2 + xi^2) / theta - N) phi_j / 2,
// phi_j = d_j theta / theta; given the normal velocity u, its mean over the
// other directions is the quadratic a0 + a1 u + a2 u^2 below, and the means of
// S = u a_n + v a_t (+ A) times 1, c_t and c_t^2 + xi^2 are the polynomials
// p, q and (N - 1) theta [p + phi_n u + phi_E] + 2 theta d_t U_t, so that only
// the half moments <u^k>, k <= 6, enter.  About 200 FP64 instructions a side
// where the moment tables took about 900.
struct CentralSlope {
  double a0, a1, a2;
};
__device__ __forceinline__ CentralSlope central_slope(double U, double ith, double r, double dU, double phi) {
  CentralSlope a;
  const double g = phi * ith;
  a.a2 = 0.5 * g;
  a.a1 = dU * ith - g * U;
  a.a0 = r - 0.5 * phi - U * (a.a1 + a.a2 * U);
  return a;
}
// One side's share of the rho-weighted moments, over u > 0 (sgn = +1) or u < 0
// (-1); X[k] for k = 0: 1, 1: a.u, 2: a.u + A, of psi (P) and u psi (Q).
// Returns the pressure.
template <bool ADD>
__device__ __forceinline__ double full_side(const KC<double> &kc, const double W[NV], const double dn[NV],
                                            const double dt[NV], int sgn, double P[3][NV], double Q[3][NV]) {
  const double c2 = kc.c2K, N1 = 2.0 * kc.hN - 1.0;
  const double rho = W[0], ir = d_rcp(rho);
  const double U = W[1] * ir, V = W[2] * ir, E = W[3] * ir;
  const double th = c2 * (E - 0.5 * (U * U + V * V)), ith = d_rcp(th);
  double sl, isp, mu[7];
  sqrt_lambda(th, sl, isp);
  half_moments<double, 6>(U, th, sl, isp, sgn, mu);
  // derivatives of ln rho, U, V, theta along n and t, and in time (Euler)
  const double rn = dn[0] * ir, rt = dt[0] * ir;
  const double Un = dn[1] * ir - U * rn, Ut = dt[1] * ir - U * rt;
  const double Vn = dn[2] * ir - V * rn, Vt = dt[2] * ir - V * rt;
  const double Tn = c2 * (dn[3] * ir - E * rn - U * Un - V * Vn), Tt = c2 * (dt[3] * ir - E * rt - U * Ut - V * Vt);
  const double div = Un + Vt;
  const double r_ = -(U * rn + V * rt + div);
  const double U_ = -(U * Un + V * Ut + th * rn + Tn);
  const double V_ = -(U * Vn + V * Vt + th * rt + Tt);
  const double T_ = -(U * Tn + V * Tt + c2 * th * div);
  const double fn = Tn * ith, ft = Tt * ith, f_ = T_ * ith;
  const CentralSlope an = central_slope(U, ith, rn, Un, fn), at = central_slope(U, ith, rt, Ut, ft),
                     aA = central_slope(U, ith, r_, U_, f_);
  const double Nt = N1 * th, e2 = V * V + Nt;
  // S = u a_n + v a_t
  const double p0 = V * at.a0 + Vt, p1 = an.a0 + V * at.a1, p2 = an.a1 + V * at.a2, p3 = an.a2;
  const double q2 = 0.5 * ft, q1 = Vn + Ut - ft * U, q0 = V * Vt + th * (rt + q2) - U * (Ut - q2 * U);
  const double k1 = Nt * fn, k0 = Nt * V * ft + 2.0 * th * Vt, kA = Nt * f_;
  double S[4], A[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    S[k] = p0 * mu[k] + p1 * mu[k + 1] + p2 * mu[k + 2] + p3 * mu[k + 3];
    A[k] = aA.a0 * mu[k] + aA.a1 * mu[k + 1] + aA.a2 * mu[k + 2];
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {   // weight 1 (P), u (Q)
    double(*X)[NV] = k == 0 ? P : Q;
    const double ct = q0 * mu[k] + q1 * mu[k + 1] + q2 * mu[k + 2], cA = V_ * mu[k];
    const double x0[NV] = { mu[k], mu[k + 1], V * mu[k], 0.5 * (mu[k + 2] + e2 * mu[k]) };
    const double x1[NV] = { S[k], S[k + 1], V * S[k] + ct,
                            0.5 * (S[k + 2] + e2 * S[k] + k1 * mu[k + 1] + k0 * mu[k]) + V * ct };
    const double x2[NV] = { A[k], A[k + 1], V * A[k] + cA, 0.5 * (A[k + 2] + e2 * A[k] + kA * mu[k]) + V * cA };
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const double s = x1[v] + x2[v];
      if (ADD) { X[0][v] += rho * x0[v]; X[1][v] += rho * x1[v]; X[2][v] += rho * s; }
      else { X[0][v] = rho * x0[v]; X[1][v] = rho * x1[v]; X[2][v] = rho * s; }
    }
  }
  return rho * th;
}
// Coefficients of Eq. (2nd-flux)'s pieces at time t for the flux integrated
// over [0, t] (fi) and the state at t (wi): equilibrium 1, viscous part, A;
// sides 1, a.u, a.u + A (see gks_full).  om = 1 - exp(-t / tau_n).
__device__ __forceinline__ void full_coeffs(double t, double tau, double taun, double om, double fi[6], double wi[6]) {
  const double e = 1.0 - om;
  const double ie = taun * om, ite = taun * (ie - t * e);
  const double c2 = ite + tau * ie - tau * t;
  fi[0] = t - ie;
  fi[1] = c2;
  fi[2] = 0.5 * t * t - tau * t + tau * ie - c2;
  fi[3] = ie;
  fi[4] = -ite;
  fi[5] = -tau * ie;
  const double te = t * e;
  wi[0] = om;
  wi[1] = 0.0;
  wi[2] = (t - tau + tau * e) - (te + tau * e - tau);
  wi[3] = e;
  wi[4] = -te;
  wi[5] = -tau * e;
}
// The linear-in-time form of the time schemes from the integrals over [0, dt]
// and [0, dt/2] (flux) and the values at dt/2 and dt (state): the six pieces'
// coefficients for F0, F1, Wc, Wt.
struct FullCoeffs {
  double F0[6], F1[6], Wc[6], Wt[6];
};
__device__ __forceinline__ void full_time_fit(double dt, double tau, double taun, FullCoeffs &C) {
  // exp(-dt / tau_n) from its value at dt/2: om(dt) = om (2 - om)
  const double omh = taun > 0.0 ? -expm1(-0.5 * dt / taun) : 1.0, omd = omh * (2.0 - omh);
  double fd[6], wd[6], fh[6], wh[6];
  full_coeffs(dt, tau, taun, omd, fd, wd);
  full_coeffs(0.5 * dt, tau, taun, omh, fh, wh);
  const double idt = d_rcp(dt), i2 = 4.0 * idt * idt;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    C.F0[k] = (4.0 * fh[k] - fd[k]) * idt;
    C.F1[k] = (fd[k] - 2.0 * fh[k]) * i2;
    C.Wc[k] = 2.0 * wh[k] - wd[k];
    C.Wt[k] = 2.0 * (wd[k] - wh[k]) * idt;
  }
}
// Full gas-kinetic flux at one Gauss point (see gks_full_point_local): side
// states and derivatives along n and t in the face frame, G the mean
// derivatives of the sides plus the jump term in the global frame; results in
// the global frame.
__device__ __forceinline__ void gks_full(const KC<double> &kc, double mu_visc, double dt, double tc1, double tc2,
                                         double nx, double ny, const double Wl[NV], const double Wr[NV],
                                         const double dnl[NV], const double dtl[NV], const double dnr[NV],
                                         const double dtr[NV], const double G[2][NV], double F0[NV], double F1[NV],
                                         double Wc[NV], double Wt[NV]) {
  double P[3][NV], Q[3][NV];
  const double pl = full_side<false>(kc, Wl, dnl, dtl, +1, P, Q);
  const double pr = full_side<true>(kc, Wr, dnr, dtr, -1, P, Q);
  double W0[NV], Fe[NV], X2[NV], Y2[NV], Hv[NV], p;
  rot_out(nx, ny, P[0], W0);
  gks_centre(kc, nx, ny, W0, G, true, Fe, X2, Y2, Hv, p);
  const double tau = mu_visc * d_rcp(p);
  const double taun = tau + tc1 * dt + tc2 * dt * fabs(pl - pr) * d_rcp(pl + pr);
  FullCoeffs C;
  full_time_fit(dt, tau, taun, C);
  auto combine = [&](const double c[6], const double X0[NV], const double *X1, const double Xc2[NV],
                     const double X[3][NV], double out[NV]) {
    double s[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) s[v] = c[3] * X[0][v] + c[4] * X[1][v] + c[5] * X[2][v];
    rot_out(nx, ny, s, out);
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      out[v] += c[0] * X0[v] + c[2] * Xc2[v];
      if (X1 && v > 0) out[v] += (c[1] * p) * X1[v];
    }
  };
  combine(C.F0, Fe, Hv, X2, Q, F0);
  combine(C.F1, Fe, Hv, X2, Q, F1);
  combine(C.Wc, W0, nullptr, Y2, P, Wc);
  combine(C.Wt, W0, nullptr, Y2, P, Wt);
}

// Cell-average primitives used by the low level (one set per cell and
// implicit step): rho, u, v, p, 1/(2 lambda), sqrt(lambda), 1/sqrt(pi
// lambda), sound speed c.
template <typename T>
struct Prim {
  T rho, u, v, p, i2l, sl, isp, c;
};
// c = sqrt(gamma p / rho); in FP64 from sqrt(lambda): p / rho = 1/(2 lambda)
__device__ __forceinline__ float sound_speed(const KC<float> &, float gamma, float p, float ir, float, float) {
  return sqrtf(gamma * p * ir);
}
__device__ __forceinline__ double sound_speed(const KC<double> &kc, double, double, double, double i2l, double sl) {
  return __dmul_rn(kc.sq2g, i2l * sl);
}
template <typename T>
__device__ __forceinline__ Prim<T> prim_of(const T W[NV], T gamma, const KC<T> &kc) {
  Prim<T> q;
  const T ir = d_rcp(W[0]);
  q.rho = W[0];
  q.u = prod(W[1], ir);
  q.v = prod(W[2], ir);
  const T eps = mad(T(-0.5) * q.rho, dot2(q.u, q.u, q.v, q.v), W[3]);
  q.p = prod(gamma - T(1), eps);
  q.i2l = kc.c2K * eps * ir;
  sqrt_lambda(q.i2l, q.sl, q.isp);
  q.c = sound_speed(kc, gamma, q.p, ir, q.i2l, q.sl);
  return q;
}

// First-order KFVS flux of two cell-average states, local frame, from
// their primitives (normal / tangential velocities already rotated).
template <typename T>
__device__ __forceinline__ void kfvs_prims(T K, T rl, T unl, T utl, T i2ll, T sll, T ispl,
                                           T rr, T unr, T utr, T i2lr, T slr, T ispr, T F[NV]) {
  T ml[4], mr[4];
  half_moments<T, 3>(unl, i2ll, sll, ispl, +1, ml);
  half_moments<T, 3>(unr, i2lr, slr, ispr, -1, mr);
  T el = utl * utl + (K + T(1)) * i2ll;
  T er = utr * utr + (K + T(1)) * i2lr;
  F[0] = rl * ml[1] + rr * mr[1];
  F[1] = rl * ml[2] + rr * mr[2];
  F[2] = rl * ml[1] * utl + rr * mr[1] * utr;
  F[3] = rl * T(0.5) * (ml[3] + ml[1] * el) + rr * T(0.5) * (mr[3] + mr[1] * er);
}

// F_n(U + dU) - F_n(U) of the Euler normal flux, written so that every
// term is proportional to the increment (no cancellation between two
// nearly equal fluxes): exact algebra, accurate to the working precision
// relative to the difference itself.  Base state: conservative W, velocity
// (u, v), pressure p; dW the increment; (nx, ny) the normal.
template <typename T>
__device__ __forceinline__ void euler_flux_delta(T gamma, const T W[NV], T u, T v, T p, const T dW[NV],
                                                 T nx, T ny, T dF[NV]) {
  const T rho = W[0], r1 = W[0] + dW[0];
  const T inv = T(1) / (rho * r1);
  const T mn = W[1] * nx + W[2] * ny, dmn = dW[1] * nx + dW[2] * ny;
  const T un = u * nx + v * ny;
  const T dun = (rho * dmn - mn * dW[0]) * inv;                       // (un)' - un
  const T un1 = un + dun;
  const T m2 = W[1] * W[1] + W[2] * W[2];
  const T dm2 = T(2) * (W[1] * dW[1] + W[2] * dW[2]) + dW[1] * dW[1] + dW[2] * dW[2];
  const T dke = T(0.5) * (rho * dm2 - m2 * dW[0]) * inv;              // d(|m|^2 / (2 rho))
  const T dp = (gamma - T(1)) * (dW[3] - dke);
  dF[0] = dmn;
  dF[1] = dW[1] * un1 + W[1] * dun + dp * nx;
  dF[2] = dW[2] * un1 + W[2] * dun + dp * ny;
  dF[3] = (dW[3] + dp) * un1 + (W[3] + p) * dun;
}

// ---------------- boundary ghost states (local frame) ----------------
// Wall velocity (wn, wt) and free stream (rho, un, ut, p) are given in the
// face frame of the boundary face.
template <typename T>
__device__ __forceinline__ void ghost_slip(const T W[NV], const T dn[NV], const T dt[NV],
                                           T Wg[NV], T dng[NV], T dtg[NV]) {
  // rho, rho u_t, rho E even across the wall, rho u_n odd
  Wg[0] = W[0]; Wg[1] = -W[1]; Wg[2] = W[2]; Wg[3] = W[3];
  dng[0] = -dn[0]; dng[1] = dn[1]; dng[2] = -dn[2]; dng[3] = -dn[3];
  dtg[0] = dt[0]; dtg[1] = -dt[1]; dtg[2] = dt[2]; dtg[3] = dt[3];
}

template <typename T>
__device__ __forceinline__ void ghost_noslip(T gamma, T wn, T wt, const T W[NV], const T dn[NV],
                                             const T dt[NV], T Wg[NV], T dng[NV], T dtg[NV]) {
  // rho, p even; u_g = 2 u_w - u  (derivatives: along n kept, along t flipped)
  T rho = W[0], ir = T(1) / rho;
  T u = W[1] * ir, v = W[2] * ir;
  T ke = T(0.5) * (u * u + v * v);
  T p = (gamma - T(1)) * (W[3] - rho * ke);
  T ug = T(2) * wn - u, vg = T(2) * wt - v;
  T keg = T(0.5) * (ug * ug + vg * vg);
  Wg[0] = rho; Wg[1] = rho * ug; Wg[2] = rho * vg; Wg[3] = p / (gamma - T(1)) + rho * keg;
  const T *D[2] = { dn, dt };
  T *G[2] = { dng, dtg };
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    T dr = D[b][0];
    T du = (D[b][1] - u * dr) * ir, dv = (D[b][2] - v * dr) * ir;
    T dp = (gamma - T(1)) * (D[b][3] - ke * dr - rho * (u * du + v * dv));
    T s = b == 0 ? T(-1) : T(1);   // scalars: normal derivative flips
    T drg = s * dr, dpg = s * dp;
    T dug = -s * du, dvg = -s * dv;  // velocity: tangential derivative flips
    G[b][0] = drg;
    G[b][1] = ug * drg + rho * dug;
    G[b][2] = vg * drg + rho * dvg;
    G[b][3] = dpg / (gamma - T(1)) + keg * drg + rho * (ug * dug + vg * dvg);
  }
}

// FP64: the mirror image of a wall as the linear map it is, in the global
// frame.  Pointwise, slip: m -> m - 2 n (n.m); no-slip, u -> 2 u_w - u at the
// same density and pressure: m -> 2 rho u_w - m, rho E -> rho E + 2 |u_w|^2 rho
// - 2 u_w.m.  A gradient flips along n, then maps like the state.  35 FP64
// instructions for one variable, 60 for all, where the way through the face
// frame and primitive variables took some 400 (3-D) with IEEE divisions: most
// of the reconstruction's time in small meshes, where every warp has a wall.
template <int ND>
struct WallMap {
  static constexpr int V = ND + 2;
  double n[ND], a[ND], e;   // normal; no-slip: 2 u_w, 2 |u_w|^2
  bool slip;
  __device__ __forceinline__ WallMap(int kind, const double *uw, const double *normal) : e(0.0) {
    slip = kind == CGKS_BC_SLIP;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      n[d] = normal[d];
      a[d] = 2.0 * uw[d];
      e = fma(0.5 * a[d], a[d], e);
    }
  }
  // the ghost's values
  __device__ __forceinline__ void apply(const double w[V], double g[V]) const {
    g[0] = w[0];
    g[V - 1] = w[V - 1];
    if (slip) {
      double mn = 0.0;
#pragma unroll
      for (int d = 0; d < ND; ++d) mn = fma(n[d], w[1 + d], mn);
#pragma unroll
      for (int d = 0; d < ND; ++d) g[1 + d] = fma(-2.0 * mn, n[d], w[1 + d]);
    } else {
      g[V - 1] = fma(e, w[0], g[V - 1]);
#pragma unroll
      for (int d = 0; d < ND; ++d) {
        g[1 + d] = fma(a[d], w[0], -w[1 + d]);
        g[V - 1] = fma(-a[d], w[1 + d], g[V - 1]);
      }
    }
  }
  __device__ __forceinline__ void apply_gradient(const double g[ND][V], double gg[ND][V]) const {
    double x[ND][V];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      double gn = 0.0;
#pragma unroll
      for (int d = 0; d < ND; ++d) gn = fma(n[d], g[d][v], gn);
#pragma unroll
      for (int d = 0; d < ND; ++d) x[d][v] = fma(-2.0 * gn, n[d], g[d][v]);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) apply(x[d], gg[d]);
  }
  // variable v of the ghost minus the cell's in b0, its gradient in b; W, Wx: the
  // cell's arrays with stride len
  __device__ __forceinline__ void one(int v, const double *W, const double *Wx, int len, double &b0,
                                      double b[ND]) const {
    double t[V], s[ND], w = 0.0, sn = 0.0;
#pragma unroll
    for (int k = 0; k < V; ++k) {   // row v of the map
      const bool mom = k >= 1 && k < V - 1;
      const double own = k == v ? 1.0 : 0.0;
      if (slip) {
        double nv = 0.0;
#pragma unroll
        for (int d = 0; d < ND; ++d) nv = v == 1 + d ? n[d] : nv;
        t[k] = mom ? fma(-2.0 * n[mom ? k - 1 : 0], nv, own) : own;
      } else if (k == 0) {
        t[k] = v == 0 ? 1.0 : e;
#pragma unroll
        for (int d = 0; d < ND; ++d) t[k] = v == 1 + d ? a[d] : t[k];
      } else {
        t[k] = mom ? (v == V - 1 ? -a[mom ? k - 1 : 0] : -own) : own;
      }
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) s[d] = 0.0;
    double wv = 0.0;
#pragma unroll
    for (int k = 0; k < V; ++k) {
      const double x = W[k * len];
      wv = k == v ? x : wv;
      w = fma(t[k], x, w);
#pragma unroll
      for (int d = 0; d < ND; ++d) s[d] = fma(t[k], Wx[(d * V + k) * len], s[d]);
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) sn = fma(n[d], s[d], sn);
#pragma unroll
    for (int d = 0; d < ND; ++d) b[d] = fma(-2.0 * sn, n[d], s[d]);
    b0 = w - wv;
  }
};

// FP64: the far-field state on the boundary from the Riemann invariants of the
// normal velocities ui, ue and sound speeds ci, ce (inside, free stream), where
// the flow is normally subsonic: velocity un and, from the side x the flow comes
// from, density and pressure rho_x y^N and p_x y^(N+2) with y = c_b / c_x and
// N = 2/(gamma - 1), the same as rho = (c_b^2 / (gamma s))^(1/(gamma-1)) with the
// entropy s = p_x / rho_x^gamma.  N is a whole number for the gases in use (5
// for gamma = 1.4), so no pow: three took about 500 FP64 instructions, a
// boundary face's warp four times as long as an inner one's.
struct FarState {
  bool out;      // flow leaves: entropy and tangential velocity of the inside
  double un, r, p;
};
__device__ __forceinline__ double d_sqrt3(double x) { return x * d_rsqrt3(x); }
// the same with the library's root for zero and everything out of the normal range
__device__ __forceinline__ double sqrt_fast(double x) { return x > 1e-290 && x < 1e290 ? d_sqrt3(x) : sqrt(x); }
__device__ __forceinline__ FarState far_state(const KC<double> &kc, double ri, double pi, double ui, double ci,
                                              double re, double pe, double ue, double ce) {
  const double N = 2.0 * kc.hN;
  const double Rp = mad(N, ci, ui), Rm = mad(-N, ce, ue);
  FarState f;
  f.un = 0.5 * (Rp + Rm);
  f.out = f.un >= 0.0;
  const double cb = fabs(0.25 * kc.c2K * (Rp - Rm));
  const double y = cb * d_rcp(f.out ? ci : ce);
  double yn;
  if (kc.iN > 0) {
    yn = 1.0;
    double b = y;
    for (int n = kc.iN; n; n >>= 1) {
      if (n & 1) yn *= b;
      b *= b;
    }
  } else {
    yn = pow(y, N);
  }
  f.r = (f.out ? ri : re) * yn;
  f.p = (f.out ? pi : pe) * (y * y) * yn;
  return f;
}
__device__ __forceinline__ void ghost_farfield(const KC<double> &kc, double gamma, double re, double une, double ute,
                                               double pe, const double W[NV], double Wg[NV]) {
  const double ri = W[0], ir = d_rcp(ri);
  const double uni = prod(W[1], ir), uti = prod(W[2], ir);
  const double pi = (gamma - 1.0) * mad(-0.5 * ri, dot2(uni, uni, uti, uti), W[3]);
  const double ci = d_sqrt3(gamma * pi * ir), ce = d_sqrt3(gamma * pe * d_rcp(re));
  double rb, unb, utb, pb;
  if (uni <= -ci) {
    rb = re; unb = une; utb = ute; pb = pe;
  } else if (uni >= ci) {
    rb = ri; unb = uni; utb = uti; pb = pi;
  } else {
    const FarState f = far_state(kc, ri, pi, uni, ci, re, pe, une, ce);
    rb = f.r; unb = f.un; pb = f.p;
    utb = f.out ? uti : ute;
  }
  Wg[0] = rb; Wg[1] = rb * unb; Wg[2] = rb * utb;
  Wg[3] = dot2(pb, kc.hN, 0.5 * rb, dot2(unb, unb, utb, utb));   // 1 / (gamma - 1) = N / 2
}

// 1-D Riemann invariants normal to the face between the interior state W
// and the free stream (rho_e, une, ute, pe); local frame.
template <typename T>
__device__ __forceinline__ void ghost_farfield(const KC<T> &, T gamma, T re, T une, T ute, T pe, const T W[NV],
                                               T Wg[NV]) {
  T ri = W[0], ir = T(1) / ri;
  T uni = W[1] * ir, uti = W[2] * ir;
  T pi = (gamma - T(1)) * (W[3] - T(0.5) * ri * (uni * uni + uti * uti));
  T ci = d_sqrt(gamma * pi / ri), ce = d_sqrt(gamma * pe / re);
  T rb, unb, utb, pb;
  if (uni <= -ci) {
    rb = re; unb = une; utb = ute; pb = pe;
  } else if (uni >= ci) {
    rb = ri; unb = uni; utb = uti; pb = pi;
  } else {
    T Rp = uni + T(2) * ci / (gamma - T(1));
    T Rm = une - T(2) * ce / (gamma - T(1));
    unb = T(0.5) * (Rp + Rm);
    T cb = T(0.25) * (gamma - T(1)) * (Rp - Rm);
    T s;
    if (unb >= T(0)) { s = pi / pow(ri, gamma); utb = uti; }
    else { s = pe / pow(re, gamma); utb = ute; }
    rb = pow(cb * cb / (gamma * s), T(1) / (gamma - T(1)));
    pb = rb * cb * cb / gamma;
  }
  Wg[0] = rb; Wg[1] = rb * unb; Wg[2] = rb * utb;
  Wg[3] = pb / (gamma - T(1)) + T(0.5) * rb * (unb * unb + utb * utb);
}

}  // namespace dev
}  // namespace cgks
