// A solve's device tables, derived on the device.
//
// Placing a solve uploads its preprocessed mesh as it is (about 300 bytes per
// cell) straight into its cell and face ranges; these kernels turn indices
// into batch indices and form what follows from the mesh: inverses, slot
// areas, the compact least-squares operator (70 values per cell) and, in the
// mixed path, the FP32 tables.  Forming them on the host and uploading them
// (1.7 KB per cell) took most of a served request's time: 44 ms for six
// requests of 62,804 cells together, under 2 ms now (with the first V-cycle 2.2).
#pragma once

#include "cgks_kernels.cuh"

namespace cgks {
namespace kern {

// device tables of a batch (views into its arena)
struct DevArrays {
  double *vol, *ivol, *per, *ih, *m2, *op, *fn, *fS, *fjump, *fxi, *snx, *sny, *sS, *fidl = nullptr;
  double *mu, *bcuw, *bcrho, *bcu, *bcp;
  int *cface, *cnbr, *fc0, *fc1, *csid, *fsid, *bckind;
  unsigned char *ccol, *wenok;
  float *f_ivol = nullptr, *f_ih = nullptr, *f_m2 = nullptr, *f_op = nullptr, *f_fn = nullptr, *f_fS = nullptr,
        *f_fjump = nullptr, *f_fidl = nullptr, *f_fxi = nullptr, *f_snx = nullptr, *f_sny = nullptr, *f_shs = nullptr, *f_mu = nullptr,
        *f_bcuw = nullptr, *f_bcrho = nullptr, *f_bcu = nullptr, *f_bcp = nullptr;
};

constexpr int kMaxColours = 32;   // the greedy colouring's mask has 32 bits
// where a solve sits and what its tables depend on besides the mesh
struct Place {
  int slot, nc, np, nf, co, fo, N, F;   // cells, padded cells, faces; offsets; capacities (strides)
  int n_colours, colour_start[kMaxColours + 1];
  unsigned wall;                        // bit t: boundary tag t mirrors the state (enters the operator)
  double alpha, mu;
  double uw[2 * kTagsPerSolve], rho[kTagsPerSolve], u[2 * kTagsPerSolve], p[kTagsPerSolve];
  int kind[kTagsPerSolve];
};

constexpr int kRows = kNCol;   // least-squares rows: one per operator column, rows of absent slots zero

// Operator of the compact quadratic of local cell k: rows per stencil slot =
// mean of the neighbour (or wall mirror cell) and h times its two mean
// gradients, plus h times the own mean gradient; unknowns the 5 coefficients
// of the monomials minus their own means.  Pseudo-inverse by modified
// Gram-Schmidt and back substitution.  Linear, from the own gradient, with
// fewer than two stencil cells or a rank-deficient fit (returns false).
// xc, c2: [2][nc], [3][nc] of the mesh; fc1 as uploaded (-1 - tag).
__device__ __forceinline__ bool operator_of(const Place &pl, const DevArrays &d, const double *xc, const double *c2,
                                            int k, double h, double Q[kRows][kNM], double R[kNM][kNM]) {
  const int nc = pl.nc, N = pl.N, F = pl.F, i = pl.co + k;
  const double x0 = xc[k], y0 = xc[nc + k], ih = 1.0 / h, ih2 = ih * ih;
  double own[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) own[q] = d.m2[q * N + i];
  int slots = 0;
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
#pragma unroll
    for (int r = 0; r < 3; ++r)
#pragma unroll
      for (int q = 0; q < kNM; ++q) Q[3 * s + r][q] = 0.0;
    const int fs = d.cface[s * N + i];
    if (fs == kNoFace) continue;
    const int f = pl.fo + (fs >= 0 ? fs : ~fs), j = d.cnbr[s * N + i];
    double dx, dy, Ixx, Ixy, Iyy;   // centre offset and central moments of the stencil cell
    if (j >= 0) {
      dx = xc[j] - x0; dy = xc[nc + j] - y0;
      Ixx = c2[j]; Ixy = c2[nc + j]; Iyy = c2[2 * nc + j];
    } else {
      if (!(pl.wall >> (-1 - d.fc1[f]) & 1u)) continue;
      // mirror image of the cell across the wall line: R = 1 - 2 n n, R C R
      const double nx = d.fn[f], ny = d.fn[F + f];
      const double off = d.fxi[f] * h * nx + d.fxi[F + f] * h * ny;   // along n to a point of the wall
      dx = 2.0 * off * nx; dy = 2.0 * off * ny;
      const double a = 1.0 - 2.0 * nx * nx, b = -2.0 * nx * ny, e = 1.0 - 2.0 * ny * ny;
      const double Cxx = c2[k], Cxy = c2[nc + k], Cyy = c2[2 * nc + k];
      const double p0 = a * Cxx + b * Cxy, p1 = a * Cxy + b * Cyy, q0 = b * Cxx + e * Cxy, q1 = b * Cxy + e * Cyy;
      Ixx = p0 * a + p1 * b; Ixy = p0 * b + p1 * e; Iyy = q0 * b + q1 * e;
    }
    const double ex = dx * ih, ey = dy * ih;
    Q[3 * s][0] = ex;
    Q[3 * s][1] = ey;
    Q[3 * s][2] = Ixx * ih2 + ex * ex - own[0];
    Q[3 * s][3] = Ixy * ih2 + ex * ey - own[1];
    Q[3 * s][4] = Iyy * ih2 + ey * ey - own[2];
    Q[3 * s + 1][0] = 1.0; Q[3 * s + 1][2] = 2.0 * ex; Q[3 * s + 1][3] = ey;
    Q[3 * s + 2][1] = 1.0; Q[3 * s + 2][3] = ex; Q[3 * s + 2][4] = 2.0 * ey;
    ++slots;
  }
#pragma unroll
  for (int q = 0; q < kNM; ++q) {
    Q[kRows - 2][q] = q == 0 ? 1.0 : 0.0;
    Q[kRows - 1][q] = q == 1 ? 1.0 : 0.0;
  }
  bool ok = slots >= 2;
  // Q R = A; R[j][j] holds the inverse of the norm
#pragma unroll
  for (int j = 0; j < kNM; ++j) {
#pragma unroll
    for (int p = 0; p < j; ++p) {
      double s = 0.0;
#pragma unroll
      for (int r = 0; r < kRows; ++r) s += Q[r][p] * Q[r][j];
      R[p][j] = s;
#pragma unroll
      for (int r = 0; r < kRows; ++r) Q[r][j] -= s * Q[r][p];
    }
    double n2 = 0.0;
#pragma unroll
    for (int r = 0; r < kRows; ++r) n2 += Q[r][j] * Q[r][j];
    const double nrm = sqrt(n2);
    ok = ok && nrm > 1e-13;
    R[j][j] = 1.0 / nrm;
#pragma unroll
    for (int r = 0; r < kRows; ++r) Q[r][j] *= R[j][j];
  }
  return ok;
}

// Cells of a solve (thread k: local cell k; k >= nc: padding).  Uploaded in
// place: vol, per, h (in ih), m2, cface, cnbr (local indices), fn, fS, fxi, fc1.
__global__ void __launch_bounds__(64) k_insert_cells(const __grid_constant__ Place pl,
                                                     const __grid_constant__ DevArrays d, int *perm,
                                                     const double *xc, const double *c2) {
  const int k = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (k >= pl.np) return;
  const int N = pl.N, F = pl.F, i = pl.co + k;
  const bool in = k < pl.nc, mixed = d.f_op != nullptr;
  const double h = in ? d.ih[i] : 1.0;
  auto put_op = [&](int col, int q, double v) {
    d.op[(col * kNM + q) * N + i] = v;
    if (mixed) d.f_op[(col * kNM + q) * N + i] = static_cast<float>(v);
  };
  {
    double Q[kRows][kNM], R[kNM][kNM];
    const bool quad = in && operator_of(pl, d, xc, c2, k, h, Q, R);
    d.wenok[i] = quad ? 1 : 0;
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      const double g = r % 3 != 0 || r >= 3 * kMaxFace ? h : 1.0;   // h folded into the gradient columns
      double y[kNM];
#pragma unroll
      for (int q = kNM - 1; q >= 0; --q) {
        double v = Q[r][q];
#pragma unroll
        for (int p = q + 1; p < kNM; ++p) v -= R[q][p] * y[p];
        y[q] = v * R[q][q];
      }
      // an absent slot's rows are zero
#pragma unroll
      for (int q = 0; q < kNM; ++q)
        put_op(r, q, quad ? y[q] * g : in && r == kRows - 2 + q ? h : 0.0);
    }
  }
  const double iv = in ? 1.0 / d.vol[i] : 1.0, ih = in ? 1.0 / h : 1.0;
  d.ivol[i] = iv;
  d.ih[i] = ih;
  if (mixed) { d.f_ivol[i] = static_cast<float>(iv); d.f_ih[i] = static_cast<float>(ih); }
  if (!in) { d.vol[i] = 1.0; d.per[i] = 4.0; perm[i] = 0; }
  d.csid[i] = in ? pl.slot : -1;
  int c = 0;
  while (in && k >= pl.colour_start[c + 1]) ++c;
  d.ccol[i] = in ? static_cast<unsigned char>(c) : 255;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (!in) d.m2[q * N + i] = 0.0;
    if (mixed) d.f_m2[q * N + i] = static_cast<float>(d.m2[q * N + i]);
  }
#pragma unroll
  for (int s = 0; s < kMaxFace; ++s) {
    const int o = s * N + i, fs = in ? d.cface[o] : kNoFace;
    double nx = 0.0, ny = 0.0, S = 0.0;
    int face = kNoFace, nbr = -1;
    if (fs != kNoFace) {
      const int f = pl.fo + (fs >= 0 ? fs : ~fs), j = d.cnbr[o];
      face = fs >= 0 ? f : ~f;
      nbr = j >= 0 ? j + pl.co : -1;
      S = d.fS[f];
      nx = fs >= 0 ? d.fn[f] : -d.fn[f];
      ny = fs >= 0 ? d.fn[F + f] : -d.fn[F + f];
    }
    d.cface[o] = face;
    d.cnbr[o] = nbr;
    d.snx[o] = nx * (0.5 * S);
    d.sny[o] = ny * (0.5 * S);
    d.sS[o] = S;
    if (mixed) {
      d.f_snx[o] = static_cast<float>(nx);
      d.f_sny[o] = static_cast<float>(ny);
      d.f_shs[o] = static_cast<float>(0.5 * S);
    }
  }
}

// Faces of a solve, after its cells (which read fc1 as uploaded).  Uploaded in
// place: fc0, fc1, fn, fS, fxi and the centre distance (in fidl).
__global__ void __launch_bounds__(128) k_insert_faces(const __grid_constant__ Place pl,
                                                      const __grid_constant__ DevArrays d) {
  const int k = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  const bool mixed = d.f_op != nullptr;
  if (blockIdx.x == 0 && threadIdx.x < kTagsPerSolve) {
    const int t = threadIdx.x, T = kTagsPerSolve, g = T * pl.slot + t;
    auto put = [&](double *x, float *x32, int at, double v) {
      x[at] = v;
      if (mixed) x32[at] = static_cast<float>(v);
    };
    if (t == 0) put(d.mu, d.f_mu, pl.slot, pl.mu);
    d.bckind[g] = pl.kind[t];
    put(d.bcrho, d.f_bcrho, g, pl.rho[t]);
    put(d.bcp, d.f_bcp, g, pl.p[t]);
    for (int q = 0; q < 2; ++q) {
      put(d.bcuw, d.f_bcuw, 2 * g + q, pl.uw[2 * t + q]);
      put(d.bcu, d.f_bcu, 2 * g + q, pl.u[2 * t + q]);
    }
  }
  if (k >= pl.nf) return;
  const int F = pl.F, f = pl.fo + k;
  const double delta = d.fidl[f];
  const double jump = delta > 0.0 ? pl.alpha / delta : 0.0, idl = delta > 0.0 ? 1.0 / delta : 0.0;
  const int c1 = d.fc1[f];
  d.fc0[f] += pl.co;
  d.fc1[f] = c1 >= 0 ? c1 + pl.co : c1 - pl.slot * kTagsPerSolve;   // -1 - (slot T + tag)
  d.fsid[f] = pl.slot;
  d.fjump[f] = jump;
  d.fidl[f] = idl;
  if (mixed) {
    d.f_fjump[f] = static_cast<float>(jump);
    d.f_fidl[f] = static_cast<float>(idl);
    d.f_fS[f] = static_cast<float>(d.fS[f]);
#pragma unroll
    for (int q = 0; q < 2; ++q) d.f_fn[q * F + f] = static_cast<float>(d.fn[q * F + f]);
#pragma unroll
    for (int q = 0; q < 8; ++q) d.f_fxi[q * F + f] = static_cast<float>(d.fxi[q * F + f]);
  }
}

}  // namespace kern
}  // namespace cgks
