// Persistent fused low-order solve (included by cgks_device.cu only).
//
// One cooperative launch runs the whole low-order level of a V-cycle
// (Section 3, steps 3-4): n_implicit backward-Euler steps, each = base
// records (and U += dU), KFVS faces, right-hand side with the first
// colour pass, then the remaining colour passes of Algorithm 1, and the
// final U += dU.  Phases are separated by a grid barrier instead of kernel
// boundaries.  Every value produced inside the launch is read with
// ld.global.cg (L2, never a stale L1 line); each phase runs the device
// functions of the per-phase kernels of cgks_kernels.cuh.
//
// Measured on GB300 (57k-cell cylinder V-cycle): slower than the per-phase
// kernels replayed from a CUDA graph (FP64 1.31 vs 0.92 ms, mixed 0.47 vs
// 0.26 ms): the resident grid holds fewer warps per SM than the separate
// launches and the graph already hides their launch gaps, so the library
// uses it only when asked (cgks_params.low_order_fused).
//
// The barrier spins with a bound: past the launch's spin limit (kSpinLimit
// unless the caller sets one) a block records kBarrierTimeout in the status
// word of every slot of the batch and leaves; every other block then times
// out at its next barrier, so the launch always ends.  The host clears the
// barrier before every launch, so a launch that timed out leaves nothing
// behind for the next one.
#pragma once

#include "cgks_kernels.cuh"

namespace cgks {
namespace kern {

constexpr int kPersistBlock = 256;
constexpr int kBarrierTimeout = 2;              // bit of the status word
constexpr long long kSpinLimit = 1ll << 22;     // ~4M polls of ~0.1-1 us: seconds, far above any phase

struct GridBarrier {
  unsigned int count, gen;
};

// a load that observes other blocks' writes (acquire, GPU scope)
__device__ __forceinline__ unsigned ld_acquire(const unsigned *p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// all blocks of the grid; returns false after a timeout (status bit set in
// each of the n_err status words)
__device__ __forceinline__ bool grid_barrier(GridBarrier *gb, long long spin_limit, int *err, int n_err) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    ok = 1;
    __threadfence();
    const unsigned my_gen = ld_acquire(&gb->gen);
    const unsigned arrived = atomicAdd(&gb->count, 1u) + 1u;
    if (arrived == gridDim.x) {
      atomicExch(&gb->count, 0u);
      __threadfence();
      atomicAdd(&gb->gen, 1u);
    } else {
      long long it = 0;
      while (ld_acquire(&gb->gen) == my_gen) {
        if (++it > spin_limit) {
          for (int k = 0; k < n_err; ++k) atomicOr(&err[k], kBadState | kBarrierTimeout);
          ok = 0;
          break;
        }
        __nanosleep(32);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// per-colour cell ranges of the batch in device memory (any number of solves)
struct ColourRanges {
  const int *rstart;   // [C + 1] first range of each colour
  const int *rbegin;   // [R] first cell of each range
  const int *rpre;     // [R + C] cells of the colour before each range (per colour, R_c + 1 entries)
};

template <typename TF>
struct LoArgs {
  MeshT<double> dm;
  MeshT<TF> fm;
  ParamsT<double> dp;
  ParamsT<TF> fp;
  int n_implicit, colour0, n_seq;
  int n_cells, n_faces;              // extents of the solves present (arrays are strided by capacity)
  int seq[48];                       // colour order after the first pass (n_sweeps x 2 x colours)
  ColourRanges cr;
  const double *Wp0, *Rp0;
  double *U, *Src;
  TF *delta, *base, *Flo, *Rk, *invD, *lamS;
  GridBarrier *gb;
  long long spin_limit;              // polls per barrier wait before giving up
  int *err;                          // [n_err] status words of the batch's slots
  int n_err;
};

// cell of the g-th position of colour c, or -1 past its end
__device__ __forceinline__ int colour_cell(const ColourRanges &cr, int c, int g) {
  const int r0 = cr.rstart[c], r1 = cr.rstart[c + 1];
  const int *pre = cr.rpre + r0 + c;            // r1 - r0 + 1 prefix entries
  if (g >= pre[r1 - r0]) return -1;
  int lo = 0, hi = r1 - r0 - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= g) lo = mid; else hi = mid - 1;
  }
  return cr.rbegin[r0 + lo] + (g - pre[lo]);
}

template <typename TF>
__global__ void __launch_bounds__(kPersistBlock, 2) k_lo_solve(const __grid_constant__ LoArgs<TF> a) {
  const int n = a.n_cells, nf = a.n_faces;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  for (int k = 0; k < a.n_implicit; ++k) {
    for (int i = tid; i < n; i += nth) lo_cell_at<TF, true>(a.dm.nc, a.fp, k == 0, a.Wp0, a.U, a.delta, a.base, i);
    if (!grid_barrier(a.gb, a.spin_limit, a.err, a.n_err)) return;
    for (int f = tid; f < nf; f += nth)
      lo_face_at<TF, true>(a.fm, a.fp, lo_face_geo(a.fm, a.fp, f), a.base, a.Flo, f);
    if (!grid_barrier(a.gb, a.spin_limit, a.err, a.n_err)) return;
    for (int i = tid; i < n; i += nth)
      lo_rhs_at<TF, true>(a.dm, a.dp, a.fp.gamma, rhs_geo(a.dm, i, a.colour0), k == 0, a.base, a.Flo, a.Rp0, a.Src,
                          a.Rk, a.invD, a.delta, a.lamS, i);
    if (!grid_barrier(a.gb, a.spin_limit, a.err, a.n_err)) return;
    for (int q = 0; q < a.n_seq; ++q) {
      const int c = a.seq[q];
      const int total = a.cr.rpre[a.cr.rstart[c + 1] + c];
      // Four lanes per cell, 8 cells of a warp iterating together.  One thread per
      // cell spilled in FP64 and left most of the resident warps idle below 20,000
      // cells of a colour: us per V-cycle, one / four, 2,048 cells FP64 878 / 714,
      // mixed 425 / 368; 57,344 1638 / 1336, 522 / 475; 131,072 2220 / 2261,
      // 681 / 684.
      const int s = threadIdx.x % 4;
      for (int g0 = tid / 32 * 8; g0 < total; g0 += nth / 4) {
        const int g = g0 + static_cast<int>(threadIdx.x % 32 / 4), i = g < total ? colour_cell(a.cr, c, g) : -1;
        sweep_quad<TF, true, true>(a.fm, a.fp.gamma, slot_geo(a.fm, i, s), i, s, a.base, a.Rk, a.invD, a.lamS,
                                   [&](int) -> const TF * { return a.delta; }, a.delta);
      }
      if (!grid_barrier(a.gb, a.spin_limit, a.err, a.n_err)) return;
    }
  }
  if (a.n_implicit > 0)
    for (int i = tid; i < n; i += nth) lo_cell_at<TF, true>(a.dm.nc, a.fp, 0, a.Wp0, a.U, a.delta, a.base, i);
}

}  // namespace kern
}  // namespace cgks
