// Launch shapes of the tunable kernels (shared by the kernels and the
// runtimes).  A shape is (threads per block, items per thread, minimum
// resident blocks per SM); an item is a cell or a face (a face's Gauss point,
// a lane group's cell), one per thread in every shape.  The block size is a
// launch argument, so one compiled kernel serves every shape: it changes only
// which thread does the work, never the result.  (A compilation per shape let
// the compiler fuse multiplies and adds differently in each; a runtime count
// of items per thread cost the short FP32 kernels 5-20%.)
#pragma once

#include "../../include/cgks.h"
#ifdef __CUDACC__
#include "cgks_pdl.cuh"
#endif

namespace cgks {

constexpr int kNShape = CGKS_TUNE_SHAPES;
constexpr int kMaxShapeBlock = 256;   // the largest block of any shape

__host__ __device__ constexpr int shape_bs(int s) {
  return s == 1 ? 64 : s == 2 ? 256 : s == 3 ? 96 : s == 4 ? 192 : 128;
}

// tunable kernels
enum TuneKernel { TK_RECON = 0, TK_FACE, TK_LOFACE, TK_SWEEP, TK_COUNT };
static_assert(TK_COUNT == CGKS_TUNE_KERNELS, "tunable kernel count");
// shapes used without the autotuner: 256-thread cell kernels, 128-thread
// face flux and sweeps
constexpr int kDefaultShape[TK_COUNT] = { 2, 0, 2, 0 };

#ifdef __CUDACC__
// the item of this thread in a launch over n items
template <typename F>
__device__ __forceinline__ void for_items(const int n, F &&f) {
  const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (i < n) f(i);
}

// The same, for a kernel launched as a programmatic dependent launch: geo(i)
// reads the item's mesh data (which no kernel of a cycle writes), then the
// thread waits for the predecessor kernel before f(i, g) touches anything
// else.  Every thread waits, so the grid completes only after its
// predecessor has.
template <typename G, typename F>
__device__ __forceinline__ void for_items_pdl(const int n, G &&geo, F &&f) {
  const int i = static_cast<int>(blockIdx.x * blockDim.x + threadIdx.x);
  if (i < n) {
    const auto g = geo(i);
    pdl_enter();
    f(i, g);
  }
  pdl_enter();   // threads without items wait too: this grid ends after its predecessor
}
#endif

}  // namespace cgks
