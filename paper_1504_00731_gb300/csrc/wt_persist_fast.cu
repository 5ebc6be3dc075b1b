// Persistent 1D kernels (resident and step-blocked) of the fast policy, a translation unit of their own so
// that the library's units compile in parallel.
#include "wt_kernels.cuh"
#include "wt_math_fast.cuh"

namespace wt {

cudaError_t launch_persist1d_fast(int flux, int tile, const PersistArgs& p, int grid, cudaStream_t st) {
  return launch_persist1d_policy<FastMath>(flux, tile, p, grid, st);
}

int persist1d_capacity_fast(int flux, int tile) { return persist1d_capacity_policy<FastMath>(flux, tile); }

cudaError_t launch_stepblock1d_fast(int flux, int tile, const PersistArgs& p, int grid, cudaStream_t st) {
  return launch_stepblock1d_policy<FastMath>(flux, tile, p, grid, st);
}

int stepblock1d_capacity_fast(int flux, int tile) { return stepblock1d_capacity_policy<FastMath>(flux, tile); }

}  // namespace wt
