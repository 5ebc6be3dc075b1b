// Persistent 1D kernels (resident and step-blocked) of the strict policy, a translation unit of their own so
// that the library's units compile in parallel.  Built with -fmad=false.
#include "wt_kernels.cuh"
#include "wt_math_strict.cuh"

namespace wt {

cudaError_t launch_persist1d_strict(int flux, int tile, const PersistArgs& p, int grid, cudaStream_t st) {
  return launch_persist1d_policy<StrictMath>(flux, tile, p, grid, st);
}

int persist1d_capacity_strict(int flux, int tile) { return persist1d_capacity_policy<StrictMath>(flux, tile); }

cudaError_t launch_stepblock1d_strict(int flux, int tile, const PersistArgs& p, int grid, cudaStream_t st) {
  return launch_stepblock1d_policy<StrictMath>(flux, tile, p, grid, st);
}

int stepblock1d_capacity_strict(int flux, int tile) { return stepblock1d_capacity_policy<StrictMath>(flux, tile); }

}  // namespace wt
