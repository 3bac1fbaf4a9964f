// FP64 instances of the persistent evolve kernel with plain staging (every
// model x stencil, any lattice side).
#include "persist_kernel.cuh"

namespace pycool {
cudaError_t launch_persist_fp64_plain(int model, int stencil, int vx, const PParams& p, int grid,
                                    cudaStream_t s, int* bps) {
  return launch_persist_impl<PREC_FP64, false, true>(model, stencil, vx, p, grid, s, bps);
}
}  // namespace pycool
