// Instantiation unit: generation with one chain per warp, rows of three words, L = 68 to 80.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_3a(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 68: return launch_warp_rows<Words<3, 68>, 68>(j, warps, ts, t0, S, trace, st);
    case 72: return launch_warp_rows<Words<3, 72>, 72>(j, warps, ts, t0, S, trace, st);
    case 76: return launch_warp_rows<Words<3, 76>, 76>(j, warps, ts, t0, S, trace, st);
    case 80: return launch_warp_rows<Words<3, 80>, 80>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
