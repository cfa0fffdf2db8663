// Instantiation unit: generation with one chain per warp, rows of three words, L = 84 to 96.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_3b(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 84: return launch_warp_rows<Words<3, 84>, 84>(j, warps, ts, t0, S, trace, st);
    case 88: return launch_warp_rows<Words<3, 88>, 88>(j, warps, ts, t0, S, trace, st);
    case 92: return launch_warp_rows<Words<3, 92>, 92>(j, warps, ts, t0, S, trace, st);
    case 96: return launch_warp_rows<Words<3, 96>, 96>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
