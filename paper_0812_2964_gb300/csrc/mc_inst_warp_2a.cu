// Instantiation unit: generation with one chain per warp, rows of two words, L = 36 to 48.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_2a(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 36: return launch_warp_rows<TwoWords<1, 36>, 36>(j, warps, ts, t0, S, trace, st);
    case 40: return launch_warp_rows<TwoWords<1, 40>, 40>(j, warps, ts, t0, S, trace, st);
    case 44: return launch_warp_rows<TwoWords<1, 44>, 44>(j, warps, ts, t0, S, trace, st);
    case 48: return launch_warp_rows<TwoWords<1, 48>, 48>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
