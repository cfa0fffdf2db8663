// Instantiation unit: generation with one chain per warp, rows of four words, L = 100 to 112.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_4a(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 100: return pairs ? launch_warp_rows<TwoWords<2, 100>, 100>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 100>, 100>(j, warps, ts, t0, S, trace, st);
    case 104: return pairs ? launch_warp_rows<TwoWords<2, 104>, 104>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 104>, 104>(j, warps, ts, t0, S, trace, st);
    case 108: return pairs ? launch_warp_rows<TwoWords<2, 108>, 108>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 108>, 108>(j, warps, ts, t0, S, trace, st);
    case 112: return pairs ? launch_warp_rows<TwoWords<2, 112>, 112>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 112>, 112>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
