// Instantiation unit: generation with one chain per warp, rows of two words, L = 52 to 64.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_2b(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 52: return launch_warp_rows<TwoWords<1, 52>, 52>(j, warps, ts, t0, S, trace, st);
    case 56: return launch_warp_rows<TwoWords<1, 56>, 56>(j, warps, ts, t0, S, trace, st);
    case 60: return launch_warp_rows<TwoWords<1, 60>, 60>(j, warps, ts, t0, S, trace, st);
    case 64: return launch_warp_rows<TwoWords<1, 64>, 64>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
