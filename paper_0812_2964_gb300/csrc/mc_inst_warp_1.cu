// Instantiation unit: generation with one chain per warp, rows of one word.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_1(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                cudaStream_t st) {
  switch (j.L) {
    case 4: return launch_warp_rows<Words<1, 4>, 4>(j, warps, ts, t0, S, trace, st);
    case 8: return launch_warp_rows<ShortRows<8>, 8>(j, warps, ts, t0, S, trace, st);
    case 12: return launch_warp_rows<ShortRows<12>, 12>(j, warps, ts, t0, S, trace, st);
    case 16: return launch_warp_rows<ShortRows<16>, 16>(j, warps, ts, t0, S, trace, st);
    case 20: return launch_warp_rows<Words<1, 20>, 20>(j, warps, ts, t0, S, trace, st);
    case 24: return launch_warp_rows<Words<1, 24>, 24>(j, warps, ts, t0, S, trace, st);
    case 28: return launch_warp_rows<Words<1, 28>, 28>(j, warps, ts, t0, S, trace, st);
    case 32: return launch_warp_rows<Words<1, 32>, 32>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
