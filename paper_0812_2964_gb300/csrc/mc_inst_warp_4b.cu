// Instantiation unit: generation with one chain per warp, rows of four words, L = 116 to 128.
#include "mc_warp_chain.cuh"

namespace mcgpu {

cudaError_t chain_kernels_warp_4b(const DevJob& j, int warps, bool ts, bool pairs, uint64_t t0, int64_t S, bool trace,
                                 cudaStream_t st) {
  switch (j.L) {
    case 116: return pairs ? launch_warp_rows<TwoWords<2, 116>, 116>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 116>, 116>(j, warps, ts, t0, S, trace, st);
    case 120: return pairs ? launch_warp_rows<TwoWords<2, 120>, 120>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 120>, 120>(j, warps, ts, t0, S, trace, st);
    case 124: return pairs ? launch_warp_rows<TwoWords<2, 124>, 124>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 124>, 124>(j, warps, ts, t0, S, trace, st);
    case 128: return pairs ? launch_warp_rows<TwoWords<2, 128>, 128>(j, warps, ts, t0, S, trace, st)
                         : launch_warp_rows<Words<4, 128>, 128>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
