// The joint of a recorded round: one instantiation serves every L, since
// nothing in it depends on the lattice size at compile time.
#include "mc_joint_kept.cuh"

namespace mcgpu {

// Samples per segment: a lane's work item.  With nothing to restore at its
// start it is as short as spreads the round over the GPU's lanes, down to 128
// samples (a small round's passes last as long as one lane takes for its
// segment: an iteration of L = 16, p = 512, S = 20 takes 443 us with 256, 424
// with 128, 428 with 64), up to 2048 (an item's set-up then costs a few percent).
cudaError_t chain_kernels_record(const DevJob& j, int64_t S, uint32_t r, cudaStream_t st) {
  DevJob jr = j;
  const int64_t M = S * j.N;
  const int64_t spread = static_cast<int64_t>(j.p) * M / (152 * 512);
  jr.seg_len = std::min<int64_t>(2048, std::max<int64_t>(128, spread & ~31ll));
  jr.ck_K = static_cast<int>((M + jr.seg_len - 1) / jr.seg_len);
  // full warps, four a block; shared memory holds only the level weights (or counts)
  return launch_join_kept<SourceRec>(jr, LaunchShape{kPlaceReg, 32, 4}, S, r, st);
}

}  // namespace mcgpu
