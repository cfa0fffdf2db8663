// The joint of a round that kept its flips, rows of 1 to 4 words.
#include "mc_joint_kept.cuh"

namespace mcgpu {

// A lane rebuilds its segment's levels from the segment's lattice (in shared
// memory, as the replays' runners keep it) and the recorded flips: with the
// flips known nothing is serial but the sum of the level changes.  Bit masks
// give every site's change (its aligned neighbours - 2 if it flipped), four
// sites are summed at once as bytes of one multiplication: about 6
// operations a site, against 35 and a chain of dependent loads for running
// the chain again.
template <int WD>
struct SourceFlip {
  static constexpr int kPlacement = kPlaceSmem;
  template <class Hook>
  __device__ __forceinline__ static void segment(const DevJob& j, const BlockCtx& b, int i, int seg, int64_t S,
                                                 Hook& hk) {
    const int L = j.L, lw = L - 32 * (WD - 1), stride = b.nslot;
    uint32_t* lat = b.lat + b.slot;
    const uint32_t* ck = j.ckpt + static_cast<size_t>(seg) * L * WD * j.p + i;
    for (int q = 0; q < L * WD; ++q) lat[q * stride] = __ldg(ck + static_cast<size_t>(q) * j.p);
    int m4 = 4 * j.ckm[static_cast<size_t>(seg) * j.p + i];
    const int64_t s0 = static_cast<int64_t>(seg) * j.ck_C;
    const int sweeps = static_cast<int>(min(S - s0, static_cast<int64_t>(j.ck_C)));
    const uint32_t* flips = j.flips + static_cast<size_t>(i) * flip_words(L, S) + s0 * L * WD;
    for (int s = 0; s < sweeps && !hk.done; ++s) {
      uint32_t up[WD], cur[WD], F[WD];
#pragma unroll
      for (int w = 0; w < WD; ++w) {
        up[w] = lat[((L - 1) * WD + w) * stride];
        cur[w] = lat[w * stride];
        F[w] = __ldg(flips + w);
      }
#pragma unroll 1
      for (int y = 0; y < L && !hk.done; ++y) {
        uint32_t dn[WD], nF[WD];
        const int yp = y + 1 == L ? 0 : y + 1;
#pragma unroll
        for (int w = 0; w < WD; ++w) {
          dn[w] = lat[(yp * WD + w) * stride];
          nF[w] = y + 1 < L ? __ldg(flips + WD + w) : 0u;
        }
        flips += WD;
#pragma unroll
        for (int w = 0; w < WD; ++w) {
          const bool lastw = w == WD - 1;
          const int nb = lastw ? lw : 32;
          const uint32_t c = cur[w], f = F[w];
          // agreements at each site's own attempt: up and left as swept, right not yet (but the row's
          // last site sees site 0 as swept)
          const uint32_t first = WD == 1 ? c ^ f : cur[0];
          const uint32_t right = (c >> 1) | (lastw ? ((first & 1u) << (lw - 1)) : (cur[(w + 1) % WD] << 31));
          const uint32_t left = ((c ^ f) << 1) | (w > 0 ? (cur[(w + WD - 1) % WD] >> 31) : ((cur[WD - 1] >> (lw - 1)) & 1u));
          const uint32_t eu = ~(c ^ up[w]), ed = ~(c ^ dn[w]), er = ~(c ^ right), el = ~(c ^ left);
          const uint32_t p0 = f & (eu ^ ed ^ er), p1 = f & el;
          const uint32_t n2 = f & ~((eu & ed) | (er & (eu ^ ed)));
          hk.word(nb);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            if (4 * q < nb) {
              // bytes: change + 2 of the four sites, then 4 times their running sums (at most 64)
              const uint32_t d = spread4((p0 >> (4 * q)) & 0xFu) + spread4((p1 >> (4 * q)) & 0xFu) + 0x02020202u -
                                 2u * spread4((n2 >> (4 * q)) & 0xFu);
              const uint32_t sum = d * 0x04040404u;
#pragma unroll
              for (int b4 = 0; b4 < 4; ++b4)
                hk.sample(m4 + static_cast<int>(prmt(sum, 0x4440u | static_cast<uint32_t>(b4))) - 8 * (b4 + 1), 4 * q + b4);
              m4 += static_cast<int>(sum >> 24) - 32;
            }
          }
          cur[w] = c ^ f;
        }
#pragma unroll
        for (int w = 0; w < WD; ++w) {
          lat[(y * WD + w) * stride] = up[w] = cur[w];
          cur[w] = dn[w];
          F[w] = nF[w];
        }
      }
      hk.poll();
    }
  }
  // the samples whose levels are at hand: each segment's last
  __device__ __forceinline__ static int seeds(const DevJob& j, int64_t) { return j.ck_K; }
  __device__ __forceinline__ static int seed(const DevJob& j, int i, int a, int n, int64_t M, int64_t* k) {
    if (a == n - 1) {
      *k = M - 1;
      return j.m[i];
    }
    *k = static_cast<int64_t>(a + 1) * j.seg_len - 1;
    return j.ckm[static_cast<size_t>(a + 1) * j.p + i];
  }
};

// As many lanes a block as leave room for a second block beside it, or as fit.
static LaunchShape flip_shape(int L) {
  LaunchShape s{kPlaceSmem, 32, 4};
  const size_t half = 113 * 1024;
  if (plan_bytes(L, s, false, true) <= half) return s;
  while (s.cpw > 1 && plan_bytes(L, s, false, true) > kMaxSmem - 2048) --s.cpw;   // (the kernels' own variables)
  return s;
}

cudaError_t chain_kernels_flips(const DevJob& j, int64_t S, uint32_t r, cudaStream_t st) {
  const LaunchShape s = flip_shape(j.L);
  switch (j.wd) {
    case 1: return launch_join_kept<SourceFlip<1>>(j, s, S, r, st);
    case 2: return launch_join_kept<SourceFlip<2>>(j, s, S, r, st);
    case 3: return launch_join_kept<SourceFlip<3>>(j, s, S, r, st);
    case 4: return launch_join_kept<SourceFlip<4>>(j, s, S, r, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
