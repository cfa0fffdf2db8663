// The joint (Sec. 2 steps 3-5) of a round whose samples generation kept: the
// kernels read every sample's level from a source (the round record, or the
// flip record) instead of running the chains again.
//
// Flow: a search for every chain's first accepted sample under the
// speculated input (first segment, then the later segments of the chains
// without a hit), resolution passes for the chains whose actual input
// differs, then -- if chains are still pending, or straight away after a
// joint that rejected many chains -- the heights of all chains from the first
// pending one on (mc_height.cuh), which settle every input at once, and one
// search for the chains that keep samples under a new input.  Discarded (or,
// when they are fewer, kept) samples are counted last.  About 25 launches,
// most of which return at once in a round with little to resolve: a queue's
// reset, the selection of a pass's results and the list of chains without a
// hit are folded into the kernels around them (they were 60 launches of 2 to
// 7 us, half of a small round's time).
//
// The joint test needs no threshold table: a sample passes iff
// u < 2^32 exp(W[m] - W[x]), and a float filter (level weights in shared
// memory, one exponential) rejects all but the samples within a percent of
// the line, which the exact test then decides.
#pragma once
#include "mc_chain_kernels.cuh"
#include "mc_height.cuh"
#include "mc_launch.cuh"

namespace mcgpu {

// ------------------------------------------------------------------ sources
// The round record: levels as uint16 (layout rec_index), read four samples at
// a time, the next 32 samples' groups loaded while the current ones are
// tested.  Segments start on multiples of 16 samples and hold multiples of
// 16, so a segment is whole words of 32 and at most one of 16.
struct SourceRec {
  static constexpr int kPlacement = kPlaceReg;   // (no lattice)
  template <int NB, class Hook>
  __device__ __forceinline__ static void word(const uint2 (&v)[8], Hook& hk) {
    hk.word(NB);
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const uint32_t pair = (b & 2) ? v[b >> 2].y : v[b >> 2].x;
      const uint32_t lv = (b & 1) ? (pair >> 16) : (pair & 0xFFFFu);
      hk.sample(4 * static_cast<int>(lv), b);
    }
  }
  template <class Hook>
  __device__ __forceinline__ static void segment(const DevJob& j, const BlockCtx&, int i, int seg, int64_t S, Hook& hk) {
    const int64_t M = S * j.N;
    const int64_t k0 = static_cast<int64_t>(seg) * j.seg_len;
    const int n = static_cast<int>(min(M - k0, j.seg_len));
    // group g (samples 4g .. 4g+3 of the segment) of the chain is grp[g * kRecTile]
    const uint2* grp = reinterpret_cast<const uint2*>(j.rec + rec_index(i, k0, M));
    uint2 v[8], nv[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 4 * q < n ? __ldg(grp + q * kRecTile) : make_uint2(0u, 0u);
    int left = n;
    for (; left >= 32 && !hk.done; left -= 32) {
      grp += 8 * kRecTile;
#pragma unroll
      for (int q = 0; q < 8; ++q) nv[q] = left > 32 + 4 * q ? __ldg(grp + q * kRecTile) : make_uint2(0u, 0u);
      word<32>(v, hk);
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = nv[q];
      if ((left & 1023) < 32) hk.poll();
    }
    if (left && !hk.done) word<16>(v, hk);
  }
  // up to 1024 samples spread over the chain: how many, and the a-th one's index and level
  __device__ __forceinline__ static int seeds(const DevJob&, int64_t M) {
    return static_cast<int>(min(static_cast<int64_t>(1024), M / 32)) & ~31;
  }
  __device__ __forceinline__ static int seed(const DevJob& j, int i, int a, int n, int64_t M, int64_t* k) {
    *k = static_cast<int64_t>(a) * (M / n);
    return j.rec[rec_index(i, *k, M)];
  }
};

// ------------------------------------------------------------------ hooks
// The exact test of one sample (off the main path: one call per candidate).
static __device__ __noinline__ bool joint_test(const double* __restrict__ W, int m, double wx, uint32_t u) {
  return u <= threshold_det(__dsub_rn(W[m], wx));
}

// First sample that passes against the input's weight wx.
struct TestHook {
  const float* wl;                  // level weights (shared memory, log2 units)
  const double* __restrict__ W;
  const unsigned long long* kmin;   // the chain's earliest hit: at or before `stop`, the search ends
  unsigned long long stop;
  double wx;
  float bl;                         // the input's, lowered by the floats' errors
  int64_t k, kw, found;
  uint32_t chain, r, k0, k1;
  uint32_t blk;
  int mq[4];
  bool done;
  __device__ __forceinline__ void word(int nb) {
    blk = static_cast<uint32_t>(static_cast<uint64_t>(k) >> 2);
    kw = k;
    k += nb;
  }
  __device__ __forceinline__ void sample(int m4, int b) {   // (by fours, as in HeightHook)
    mq[b & 3] = m4;
    if ((b & 3) != 3) return;
    const uint4 u = philox4x32_10(make_uint4(blk + static_cast<uint32_t>(b >> 2), r, chain, kTagJoint), k0, k1);
    if (height_filter4(wl, mq, bl, u)) {
#pragma unroll 1
      for (uint32_t left = height_passing(wl, mq, bl, u); left && !done; left &= left - 1u) {
        const int q = __ffs(static_cast<int>(left)) - 1;
        const int mm = q == 0 ? mq[0] : (q == 1 ? mq[1] : (q == 2 ? mq[2] : mq[3]));
        if (joint_test(W, mm >> 2, wx, uint4_word(u, static_cast<uint32_t>(q)))) {
          found = kw + (b - 3 + q) + 1;
          done = true;
        }
      }
    }
  }
  __device__ __forceinline__ void poll() {
    if (kmin && __ldcg(kmin) <= stop) done = true;
  }
};

// Counts the samples [lo, lo + n) of a segment (indices from its start).
struct CountHook {
  uint32_t* hist;
  int lo;
  uint32_t n;
  int at;        // samples of the words seen so far
  bool done;
  int base = 0;
  __device__ __forceinline__ void poll() {}
  __device__ __forceinline__ void word(int nb) {
    base = at - lo;
    at += nb;
    done = at >= lo + static_cast<int>(n);
  }
  __device__ __forceinline__ void sample(int m4, int b) {
    if (static_cast<uint32_t>(base + b) < n) red_shared_add(hist, m4, 1u);
  }
};

// ------------------------------------------------------------------ kernels
constexpr int kKeptWarps = 12;   // a block's most (two such blocks an SM: 80 registers)

__device__ __forceinline__ unsigned long long* kept_queue(const DevJob& j, int which) {
  return reinterpret_cast<unsigned long long*>(&j.stats[which]);
}

// The level weights of the block's chains into shared memory.
__device__ __forceinline__ float* kept_weights(const DevJob& j, const BlockCtx& b) {
  float* wl = reinterpret_cast<float*>(b.hist);
  const float* g = level_weights(j);
  for (int m = threadIdx.x; m < j.np1; m += blockDim.x) wl[m] = g[m];
  __syncthreads();
  return wl;
}

__device__ __forceinline__ void kept_test_setup(const DevJob& j, TestHook& hk, const float* wl, float slack, int i,
                                                int x, int64_t k, uint32_t r) {
  hk.wl = wl;
  hk.W = j.W;
  hk.wx = j.W[x];
  hk.bl = input_weight(level_weights(j)[x]) - slack;
  hk.k = k;
  hk.kw = k;
  hk.found = 0;
  hk.chain = static_cast<uint32_t>(i);
  hk.r = r;
  hk.k0 = j.key0;
  hk.k1 = j.key1;
  hk.done = false;
  hk.kmin = &j.kmin[i];
  hk.stop = static_cast<unsigned long long>(k);
}

// Joint search: items (chain, segment) of the chains of the list (all, or
// work[]) -- their first segments, or (later) the later segments of the
// chains without a hit there.  Persistent: each warp takes cpw consecutive
// items (segment-major) from the queue, its lanes read them side by side.  A
// segment is skipped, or left at the next poll, once an earlier one of its
// chain has a hit.
template <class Src>
__global__ void __launch_bounds__(32 * kKeptWarps, 2) kept_search_kernel(const DevJob j, const int cpw, const int64_t S,
                                                          const uint32_t r, const int listed, const int later,
                                                          const int exact_first) {
  after_previous();
  if (exact_first && rough_last_joint(j, j.stats[kStatRejected])) return;   // (the first search only)
  const int nchains = later ? static_cast<int>(j.stats[kStatNoHit]) : (listed ? static_cast<int>(j.stats[kStatPending]) : j.p);
  const int segs = later ? j.ck_K - 1 : 1;
  const long long items = static_cast<long long>(nchains) * segs;
  if (items == 0) return;
  unsigned long long* queue = kept_queue(j, later ? kStatQueueB : kStatQueueA);
  __shared__ int s_dry;
  if (threadIdx.x == 0) s_dry = static_cast<long long>(__ldcg(queue)) >= items;
  __syncthreads();
  if (s_dry) return;
  const SmemPlan sp = smem_plan(j.L, Src::kPlacement, cpw, blockDim.x >> 5, false, true);
  BlockCtx b = block_setup<false>(j, sp, cpw, 0, false);
  const float* wl = kept_weights(j, b);
  const float slack = height_slack(j);
  long long searched = 0;
  for (;;) {
    long long base = 0;
    if (b.lane == 0) base = static_cast<long long>(atomicAdd(queue, static_cast<unsigned long long>(cpw)));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (base >= items) break;
    const long long item = base + b.lane;
    if (b.lane < cpw && item < items) {
      const int seg = later + static_cast<int>(item / nchains);
      const int q = static_cast<int>(item % nchains);
      const int i = later ? j.work2[q] : (listed ? j.work[q] : q);
      const int64_t seg_start = static_cast<int64_t>(seg) * j.seg_len;
      int64_t found = 0;
      if (__ldcg(&j.kmin[i]) > static_cast<unsigned long long>(seg_start)) {   // no accepted sample before this segment yet
        const int x = j.xused[i];
        if (x < 0) {
          found = 1;   // job's first joint: chain 0 is kept whole
        } else {
          TestHook hk;
          kept_test_setup(j, hk, wl, slack, i, x, seg_start, r);
          Src::segment(j, b, i, seg, S, hk);
          found = hk.found;
          searched += hk.k - seg_start;
        }
        if (found > 0) atomicMin(&j.kmin[i], static_cast<unsigned long long>(found));
        else if (!later) j.work2[atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatNoHit]), 1ull)] = i;
      }
    }
    __syncwarp();
  }
  if (searched)
    atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatSearched]), static_cast<unsigned long long>(searched));
}

// A lower bound of every chain's second-best v before the pass over its
// samples, so that the pass's filter is tight from the start (without it each
// segment's first samples pass: 15 of 2048 a lane, a quarter of the warps'
// iterations): the second best of up to 1024 samples spread over the chain,
// one warp a chain.  Starts the chain's entry; the chains before the first
// pending one are marked settled.
__device__ __forceinline__ void height_top2(float v, float& best, float& second) {
  second = fmaxf(second, fminf(best, v));
  best = fmaxf(best, v);
}
template <class Src>
__global__ void __launch_bounds__(128) kept_seed_kernel(const DevJob j, const int64_t S, const uint32_t r) {
  after_previous();
  if (j.stats[kStatPending] == 0) return;
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const float* wl = level_weights(j);
  const int lane = threadIdx.x & 31;
  const int64_t M = S * j.N;
  const int n = Src::seeds(j, M);
  const int nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < j.p; q += nwarps) {
    const int i = j.perm[q];
    if (q < f) {   // (its answer stands)
      if (lane == 0) {
        Height h = height_none();
        h.m = kSettled;
        heights(j)[i] = h;
      }
      continue;
    }
    float best = height_none().best, second = best;
    for (int a = lane; a < n; a += 32) {
      int64_t k;   // distinct samples (0-based)
      const int m = Src::seed(j, i, a, n, M, &k);
      const uint4 v = philox4x32_10(make_uint4(static_cast<uint32_t>(k >> 2), r, static_cast<uint32_t>(i), kTagJoint),
                                    j.key0, j.key1);
      height_top2(wl[m] + height_draw(uint4_word(v, static_cast<uint32_t>(k & 3))), best, second);
    }
    for (int o = 16; o > 0; o >>= 1) {
      const float b2 = __shfl_xor_sync(0xFFFFFFFFu, best, o), s2 = __shfl_xor_sync(0xFFFFFFFFu, second, o);
      height_top2(b2, best, second);
      second = fmaxf(second, s2);
    }
    if (lane == 0) {
      Height h = height_none();
      h.second = second;
      heights(j)[i] = h;
    }
  }
}

// Heights of the chains from the first pending one on: items as in the
// search, all segments.  Lanes take the chains by index, whatever the joint's
// order, so that a warp reads whole runs of the record (taken in the order of
// an ordered joint, a warp's loads were 32 separate sectors each: L = 52,
// p = 1000, S = 100 0.75 ms a pass, 0.33 now).
template <class Src>
__global__ void __launch_bounds__(32 * kKeptWarps, 2) kept_height_kernel(const DevJob j, const int cpw, const int64_t S,
                                                          const uint32_t r) {
  after_previous();
  if (j.stats[kStatPending] == 0) return;
  const long long items = static_cast<long long>(j.p) * j.ck_K;
  const SmemPlan sp = smem_plan(j.L, Src::kPlacement, cpw, blockDim.x >> 5, false, true);
  BlockCtx b = block_setup<false>(j, sp, cpw, 0, false);
  const float* wl = kept_weights(j, b);
  const float slack = height_slack(j);
  unsigned long long* queue = kept_queue(j, kStatQueueSearch);
  long long searched = 0;
  for (;;) {
    long long base = 0;
    if (b.lane == 0) base = static_cast<long long>(atomicAdd(queue, static_cast<unsigned long long>(cpw)));
    base = __shfl_sync(0xFFFFFFFFu, base, 0);
    if (base >= items) break;
    const long long item = base + b.lane;
    const int i = static_cast<int>(item % j.p), seg = static_cast<int>(item / j.p);
    if (b.lane < cpw && item < items && __ldcg(&heights(j)[i].m) != kSettled) {
      HeightHook hk;
      hk.wl = wl;
      hk.entry = heights(j) + i;
      hk.slack = slack;
      hk.k = static_cast<int64_t>(seg) * j.seg_len;
      hk.chain = static_cast<uint32_t>(i);
      hk.r = r;
      hk.k0 = j.key0;
      hk.k1 = j.key1;
      hk.done = false;
      hk.begin();
      const int64_t k_begin = hk.k;
      Src::segment(j, b, i, seg, S, hk);
      if (hk.h.m != kNoLevel) height_store_max(heights(j) + i, hk.h);
      searched += hk.k - k_begin;
    }
    __syncwarp();
  }
  if (searched)
    atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatSearched]), static_cast<unsigned long long>(searched));
}

// The samples to count into dpre: the kept ones where they are fewer than
// the discarded ones (kStatCountKept), else the discarded ones (the samples
// before k_i, the whole chain if nothing is kept), of the chains listed in
// work2.  Every (segment, chain) pair, dealt out in turn, segment-major; a
// block counts at most its share of the round (below 2^32: the rounds kept
// hold at most 2^36 samples, and a grid is smaller than the chip only when
// there are few items).
template <class Src>
__global__ void __launch_bounds__(32 * kKeptWarps, 2) kept_count_kernel(const DevJob j, const int cpw, const int64_t S) {
  after_previous();
  const int nchains = static_cast<int>(j.stats[kStatNoHit]);
  const long long items = static_cast<long long>(nchains) * j.ck_K;
  const int slots = (blockDim.x >> 5) * cpw;
  if (static_cast<long long>(blockIdx.x) * slots >= items) return;
  const SmemPlan sp = smem_plan(j.L, Src::kPlacement, cpw, blockDim.x >> 5, false, true);
  BlockCtx b = block_setup<false>(j, sp, cpw, 0, true);
  __syncthreads();
  const int64_t M = S * j.N;
  const bool kept = j.stats[kStatCountKept] != 0;
  for (long long base = static_cast<long long>(blockIdx.x) * slots; base < items;
       base += static_cast<long long>(gridDim.x) * slots) {
    const long long item = base + b.slot;
    if (b.lane < cpw && item < items) {
      const int i = j.work2[item % nchains], seg = static_cast<int>(item / nchains);
      const int64_t k = j.k[i];
      int64_t lo = kept ? (k > 0 ? k - 1 : M) : 0;                // 0-based, [lo, hi)
      int64_t hi = kept ? M : (k > 0 ? k - 1 : M);
      const int64_t s0 = static_cast<int64_t>(seg) * j.seg_len, s1 = min(M, s0 + j.seg_len);
      lo = max(lo, s0);
      hi = min(hi, s1);
      if (lo < hi) {
        CountHook hk{b.hist, static_cast<int>(lo - s0), static_cast<uint32_t>(hi - lo), 0, false};
        Src::segment(j, b, i, seg, S, hk);
      }
    }
    __syncwarp();
  }
  asm volatile("" ::: "memory");
  __syncthreads();
  for (int m = threadIdx.x; m < j.np1; m += blockDim.x) {
    const uint32_t v = b.hist[m];
    if (v) atomicAdd(&j.dpre[m], static_cast<unsigned long long>(v));
  }
}

// The last resort (an answer the heights could not give): search the pending
// chains, one block, until no input changes.
template <class Src>
__global__ void __launch_bounds__(128) kept_resolve_kernel(const DevJob j, const int cpw, const int64_t S,
                                                           const uint32_t r) {
  after_previous();
  if (j.stats[kStatPending] == 0) return;
  const SmemPlan sp = smem_plan(j.L, Src::kPlacement, cpw, blockDim.x >> 5, false, true);
  BlockCtx b = block_setup<false>(j, sp, cpw, 0, false);
  const float* wl = kept_weights(j, b);
  const float slack = height_slack(j);
  __shared__ int s_tmp[128];
  __shared__ int s_count;
  __shared__ unsigned long long s_sum;
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  const int64_t M = S * j.N;
  long long searched = 0;
  int passes = 0, mism_total = 0;
  for (;;) {
    block_last_accepted(j, s_tmp, j.work);
    if (threadIdx.x == 0) s_count = 0;
    __syncthreads();
    for (int q = threadIdx.x; q < j.p; q += blockDim.x) {   // positions in the joint
      const int last = j.work[q];
      const int x = (last >= 0) ? j.m[j.perm[last]] : carry_in;
      const int i = j.perm[q];
      if (x != j.xused[i] || j.k[i] < 0) {
        j.xused[i] = x;
        j.k[i] = -1;   // marked: to be searched (again)
        atomicAdd(&s_count, 1);
      }
    }
    __syncthreads();
    const int count = s_count;
    if (count == 0 || passes > j.p) break;
    ++passes;
    mism_total += count;
    if (threadIdx.x == 0) {
      int n = 0;
      for (int i = 0; i < j.p; ++i)
        if (j.k[i] == -1) j.work[n++] = i;
    }
    __syncthreads();
    if (b.lane < cpw) {
      for (int q = b.slot; q < count; q += b.nslot) {
        const int i = j.work[q];
        if (j.xused[i] < 0) {
          j.k[i] = 1;
          continue;
        }
        TestHook hk;
        kept_test_setup(j, hk, wl, slack, i, j.xused[i], 0, r);
        hk.kmin = nullptr;
        for (int sg = 0; sg < j.ck_K && !hk.done; ++sg) Src::segment(j, b, i, sg, S, hk);
        j.k[i] = hk.found;
        searched += hk.k;
      }
    }
    __syncthreads();
  }
  // the carry for the next round, and what to count
  if (threadIdx.x == 0) s_sum = 0ull;
  __syncthreads();
  unsigned long long sum = 0;
  for (int i = threadIdx.x; i < j.p; i += blockDim.x) sum += j.k[i] > 0 ? static_cast<unsigned long long>(M - j.k[i] + 1) : 0ull;
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(&s_sum, sum);
  __syncthreads();
  if (threadIdx.x == 0) {
    int last = -1;
    for (int q = j.p - 1; q >= 0 && last < 0; --q)
      if (j.k[j.perm[q]] > 0) last = j.perm[q];
    if (last >= 0) {
      j.stats[kStatCarry] = j.m[last];
      j.stats[kStatCarryValid] = 1;
    }
    j.stats[kStatCountKept] = 2ull * s_sum < static_cast<unsigned long long>(j.p) * static_cast<unsigned long long>(M);
    j.stats[kStatMismatch] += mism_total;
    j.stats[kStatPasses] += passes;
    j.stats[kStatNoHit] = 0;
  }
  __syncthreads();
  kept_list_counted(j);
  if (searched) atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatSearched]),
                          static_cast<unsigned long long>(searched));
}

// ------------------------------------------------------------------ host side
// Warps a block of a pass over so many items: the passes wait on each warp's
// own chain of operations, so what counts is the warps an SM holds, and a
// block's warps share one copy of the level weights (64 KiB at L = 128).  From
// four warps up to kKeptWarps, as many as let an SM hold more of them -- where
// the items fill the chip (fewer are spread over it in small blocks).
// Measured, four warps a block and then this: L = 64, 1.7e10 samples, flips (64
// KiB of lattices each four warps: 8 warps an SM, 12 now) heights 20.6 -> 19.3
// ms, counts 3.8 -> 1.7; L = 128, 3.4e9 samples, recorded (12 warps an SM, 24
// now) heights 3.0 -> 3.0 ms, counts 1.10 -> 0.66.
inline LaunchShape kept_shape(const DevJob& j, LaunchShape s, long long items) {
  const auto held = [&](int wpb) {
    const LaunchShape t{s.placement, s.cpw, wpb};
    return std::min<int>(2 * kKeptWarps, static_cast<int>((kMaxSmem + 1024) / (plan_bytes(j.L, t, false, true) + 2048)) * wpb);
  };
  const int base = s.wpb;
  if (items < 152ll * s.cpw * std::max(1, held(base))) return s;
  for (int wpb = 2 * base; wpb <= kKeptWarps; wpb += base)
    if (held(wpb) > held(s.wpb)) s.wpb = wpb;
  return s;
}

// s: lanes a warp and warps a block of the passes over segments (Src's
// lattices and the level weights fit in shared memory).
template <class Src>
inline cudaError_t launch_join_kept(const DevJob& j, const LaunchShape& s, int64_t S, uint32_t r, cudaStream_t st) {
  auto kq = kept_search_kernel<Src>;
  auto kh = kept_height_kernel<Src>;
  auto kc = kept_count_kernel<Src>;
  auto kr = kept_resolve_kernel<Src>;
  cudaError_t e;
  const long long items = static_cast<long long>(j.p) * j.ck_K;
  const LaunchShape all = kept_shape(j, s, items), one = kept_shape(j, s, j.p);   // all segments; one a chain
  const size_t bytes = plan_bytes(j.L, s, false, true), all_bytes = plan_bytes(j.L, all, false, true),
               one_bytes = plan_bytes(j.L, one, false, true);
  if ((e = allow_smem(kq)) != cudaSuccess || (e = allow_smem(kh)) != cudaSuccess || (e = allow_smem(kc)) != cudaSuccess ||
      (e = allow_smem(kr)) != cudaSuccess)
    return e;
  const auto grid = [&](auto kern, const LaunchShape& t, size_t b, long long n) {
    return static_cast<unsigned>(std::max<long long>(
        1, std::min<long long>(blocks_for(n, t.cpw * t.wpb), resident_blocks(kern, 32 * t.wpb, b))));
  };
  const unsigned grid_one = grid(kq, one, one_bytes, j.p), grid_later = grid(kq, all, all_bytes, items);
  // (the default limit is the replays': a kept round of any size may take the exact path)
  const bool exact = static_cast<long long>(j.p) * S * j.N <= j.scan_max_samples || j.scan_max_samples == kScanMaxSamples;
  auto search = [&](int listed, int first) -> cudaError_t {
    launch_next(kq, grid_one, 32 * one.wpb, one_bytes, st, j, one.cpw, S, r, listed, 0, first);
    launches_add(1);
    if (j.ck_K > 1) {
      launch_next(kq, grid_later, 32 * all.wpb, all_bytes, st, j, all.cpw, S, r, listed, 1, first);
      launches_add(1);
    }
    return cudaGetLastError();
  };
  int select = exact ? kMarkExactFirst : 0;   // how the next mark takes the last search's results
  const auto mark = [&](int flags) -> cudaError_t {
    const cudaError_t e2 = kept_mark(j, S, select | flags, st);
    select = kMarkListed;
    return e2;
  };
  const auto passes = [&](int n, int flags) -> cudaError_t {
    for (int q = 0; q < n; ++q) {
      cudaError_t e2 = mark(flags);
      if (e2 == cudaSuccess) e2 = search(1, 0);
      if (e2 != cudaSuccess) return e2;
    }
    return cudaSuccess;
  };
  if ((e = kept_prelude(j, st)) != cudaSuccess) return e;
  if ((e = search(0, exact ? 1 : 0)) != cudaSuccess) return e;
  if (exact) {
    // Passes before the heights: a pass reads the pending chains only, and past the replays' limit the heights
    // of all chains cost more than the passes that replays take there (L = 64, 4096 chains of 4000 sweeps, 279
    // rejected: 131 ms with two passes, 53 with up to ten, 50 replayed; L = 128, 1024 of 3000, 160 rejected:
    // 436, 240, 200)
    const bool large = static_cast<long long>(j.p) * S * j.N > j.scan_max_samples;
    if ((e = passes(large ? j.passes_plain : j.passes_scan, large ? kMarkDeferLate : kMarkDefer)) != cudaSuccess) return e;
    if ((e = mark(0)) != cudaSuccess) return e;
    launch_next(kept_seed_kernel<Src>, std::min(2432u, blocks_for(j.p, 4)), 128, 0, st, j, S, r);
    launch_next(kh, grid(kh, all, all_bytes, items), 32 * all.wpb, all_bytes, st, j, all.cpw, S, r);
    launches_add(2);
    if ((e = kept_scan(j, st)) != cudaSuccess) return e;
    if ((e = search(1, 0)) != cudaSuccess) return e;
    if (j.passes_scan > 0) {   // the first pass goes on from an undecided chain, now searched
      if ((e = kept_mark_scan(j, S, kMarkListed, st)) != cudaSuccess) return e;
      if ((e = search(1, 0)) != cudaSuccess) return e;
    }
    if ((e = passes(j.passes_scan - 1, 0)) != cudaSuccess) return e;
  } else {
    if ((e = passes(j.passes_plain, 0)) != cudaSuccess) return e;
  }
  if ((e = mark(kMarkFinal)) != cudaSuccess) return e;
  launch_next(kr, 1, 32 * s.wpb, bytes, st, j, s.cpw, S, r);
  launch_next(kc, grid(kc, all, all_bytes, items), 32 * all.wpb, all_bytes, st, j, all.cpw, S);
  launches_add(2);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  return join_finalize(j, S, st);
}

}  // namespace mcgpu
