// Generation with one chain per warp (Sec. 2 step 2): the 32 sites of a
// lattice word are resolved together, one site a lane.
//
// A chain's attempts are serial -- the level after each decides the next
// one's threshold, and its flip the right neighbour's aligned count -- but
// most decisions do not hang on the exact level: thresholds of neighbouring
// levels lie close together.  So a word is resolved by a fixed-point
// iteration over its flip mask F.  Given any F, every site's level before
// its attempt and its aligned count follow from the sites before it
// (bit masks and population counts), so every lane can evaluate its
// decision at once, and the mask of the decisions is the next F.  The
// decision at site b depends on F only through the sites before b; hence
// after n evaluations the first n sites are those of the serial chain, a
// mask that reproduces itself is the serial chain's, and it is reached after
// at most one evaluation per site.
//
// The first F comes from a solve that is exact in the left neighbour's flip
// and takes the level at the word's start for every site: with both
// outcomes' decisions known (G0 if the left neighbour did not flip, G1 if it
// did), the nearest site at or before b where they agree fixes the flip
// there, and each site between where exactly the unflipped neighbour lets
// the site flip (G0 and not G1) inverts it.  Measured on the CPU for grown
// weights at L = 32..128: the solve and 1.6 evaluations a word on average
// (3.0 to 3.4 evaluations without the solve, 12 for a young weight whose
// visited range ends in a cliff).
//
// What bounds it: few chains (fewer than about four warps a scheduler) --
// the latency of the solve and of each evaluation (two dependent population
// counts, a table load, a compare, a vote); more chains -- instruction
// issue, about 100 instructions a word.  One chain per lane (mc_chain.cuh)
// issues about 35 a site for 32 chains and takes 59 (table in shared memory)
// to 108 (table through L1) cycles a site however few chains there are, so
// this form is the better one up to the chain counts of warp_chain_better().
#pragma once
#include <algorithm>

#include "mc_chain.cuh"
#include "mc_internal.h"

namespace mcgpu {

constexpr int kRingWords = 256;      // uniforms in flight a warp (two batches of 128 attempts)
constexpr int kTablePad = 64;        // a mask on the way to the fixed point may put a site up to
                                     // 62 levels outside [0, N]: words a table read may stray

// Shared memory of a block: [rings][table (opt.)][pad][histogram][lattices], in words.
struct WarpPlan {
  int ring, table, hist, lat, total;
};

__host__ __device__ inline WarpPlan warp_plan(int L, int warps, bool tsmem) {
  const int np1 = L * L + 1, wd = (L + 31) / 32;
  WarpPlan w;
  w.ring = 0;
  w.table = kRingWords * warps;
  w.hist = w.table + (tsmem ? ((5 * np1 + 3) & ~3) + kTablePad : 0);
  w.lat = w.hist + ((np1 + 3) & ~3);
  w.total = w.lat + warps * L * wd;
  return w;
}

constexpr int kWarpChainBlock = 32;   // most warps (chains) a block: 64 registers a thread

// Sweeps between flushes of the block's u32 level counters (0: the round fits).
inline int64_t warp_flush_sweeps(int warps, int N, int64_t S) {
  const int64_t f = 0xFFFFFFFFll / (static_cast<int64_t>(warps) * N);
  return S > f ? f : 0;
}

// Warps a block and the table's place.  The time of a round is set by the
// fullest scheduler (four an SM, a block's warps dealt out in turn), so up to
// one warp a scheduler the chains are spread over the SMs, and above that the
// block size (a multiple of four) with the fewest warps on the fullest SM is
// taken, the larger block where two tie: its chains share one histogram and
// leave more of the SM's memory to the L1 copy of the table.  (Blocks of 14
// put 8 of 28 warps on two schedulers and 6 on the others.)  All blocks are
// resident at once where shared memory allows; the table goes there too if
// that costs no residency.
inline void warp_chain_shape(int L, int p, int num_sms, int* warps, bool* tsmem) {
  const auto bytes = [&](int w, bool ts) { return 4ll * warp_plan(L, w, ts).total + 1024; };
  const long long sm_bytes = 228 * 1024;
  int best = 1, blocks = 1;   // blocks: on the fullest SM
  if (p <= 4 * num_sms) {
    best = (p + num_sms - 1) / num_sms;
  } else {
    int best_load = 1 << 30;
    for (int w = 4; w <= kWarpChainBlock; w += 4) {
      const int resident = static_cast<int>(std::min<long long>(sm_bytes / bytes(w, false), 32 / w));
      if (resident < 1) break;
      const int n = ((p + w - 1) / w + num_sms - 1) / num_sms;   // blocks on the fullest SM
      // blocks that do not fit at once run in whole waves
      const int load = n <= resident ? n * w : (n + resident - 1) / resident * resident * w + w;
      if (load <= best_load) best_load = load, best = w, blocks = std::min(n, resident);
    }
  }
  *warps = best;
  *tsmem = bytes(best, true) <= 227 * 1024 && blocks * bytes(best, true) <= sm_bytes;
}

// Whether p chains run faster one a warp than one a lane.  The line is drawn
// in chains per scheduler (p / (4 SMs)); up to 8 are resident.  Measured, ns a
// site (one a warp / one a lane, rounds of 10 to 200 sweeps, grown weights,
// 152 SMs):
//   L = 8     35 / 37 at 300 chains (a row fills 8 of 32 lanes: left to the lanes)
//   L = 16    19 / 33 at 600, 27 / 33 at 2048, 35 / 33 at 3000
//   L = 20    16 / 33 at 1200, 25 / 33 at 3000
//   L = 32    8.9 / 28 at 512 or fewer, 13 / 28 at 2048, 21 / 28 at 4096, 41 / 29 at 5500
//   L = 36    19 / 96 at 2048 (no lane kernel with L fixed at compile time)
//   L = 64    9.4 / 26 at 1024, 20 / 29 at 4096, 33 / 42 at 5500, 37 / 42 at 8192
//   L = 76    39 / 80 at 6000, 50 / 80 at 9000
//   L = 96    13 / 44 at 1280, 19 / 45 at 4096, 40 / 52 at 8192
//   L = 100   12 / 53 at 32, 23 / 76 at 4096, 46 / 169 at 8000
//   L = 128   12 / 53 at 1024, 25 / 64 at 4096, 59 / 69 at 6000, 88 / 75 at 8192
inline bool warp_chain_better(int L, int p, int num_sms) {
  int most = 8;                                               // one wave
  if (L < 12) most = 0;
  else if (L <= 16) most = 4;
  else if (L <= 24) most = 6;
  else if (L == 48 || L == 64 || L == 96) most = 12;          // two waves
  else if (L > 32 && L <= 100) most = 16;
  return p <= most * 4 * num_sms;
}

#ifdef __CUDACC__

// Threshold at a byte offset.  In shared memory `off` is an address of the
// shared window; the table lies between the rings and the pad, so a stray
// read stays inside the block's memory.  In global memory it is an offset
// into the planar table, clamped into it.
template <bool TSMEM>
__device__ __forceinline__ uint32_t warp_threshold(const uint32_t* __restrict__ T, int off, uint32_t last) {
  if constexpr (TSMEM) {
    uint32_t v;
    asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(off));   // (the table never changes during the kernel)
    return v;
  } else {
    return __ldg(reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(T) + min(static_cast<uint32_t>(off), last)));
  }
}

// Evaluate the flip mask F until it reproduces itself (at most one
// evaluation a site: the sites before the first wrong one stay right).
// Returns this lane's level change before its site (lane 0: of the whole
// word).  Written as one PTX block so that the loop's branch is uniform.
#define MC_EVAL(WRAP_, LOAD_)                                        \
  "{\n\t"                                                            \
  ".reg .pred p, q, v;\n\t"                                          \
  ".reg .b32 fs, x, a, b, c, at, t, fn;\n\t"                         \
  "setp.ne.u32 v, %12, 0;\n\t"                                       \
  "EVAL:\n\t"                                                        \
  "shl.b32 fs, %0, 1;\n\t"                                           \
  "and.b32 x, %0, %5;\n\t"                                           \
  "and.b32 a, x, %2;\n\t"                                            \
  "lop3.b32 b, fs, %4, x, 0x28;\n\t"                                 \
  "and.b32 c, x, %3;\n\t"                                            \
  "popc.b32 a, a;\n\t"                                               \
  "popc.b32 b, b;\n\t"                                               \
  "popc.b32 c, c;\n\t"                                               \
  "and.b32 t, fs, %6;\n\t"                                           \
  "setp.ne.u32 q, t, 0;\n\t"                                         \
  "selp.b32 at, %8, %7, q;\n\t" WRAP_                                \
  "add.s32 a, a, b;\n\t"                                             \
  "mad.lo.s32 %1, c, -2, a;\n\t"                                     \
  "mad.lo.s32 at, %1, %9, at;\n\t" LOAD_                             \
  "setp.le.and.u32 p, %11, t, v;\n\t"                                \
  "vote.sync.ballot.b32 fn, p, 0xffffffff;\n\t"                      \
  "setp.ne.u32 q, fn, %0;\n\t"                                       \
  "mov.b32 %0, fn;\n\t"                                              \
  "@q bra.uni EVAL;\n\t"                                             \
  "}"
#define MC_EVAL_WRAP                       \
  "and.b32 t, %0, 1;\n\t"                  \
  "setp.eq.u32 q, t, 0;\n\t"               \
  "@q add.s32 at, at, %10;\n\t"
#define MC_EVAL_SHARED "ld.shared.u32 t, [at];\n\t"
#define MC_EVAL_GLOBAL                     \
  "min.u32 at, at, %14;\n\t"               \
  "{ .reg .b64 g; cvt.u64.u32 g, at; add.s64 g, g, %13; ld.global.nc.u32 t, [g]; }\n\t"
template <bool WRAP, bool TSMEM>
__device__ __forceinline__ int warp_fixed_point(uint32_t& F, uint32_t s0, uint32_t ns1, uint32_t el, uint32_t before,
                                                uint32_t bit, int row, int row1, int dwrap, int scale, uint32_t u,
                                                bool valid, const uint32_t* __restrict__ T, uint32_t last) {
  int d;
#define MC_EVAL_ARGS                                                                                            \
  : "+r"(F), "=&r"(d)                                                                                           \
  : "r"(s0), "r"(ns1), "r"(el), "r"(before), "r"(bit), "r"(row), "r"(row1), "r"(scale), "r"(dwrap), "r"(u),     \
    "r"(static_cast<uint32_t>(valid)), "l"(T), "r"(last)
  if constexpr (WRAP) {
    if constexpr (TSMEM) asm volatile(MC_EVAL(MC_EVAL_WRAP, MC_EVAL_SHARED) MC_EVAL_ARGS);
    else asm volatile(MC_EVAL(MC_EVAL_WRAP, MC_EVAL_GLOBAL) MC_EVAL_ARGS);
  } else {
    if constexpr (TSMEM) asm volatile(MC_EVAL("", MC_EVAL_SHARED) MC_EVAL_ARGS);
    else asm volatile(MC_EVAL("", MC_EVAL_GLOBAL) MC_EVAL_ARGS);
  }
#undef MC_EVAL_ARGS
  return d;
}
#undef MC_EVAL
#undef MC_EVAL_WRAP
#undef MC_EVAL_SHARED
#undef MC_EVAL_GLOBAL

// 2-byte store of the round record, opaque to the compiler's memory ordering (nothing here reads it)
__device__ __forceinline__ void st_record1(uint16_t* p, int lvl) {
  asm volatile("st.global.u16 [%0], %1;" ::"l"(p), "h"(static_cast<uint16_t>(lvl)));
}

// One block of the round: `warps` chains, chain blockIdx-wise first + warp.
template <int WD, bool TSMEM, bool REC>
__device__ __forceinline__ void warp_gen_body(const DevJob& j, const uint64_t t0, const int64_t S,
                                              const int64_t flushF, const int do_trace, const int block) {
  extern __shared__ __align__(16) uint32_t smem[];
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  const int L = j.L, np1 = j.np1;
  const WarpPlan pl = warp_plan(L, nthr >> 5, TSMEM);
  uint32_t* ring = smem + pl.ring + warp * kRingWords;
  uint32_t* hist = smem + pl.hist;
  uint32_t* lat = smem + pl.lat + warp * L * WD;
  if constexpr (TSMEM)
    for (int i = tid; i < 5 * np1; i += nthr) smem[pl.table + i] = j.T[i];
  for (int i = tid; i < np1; i += nthr) hist[i] = 0u;
  const uint32_t* __restrict__ T = j.T;
  const uint32_t t_last = static_cast<uint32_t>(4 * (5 * np1 - 1));
  const int t_base = TSMEM ? static_cast<int>(__cvta_generic_to_shared(smem + pl.table)) : 0;
  const int chain = block * (nthr >> 5) + warp;
  const bool active = chain < j.p;   // (uniform in a warp)
  int m = 0;
  if (active) {
    const uint32_t* g = j.spins + static_cast<size_t>(chain) * L * WD;
    for (int i = lane; i < L * WD; i += 32) lat[i] = g[i];
    m = j.m[chain];
  }
  __syncthreads();
  const int lw = L - 32 * (WD - 1);
  const uint32_t bit = 1u << lane, lt = bit - 1u, le = (bit << 1) - 1u;
  // lane 0 sums the whole word's level changes instead of the (none) before its site
  const uint32_t before = lane ? lt : 0xFFFFFFFFu;
  const int scale = lane ? 4 : 0;
  const int r1 = 4 * np1, r1z = lane ? r1 : 0;   // a row of the table in bytes; none for site 0's left neighbour
  const int row2 = 2 * r1 + t_base;
  const bool in_last = lane < lw;                // this lane has a site in the row's last word
  const bool wrap = WD == 1 && lane == lw - 1;   // ... the site that sees site 0 of the same word
  int avail = 0;                                 // uniforms in the ring not used yet
  uint32_t fill_at = 0, use_at = 4u * lane;      // ring positions, bytes
  const uint32_t hist_a = static_cast<uint32_t>(__cvta_generic_to_shared(hist));
  uint64_t blk = (t0 >> 2) + static_cast<uint64_t>(lane);   // this lane's next Philox block
  uint16_t* rec = nullptr;
  if constexpr (REC)
    rec = j.rec + rec_index(active ? chain : 0, 0, S * j.N) + (lane >> 2) * kRecGroupStride + (lane & 3);
  int ck_left = 0, seg = 0;
  int64_t fl_left = flushF;
  for (int64_t s = 0; s < S; ++s) {
    if (active) {
      if (j.ckpt && ck_left == 0) {
        // lattice and level at the start of segment s / C, for the joint's replays
        uint32_t* ck = j.ckpt + static_cast<size_t>(seg) * L * WD * j.p + chain;
        for (int i = lane; i < L * WD; i += 32) ck[static_cast<size_t>(i) * j.p] = lat[i];
        if (lane == 0) j.ckm[static_cast<size_t>(seg) * j.p + chain] = m;
      }
      uint32_t up[WD], cur[WD];
#pragma unroll
      for (int w = 0; w < WD; ++w) {
        up[w] = lat[(L - 1) * WD + w];
        cur[w] = lat[w];
      }
#pragma unroll 1
      for (int y = 0; y < L; ++y) {
        uint32_t dn[WD];
        const int yp = (y + 1 == L) ? 0 : y + 1;
#pragma unroll
        for (int w = 0; w < WD; ++w) dn[w] = lat[yp * WD + w];
#pragma unroll
        for (int w = 0; w < WD; ++w) {
          const bool lastw = w == WD - 1;
          const int nb = lastw ? lw : 32;
          const bool valid = lastw ? in_last : true;
          if (avail < nb) {   // the next 128 uniforms, a Philox block a lane
            const uint4 v = philox4x32_10(
                make_uint4(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32), static_cast<uint32_t>(chain),
                           kTagFlip),
                j.key0, j.key1);
            blk += 32;
            *reinterpret_cast<uint4*>(ring + (fill_at >> 2) + 4 * lane) = v;
            fill_at ^= 512u;
            avail += 128;
            __syncwarp();
          }
          const uint32_t u = *reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(ring) + use_at);
          use_at = (use_at + 4u * nb) & (4u * kRingWords - 1u);
          avail -= nb;
          // agreements with the neighbours: up and left as swept, down and right as they are
          // (the last site of a row sees site 0 as swept: in a one-word row it is taken as flipped,
          // as most attempts are accepted, and corrected where F says otherwise)
          const uint32_t c = cur[w];
          const uint32_t right =
              (c >> 1) | (lastw ? (((WD == 1 ? ~c : cur[0]) & 1u) << (lw - 1)) : (cur[(w + 1) % WD] << 31));
          const uint32_t left =
              (c << 1) | (w > 0 ? (cur[(w + WD - 1) % WD] >> 31) : ((cur[WD - 1] >> (lw - 1)) & 1u));
          const uint32_t eu = ~(c ^ up[w]), ed = ~(c ^ dn[w]), er = ~(c ^ right), el = ~(c ^ left);
          const uint32_t s0 = eu ^ ed ^ er;
          const uint32_t ns1 = ~((eu & ed) | (er & (eu ^ ed)));
          // entry of the table at the word's first level for an unflipped and a flipped left neighbour
          // (site 0's left neighbour is outside the word: the same)
          int row = 4 * m + row2, row1 = r1z;
          if (s0 & bit) row += r1;
          if (ns1 & bit) row -= 2 * r1;
          if (el & bit) {
            row += r1;
            row1 = -r1z;
          }
          row1 += row;
          const int dwrap = wrap ? ((er & bit) ? -r1 : r1) : 0;
          // solve with every site at the word's first level
          const uint32_t ta = warp_threshold<TSMEM>(T, row, t_last);
          const uint32_t tb = warp_threshold<TSMEM>(T, row1, t_last);
          const uint32_t G0 = __ballot_sync(0xFFFFFFFFu, valid && u <= ta);
          const uint32_t G1 = __ballot_sync(0xFFFFFFFFu, valid && u <= tb);
          const uint32_t dif = G0 ^ G1;
          const int anchor = 31 - __clz(~dif & le);   // (bit 0 always agrees)
          const uint32_t inv = dif & G0 & le & (0xFFFFFFFEu << anchor);
          uint32_t F = __ballot_sync(0xFFFFFFFFu, ((G0 >> anchor) ^ __popc(inv)) & 1u);
          // evaluate until the mask reproduces itself (at most one evaluation a site)
          const int d = warp_fixed_point<WD == 1, TSMEM>(F, s0, ns1, el, before, bit, row, row1, dwrap, scale, u,
                                                         lastw ? in_last : true, T, t_last);
          // the samples' levels: what the next site finds before its attempt, lane 0's sum after the last
          int lvl = m + __shfl_sync(0xFFFFFFFFu, d, (lane + 1) & 31);
          int m1 = m + __shfl_sync(0xFFFFFFFFu, d, 0);
          if constexpr (WD == 1) {
            if (!(F & 1u) && ((F >> (lw - 1)) & 1u)) {   // the last site's move, with site 0 as it is
              const int fix = ((er >> (lw - 1)) & 1u) ? -1 : 1;
              m1 += fix;
              if (wrap) lvl += fix;
            }
          }
          m = m1;
          if (valid) asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(hist_a + 4u * lvl), "r"(1u));
          if constexpr (REC) {
            if (valid) st_record1(rec, lvl);
            rec += (nb >> 2) * kRecGroupStride;
          }
          cur[w] = c ^ F;
        }
        // (every lane stores the same words)
#pragma unroll
        for (int w = 0; w < WD; ++w) {
          lat[y * WD + w] = cur[w];
          up[w] = cur[w];
          cur[w] = dn[w];
        }
        __syncwarp();
      }
      if (do_trace && lane == 0) j.trace[s * j.p + chain] = 4 * m - 2 * j.N;
    }
    if (ck_left == 0) {
      ck_left = j.ck_C;
      ++seg;
    }
    --ck_left;
    if (flushF > 0 && --fl_left == 0 && s + 1 < S) {
      fl_left = flushF;
      asm volatile("" ::: "memory");
      __syncthreads();
      for (int i = tid; i < np1; i += nthr) {
        const uint32_t v = hist[i];
        if (v) {
          atomicAdd(&j.hgen[i], static_cast<unsigned long long>(v));
          hist[i] = 0u;
        }
      }
      __syncthreads();
    }
  }
  if (active) {
    uint32_t* g = j.spins + static_cast<size_t>(chain) * L * WD;
    for (int i = lane; i < L * WD; i += 32) g[i] = lat[i];
    if (lane == 0) j.m[chain] = m;
  }
  asm volatile("" ::: "memory");
  __syncthreads();
  for (int i = tid; i < np1; i += nthr) {
    const uint32_t v = hist[i];
    if (v) atomicAdd(&j.hgen[i], static_cast<unsigned long long>(v));
  }
}

#endif  // __CUDACC__

}  // namespace mcgpu
