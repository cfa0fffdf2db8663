// Generation with one chain per warp (Sec. 2 step 2): the sites of a window
// of the row are resolved together: a lattice word, one site a lane (Words),
// 64 sites, two neighbouring ones a lane (TwoWords; warp_pairs), or several
// rows of a small lattice (ShortRows).
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
// the latency of the solve and of each evaluation (population counts, a table
// load, a compare, a vote), 600 cycles a word, 900 a window of 64; more
// chains -- instruction issue and the integer pipe, 135 instructions a word,
// 270 a window of 64 (at L = 64 and 4096 chains 77 % of the issue slots, the
// integer pipe 77 % busy).  One chain per lane (mc_chain.cuh)
// issues about 35 a site for 32 chains and takes 59 (table in shared memory)
// to 108 (table through L1) cycles a site however few chains there are, so
// this form is the better one up to the chain counts of warp_chain_better().
#pragma once
#include <algorithm>

#include "mc_chain_kernels.cuh"

namespace mcgpu {

constexpr int kRingWords = 256;      // uniforms in flight a warp (two batches of 128 attempts)
constexpr int kTablePad = 160;       // a mask on the way to the fixed point may put a site up to
                                     // 126 levels outside [0, N]: words a table read may stray
static_assert(kRingWords > 128, "the ring before the table takes the strays below it");

// Words a row of the block's own lattice copy (two sites a lane: an even and
// an odd word per window of 64 sites -- as many for the sizes that use it).
__host__ __device__ inline int warp_row_words(int L) { return (L + 31) / 32; }

// Shared memory of a block: [rings][table (opt.)][pad][histogram][lattices], in words.
struct WarpPlan {
  int ring, table, hist, lat, total;
};

__host__ __device__ inline WarpPlan warp_plan(int L, int warps, bool tsmem) {
  const int np1 = L * L + 1;
  WarpPlan w;
  w.ring = 0;
  w.table = kRingWords * warps;
  w.hist = w.table + (tsmem ? ((5 * np1 + 3) & ~3) + kTablePad : 0);
  w.lat = w.hist + ((np1 + 3) & ~3);
  w.total = w.lat + warps * L * warp_row_words(L);
  return w;
}

constexpr int kWarpChainBlock = 32;   // most warps (chains) a block: 64 registers a thread

// Sweeps between flushes of the block's u32 level counters (0: the round fits).
inline int64_t warp_flush_sweeps(int warps, int N, int64_t S) {
  const int64_t f = 0xFFFFFFFFll / (static_cast<int64_t>(warps) * N);
  return S > f ? f : 0;
}

// Two sites a lane (windows of 64) or one (a window a word).  A window of 64
// takes 1.5 times a word's latency, so it wins where it halves the windows of
// a row and latency is the bound: rows of two words at any number of chains
// (9 against 10 ns a site at 1024 chains and L = 64, the same 19 at 4096),
// rows of four with at most two warps a scheduler (L = 100, 32 chains: 9.0
// against 11.8; L = 128, 1024 chains: 9.7 against 11.7; 4096 chains: 31
// against 26).  Rows of three words would still be two windows: one a lane
// (L = 96, 1280 chains: 12.0 against 15.7).
__host__ __device__ inline bool warp_pairs(int L, int p, int num_sms) {
  const int wd = (L + 31) / 32;
  return wd == 2 || (wd == 4 && p <= 8 * num_sms);
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
// in chains per scheduler (p / (4 SMs)); up to 8 are resident.  A job begins
// with young weights, whose visited range ends in cliffs: 2 to 4 evaluations a
// window instead of 1.5, which count where instruction issue is the bound.  So
// the line is where the first ten iterations from W = 0 together are not
// slower, and grown weights have room to spare; past it the form lost (L = 16
// at 4864 36 / 33, L = 48 at 5472 47 / 40, L = 64 at 7296 53 / 41, L = 96 there
// 53 / 51).  L = 64 between 3600 and 4900 chains is the exception: 28 to 35 /
// 28 to 31 over ten iterations, even after 24, 1.2 to 1.5 times faster grown
// (an iteration with its joint is no slower at any of them than it was with
// one chain a lane and the joint of that time).  Measured, ns a site (one a
// warp / one a lane, 152 SMs), the mean of a job's first ten iterations:
//   L = 8     22 / 37 at 1824, 25 / 37 at 2432, 28 / 37 at 3040
//   L = 12    22 / 34 at 1824, 25 / 34 at 2432
//   L = 16    20 / 32 at 2432, 28 / 32 at 3648, 31 / 32 at 4256
//   L = 20    22 / 33 at 2432, 29 / 32 at 3648
//   L = 28    20 / 31 at 3040, 29 / 31 at 4256, 33 / 31 at 4864
//   L = 32    25 / 29 at 3648, 29 / 31 at 4864
//   L = 40    41 / 91 at 4864, 81 / 108 at 8512, 88 / 108 at 9728
//   L = 48    29 / 47 at 3648, 35 / 51 at 4864
//   L = 56    54 / 84 at 7296, 83 / 84 at 9728
//   L = 64    18 / 26 at 2432, 23 / 27 at 3040, 41 / 41 at 5472
//   L = 76    60 / 79 at 7296, 76 / 79 at 9728
//   L = 96    35 / 48 at 4864, 48 / 51 at 6080
// and with grown weights (rounds of 10 to 200 sweeps):
//   L = 8     16 / 37 at 608 or fewer, 25 / 37 at 2432, 33 / 37 at 3600
//   L = 12    15 / 33 at 64, 24 / 33 at 2432, 28 / 35 at 3040, 46 / 33 at 4800
//   L = 16    12 / 33 at 512, 18 / 33 at 2432, 31 / 33 at 4800
//   L = 20    13 / 33 at 512, 27 / 33 at 3600, 35 / 33 at 4800
//   L = 24    23 / 32 at 3600, 30 / 52 at 4800 (lane groups of 4)
//   L = 32    8.0 / 28 at 512 or fewer, 12 / 28 at 2048, 19 / 28 at 4096, 41 / 29 at 5500
//   L = 36    19 / 96 at 2048 (no lane kernel with L fixed at compile time)
//   L = 64    8.1 / 26 at 1024, 19 / 29 at 4096, 33 / 42 at 5500, 43 / 42 at 8192
//   L = 76    39 / 80 at 6000, 50 / 80 at 9000
//   L = 96    13 / 44 at 1280, 19 / 45 at 4096, 40 / 52 at 8192
//   L = 100   8.8 / 53 at 32, 21 / 76 at 4096, 46 / 169 at 8000
//   L = 128   9.2 / 53 at 1024, 20 / 64 at 4096, 59 / 69 at 6000, 88 / 75 at 8192
inline bool warp_chain_better(int L, int p, int num_sms) {
  int most = 8;                                               // one wave
  if (L < 8) most = 0;
  else if (L == 8) most = 6;
  else if (L == 12) most = 5;
  else if (L == 16 || L == 28) most = 7;
  else if (L == 20) most = 6;
  else if (L == 64 || L == 96) most = 10;                     // two waves
  else if (L > 32 && L <= 100 && L != 48) most = 16;
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

// Flips along a row of sites of which lane l's flips iff its left neighbour
// (lane l - 1) did and H1 says so, or did not and H0 says so; H0 and H1 agree
// at lane 0.  The nearest lane at or before l where they agree fixes the
// flip there; each lane between where only the unflipped neighbour lets the
// site flip inverts it.
__device__ __forceinline__ uint32_t warp_solve(uint32_t H0, uint32_t H1, uint32_t le) {
  const uint32_t dif = H0 ^ H1;
  const int anchor = 31 - __clz(~dif & le);
  const uint32_t inv = dif & H0 & le & (0xFFFFFFFEu << anchor);
  return __ballot_sync(0xFFFFFFFFu, ((H0 >> anchor) ^ __popc(inv)) & 1u);
}

// The fixed-point loops, written as PTX blocks so that their branch is
// uniform (as C++ loops the compiler re-converged the warp at every vote: 10 %
// slower).  Both end after at most one evaluation a site: the sites before
// the first wrong one stay right.
#define MC_LOAD_SHARED(at, to) "ld.shared.u32 " to ", [" at "];\n\t"
#define MC_LOAD_GLOBAL(at, to, T, last)            \
  "min.u32 " at ", " at ", " last ";\n\t"          \
  "{ .reg .b64 g; cvt.u64.u32 g, " at "; add.s64 g, g, " T "; ld.global.nc.u32 " to ", [g]; }\n\t"

// One site a lane.  Returns this lane's level change before its site (lane 0,
// whose `before` is the whole word: of the word).
#define MC_EVAL1(WRAP_, LOAD_)                                       \
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
#define MC_EVAL_WRAP(at, F, delta)         \
  "and.b32 x, " F ", 1;\n\t"               \
  "setp.eq.u32 q, x, 0;\n\t"               \
  "@q add.s32 " at ", " at ", " delta ";\n\t"
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
    if constexpr (TSMEM) asm volatile(MC_EVAL1(MC_EVAL_WRAP("at", "%0", "%10"), MC_LOAD_SHARED("at", "t")) MC_EVAL_ARGS);
    else asm volatile(MC_EVAL1(MC_EVAL_WRAP("at", "%0", "%10"), MC_LOAD_GLOBAL("at", "t", "%13", "%14")) MC_EVAL_ARGS);
  } else {
    if constexpr (TSMEM) asm volatile(MC_EVAL1("", MC_LOAD_SHARED("at", "t")) MC_EVAL_ARGS);
    else asm volatile(MC_EVAL1("", MC_LOAD_GLOBAL("at", "t", "%13", "%14")) MC_EVAL_ARGS);
  }
#undef MC_EVAL_ARGS
  return d;
}
#undef MC_EVAL1

// Two sites a lane: masks of the even and of the odd sites; the even site's
// left neighbour is the odd site of the lane before, the odd site's is the
// lane's own even site.  Returns the level change before the even site (lane
// 0: of the window) and, in `mid`, 4 times the change before the odd one.
#define MC_EVAL2(WRAP_, LOAD_E_, LOAD_O_)                            \
  "{\n\t"                                                            \
  ".reg .pred p, q, r, v;\n\t"                                       \
  ".reg .b32 fs, x, a, b, c, e, f, g, t, ae, ao, mv;\n\t"            \
  "setp.ne.u32 v, %22, 0;\n\t"                                       \
  "EVAL:\n\t"                                                        \
  "shl.b32 fs, %1, 1;\n\t"                                           \
  "and.b32 x, %0, %10;\n\t"                                          \
  "and.b32 t, %1, %10;\n\t"                                          \
  "and.b32 a, x, %4;\n\t"                                            \
  "lop3.b32 b, fs, %6, x, 0x28;\n\t"                                 \
  "and.b32 c, x, %5;\n\t"                                            \
  "and.b32 e, t, %7;\n\t"                                            \
  "lop3.b32 f, %0, %9, t, 0x28;\n\t"                                 \
  "and.b32 g, t, %8;\n\t"                                            \
  "popc.b32 a, a;\n\t"                                               \
  "popc.b32 b, b;\n\t"                                               \
  "popc.b32 c, c;\n\t"                                               \
  "popc.b32 e, e;\n\t"                                               \
  "popc.b32 f, f;\n\t"                                               \
  "popc.b32 g, g;\n\t"                                               \
  "and.b32 x, fs, %11;\n\t"                                          \
  "setp.ne.u32 q, x, 0;\n\t"                                         \
  "and.b32 x, %0, %11;\n\t"                                          \
  "setp.ne.u32 r, x, 0;\n\t"                                         \
  "selp.b32 ae, %13, %12, q;\n\t"                                    \
  "selp.b32 ao, %15, %14, r;\n\t"                                    \
  "selp.b32 mv, %17, %16, q;\n\t"                                    \
  "selp.b32 mv, mv, 0, r;\n\t" WRAP_                                 \
  "add.s32 a, a, b;\n\t"                                             \
  "add.s32 e, e, f;\n\t"                                             \
  "add.s32 c, c, g;\n\t"                                             \
  "add.s32 a, a, e;\n\t"                                             \
  "mad.lo.s32 %2, c, -2, a;\n\t"                                     \
  "mad.lo.s32 ae, %2, %18, ae;\n\t"                                  \
  "mad.lo.s32 %3, %2, %18, mv;\n\t"                                  \
  "add.s32 ao, ao, %3;\n\t" LOAD_E_ LOAD_O_                          \
  "setp.le.and.u32 p, %19, a, v;\n\t"                                \
  "setp.le.and.u32 q, %20, b, v;\n\t"                                \
  "vote.sync.ballot.b32 a, p, 0xffffffff;\n\t"                       \
  "vote.sync.ballot.b32 b, q, 0xffffffff;\n\t"                       \
  "xor.b32 c, a, %0;\n\t"                                            \
  "lop3.b32 c, b, %1, c, 0xBE;\n\t"                                  \
  "setp.ne.u32 q, c, 0;\n\t"                                         \
  "mov.b32 %0, a;\n\t"                                               \
  "mov.b32 %1, b;\n\t"                                               \
  "@q bra.uni EVAL;\n\t"                                             \
  "}"
template <bool WRAP, bool TSMEM>
__device__ __forceinline__ int warp_fixed_point2(uint32_t& FE, uint32_t& FO, int& mid, uint32_t s0E, uint32_t nsE,
                                                 uint32_t elE, uint32_t s0O, uint32_t nsO, uint32_t elO,
                                                 uint32_t before, uint32_t bit, int rowE, int rowE1, int rowO,
                                                 int rowO1, int moveE, int moveE1, int scale, uint32_t uE, uint32_t uO,
                                                 int dwrap, bool valid, const uint32_t* __restrict__ T, uint32_t last) {
  int d;
#define MC_EVAL_ARGS                                                                                              \
  : "+r"(FE), "+r"(FO), "=&r"(d), "=&r"(mid)                                                                      \
  : "r"(s0E), "r"(nsE), "r"(elE), "r"(s0O), "r"(nsO), "r"(elO), "r"(before), "r"(bit), "r"(rowE), "r"(rowE1),     \
    "r"(rowO), "r"(rowO1), "r"(moveE), "r"(moveE1), "r"(scale), "r"(uE), "r"(uO), "r"(dwrap),                     \
    "r"(static_cast<uint32_t>(valid)), "l"(T), "r"(last)
  if constexpr (TSMEM) {
    if constexpr (WRAP)
      asm volatile(MC_EVAL2(MC_EVAL_WRAP("ao", "%0", "%21"), MC_LOAD_SHARED("ae", "a"), MC_LOAD_SHARED("ao", "b")) MC_EVAL_ARGS);
    else
      asm volatile(MC_EVAL2("", MC_LOAD_SHARED("ae", "a"), MC_LOAD_SHARED("ao", "b")) MC_EVAL_ARGS);
  } else {
    if constexpr (WRAP)
      asm volatile(MC_EVAL2(MC_EVAL_WRAP("ao", "%0", "%21"), MC_LOAD_GLOBAL("ae", "a", "%23", "%24"), MC_LOAD_GLOBAL("ao", "b", "%23", "%24")) MC_EVAL_ARGS);
    else
      asm volatile(MC_EVAL2("", MC_LOAD_GLOBAL("ae", "a", "%23", "%24"), MC_LOAD_GLOBAL("ao", "b", "%23", "%24")) MC_EVAL_ARGS);
  }
#undef MC_EVAL_ARGS
  return d;
}
#undef MC_EVAL2
#undef MC_EVAL_WRAP

// One site a lane, several short rows a window: F also flips the sites above
// (a row earlier) and, at the row's end, the site at its start, so the masks
// are made from F each time.
#define MC_EVALR(LOAD_)                                              \
  "{\n\t"                                                            \
  ".reg .pred p, q, v;\n\t"                                          \
  ".reg .b32 fu, fr, el, s0, n1, x, a, b, c, at, t, fn;\n\t"         \
  "setp.ne.u32 v, %16, 0;\n\t"                                       \
  "EVAL:\n\t"                                                        \
  "shl.b32 fu, %0, %8;\n\t"                                          \
  "and.b32 fr, %0, %7;\n\t"                                          \
  "shl.b32 fr, fr, %9;\n\t"                                          \
  "shl.b32 el, %0, 1;\n\t"                                           \
  "lop3.b32 el, el, %7, %6, 0x9A;\n\t"                               \
  "lop3.b32 s0, %2, fu, fr, 0x96;\n\t"                               \
  "xor.b32 fu, %3, fu;\n\t"                                          \
  "xor.b32 fr, %5, fr;\n\t"                                          \
  "lop3.b32 n1, fu, %4, fr, 0x17;\n\t"                               \
  "and.b32 x, %0, %10;\n\t"                                          \
  "and.b32 a, x, s0;\n\t"                                            \
  "and.b32 b, x, el;\n\t"                                            \
  "and.b32 c, x, n1;\n\t"                                            \
  "popc.b32 a, a;\n\t"                                               \
  "popc.b32 b, b;\n\t"                                               \
  "popc.b32 c, c;\n\t"                                               \
  "mov.b32 at, %12;\n\t"                                             \
  "and.b32 t, s0, %11;\n\t"                                          \
  "setp.ne.u32 q, t, 0;\n\t"                                         \
  "@q add.s32 at, at, %13;\n\t"                                      \
  "and.b32 t, el, %11;\n\t"                                          \
  "setp.ne.u32 q, t, 0;\n\t"                                         \
  "@q add.s32 at, at, %13;\n\t"                                      \
  "and.b32 t, n1, %11;\n\t"                                          \
  "setp.ne.u32 q, t, 0;\n\t"                                         \
  "@q mad.lo.s32 at, %13, -2, at;\n\t"                               \
  "add.s32 a, a, b;\n\t"                                             \
  "mad.lo.s32 %1, c, -2, a;\n\t"                                     \
  "mad.lo.s32 at, %1, %14, at;\n\t" LOAD_                            \
  "setp.le.and.u32 p, %15, t, v;\n\t"                                \
  "vote.sync.ballot.b32 fn, p, 0xffffffff;\n\t"                      \
  "setp.ne.u32 q, fn, %0;\n\t"                                       \
  "mov.b32 %0, fn;\n\t"                                              \
  "@q bra.uni EVAL;\n\t"                                             \
  "}"
template <int L, uint32_t COL0, bool TSMEM>
__device__ __forceinline__ int warp_fixed_point_rows(uint32_t& F, uint32_t e0, uint32_t eu, uint32_t ed, uint32_t er,
                                                     uint32_t el, uint32_t before, uint32_t bit, int base, int r1, int scale, uint32_t u, bool valid,
                                                     const uint32_t* __restrict__ T, uint32_t last) {
  int d;
#define MC_EVAL_ARGS                                                                                            \
  : "+r"(F), "=&r"(d)                                                                                           \
  : "r"(e0), "r"(eu), "r"(ed), "r"(er), "r"(el), "n"(COL0), "n"(L), "n"(L - 1), "r"(before), "r"(bit),          \
    "r"(base), "r"(r1), "r"(scale), "r"(u), "r"(static_cast<uint32_t>(valid)), "l"(T), "r"(last)
  if constexpr (TSMEM) asm volatile(MC_EVALR(MC_LOAD_SHARED("at", "t")) MC_EVAL_ARGS);
  else asm volatile(MC_EVALR(MC_LOAD_GLOBAL("at", "t", "%17", "%18")) MC_EVAL_ARGS);
#undef MC_EVAL_ARGS
  return d;
}
#undef MC_EVALR
#undef MC_LOAD_SHARED
#undef MC_LOAD_GLOBAL

// What every window needs of the block and the lane.
struct WarpLane {
  int lane;
  uint32_t bit, lt, le, before;   // this lane, those before it, and it; `before` is everything for lane 0
  int scale;                      // 4; 0 for lane 0, whose sum is the window's
  int r1, r1z, row2;              // a table row in bytes; 0 for lane 0; row 2 at level 0
  const uint32_t* T;
  uint32_t t_last;                // last byte offset of the table (global memory)
  uint32_t hist_a;                // shared address of the level counters
  uint16_t* rec;                  // this lane's place in the round record
  uint32_t* flip;                 // the chain's place in the flip record
};

// Uniforms: a ring in shared memory, filled 128 at a time, a Philox block a lane.
struct WarpRing {
  char* ring;
  int avail = 0;
  uint32_t fill_at = 0, use_at;
  uint64_t blk;
  uint32_t chain, k0, k1;
  __device__ __forceinline__ void need(int nb, int lane) {
    if (avail < nb) {
      const uint4 v =
          philox4x32_10(make_uint4(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32), chain, kTagFlip), k0, k1);
      blk += 32;
      *reinterpret_cast<uint4*>(ring + fill_at + 16 * lane) = v;
      fill_at ^= 512u;
      avail += 128;
      __syncwarp();
    }
    avail -= nb;
  }
  __device__ __forceinline__ void step(int nb) { use_at = (use_at + 4u * nb) & (4u * kRingWords - 1u); }
};

// stores of the round record, opaque to the compiler's memory ordering (nothing here reads it)
__device__ __forceinline__ void st_record1(uint16_t* p, int lvl) {
  asm volatile("st.global.u16 [%0], %1;" ::"l"(p), "h"(static_cast<uint16_t>(lvl)));
}
__device__ __forceinline__ void st_record2(uint16_t* p, uint32_t pair) {
  asm volatile("st.global.u32 [%0], %1;" ::"l"(p), "r"(pair));
}
__device__ __forceinline__ void warp_count(uint32_t addr) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(1u));
}

// Rows of WD words, a window a word: lane l holds site l of the word.
// (L at compile time: 10 % off a window.)
template <int WD, int L>
struct Words {
  static constexpr int kRowWords = WD, kSitesPerLane = 1;
  static constexpr int lw = L - 32 * (WD - 1);   // sites of the last word
  __device__ __forceinline__ static int step() { return 1; }
  uint32_t up[WD], cur[WD];
  __device__ __forceinline__ void begin(const uint32_t* lat) {
#pragma unroll
    for (int w = 0; w < WD; ++w) {
      up[w] = lat[(L - 1) * WD + w];
      cur[w] = lat[w];
    }
  }
  __device__ __forceinline__ static void load(uint32_t* lat, const uint32_t* g, int lane) {
    for (int i = lane; i < L * WD; i += 32) lat[i] = g[i];
  }
  __device__ __forceinline__ static void store(uint32_t* g, size_t stride, const uint32_t* lat, int lane) {
    for (int i = lane; i < L * WD; i += 32) g[i * stride] = lat[i];
  }
  template <bool TSMEM, int KEEP>
  __device__ __forceinline__ void row(uint32_t* lat, int y, int& m, WarpLane& w, WarpRing& ring) {
    const int yp = y + 1 == L ? 0 : y + 1;
    uint32_t dn[WD];
#pragma unroll
    for (int v = 0; v < WD; ++v) dn[v] = lat[yp * WD + v];
#pragma unroll
    for (int v = 0; v < WD; ++v) {
      const bool lastv = v == WD - 1;
      const int nb = lastv ? lw : 32;
      const bool valid = lastv ? w.lane < lw : true, wrap = WD == 1 && w.lane == lw - 1;
      ring.need(nb, w.lane);
      const uint32_t u = *reinterpret_cast<const uint32_t*>(ring.ring + ring.use_at);
      ring.step(nb);
      // agreements with the neighbours: up and left as swept, down and right as they are (the last site of
      // the row sees site 0 as swept: in a one-word row that is taken as flipped, as most attempts are
      // accepted, and corrected where F says otherwise)
      const uint32_t c = cur[v];
      const uint32_t right =
          (c >> 1) | (lastv ? (((WD == 1 ? ~c : cur[0]) & 1u) << (lw - 1)) : (cur[(v + 1) % WD] << 31));
      const uint32_t left =
          (c << 1) | (v > 0 ? (cur[(v + WD - 1) % WD] >> 31) : ((cur[WD - 1] >> (lw - 1)) & 1u));
      const uint32_t eu = ~(c ^ up[v]), ed = ~(c ^ dn[v]), er = ~(c ^ right), el = ~(c ^ left);
      const uint32_t s0 = eu ^ ed ^ er;
      const uint32_t ns1 = ~((eu & ed) | (er & (eu ^ ed)));
      // table entries at the word's first level for an unflipped and a flipped left neighbour (the first
      // site's left neighbour is outside the word: the same)
      int off = w.row2, off1 = w.r1z;
      if (s0 & w.bit) off += w.r1;
      if (ns1 & w.bit) off -= 2 * w.r1;
      if (el & w.bit) {
        off += w.r1;
        off1 = -w.r1z;
      }
      const int dwrap = wrap ? ((er & w.bit) ? -w.r1 : w.r1) : 0;
      const int row = 4 * m + off, row1 = row + off1;
      const uint32_t ta = warp_threshold<TSMEM>(w.T, row, w.t_last);
      const uint32_t tb = warp_threshold<TSMEM>(w.T, row1, w.t_last);
      const uint32_t G0 = __ballot_sync(0xFFFFFFFFu, valid && u <= ta);
      const uint32_t G1 = __ballot_sync(0xFFFFFFFFu, valid && u <= tb);
      uint32_t F = warp_solve(G0, G1, w.le);
      const int d = warp_fixed_point<WD == 1, TSMEM>(F, s0, ns1, el, w.before, w.bit, row, row1, dwrap, w.scale, u,
                                                     valid, w.T, w.t_last);
      // the samples' levels: what the next site finds before its attempt, lane 0's sum after the last
      int lvl = m + __shfl_sync(0xFFFFFFFFu, d, (w.lane + 1) & 31);
      int m1 = m + __shfl_sync(0xFFFFFFFFu, d, 0);
      if constexpr (WD == 1) {
        if (!(F & 1u) && ((F >> (lw - 1)) & 1u)) {   // the last site's move, with site 0 as it is
          const int fix = ((er >> (lw - 1)) & 1u) ? -1 : 1;
          m1 += fix;
          if (wrap) lvl += fix;
        }
      }
      m = m1;
      if (valid) warp_count(w.hist_a + 4u * lvl);
      if constexpr (KEEP == kKeepLevels) {
        if (valid) st_record1(w.rec, lvl);
        w.rec += (nb >> 2) * kRecGroupStride;
      }
      cur[v] = c ^ F;
      if constexpr (KEEP == kKeepFlips) {
        if (w.lane == 0) __stcs(w.flip, F);
        ++w.flip;
      }
    }
    // (every lane stores the same words)
#pragma unroll
    for (int v = 0; v < WD; ++v) {
      lat[y * WD + v] = up[v] = cur[v];
      cur[v] = dn[v];
    }
  }
};

// Even bits of x in the low half, and back.
__device__ __forceinline__ uint32_t bits_even(uint32_t x) {
  x &= 0x55555555u;
  x = (x | (x >> 1)) & 0x33333333u;
  x = (x | (x >> 2)) & 0x0F0F0F0Fu;
  x = (x | (x >> 4)) & 0x00FF00FFu;
  return (x | (x >> 8)) & 0xFFFFu;
}
__device__ __forceinline__ uint32_t bits_spread(uint32_t x) {
  x &= 0xFFFFu;
  x = (x | (x << 8)) & 0x00FF00FFu;
  x = (x | (x << 4)) & 0x0F0F0F0Fu;
  x = (x | (x << 2)) & 0x33333333u;
  return (x | (x << 1)) & 0x55555555u;
}

// Rows of more than 32 sites, in windows of 64: lane l holds sites 2l and
// 2l + 1 of the window, the lattice copy the window's even and odd sites as
// two words (so that neighbours in the row are the other word, or its
// neighbour bit).  Against 32 sites a window, one a lane: half the solves and
// a third fewer evaluations a site (2.1 for 64 sites, 1.6 for 32).
template <int NW, int L>
struct TwoWords {
  static constexpr int kRowWords = 2 * NW, kSitesPerLane = 2;
  static constexpr int wd = (L + 31) / 32, nl = L - 64 * (NW - 1), hl = nl / 2;   // sites and lanes of the last window
  __device__ __forceinline__ static int step() { return 1; }
  uint32_t upE[NW], upO[NW], E[NW], O[NW];
  __device__ __forceinline__ void begin(const uint32_t* lat) {
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      upE[v] = lat[(L - 1) * 2 * NW + 2 * v];
      upO[v] = lat[(L - 1) * 2 * NW + 2 * v + 1];
      E[v] = lat[2 * v];
      O[v] = lat[2 * v + 1];
    }
  }
  __device__ __forceinline__ static void load(uint32_t* lat, const uint32_t* g, int lane) {
    for (int i = lane; i < L * NW; i += 32) {
      const int y = i / NW, v = i % NW;
      const uint32_t a = g[y * wd + 2 * v], b = 2 * v + 1 < wd ? g[y * wd + 2 * v + 1] : 0u;
      lat[2 * i] = bits_even(a) | (bits_even(b) << 16);
      lat[2 * i + 1] = bits_even(a >> 1) | (bits_even(b >> 1) << 16);
    }
  }
  __device__ __forceinline__ static void store(uint32_t* g, size_t stride, const uint32_t* lat, int lane) {
    for (int i = lane; i < L * wd; i += 32) {
      const int y = i / wd, x = i % wd, at = 2 * (y * NW + x / 2), sh = 16 * (x & 1);
      g[i * stride] = bits_spread(lat[at] >> sh) | (bits_spread(lat[at + 1] >> sh) << 1);
    }
  }
  template <bool TSMEM, int KEEP>
  __device__ __forceinline__ void row(uint32_t* lat, int y, int& m, WarpLane& w, WarpRing& ring) {
    const int yp = y + 1 == L ? 0 : y + 1;
    uint32_t dnE[NW], dnO[NW];
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      dnE[v] = lat[yp * 2 * NW + 2 * v];
      dnO[v] = lat[yp * 2 * NW + 2 * v + 1];
    }
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      const bool lastv = v == NW - 1;
      const int nb = lastv ? nl : 64;
      const bool valid = lastv ? w.lane < hl : true;
      ring.need(nb, w.lane);
      const uint2 u = *reinterpret_cast<const uint2*>(ring.ring + ring.use_at);
      ring.step(nb);
      // agreements with the neighbours, as in Words: `pair` between the lane's two sites
      const uint32_t e = E[v], o = O[v];
      const uint32_t left = (o << 1) | (v > 0 ? (O[(v + NW - 1) % NW] >> 31) : ((O[NW - 1] >> (hl - 1)) & 1u));
      const uint32_t right =
          (e >> 1) | (lastv ? (((NW == 1 ? ~e : E[0]) & 1u) << (hl - 1)) : (E[(v + 1) % NW] << 31));
      const uint32_t pair = ~(e ^ o), elE = ~(e ^ left), erO = ~(o ^ right);
      const uint32_t euE = ~(e ^ upE[v]), edE = ~(e ^ dnE[v]), euO = ~(o ^ upO[v]), edO = ~(o ^ dnO[v]);
      const uint32_t s0E = euE ^ edE ^ pair, s0O = euO ^ edO ^ erO;
      const uint32_t nsE = ~((euE & edE) | (pair & (euE ^ edE))), nsO = ~((euO & edO) | (erO & (euO ^ edO)));
      // the moves in levels (aligned neighbours - 2) with an unflipped left neighbour, and their change
      // with a flipped one (none for the window's first site)
      int mE = 0, mO = 0, cE = w.lane ? 1 : 0, cO = 1;
      if (s0E & w.bit) mE += 1;
      if (nsE & w.bit) mE -= 2;
      if (elE & w.bit) mE += 1, cE = -cE;
      if (s0O & w.bit) mO += 1;
      if (nsO & w.bit) mO -= 2;
      if (pair & w.bit) mO += 1, cO = -1;
      int dwrap = 0;
      if constexpr (NW == 1)
        if (w.lane == hl - 1) dwrap = (erO & w.bit) ? -w.r1 : w.r1;
      const int base = 4 * m + w.row2;
      const int rowE = base + mE * w.r1, rowE1 = rowE + cE * w.r1;
      const int rowO = base + mO * w.r1, rowO1 = rowO + cO * w.r1;
      const uint32_t tE0 = warp_threshold<TSMEM>(w.T, rowE, w.t_last);
      const uint32_t tE1 = warp_threshold<TSMEM>(w.T, rowE1, w.t_last);
      const uint32_t tO0 = warp_threshold<TSMEM>(w.T, rowO, w.t_last);
      const uint32_t tO1 = warp_threshold<TSMEM>(w.T, rowO1, w.t_last);
      const uint32_t GE0 = __ballot_sync(0xFFFFFFFFu, valid && u.x <= tE0);
      const uint32_t GE1 = __ballot_sync(0xFFFFFFFFu, valid && u.x <= tE1);
      const uint32_t GO0 = __ballot_sync(0xFFFFFFFFu, valid && u.y <= tO0);
      const uint32_t GO1 = __ballot_sync(0xFFFFFFFFu, valid && u.y <= tO1);
      // solve the odd sites, each pair of sites one step; the even ones follow
      uint32_t FO = warp_solve((GE0 & GO1) | (~GE0 & GO0), (GE1 & GO1) | (~GE1 & GO0), w.le);
      uint32_t FE = ((FO << 1) & GE1) | (~(FO << 1) & GE0);
      int mid;
      const int d = warp_fixed_point2<NW == 1, TSMEM>(FE, FO, mid, s0E, nsE, elE, s0O, nsO, pair, w.before, w.bit, rowE,
                                                      rowE1, rowO, rowO1, 4 * mE, 4 * (mE + cE), w.scale, u.x, u.y,
                                                      dwrap, valid, w.T, w.t_last);
      // the samples' levels: after the even site, what the odd one finds; after the odd site, what the
      // next lane finds (lane 0's sum after the last)
      const int m4 = 4 * m;
      int lo = m + __shfl_sync(0xFFFFFFFFu, d, (w.lane + 1) & 31);
      int m1 = m + __shfl_sync(0xFFFFFFFFu, d, 0);
      if constexpr (NW == 1) {
        if (!(FE & 1u) && ((FO >> (hl - 1)) & 1u)) {   // the last site's move, with site 0 as it is
          const int fix = ((erO >> (hl - 1)) & 1u) ? -1 : 1;
          m1 += fix;
          if (w.lane == hl - 1) lo += fix;
        }
      }
      m = m1;
      if (valid) {
        warp_count(w.hist_a + static_cast<uint32_t>(m4 + mid));
        warp_count(w.hist_a + 4u * lo);
      }
      if constexpr (KEEP == kKeepLevels) {
        if (valid) st_record2(w.rec, (static_cast<uint32_t>(m4 + mid) >> 2) | (static_cast<uint32_t>(lo) << 16));
        w.rec += (nb >> 2) * kRecGroupStride;
      }
      E[v] = e ^ FE;
      O[v] = o ^ FO;
      if constexpr (KEEP == kKeepFlips) {
        // the window's two words in site order: lane l votes for sites l and 32 + l
        const uint32_t half = (w.lane & 1) ? FO : FE;
        const uint32_t w0 = __ballot_sync(0xFFFFFFFFu, (half >> (w.lane >> 1)) & 1u);
        const uint32_t w1 = __ballot_sync(0xFFFFFFFFu, (half >> (16 + (w.lane >> 1))) & 1u);
        const int nw = lastv ? (nl + 31) / 32 : 2;
        if (w.lane < nw) __stcs(w.flip + w.lane, w.lane ? w1 : w0);
        w.flip += nw;
      }
    }
    // (every lane stores the same words)
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      lat[y * 2 * NW + 2 * v] = upE[v] = E[v];
      lat[y * 2 * NW + 2 * v + 1] = upO[v] = O[v];
      E[v] = dnE[v];
      O[v] = dnO[v];
    }
  }
};

// Rows of 8, 12 or 16 sites, 32 / L of them a window (a row a window would
// leave most lanes idle): lane l holds site l of the window in typewriter
// order, the lattice copy a word a window.  The first mask is solved along
// each row with every other site taken as flipped (levels and rows above
// included); 1.2 to 1.6 evaluations follow for grown weights.
template <int L>
struct ShortRows {
  static constexpr int kRowWords = 1, kSitesPerLane = 1;
  static constexpr int R = 32 / L, nb = R * L, top = nb - L, kWindows = L / R;
  static_assert(L % R == 0, "whole windows");
  static constexpr uint32_t sites = nb == 32 ? 0xFFFFFFFFu : (1u << (nb & 31)) - 1u;
  static constexpr uint32_t col0 = L == 8 ? 0x01010101u : (L == 12 ? 0x001001u : 0x00010001u);   // the rows' first sites
  uint32_t prev;
  __device__ __forceinline__ static int step() { return R; }
  __device__ __forceinline__ void begin(const uint32_t* lat) { prev = lat[kWindows - 1]; }
  __device__ __forceinline__ static void load(uint32_t* lat, const uint32_t* g, int lane) {
    for (int v = lane; v < kWindows; v += 32) {
      uint32_t x = 0u;
      for (int q = 0; q < R; ++q) x |= g[v * R + q] << (q * L);
      lat[v] = x;
    }
  }
  __device__ __forceinline__ static void store(uint32_t* g, size_t stride, const uint32_t* lat, int lane) {
    for (int y = lane; y < L; y += 32) g[y * stride] = (lat[y / R] >> ((y % R) * L)) & ((1u << L) - 1u);
  }
  template <bool TSMEM, int KEEP>
  __device__ __forceinline__ void row(uint32_t* lat, int y, int& m, WarpLane& w, WarpRing& ring) {
    const int v = y / R;
    const uint32_t c = lat[v], next = lat[v + 1 == kWindows ? 0 : v + 1];
    ring.need(nb, w.lane);
    const uint32_t u = *reinterpret_cast<const uint32_t*>(ring.ring + ring.use_at);
    ring.step(nb);
    const bool valid = w.lane < nb;
    // agreements with the neighbours, F's flips left out: the row above is the window's own but for its
    // first row, the row below but for its last
    const uint32_t up = (c << L) | (prev >> top), dn = (c >> L) | (next << top);
    const uint32_t right = ((c >> 1) & ~(col0 << (L - 1))) | ((c & col0) << (L - 1));
    const uint32_t left = ((c << 1) & ~col0) | ((c >> (L - 1)) & col0);
    const uint32_t eu = ~(c ^ up), ed = ~(c ^ dn), er = ~(c ^ right), el = ~(c ^ left);
    const uint32_t e0 = eu ^ ed ^ er;
    const int base = 4 * m + w.row2;
    // the first mask: everything flipped but each site's left neighbour, which is solved
    constexpr uint32_t fr = (sites & col0) << (L - 1);
    const uint32_t s1 = e0 ^ (sites << L) ^ fr, eu1 = eu ^ (sites << L), er1 = er ^ fr;
    const uint32_t n1 = ~((eu1 & ed) | (er1 & (eu1 ^ ed))), el1 = el ^ ((sites << 1) & ~col0);
    const uint32_t X = sites & w.before;
    int at = base + w.scale * (__popc(X & s1) + __popc(X & el1) - 2 * __popc(X & n1));
    if (s1 & w.bit) at += w.r1;
    if (n1 & w.bit) at -= 2 * w.r1;
    int at0 = at;   // left neighbour not flipped
    if (el & w.bit) at0 += w.r1;
    if (el1 & w.bit) at += w.r1;
    const uint32_t t0 = warp_threshold<TSMEM>(w.T, at0, w.t_last);
    const uint32_t t1 = warp_threshold<TSMEM>(w.T, at, w.t_last);
    const uint32_t G0 = __ballot_sync(0xFFFFFFFFu, valid && u <= t0);
    const uint32_t G1 = __ballot_sync(0xFFFFFFFFu, valid && u <= t1);
    uint32_t F = warp_solve(G0, G1, w.le);
    const int d = warp_fixed_point_rows<L, col0, TSMEM>(F, e0, eu, ed, er, el, w.before, w.bit, base, w.r1, w.scale,
                                                        u, valid, w.T, w.t_last);
    const int lvl = m + __shfl_sync(0xFFFFFFFFu, d, (w.lane + 1) & 31);
    m += __shfl_sync(0xFFFFFFFFu, d, 0);
    if (valid) warp_count(w.hist_a + 4u * lvl);
    if constexpr (KEEP == kKeepLevels) {
      if (valid) st_record1(w.rec, lvl);
      w.rec += (nb >> 2) * kRecGroupStride;
    }
    if constexpr (KEEP == kKeepFlips) {
      if (w.lane < R) __stcs(w.flip + w.lane, (F >> (w.lane * L)) & ((1u << L) - 1u));
      w.flip += R;
    }
    prev = c ^ F;
    lat[v] = prev;   // (every lane stores the same word)
  }
};

// One block of the round: its warps' chains, first + warp.
template <class Rows, int L, bool TSMEM, int KEEP>
__device__ __forceinline__ void warp_gen_body(const DevJob& j, const uint64_t t0, const int64_t S,
                                              const int64_t flushF, const int do_trace, const int block) {
  extern __shared__ __align__(16) uint32_t smem[];
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);
  constexpr int N = L * L, np1 = N + 1, wd = (L + 31) / 32;
  const WarpPlan pl = warp_plan(L, nthr >> 5, TSMEM);
  uint32_t* hist = smem + pl.hist;
  uint32_t* lat = smem + pl.lat + warp * L * Rows::kRowWords;
  if constexpr (TSMEM)
    for (int i = tid; i < 5 * np1; i += nthr) smem[pl.table + i] = j.T[i];
  for (int i = tid; i < np1; i += nthr) hist[i] = 0u;
  const int chain = block * (nthr >> 5) + warp;
  const bool active = chain < j.p;   // (uniform in a warp)
  uint32_t* spins = j.spins + static_cast<size_t>(active ? chain : 0) * L * wd;
  int m = 0;
  if (active) {
    Rows::load(lat, spins, lane);
    m = j.m[chain];
  }
  __syncthreads();
  WarpLane w;
  w.lane = lane;
  w.bit = 1u << lane;
  w.lt = w.bit - 1u;
  w.le = (w.bit << 1) - 1u;
  w.before = lane ? w.lt : 0xFFFFFFFFu;
  w.scale = lane ? 4 : 0;
  w.r1 = 4 * np1;
  w.r1z = lane ? w.r1 : 0;
  w.row2 = 2 * w.r1 + (TSMEM ? static_cast<int>(__cvta_generic_to_shared(smem + pl.table)) : 0);
  w.T = j.T;
  w.t_last = static_cast<uint32_t>(4 * (5 * np1 - 1));
  w.hist_a = static_cast<uint32_t>(__cvta_generic_to_shared(hist));
  w.rec = nullptr;
  w.flip = nullptr;
  if constexpr (KEEP == kKeepFlips) w.flip = j.flips + static_cast<size_t>(active ? chain : 0) * flip_words(L, S);
  if constexpr (KEEP == kKeepLevels) {
    const int k = Rows::kSitesPerLane * lane;   // this lane's first sample in a window
    w.rec = j.rec + rec_index(active ? chain : 0, 0, S * N) + (k >> 2) * kRecGroupStride + (k & 3);
  }
  WarpRing ring;
  ring.ring = reinterpret_cast<char*>(smem + pl.ring + warp * kRingWords);
  ring.use_at = 4u * Rows::kSitesPerLane * lane;
  ring.blk = (t0 >> 2) + static_cast<uint64_t>(lane);
  ring.chain = static_cast<uint32_t>(chain);
  ring.k0 = j.key0;
  ring.k1 = j.key1;
  int ck_left = 0, seg = 0;
  int64_t fl_left = flushF;
  for (int64_t s = 0; s < S; ++s) {
    if (active) {
      if (j.ckpt && ck_left == 0) {
        // lattice and level at the start of segment s / C, for the joint's replays
        Rows::store(j.ckpt + static_cast<size_t>(seg) * L * wd * j.p + chain, static_cast<size_t>(j.p), lat, lane);
        if (lane == 0) j.ckm[static_cast<size_t>(seg) * j.p + chain] = m;
      }
      Rows rows;
      rows.begin(lat);
#pragma unroll 1
      for (int y = 0; y < L; y += Rows::step()) {
        rows.template row<TSMEM, KEEP>(lat, y, m, w, ring);
        __syncwarp();
      }
      if (do_trace && lane == 0) j.trace[s * j.p + chain] = 4 * m - 2 * N;
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
    Rows::store(spins, 1, lat, lane);
    if (lane == 0) j.m[chain] = m;
  }
  asm volatile("" ::: "memory");
  __syncthreads();
  for (int i = tid; i < np1; i += nthr) {
    const uint32_t v = hist[i];
    if (v) atomicAdd(&j.hgen[i], static_cast<unsigned long long>(v));
  }
}

template <class Rows, int L, bool TSMEM, int KEEP>
__global__ void __launch_bounds__(32 * kWarpChainBlock, 1)
    warp_gen_kernel(const DevJob j, const uint64_t t0, const int64_t S, const int64_t flushF, const int do_trace) {
  warp_gen_body<Rows, L, TSMEM, KEEP>(j, t0, S, flushF, do_trace, blockIdx.x);
}

template <class Rows, int L>
inline cudaError_t launch_warp_rows(const DevJob& j, int warps, bool ts, uint64_t t0, int64_t S, bool trace,
                                    cudaStream_t st) {
  auto kern = ts ? warp_gen_kernel<Rows, L, true, kKeepNone> : warp_gen_kernel<Rows, L, false, kKeepNone>;
  if (j.rec) kern = ts ? warp_gen_kernel<Rows, L, true, kKeepLevels> : warp_gen_kernel<Rows, L, false, kKeepLevels>;
  else if (j.flips) kern = ts ? warp_gen_kernel<Rows, L, true, kKeepFlips> : warp_gen_kernel<Rows, L, false, kKeepFlips>;
  const size_t bytes = 4ull * warp_plan(L, warps, ts).total;
  const cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  kern<<<blocks_for(j.p, warps), 32 * warps, bytes, st>>>(j, t0, S, warp_flush_sweeps(warps, j.N, S), trace ? 1 : 0);
  launches_add(1);
  return cudaGetLastError();
}

#endif  // __CUDACC__

}  // namespace mcgpu
