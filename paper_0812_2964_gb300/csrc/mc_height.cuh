// The joint's exact path for recorded rounds: acceptance heights.
//
// Chain i keeps samples for input level x iff some sample k passes the joint
// test u_k <= thr(W[m_k] - W[x]) (Sec. 2 step 4), that is iff
// u_k < 2^32 exp(W[m_k] - W[x]), that is iff
//     W[x] < max_k v_k,   v_k = W[m_k] - ln(u_k / 2^32).
// So one number per chain -- its height, the largest v_k -- answers every
// input, and the serial rule over chains becomes "the next chain that keeps
// samples after chain q is the first one whose height exceeds W[m_q]": all
// those successors are found independently, and the chains that keep
// samples are the ones reached from the round's input by following them
// (pointer doubling).  Nothing is carried chain by chain.
//
// Heights are kept in floating point, so decisions close to the line are
// made on the sample itself: the chain's entry holds the best sample's level
// and uniform (tested exactly, by the threshold function of the joint) and the
// second-best v, whose upper estimate says whether any other sample could
// pass where the best does not.  What neither settles (the two samples and
// W[x] within rounding of one another) is undecided, and the ordinary
// resolution passes finish from that chain on.
//
// What bounds the pass over the samples: instruction issue and the integer
// pipes -- 24 instructions a sample, most of them the Philox block of four
// samples.  Four samples share one filter (the largest weight against the
// smallest uniform, one exponential) that lets them through to the exact
// bookkeeping only if one may be among the chain's two best.  The uniforms
// are drawn four at a time where they are used: with a lattice word's 32 held
// in registers an SM held 16 warps instead of 24.  Measured, one filter a
// sample and 32 uniforms ahead, and now: L = 32, p = 16384, S = 1000 (flips)
// 18.1 -> 16.0 ms; L = 64, p = 4096, S = 1000 23.8 -> 19.3.  (No sample's
// uniform can be left undrawn however low its level's weight: a uniform of 0
// passes every test.)
#pragma once
#include "mc_chain.cuh"
#include "mc_internal.h"

namespace mcgpu {

// best and second in log2 units relative to the joint's reference weight:
// (W[m] - Wref) / ln 2 + 32 - log2 u
struct alignas(16) Height {
  uint32_t m, u;        // best sample: its level (kNoLevel: none yet) and joint uniform
  float best, second;   // the two largest v
};
constexpr uint32_t kNoLevel = 0xFFFFFFFFu;
constexpr uint32_t kSettled = 0xFFFFFFFEu;   // the level of a chain whose height nothing needs
// |height_value - exact v| stays below half of this: log2 of a float (relative
// error 2^-22 of at most 32, plus the rounding of u) and the rounding of W
constexpr double kHeightEps = 1e-4;

#ifdef __CUDACC__

__device__ __forceinline__ Height* heights(const DevJob& j) { return reinterpret_cast<Height*>(j.summ); }

// The levels' weights (W[m] - Wref) / ln 2, built at the start of the joint
// in the scratch of the energy ordering; Wref is the weight of a level that
// the round met.  A grown job's lie within 2^15 of it; the floats of weights
// further away than kWeightSpan (levels masked by a huge value) would be too
// coarse, or infinite.  As a sample's weight they are replaced by bounds from
// above, infinity or kWeightLow, as the input's by bounds from below: the
// filters then let such samples through, the second-best v stays an upper
// estimate, and the answers are the exact test's, or undecided.
constexpr float kWeightSpan = 1048576.0f;
constexpr float kWeightLow = 1.0f - kWeightSpan;   // (1 above: more than the rounding of sums with it)
__device__ __forceinline__ float level_weight(float v) {
  return v > kWeightSpan ? __int_as_float(0x7F800000) : (v >= -kWeightSpan ? v : kWeightLow);
}
__device__ __forceinline__ float input_weight(float level) {
  return level == kWeightLow ? __int_as_float(static_cast<int>(0xFF800000)) : fminf(level, kWeightSpan);
}
__device__ __forceinline__ float* level_weights(const DevJob& j) { return reinterpret_cast<float*>(j.lvcnt); }
__device__ __forceinline__ double reference_weight(const DevJob& j) { return j.W[j.m[0]]; }

__device__ __forceinline__ Height height_none() {
  Height h;
  h.m = kNoLevel;
  h.u = 0u;
  h.best = h.second = __int_as_float(static_cast<int>(0xFF800000));
  return h;
}

// -log2(u / 2^32); a uniform of 0 passes every test
__device__ __forceinline__ float height_draw(uint32_t u) {
  return u ? 32.0f - __log2f(static_cast<float>(u)) : __int_as_float(0x7F800000);
}

// v of the entry's best sample, from its level and uniform
__device__ __forceinline__ double height_value(const DevJob& j, const Height& h) {
  if (h.m == kNoLevel) return __longlong_as_double(static_cast<long long>(0xFFF0000000000000ull));
  if (h.u == 0u) return __longlong_as_double(0x7FF0000000000000ll);
  return j.W[h.m] + static_cast<double>(height_draw(h.u)) * 0.6931471805599453;
}

// Error of the float weights (log2 units): twice the rounding of the largest.
__device__ __forceinline__ float weight_error(const DevJob& j) {
  return __int_as_float(static_cast<int>(j.stats[kStatWeightMax])) * 0x1p-22f;
}

// What the filters leave between a sample they drop and the line: the weights'
// error and ample room for the exponential's.
__device__ __forceinline__ float height_slack(const DevJob& j) { return 0.01f + weight_error(j); }

// Error of a second-best v: the logarithm's (within 1e-5 at up to 32, sums
// included) and the weights'.  Where the line lies between the second best and
// this above it, the answer is undecided and the scan ends there, so it is no
// wider than that: with height_slack one chain in some 2 10^6 was, and what was
// left of its joint (L = 8, 2^17 chains, one sweep) took 4.5 s instead of 2 ms.
__device__ __forceinline__ float height_error(const DevJob& j) { return 1e-4f + weight_error(j); }

// No other sample of the chain has a larger v (one that a filter dropped lies
// below the second best of that time by nearly height_slack).
__device__ __forceinline__ double height_second(const Height& h, double wref, float error) {
  return wref + (static_cast<double>(h.second) + error) * 0.6931471805599453;
}

__device__ __forceinline__ Height height_load(const Height* p) {
  const uint4 v = __ldcg(reinterpret_cast<const uint4*>(p));
  Height h;
  h.m = v.x;
  h.u = v.y;
  h.best = __uint_as_float(v.z);
  h.second = __uint_as_float(v.w);
  return h;
}

// The entry of two disjoint sets of samples.
__device__ __forceinline__ Height height_merge(const Height& a, const Height& b) {
  Height r = a.best >= b.best ? a : b;
  r.second = fmaxf(fminf(a.best, b.best), fmaxf(a.second, b.second));
  return r;
}

__device__ __forceinline__ void height_store_max(Height* p, const Height& mine) {
  Height cur = height_load(p);
  for (;;) {   // (a failed exchange means another lane's succeeded: at most one retry per lane that merges)
    const Height nw = height_merge(cur, mine);
    if (nw.m == cur.m && nw.u == cur.u && nw.second == cur.second) return;
    const Height old = atomicCAS(p, cur, nw);
    if (old.m == cur.m && old.u == cur.u && __float_as_uint(old.best) == __float_as_uint(cur.best) &&
        __float_as_uint(old.second) == __float_as_uint(cur.second))
      return;
    cur = old;
  }
}

// Whether a sample may pass u / 2^32 < 2^x, x within the filter's slack of
// exact: 1 + u / 2^32 rounded down to 23 bits, against 1 + 2^x and the
// rounding (a NaN passes).
__device__ __forceinline__ bool height_filter(float x, uint32_t u) {
  float e;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(e) : "f"(x));
  const float u1 = __uint_as_float(__funnelshift_r(u, 0x7Fu, 9));
  return !(u1 >= e + 1.0000005f);
}

// The same for any of four samples: the largest weight against the smallest
// uniform.  One exponential for four, and a third of the operations of four
// tests (the exponential's unit takes 8 cycles a warp).
__device__ __forceinline__ bool height_filter4(const float* wl, const int (&m4)[4], float bl, const uint4& u) {
  float w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) w[q] = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(wl) + m4[q]);
  float top;   // (a NaN stays one)
  asm("{.reg .f32 t;\n\tmax.NaN.f32 t, %1, %2, %3;\n\tmax.NaN.f32 %0, t, %4;}"
      : "=f"(top) : "f"(w[0]), "f"(w[1]), "f"(w[2]), "f"(w[3]));
  return height_filter(top - bl, min(__vimin3_u32(u.x, u.y, u.z), u.w));
}

// Which of the four pass it by themselves.
__device__ __forceinline__ uint32_t height_passing(const float* wl, const int (&m4)[4], float bl, const uint4& u) {
  uint32_t r = 0u;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float w = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(wl) + m4[q]);
    if (height_filter(w - bl, uint4_word(u, static_cast<uint32_t>(q)))) r |= 1u << q;
  }
  return r;
}

// Hook of the pass over a segment's samples.  wl[m] = (W[m] - Wref) / ln 2 as
// a float; a sample can be among the best two only if u / 2^32 <
// 2^(wl[m] - bl), bl below the second-best v found so far by more than the
// float weights' and the exponential's errors.
struct HeightHook {
  const float* wl;      // shared memory
  const Height* entry;  // the chain's entry (polled for the other segments' second best)
  float slack, bl;
  int64_t k;
  uint32_t chain, r, k0, k1;
  uint32_t blk;         // the word's first Philox block
  Height h;
  int mq[4];            // the current group of four samples: levels (times 4)
  bool done;            // never set: the whole segment is read
  __device__ __forceinline__ void begin() {
    h = height_none();
    bl = height_load(entry).second - slack;
  }
  __device__ __forceinline__ void poll() { bl = fmaxf(bl, height_load(entry).second - slack); }
  __device__ __forceinline__ void word(int nb) {
    blk = static_cast<uint32_t>(static_cast<uint64_t>(k) >> 2);
    k += nb;
  }
  // (one test, one branch and one copy of the bookkeeping per four samples:
  // unrolled a word at a time, a copy a sample overran the instruction cache)
  __device__ __forceinline__ void sample(int m4, int b) {
    mq[b & 3] = m4;
    if ((b & 3) != 3) return;
    const uint4 u = philox4x32_10(make_uint4(blk + static_cast<uint32_t>(b >> 2), r, chain, kTagJoint), k0, k1);
    if (height_filter4(wl, mq, bl, u)) {
      // (in small rounds every second group has a lane that passes: one turn per passing
      // sample, 28 us a pass at L = 16, p = 512, S = 20 instead of 36 with all four)
#pragma unroll 1
      for (uint32_t left = height_passing(wl, mq, bl, u); left; left &= left - 1u) {
        const int q = __ffs(static_cast<int>(left)) - 1;
        const int mm = q == 0 ? mq[0] : (q == 1 ? mq[1] : (q == 2 ? mq[2] : mq[3]));
        const uint32_t uq = uint4_word(u, static_cast<uint32_t>(q));
        const float wq = *reinterpret_cast<const float*>(reinterpret_cast<const char*>(wl) + mm);
        const float v = uq ? wq + height_draw(uq) : __int_as_float(0x7F800000);
        if (v > h.second) {
          const bool top = v > h.best;
          h.second = top ? h.best : v;
          if (top) {
            h.best = v;
            h.m = static_cast<uint32_t>(mm) >> 2;
            h.u = uq;
          }
        }
      }
      bl = fmaxf(bl, h.second - slack);
    }
  }
};

// The chains whose samples kept_count_kernel counts, into work2 (one block;
// work2 and its counter are free once nothing is searched any more).
__device__ __forceinline__ void kept_list_counted(const DevJob& j) {
  const bool kept = j.stats[kStatCountKept] != 0;
  for (int i = threadIdx.x; i < j.p; i += blockDim.x) {
    const int64_t k = j.k[i];
    if (kept ? k > 0 : k != 1)
      j.work2[atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatNoHit]), 1ull)] = i;
  }
}

// Whether the chain whose entry is h keeps samples for an input level of
// weight wx: 1 yes, 0 no, 2 undecided.
__device__ __forceinline__ int height_accepts(const DevJob& j, const Height& h, double wx, double wref, float error) {
  const double v = height_value(j, h);
  const double eps = kHeightEps + 1e-13 * fabs(wx);
  if (v > wx + eps) return 1;
  if (!(v < wx - eps) && h.m != kNoLevel && h.u <= threshold_det(__dsub_rn(j.W[h.m], wx))) return 1;
  return height_second(h, wref, error) < wx - eps ? 0 : 2;
}

#endif  // __CUDACC__

}  // namespace mcgpu
