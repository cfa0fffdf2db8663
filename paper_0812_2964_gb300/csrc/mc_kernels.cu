// Kernels of the hot path: initial lattices, threshold table, generation of
// p independent chains (Sec. 2 step 2), the joint by detailed balance (steps
// 3-5) as speculation + resolution + segmented scan, and the weight update
// (Sec. 3.1 Eq. new_weight in logarithms, Sec. 4.2).
#include <atomic>
#include <algorithm>
#include <mutex>
#include <unordered_map>
#include <math_constants.h>

#include "mc_launch.cuh"
#include "mc_chain_kernels.cuh"
#include "mc_height.cuh"
#include "mc_scan_fsm.cuh"
#include "mc_warp_chain.cuh"

namespace mcgpu {

static std::atomic<uint64_t> g_launches{0};
uint64_t launches_add(uint64_t n) { return g_launches.fetch_add(n) + n; }

// (set again at each use: another's cudaDeviceReset puts it back to the default)
cudaError_t allow_smem(const void* kernel) {
  static std::mutex mu;
  static std::unordered_map<const void*, int> limits;   // a block's most less the kernel's own variables
  int bytes = 0;
  {
    std::lock_guard<std::mutex> lk(mu);
    const auto it = limits.find(kernel);
    if (it != limits.end()) bytes = it->second;
  }
  if (bytes == 0) {
    cudaFuncAttributes a;
    const cudaError_t e = cudaFuncGetAttributes(&a, kernel);
    if (e != cudaSuccess) return e;
    bytes = static_cast<int>(kMaxSmem - a.sharedSizeBytes);
    std::lock_guard<std::mutex> lk(mu);
    try {
      limits[kernel] = bytes;
    } catch (...) {   // (no memory: asked for again next time)
    }
  }
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}

// ------------------------------------------------------------------ init
// Step 1: C_1 all up, or random: bit (site & 31) of Philox word q & 3 at
// counter (q >> 2, 0, chain, 2), q = site >> 5, site = y L + x.
__global__ void init_lattice_kernel(const DevJob j, const int start) {
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  const long long total = static_cast<long long>(j.p) * j.L * j.wd;
  if (idx >= total) return;
  const int w = static_cast<int>(idx % j.wd);
  const long long cy = idx / j.wd;
  const int y = static_cast<int>(cy % j.L);
  const uint32_t c = static_cast<uint32_t>(cy / j.L);
  const int x0 = 32 * w, x1 = min(j.L, x0 + 32);
  uint32_t word = 0u;
  if (start == 0) {
    word = (x1 - x0 == 32) ? 0xFFFFFFFFu : ((1u << (x1 - x0)) - 1u);
  } else {
    uint32_t cached = 0xFFFFFFFFu, R = 0u;
    for (int x = x0; x < x1; ++x) {
      const uint32_t site = static_cast<uint32_t>(y * j.L + x);
      const uint32_t q = site >> 5;
      if (q != cached) {
        const uint4 v = philox4x32_10(make_uint4(q >> 2, 0u, c, kTagInit), j.key0, j.key1);
        R = uint4_word(v, q & 3u);
        cached = q;
      }
      word |= ((R >> (site & 31u)) & 1u) << (x - x0);
    }
  }
  j.spins[idx] = word;
}

// Level m = (E + 2N)/4 of each chain's lattice, E = -sum s (s_right + s_down):
// m = N - A/2 with A the aligned pairs.  A warp a chain, a lane a lattice
// word, 32 pairs of each kind at a time (one thread a chain, site by site,
// took 0.4 ms at L = 64 and 1.6 ms at L = 128 whatever the chains).
__global__ void __launch_bounds__(128) levels_kernel(const DevJob j) {
  const int lane = threadIdx.x & 31;
  const int c = static_cast<int>((blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5);
  if (c >= j.p) return;
  const int L = j.L, wd = j.wd, lw = L - 32 * (wd - 1);
  const uint32_t* lat = j.spins + static_cast<size_t>(c) * L * wd;
  int A = 0;
  for (int i = lane; i < L * wd; i += 32) {
    const int y = i / wd, w = i % wd;
    const uint32_t x = lat[i], down = lat[(y + 1 == L ? 0 : y + 1) * wd + w];
    const bool last = w == wd - 1;
    const uint32_t next = last ? lat[y * wd] : lat[i + 1];
    const uint32_t right = (x >> 1) | (next << (last ? lw - 1 : 31));
    const uint32_t sites = last && lw < 32 ? (1u << lw) - 1u : 0xFFFFFFFFu;
    A += __popc(~(x ^ right) & sites) + __popc(~(x ^ down) & sites);
  }
  A = __reduce_add_sync(0xFFFFFFFFu, A);
  if (lane == 0) j.m[c] = j.N - A / 2;
}

// T[a][m] = thr(W[m + a - 2] - W[m]); moves outside [0, N] never occur.
__global__ void table_kernel(const DevJob j) {
  after_previous();
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 5 * j.np1) return;
  const int a = idx / j.np1, m = idx % j.np1;
  const int mp = m + a - 2;
  j.T[idx] = (mp < 0 || mp > j.N) ? 0u : threshold_det(__dsub_rn(j.W[mp], j.W[m]));
}

// Eq. (new_weight) in logarithms: W -= ln h where h > 0; h cleared.
__global__ void weights_kernel(const DevJob j) {
  after_previous();
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= j.np1) return;
  const long long h = j.h[m];
  if (h > 0) {
    j.W[m] = __dsub_rn(j.W[m], log_det(static_cast<double>(h)));
    j.visited[m] = 1;
  }
  j.h[m] = 0;
}

// ------------------------------------------------------------------ part (ii)
// Statistical averages at inverse temperature beta (Sec. 3.2, Eq.
// reweighting2, with E, C, F, S of Sec. 4.1), one block per beta.  D(E) is
// proportional to 1/w(E) = e^{-W(E)} over the levels the weight iteration
// has visited; every sum is taken relative to its largest exponent (the
// logarithmic evaluation of Sec. 4.2).  D counts all 2^N states:
// ln Z = N ln 2 + ln sum e^{-W - beta E} - ln sum e^{-W}.
// C = beta^2 <(H - <H>)^2>, F = -ln Z / beta, S = beta (E - F).
// Reductions are fixed-shape trees, so repeated calls agree bit for bit.
//
// What bounds it: FP64, at two lanes a clock and SM.  So the sum over e^{-W},
// the same for every beta, is made once (thermo_norm_kernel); the exponents
// are looked over in FP32 first, and only levels within 752 of the largest
// -- below, e^x is zero -- are evaluated in FP64, once, their terms kept in
// shared memory for the second moment.  200 betas at L = 64: 47 us (169 with
// three exponentials a level and beta); 10000 at L = 128 2.4 ms (21).
constexpr int kThermoThreads = 256;
constexpr int kThermoParts = 32;          // blocks of the sum over e^{-W}
// -W as a float: -inf marks a level that was not visited (or has no weight at
// all), so one too far below for a float is no number -- which passes every
// test of the FP32 look and leaves the level to FP64.
__device__ __forceinline__ float thermo_exponent(double w) {
  const float n = static_cast<float>(-w);
  return n == -CUDART_INF_F && w < CUDART_INF ? CUDART_NAN_F : n;
}
constexpr float kThermoReach = 752.0f;    // e^{-745.2} is the smallest double; the rest covers the FP32 exponents

// Sums (or maxima) over the block: every thread's value in shared memory, one
// warp a quantity takes 8 each and folds them.  12 FP64 instructions a warp and
// quantity in all; with every warp folding its own and all threads the warps'
// it was 96, and small lattices, whose blocks do little else, took 107 us for
// 1000 betas at L = 8 (71 now; 75 before the FP32 look).  (Two in a row need no
// barrier between them but their own: the values are free once the results are
// there.)
struct BlockFold {
  double v[2][kThermoThreads];
  double r[2];
  __device__ __forceinline__ void put(int which, double x) { v[which][threadIdx.x] = x; }
  // by warp `which` of the block, after a barrier
  template <class Op>
  __device__ __forceinline__ double fold(int which, const Op& op) {
    const int lane = threadIdx.x & 31;
    double x = v[which][lane];
    for (int w = 1; w < kThermoThreads / 32; ++w) x = op(x, v[which][lane + 32 * w]);
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xFFFFFFFFu, x, o));
    if (lane == 0) r[which] = x;
    return x;
  }
};
struct AddOp {
  __device__ double operator()(double a, double b) const { return a + b; }
};
struct MaxOp {
  __device__ double operator()(double a, double b) const { return fmax(a, b); }
};

// Part q of sum e^{-W}: out[2q] = its largest exponent, out[2q + 1] = its sum
// relative to that; and -W as a float (-inf: not visited).
__global__ void __launch_bounds__(kThermoThreads) thermo_norm_kernel(const DevJob j, double* __restrict__ out,
                                                                     float* __restrict__ neg) {
  __shared__ BlockFold f;
  const int warp = threadIdx.x >> 5;
  const int per = (j.np1 + kThermoParts - 1) / kThermoParts;
  const int lo = blockIdx.x * per, hi = min(j.np1, lo + per);
  double bm = -CUDART_INF;
  for (int m = lo + threadIdx.x; m < hi; m += kThermoThreads) {
    const bool on = j.visited[m];
    if (on) bm = fmax(bm, -j.W[m]);
    neg[m] = on ? thermo_exponent(j.W[m]) : -CUDART_INF_F;
  }
  f.put(0, bm);
  __syncthreads();
  if (warp == 0) f.fold(0, MaxOp());
  __syncthreads();
  const double B = f.r[0];
  double sg = 0.0;
  for (int m = lo + threadIdx.x; m < hi; m += kThermoThreads)
    if (j.visited[m] && j.W[m] != CUDART_INF) sg += exp(-j.W[m] - B);   // (a part may hold nothing else)
  f.put(1, sg);
  __syncthreads();
  if (warp == 0) {
    const double SG = f.fold(1, AddOp());
    if (threadIdx.x == 0) {
      out[2 * blockIdx.x] = B;
      out[2 * blockIdx.x + 1] = SG;
    }
  }
}

// OWN: the block makes the sum over e^{-W} itself (small lattices: a launch
// costs more than N + 1 exponentials).
template <bool OWN>
__global__ void __launch_bounds__(kThermoThreads) thermo_kernel(const DevJob j, const double* __restrict__ betas,
                                                                const double* __restrict__ norm,
                                                                const float* __restrict__ neg_in,
                                                                double* __restrict__ out) {
  extern __shared__ double terms[];   // [np1], then (OWN) -W as floats
  __shared__ BlockFold f;
  __shared__ float s_am[kThermoThreads / 32], s_big[kThermoThreads / 32];
  __shared__ int s_lo, s_hi;
  const int t = threadIdx.x, warp = t >> 5, np1 = j.np1, N = j.N;
  const double beta = betas[blockIdx.x];
  const float bf = static_cast<float>(beta);
  float* mine = reinterpret_cast<float*>(terms + np1);
  const float* neg = OWN ? mine : neg_in;   // (each thread reads its own entries, but for the range below)
  // largest exponent, in FP32; its rounding, relative to the largest of either part
  float am = -CUDART_INF_F, big = 0.0f;
  double bm = -CUDART_INF;
  for (int m = t; m < np1; m += kThermoThreads) {
    float n;
    if constexpr (OWN) {
      const bool on = j.visited[m];
      if (on) bm = fmax(bm, -j.W[m]);
      n = on ? thermo_exponent(j.W[m]) : -CUDART_INF_F;
      mine[m] = n;
    } else {
      n = neg[m];
    }
    const float e = bf * static_cast<float>(4 * m - 2 * N);
    if (n != -CUDART_INF_F) {
      am = fmaxf(am, n - e);
      big = fmaxf(big, fmaxf(fabsf(n), fabsf(e)));
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    am = fmaxf(am, __shfl_xor_sync(0xFFFFFFFFu, am, o));
    big = fmaxf(big, __shfl_xor_sync(0xFFFFFFFFu, big, o));
  }
  if ((t & 31) == 0) {
    s_am[warp] = am;
    s_big[warp] = big;
  }
  if (t == 0) {
    s_lo = np1;
    s_hi = 0;
  }
  if constexpr (OWN) f.put(0, bm);
  __syncthreads();
  for (int w = 0; w < kThermoThreads / 32; ++w) {
    am = fmaxf(am, s_am[w]);
    big = fmaxf(big, s_big[w]);
  }
  double B = 0.0, SG = 0.0;
  if constexpr (OWN) {
    if (warp == 0) f.fold(0, MaxOp());
    __syncthreads();
    B = f.r[0];
  }
  const float low = am - kThermoReach - big * 0x1p-20f, top = am - 0.5f - big * 0x1p-20f;
  // the levels within reach lie in [lo, hi); the exact largest exponent, among those that may hold it
  int lo = np1, hi = 0;
  double xm = -CUDART_INF, sg = 0.0;
  for (int m = t; m < np1; m += kThermoThreads) {
    const float n = neg[m];
    const int E = 4 * m - 2 * N;
    const float x = n - bf * static_cast<float>(E);
    if (n != -CUDART_INF_F) {
      if (!(x < low)) {
        lo = min(lo, m);
        hi = m + 1;
        if (!(x < top)) xm = fmax(xm, -j.W[m] - beta * static_cast<double>(E));
      }
      if constexpr (OWN) sg += exp(-j.W[m] - B);
    }
  }
  lo = __reduce_min_sync(0xFFFFFFFFu, lo);
  hi = __reduce_max_sync(0xFFFFFFFFu, hi);
  if ((t & 31) == 0 && hi > 0) {
    atomicMin(&s_lo, lo);
    atomicMax(&s_hi, hi);
  }
  f.put(0, xm);
  if constexpr (OWN) f.put(1, sg);
  __syncthreads();
  if (warp == 0) f.fold(0, MaxOp());
  if constexpr (OWN)
    if (warp == 1) f.fold(1, AddOp());
  __syncthreads();
  const double A = f.r[0];
  if constexpr (OWN) SG = f.r[1];
  lo = s_lo;
  hi = s_hi;
  double z = 0.0, e1 = 0.0;
  for (int m = lo + t; m < hi; m += kThermoThreads) {
    const float n = neg[m];
    const int E = 4 * m - 2 * N;
    double w = 0.0;
    if (n != -CUDART_INF_F && !(n - bf * static_cast<float>(E) < low)) {
      w = exp(-j.W[m] - beta * static_cast<double>(E) - A);
      z += w;
      e1 += static_cast<double>(E) * w;
    }
    terms[m] = w;
  }
  f.put(0, z);
  f.put(1, e1);
  __syncthreads();
  if (warp == 0) f.fold(0, AddOp());
  if (warp == 1) f.fold(1, AddOp());
  __syncthreads();
  const double Z = f.r[0], Eav = f.r[1] / Z;
  double v = 0.0;
  for (int m = lo + t; m < hi; m += kThermoThreads) {
    const double w = terms[m];
    if (w != 0.0) {
      const double d = static_cast<double>(4 * m - 2 * N) - Eav;
      v += d * d * w;
    }
  }
  f.put(0, v);
  __syncthreads();
  if (t < 32) {
    const double V = f.fold(0, AddOp());
    if constexpr (!OWN) {   // ln sum e^{-W} from its parts
      static_assert(kThermoParts == 32, "a lane a part");
      const double b = norm[2 * t], g = norm[2 * t + 1];
      B = b;
      for (int o = 16; o > 0; o >>= 1) B = fmax(B, __shfl_xor_sync(0xFFFFFFFFu, B, o));
      SG = g == 0.0 ? 0.0 : g * exp(b - B);
      for (int o = 16; o > 0; o >>= 1) SG += __shfl_xor_sync(0xFFFFFFFFu, SG, o);
    }
    if (t == 0) {
      const double lnZ = static_cast<double>(N) * log(2.0) + A + log(Z) - (B + log(SG));
      const double F = -lnZ / beta;
      double* o = out + 4 * blockIdx.x;
      o[0] = Eav;
      o[1] = beta * beta * (V / Z);
      o[2] = F;
      o[3] = beta * (Eav - F);
    }
  }
}

// Joint thresholds for each listed chain's input level x: tj[i][m] = thr(W[m] - W[x]).
__global__ void tj_kernel(const DevJob j, const int32_t* __restrict__ list, const int n) {
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= static_cast<long long>(n) * j.np1) return;
  const int q = static_cast<int>(idx / j.np1), m = static_cast<int>(idx % j.np1);
  const int i = list ? list[q] : q;
  const int x = j.xused[i];
  if (x < 0) return;
  j.tj[static_cast<size_t>(i) * j.np1 + m] = threshold_det(__dsub_rn(j.W[m], j.W[x]));
}

// Speculated inputs: chain i is assumed to receive the last configuration of
// chain i-1 (chain 0 receives the carry from the previous round, or nothing
// in the job's first round).
__global__ void spec_inputs_kernel(const DevJob j) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // position in the joint
  if (q >= j.p) return;
  int x;
  if (q == 0)
    x = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  else
    x = j.m[j.perm[q - 1]];
  j.xused[j.perm[q]] = x;
}

// Joint order (one block): identity, or -- energy-ordered joining -- the
// chains sorted by final level, equal levels in index order: a counting sort
// whose scatter walks the chains in index order a warp at a time (ranks among
// equal levels inside a warp from __match_any_sync).
__global__ void __launch_bounds__(1024) order_kernel(const DevJob j) {
  after_previous();
  const int t = threadIdx.x, nt = blockDim.x;
  if (!j.ordered) {
    for (int q = t; q < j.p; q += nt) j.perm[q] = q;
    return;
  }
  __shared__ int s_part[1024];
  for (int v = t; v < j.np1; v += nt) j.lvcnt[v] = 0;
  __syncthreads();
  for (int c = t; c < j.p; c += nt) atomicAdd(&j.lvcnt[j.m[c]], 1);
  __syncthreads();
  // exclusive scan of the counts: contiguous ranges per thread
  const int per = (j.np1 + nt - 1) / nt;
  const int lo = min(j.np1, t * per), hi = min(j.np1, lo + per);
  int sum = 0;
  for (int v = lo; v < hi; ++v) sum += j.lvcnt[v];
  s_part[t] = sum;
  __syncthreads();
  for (int off = 1; off < nt; off <<= 1) {
    const int a = (t >= off) ? s_part[t - off] : 0;
    __syncthreads();
    s_part[t] += a;
    __syncthreads();
  }
  int run = s_part[t] - sum;
  for (int v = lo; v < hi; ++v) {
    const int c = j.lvcnt[v];
    j.lvcnt[v] = run;
    run += c;
  }
  __syncthreads();
  // stable scatter
  const int lane = t & 31, warp = t >> 5, nwarps = nt >> 5;
  for (int base = 0; base < j.p; base += nt) {
    const int c = base + t;
    const bool act = c < j.p;
    const unsigned amask = __ballot_sync(0xFFFFFFFFu, act);
    int v = -1;
    unsigned same = 0u;
    if (act) {
      v = j.m[c];
      same = __match_any_sync(amask, v);
    }
    for (int w = 0; w < nwarps; ++w) {
      if (warp == w && act) {
        const int rank = __popc(same & ((1u << lane) - 1u));
        j.perm[j.lvcnt[v] + rank] = c;
        __syncwarp(amask);
        if (rank == 0) j.lvcnt[v] += __popc(same);
      }
      __syncthreads();
    }
  }
}

// Inclusive sum over the block (1024 threads); *total = the whole block's.
__device__ __forceinline__ long long block_sum_scan(long long v, long long* s_warp, long long* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) s_warp[warp] = v;
  __syncthreads();
  long long w = s_warp[lane];
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(0xFFFFFFFFu, w, o);
    if (lane >= o) w += u;
  }
  *total = __shfl_sync(0xFFFFFFFFu, w, 31);
  if (warp > 0) v += __shfl_sync(0xFFFFFFFFu, w, warp - 1);
  __syncthreads();
  return v;
}

// Segmented scan and histogram: kept length of chain i is M - k_i + 1 (0 if
// nothing is kept); offsets are the exclusive scan (block 0, 1024 positions
// at a time); h += hgen - dpre, or += dpre where that holds the kept samples
// (the other blocks).
__global__ void __launch_bounds__(1024) finalize_kernel(const DevJob j, const int64_t M, const int may_count_kept) {
  after_previous();
  const int t = threadIdx.x;
  if (blockIdx.x > 0) {
    const bool kept = may_count_kept && j.stats[kStatCountKept];
    for (int m = (blockIdx.x - 1) * 1024 + t; m < j.np1; m += (gridDim.x - 1) * 1024) {
      const unsigned long long d = j.dpre[m];
      j.h[m] += static_cast<long long>(kept ? d : j.hgen[m] - d);
      j.hgen[m] = 0ull;
      j.dpre[m] = 0ull;
    }
    return;
  }
  __shared__ long long s_warp[32];
  long long run = 0, rej = 0;
  for (int base = 0; base < j.p; base += 1024) {
    const int q = base + t;
    const int i = q < j.p ? j.perm[q] : 0;
    const int64_t k = q < j.p ? j.k[i] : 0;
    const long long len = k > 0 ? M - k + 1 : 0;
    rej += q < j.p && k <= 0 ? 1 : 0;
    long long total;
    const long long incl = block_sum_scan(len, s_warp, &total);
    if (q < j.p) j.offsets[i] = run + incl - len;
    run += total;
  }
  long long rejected;
  block_sum_scan(rej, s_warp, &rejected);
  if (t == 0) {
    j.stats[kStatJoined] = run;
    j.stats[kStatJoinedTotal] += run;
    j.stats[kStatRejected] = rejected;
    j.stats[kStatWeightMax] = 0;
  }
}

static void launch_finalize(const DevJob& j, int64_t M, bool may_count_kept, cudaStream_t st) {
  launch_next(finalize_kernel, 1 + blocks_for(j.np1, 1024), 1024, 0, st, j, M, may_count_kept ? 1 : 0);
}

// Control experiment (no detailed balance at the joints): keep everything.
__global__ void naive_kernel(const DevJob j) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < j.p) {
    j.k[i] = 1;
    j.xused[i] = -1;
  }
  if (i == 0) {
    j.stats[kStatCarry] = j.m[j.perm[j.p - 1]];
    j.stats[kStatCarryValid] = 1;
    j.stats[kStatMismatch] = 0;
    j.stats[kStatPasses] = 0;
  }
}

__global__ void clear_stats_kernel(const DevJob j) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    j.stats[kStatSearched] = 0;
    j.stats[kStatMismatch] = 0;
    j.stats[kStatPasses] = 0;
    j.stats[kStatPending] = 0;
    j.stats[kStatQueuePrefix] = 0;
    j.stats[kStatPartial] = 0;
    j.stats[kStatWholeFill] = 0;
    j.stats[kStatScanned] = 0;
    j.stats[kStatFirstPending] = j.p;
  }
  // earliest accepted sample of each chain: none found yet
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < j.p; i += gridDim.x * blockDim.x) j.kmin[i] = kNoHit;
}

// One grid-wide resolution pass, part 1 (one block): with the current k's,
// the actual input of chain i is the last level of the nearest chain before
// it that kept samples (or the carry).  Chains whose k was computed for
// another input are queued in work[], with the new input in xused, and
// their joint thresholds are rebuilt by tj_list_kernel.
//
// defer (speculative passes ahead of the exact scan): the pass is left to
// the scan -- the pending count seen by the pass's kernels is 0 and the
// chains stay marked (k = -1), so the next mark lists them again (a chain
// with k < 0 is pending whatever its input) -- when more than p/16 chains
// are pending (rough weights: passes are unlikely to settle them) and the
// scan's serial cost, ~1.5 us per evaluated chain, is below that of two
// passes, ~70 ns per sample of a C-sweep segment replay: pending * 11 <
// C * N.  (Measured at 20 sweeps: joint L = 128 28 -> 18 ms, L = 96 15 ->
// 10 ms; L = 32 with 16384 chains, where the scan would be long, keeps the
// passes.)
__global__ void __launch_bounds__(1024) mark_kernel(const DevJob j, const int defer) {
  __shared__ int s_tmp[1024];
  __shared__ int s_count, s_first, s_new;
  block_last_accepted(j, s_tmp, j.lastacc);
  if (threadIdx.x == 0) {
    s_count = 0;
    s_first = j.p;
    s_new = 0;
  }
  __syncthreads();
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  for (int q = threadIdx.x; q < j.p; q += blockDim.x) {   // positions in the joint
    const int last = j.lastacc[q];
    const int x = (last >= 0) ? j.m[j.perm[last]] : carry_in;
    const int i = j.perm[q];
    if (x != j.xused[i]) {
      j.xused[i] = x;
      j.k[i] = -1;
      j.kmin[i] = kNoHit;
      j.work[atomicAdd(&s_count, 1)] = i;
      atomicMin(&s_first, q);
      atomicAdd(&s_new, 1);
    } else if (j.k[i] < 0) {
      j.work[atomicAdd(&s_count, 1)] = i;   // marked earlier, not searched yet
      atomicMin(&s_first, q);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const bool deferred = defer && s_count > j.p / 16 &&
                          static_cast<long long>(s_count) * 11 < static_cast<long long>(j.seg_len);
    j.stats[kStatPending] = deferred ? 0 : s_count;
    j.stats[kStatFirstPending] = s_first;
    if (s_new) {
      j.stats[kStatPasses] += 1;
      j.stats[kStatMismatch] += s_new;
    }
  }
}

// Summary replay, set-up: for the chains from the first pending one on, the
// per-level minimum of the joint uniforms (kept in tj, whose rows are
// rebuilt afterwards for the chains that still need a search) starts empty.
__global__ void summary_init_kernel(const DevJob j) {
  if (j.stats[kStatPending] == 0) return;
  const int f = static_cast<int>(j.stats[kStatFirstPending]);   // a position in the joint
  const long long n = static_cast<long long>(j.p - f) * j.np1;
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < n;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = j.perm[f + static_cast<int>(idx / j.np1)];
    j.tj[static_cast<size_t>(i) * j.np1 + static_cast<size_t>(idx % j.np1)] = 0xFFFFFFFFu;
  }
  for (int q = f + blockIdx.x * blockDim.x + threadIdx.x; q < j.p; q += gridDim.x * blockDim.x) {
    const int i = j.perm[q];
    j.summ[i] = 0x7FFFFFFF;     // lowest level visited
    j.summ[j.p + i] = -1;       // highest level visited
    j.summ[2 * j.p + i] = 0;    // a level's minimum was 0xFFFFFFFF
  }
}

// Exact resolution of the joint (Sec. 2 step 4) in chain order, from the
// first chain whose speculated input was wrong: the input x of chain i is
// the last level of the nearest earlier chain that kept samples (else the
// carry).  Chain i keeps samples for input x iff some sample k passes
// u_k <= thr(W[m_k] - W[x]), i.e. iff some visited level m has
// min{u_k : m_k = m} <= thr(W[m] - W[x]) -- exact, from the summary replay.
// Where x is the input k_i was already found for, k_i decides.  Chains that
// keep samples under a new input are listed for one search pass (their x is
// now exact, so nothing cascades); the others get k_i = 0.  A chain whose
// answer the summary cannot give (a level whose every uniform was
// 0xFFFFFFFF, against a threshold of 0xFFFFFFFF) stops the scan; the chains
// from it on keep their speculated inputs for the ordinary passes.
//
// Most inputs the scan meets are the last level of one of the few chains
// just before (the rest of them kept nothing): cand_kernel settles, in
// parallel, chain q under the input of each of the kScanCand positions
// before it (position -1: the carry).  The serial rule then becomes a small
// state machine over positions -- state d = how many positions back the
// current input came from -- whose per-position transition functions are
// composed by a block-wide prefix scan, so the scan costs O(p / 1024) and
// not O(p); only an input from further back than kScanCand positions is
// evaluated one chain at a time.  The state machine is in mc_scan_fsm.cuh.

__device__ __forceinline__ uint8_t* scan_cand(const DevJob& j) {
  return reinterpret_cast<uint8_t*>(j.summ + 3 * static_cast<size_t>(j.p));   // [p][kScanCand]
}

// Whether the chain at joint position pos keeps samples for input level
// x >= 0, from its summary: 1 yes, 0 no, 2 undecidable (a level whose every
// uniform was 0xFFFFFFFF, against a threshold of 0xFFFFFFFF).  Warp-
// collective: the 32 lanes call it with the same arguments.
__device__ __forceinline__ int scan_decide(const DevJob& j, int pos, int x) {
  const int lane = threadIdx.x & 31;
  const int ch = j.perm[pos];
  const uint32_t* um = j.tj + static_cast<size_t>(ch) * j.np1;
  const double wx = j.W[x];
  const bool flag = j.summ[2 * j.p + ch] != 0;
  int hit = 0, amb = 0;
  for (int m = j.summ[ch] + lane; m <= j.summ[j.p + ch]; m += 32) {
    const uint32_t u = um[m];
    if (u != 0xFFFFFFFFu || flag) {
      const uint32_t thr = threshold_det(__dsub_rn(j.W[m], wx));
      if (u != 0xFFFFFFFFu) hit |= (u <= thr) ? 1 : 0;
      else amb |= (thr == 0xFFFFFFFFu) ? 1 : 0;
    }
  }
  hit = __any_sync(0xFFFFFFFFu, hit);
  amb = __any_sync(0xFFFFFFFFu, amb);
  return hit ? kAnsYes : (amb ? kAnsUndecided : kAnsNo);
}

// The answer codes of chain q under the inputs of the kScanCand positions
// before it (mc_scan_fsm.cuh).
__global__ void __launch_bounds__(256) cand_kernel(const DevJob j) {
  if (j.stats[kStatPending] == 0) return;
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  uint8_t* cand = scan_cand(j);
  const int lane = threadIdx.x & 31;
  const long long nwarps = (static_cast<long long>(gridDim.x) * blockDim.x) >> 5;
  const long long n = static_cast<long long>(j.p - f) * kScanCand;
  for (long long w = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5; w < n; w += nwarps) {
    const int q = f + static_cast<int>(w / kScanCand), d = 1 + static_cast<int>(w % kScanCand);
    const int src = q - d;
    const int x = src >= 0 ? j.m[j.perm[src]] : (src == -1 ? carry_in : -1);
    int code = kAnsNone;
    if (x >= 0) {
      const int ch = j.perm[q];
      const int64_t kc = j.k[ch];
      code = (kc >= 0 && j.xused[ch] == x) ? (kc > 0 ? kAnsKnownYes : kAnsKnownNo) : scan_decide(j, q, x);
    }
    if (lane == 0) cand[static_cast<size_t>(q) * kScanCand + d - 1] = static_cast<uint8_t>(code);
  }
}

__device__ __forceinline__ unsigned long long cand_codes(const DevJob& j, int q) {
  const uint32_t* c32 = reinterpret_cast<const uint32_t*>(scan_cand(j));
  const size_t w = 2 * static_cast<size_t>(q);
  return c32[w] | (static_cast<unsigned long long>(c32[w + 1]) << 32);
}

__global__ void __launch_bounds__(1024) scan_kernel(const DevJob j) {
  if (j.stats[kStatPending] == 0) return;
  __shared__ Trans s_tr[1024];
  __shared__ int s_first, s_count, s_state, s_from, s_last, s_end;
  __shared__ unsigned long long s_scanned;
  const int t = threadIdx.x, nt = blockDim.x;
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  if (t == 0) {
    const int last = j.lastacc[f];   // position of the nearest chain before that kept samples (-1: none)
    s_state = (last < 0 && carry_in < 0) ? 0 : min(f - last, kFar);
    s_last = last;
    s_from = f;
    s_count = 0;
    s_end = -1;
    s_scanned = 0;
  }
  __syncthreads();
  unsigned long long scanned = 0;
  for (;;) {
    // a pass over positions [a, p) from state st0, each thread a range
    const int a = s_from, st0 = s_state;
    if (a >= j.p || s_end >= 0) break;
    const int len = j.p - a, per = (len + nt - 1) / nt;
    const int lo = min(j.p, a + t * per), hi = min(j.p, lo + per);
    Trans agg = tr_identity();
    for (int q = lo; q < hi; ++q) agg = tr_then(agg, tr_position(cand_codes(j, q)));
    s_tr[t] = agg;
    if (t == 0) s_first = j.p;
    __syncthreads();
    for (int off = 1; off < nt; off <<= 1) {   // inclusive prefix of the ranges' compositions
      const Trans prev = t >= off ? s_tr[t - off] : tr_identity();
      __syncthreads();
      s_tr[t] = tr_then(prev, s_tr[t]);
      __syncthreads();
    }
    const int s_in = tr_at(t > 0 ? s_tr[t - 1] : tr_identity(), st0);   // state entering this range
    // the first position entered in state kFar or kStop ends the pass
    int s = s_in;
    for (int q = lo; q < hi; ++q) {
      if (s >= kFar) {
        atomicMin(&s_first, q);
        break;
      }
      s = tr_at(tr_position(cand_codes(j, q)), s);
    }
    __syncthreads();
    const int stop_at = s_first;
    // the positions before it: inputs and outcomes, in parallel
    s = s_in;
    for (int q = lo; q < min(hi, stop_at); ++q) {
      const unsigned long long codes = cand_codes(j, q);
      const int ch = j.perm[q];
      if (s == 0) {   // no input yet: the chain is kept whole
        j.xused[ch] = -1;
        j.k[ch] = 1;
      } else {
        const int c = static_cast<int>((codes >> (8 * (s - 1))) & 0xFFu);
        if (c < kAnsKnownNo) {   // not known for this input
          const int src = q - s;
          j.xused[ch] = src >= 0 ? j.m[j.perm[src]] : carry_in;
          if (c == kAnsYes) {
            j.k[ch] = -1;   // to be searched under the exact input
            j.kmin[ch] = kNoHit;
            j.work[atomicAdd(&s_count, 1)] = ch;
          } else {
            j.k[ch] = 0;
          }
          ++scanned;
        }
      }
      s = tr_at(tr_position(codes), s);
    }
    if (stop_at >= j.p) break;   // uniform: every position is settled
    // at stop_at: kStop ends the scan; kFar (the input is the last level of
    // a chain more than kScanCand positions back) is carried one chain at a
    // time, by one warp, until a chain keeps samples
    if (t < 32) {
      const int owner = (stop_at - a) / per;   // the thread whose range holds stop_at
      int sst = tr_at(owner > 0 ? s_tr[owner - 1] : tr_identity(), st0);
      for (int q = a + owner * per; q < stop_at; ++q) sst = tr_at(tr_position(cand_codes(j, q)), sst);
      int end = -1, next_from = j.p;
      if (sst == kStop) {
        end = stop_at;
      } else {
        // the chain that kept samples last: kScanCand + 1 positions back if
        // the state became kFar in this pass, else the pass's own start
        const int last = stop_at > a ? stop_at - kFar : s_last;
        const int x = last >= 0 ? j.m[j.perm[last]] : carry_in;
        for (int q = stop_at; q < j.p; ++q) {
          const int ch = j.perm[q];
          const int64_t kc = j.k[ch];
          const int code = (kc >= 0 && j.xused[ch] == x) ? (kc > 0 ? kAnsKnownYes : kAnsKnownNo) : scan_decide(j, q, x);
          if (code == kAnsUndecided) {
            end = q;
            break;
          }
          if (t == 0 && code < kAnsKnownNo) {
            j.xused[ch] = x;
            ++scanned;
            if (code == kAnsYes) {
              j.k[ch] = -1;
              j.kmin[ch] = kNoHit;
              j.work[atomicAdd(&s_count, 1)] = ch;
            } else {
              j.k[ch] = 0;
            }
          }
          if (code == kAnsYes || code == kAnsKnownYes) {
            next_from = q + 1;
            break;
          }
        }
      }
      if (t == 0) {
        s_end = end;
        s_from = next_from;
        s_state = 1;
        s_last = next_from - 1;
      }
    }
    __syncthreads();
  }
  atomicAdd(&s_scanned, scanned);
  __syncthreads();
  // stopped early: chains still waiting for a search keep their inputs
  if (t == 0) {
    for (int q = s_end >= 0 ? s_end : j.p; q < j.p; ++q)
      if (j.k[j.perm[q]] < 0) j.work[s_count++] = j.perm[q];
    j.stats[kStatPending] = s_count;
    j.stats[kStatScanned] = static_cast<long long>(s_scanned);
  }
}

// ------------------------------------------------------------------ kept rounds (mc_joint_kept.cuh)
// For every position of the joint, the last position before it whose chain
// `keeps` (-1: none): each(q, last) for all q in [f, p); returns the last
// one of all to every thread.  One block of 1024 threads; positions are read
// 1024 at a time, coalesced, as bits of 32 positions a word.
template <class Keeps, class Each>
__device__ __forceinline__ int block_last_kept(const int f, const int p, const Keeps& keeps, const Each& each) {
  __shared__ uint32_t s_bits[1024];
  __shared__ int s_before[1024], s_warp[32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int carry = -1;
  for (int base = f; base < p; base += 32768) {
    const int its = min(32, (p - base + 1023) / 1024);
    for (int it = 0; it < its; ++it) {
      const int q = base + it * 1024 + t;
      const uint32_t b = __ballot_sync(0xFFFFFFFFu, q < p && keeps(q));
      if (lane == 0) s_bits[it * 32 + warp] = b;
    }
    __syncthreads();
    const uint32_t w = t < 32 * its ? s_bits[t] : 0u;
    int v = w ? base + 32 * t + 31 - __clz(w) : -1;
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xFFFFFFFFu, v, o);
      if (lane >= o) v = max(v, u);
    }
    if (lane == 31) s_warp[warp] = v;
    __syncthreads();
    int x = s_warp[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x = max(x, u);
    }
    const int all = __shfl_sync(0xFFFFFFFFu, x, 31);
    int before = __shfl_up_sync(0xFFFFFFFFu, v, 1);
    if (lane == 0) before = -1;
    const int warps_before = warp > 0 ? __shfl_sync(0xFFFFFFFFu, x, warp - 1) : -1;
    s_before[t] = max(carry, max(before, warps_before));
    __syncthreads();
    for (int it = 0; it < its; ++it) {
      const int q = base + it * 1024 + t;
      if (q < p) {
        const uint32_t m = s_bits[it * 32 + warp] & ((1u << lane) - 1u);
        each(q, m ? q - lane + 31 - __clz(m) : s_before[it * 32 + warp]);
      }
    }
    carry = max(carry, all);
    __syncthreads();
  }
  return carry;
}

// Start of a kept round's joint: the joint order where it is the chains' own,
// the speculated inputs (spec_inputs_kernel), nothing found yet, the level
// weights and the cleared counters.
__global__ void kept_prelude_kernel(const DevJob j) {
  after_previous();
  const int t = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  if (t == 0) {
    for (const int s : {kStatSearched, kStatMismatch, kStatPasses, kStatPending, kStatScanned, kStatNoHit,
                        kStatQueueSearch, kStatQueueA, kStatQueueB})
      j.stats[s] = 0;
    j.stats[kStatFirstPending] = j.p;
  }
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  for (int q = t; q < j.p; q += nt) {
    const int i = j.ordered ? j.perm[q] : q;
    const int prev = q > 0 ? (j.ordered ? j.perm[q - 1] : q - 1) : -1;
    if (!j.ordered) j.perm[q] = q;
    j.xused[i] = prev >= 0 ? j.m[prev] : carry_in;
    j.kmin[i] = kNoHit;
  }
  const double wref = reference_weight(j);
  float* wl = level_weights(j);
  float big = 0.0f;
  for (int m = t; m < j.np1; m += nt) {
    const float v = static_cast<float>((j.W[m] - wref) * 1.4426950408889634);
    wl[m] = level_weight(v);
    if (fabsf(v) <= kWeightSpan) big = fmaxf(big, fabsf(v));
  }
  // (0 before: finalize_kernel clears it)
  if (big > 0.0f) atomicMax(&j.stats[kStatWeightMax], static_cast<long long>(__float_as_int(big)));
}

// Results of the last search, then one resolution pass, part 1 (as
// mark_kernel, which see for `defer`): the chains whose actual input is not
// the one their k was found for go to work[], with the new input in xused.
// With kMarkFinal and nothing pending: the carry, and whether fewer samples
// are kept than discarded.
__device__ __forceinline__ void kept_mark_body(const DevJob& j, const int64_t M, const int flags) {
  __shared__ int s_count, s_first, s_new;
  __shared__ unsigned long long s_kept;
  const int t = threadIdx.x, nt = blockDim.x;
  if (t == 0) {
    s_count = 0;
    s_first = j.p;
    s_new = 0;
    s_kept = 0ull;
  }
  const bool unsearched = (flags & kMarkExactFirst) && rough_last_joint(j, j.stats[kStatRejected]);
  const int n = (flags & kMarkListed) ? static_cast<int>(j.stats[kStatPending]) : j.p;
  for (int q = t; q < n; q += nt) {
    const int i = (flags & kMarkListed) ? j.work[q] : q;
    const unsigned long long k = j.kmin[i];
    j.k[i] = unsearched ? -1 : (k == kNoHit ? 0 : static_cast<int64_t>(k));
  }
  const int carry_in = j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1;
  __syncthreads();
  unsigned long long kept = 0;
  const int last_all = block_last_kept(
      0, j.p, [&](int q) { return j.k[j.perm[q]] > 0; },
      [&](int q, int last) {
        const int x = last >= 0 ? j.m[j.perm[last]] : carry_in;
        const int i = j.perm[q];
        const int64_t k = j.k[i];
        j.lastacc[q] = last;
        if (k > 0) kept += static_cast<unsigned long long>(M - k + 1);
        const bool moved = x != j.xused[i];
        if (moved || k < 0) {
          j.work[atomicAdd(&s_count, 1)] = i;
          atomicMin(&s_first, q);
        }
        if (moved) {
          j.xused[i] = x;
          j.k[i] = -1;
          j.kmin[i] = kNoHit;
          atomicAdd(&s_new, 1);
        }
      });
  // (a warp's sum first: 64-bit shared atomics are compare-and-swap loops, 30 us when 1024 threads meet in one)
  for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xFFFFFFFFu, kept, o);
  if (kept && (t & 31) == 0) atomicAdd(&s_kept, kept);
  __syncthreads();
  if (t == 0) {
    const bool deferred = ((flags & kMarkDefer) && s_count > j.p / 16) || ((flags & kMarkDeferLate) && s_count > j.p / 4);
    j.stats[kStatPending] = deferred ? 0 : s_count;
    j.stats[kStatFirstPending] = s_first;
    if (s_new) {
      j.stats[kStatPasses] += 1;
      j.stats[kStatMismatch] += s_new;
    }
    j.stats[kStatNoHit] = 0;
    j.stats[kStatQueueSearch] = 0;
    j.stats[kStatQueueA] = 0;
    j.stats[kStatQueueB] = 0;
    if ((flags & kMarkFinal) && s_count == 0) {
      if (last_all >= 0) {
        j.stats[kStatCarry] = j.m[j.perm[last_all]];
        j.stats[kStatCarryValid] = 1;
      }
      j.stats[kStatCountKept] = 2ull * s_kept < static_cast<unsigned long long>(j.p) * static_cast<unsigned long long>(M);
    }
  }
  __syncthreads();
  if ((flags & kMarkFinal) && s_count == 0) kept_list_counted(j);
}

__global__ void __launch_bounds__(1024) kept_mark_kernel(const DevJob j, const int64_t M, const int flags) {
  after_previous();
  kept_mark_body(j, M, flags);
}

// Scratch of the scan in tj (its rows are rebuilt for the chains searched
// next): values of the heights by position (the larger of the two samples'), their maxima over 32 and 1024
// positions, successors (one more: the round's input), two jump arrays and
// the marks -- at most 21 p + 40 of the 4 (N + 1) p >= 68 p bytes.
struct HeightScratch {
  double *val, *max32, *max1024;
  int32_t *next, *jump;
  uint8_t* mark;
};
__device__ __forceinline__ HeightScratch height_scratch(const DevJob& j) {
  HeightScratch s;
  const int p = j.p;
  s.val = reinterpret_cast<double*>(j.tj);
  s.max32 = s.val + p;
  s.max1024 = s.max32 + (p + 31) / 32;
  s.next = reinterpret_cast<int32_t*>(s.max1024 + (p + 1023) / 1024);
  s.jump = s.next + p + 1;
  s.mark = reinterpret_cast<uint8_t*>(s.jump + p + 1);
  return s;
}

// Values and maxima of the positions [1024 block, 1024 block + 1024), in steps of `blocks` blocks.
__device__ __forceinline__ void height_values(const DevJob& j, int block, int blocks) {
  __shared__ double s_max[32];
  const HeightScratch hs = height_scratch(j);
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const int t = threadIdx.x;
  const double wref = reference_weight(j);
  const float error = height_error(j);
  for (int base = block * 1024; base < j.p; base += blocks * 1024) {
    const int q = base + t;
    double v = -CUDART_INF;
    if (q >= f && q < j.p) {
      const Height h = heights(j)[j.perm[q]];
      v = fmax(height_value(j, h), height_second(h, wref, error));
    }
    if (q < j.p) hs.val[q] = v;
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    if ((t & 31) == 0) {
      s_max[t >> 5] = v;
      if (q < j.p) hs.max32[q >> 5] = v;
    }
    __syncthreads();
    if (t < 32) {
      v = s_max[t];
      for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
      if (t == 0) hs.max1024[base >> 10] = v;
    }
    __syncthreads();
  }
}

// First position from q on whose chain keeps samples for an input level of
// weight wx; p if none; p + 1 + q' if that is undecided at q'.
__device__ __forceinline__ int height_next(const DevJob& j, const HeightScratch& hs, int q, double wx, double wref,
                                           float error) {
  const double low = wx - (kHeightEps + 1e-13 * fabs(wx));
  while (q < j.p) {
    if ((q & 1023) == 0 && hs.max1024[q >> 10] < low) {
      q += 1024;
      continue;
    }
    if ((q & 31) == 0 && hs.max32[q >> 5] < low) {
      q += 32;
      continue;
    }
    if (!(hs.val[q] < low)) {
      const int a = height_accepts(j, heights(j)[j.perm[q]], wx, wref, error);
      if (a) return a == 1 ? q : j.p + 1 + q;
    }
    ++q;
  }
  return j.p;
}

// The input at position f: the last level passed on (-1: none yet).
__device__ __forceinline__ int height_input(const DevJob& j, int f) {
  const int last = j.lastacc[f];
  return last >= 0 ? j.m[j.perm[last]] : (j.stats[kStatCarryValid] ? static_cast<int>(j.stats[kStatCarry]) : -1);
}

// Successors: next[q] = the next chain that keeps samples if the chain at q
// does; next[p] = the first one for the input at f (none yet: f, kept whole).
__device__ __forceinline__ void height_successors(const DevJob& j, int t, int nt) {
  const HeightScratch hs = height_scratch(j);
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const double wref = reference_weight(j);
  const float error = height_error(j);
  for (int q = f + t; q <= j.p; q += nt) {
    int nx;
    if (q < j.p) {
      nx = height_next(j, hs, q + 1, j.W[j.m[j.perm[q]]], wref, error);
    } else {
      const int x = height_input(j, f);
      nx = x < 0 ? f : height_next(j, hs, f, j.W[x], wref, error);
    }
    hs.next[q] = nx;
  }
}

// One block: mark the positions reached from the round's input (after k
// doublings the marks hold the first 2^k of them), then give every position
// its input and outcome, as scan_kernel does.
__device__ __forceinline__ void height_path(const DevJob& j) {
  __shared__ int s_end, s_count, s_scanned;
  const HeightScratch hs = height_scratch(j);
  const int t = threadIdx.x, nt = blockDim.x, p = j.p;
  const int f = static_cast<int>(j.stats[kStatFirstPending]);
  const int x0 = height_input(j, f);
  if (t == 0) {
    s_end = p;
    s_count = 0;
    s_scanned = 0;
  }
  for (int q = f + t; q < p; q += nt) hs.mark[q] = q == hs.next[p] ? 1 : 0;
  __syncthreads();
  int32_t *src = hs.next, *dst = hs.jump;
  for (long long len = 1; len < p - f; len <<= 1) {
    for (int q = f + t; q < p; q += nt) {
      const int a = src[q];
      if (a < p) {
        if (hs.mark[q]) hs.mark[a] = 1;
        dst[q] = src[a];
      } else {
        dst[q] = a;
      }
    }
    __syncthreads();
    int32_t* o = src;
    src = dst;
    dst = o;
  }
  // every jump now leads past the path's end: p, or p + 1 + the position whose answer is undecided
  if (t == 0) {
    const int start = hs.next[p];
    const int end = start < p ? src[start] : start;
    if (end > p) s_end = end - (p + 1);
  }
  __syncthreads();
  const int stop_at = s_end;
  int scanned = 0;
  block_last_kept(
      f, p, [&](int q) { return hs.mark[q] != 0; },
      [&](int q, int last) {
        const int ch = j.perm[q];
        const int64_t kc = j.k[ch];
        if (q < stop_at) {
          const int x = last >= 0 ? j.m[j.perm[last]] : x0;
          if (kc < 0 || j.xused[ch] != x) {   // not known for this input
            j.xused[ch] = x;
            if (!hs.mark[q]) {
              j.k[ch] = 0;
            } else if (x < 0) {               // no input yet: the chain is kept whole
              j.k[ch] = 1;
            } else {
              j.k[ch] = -1;                   // to be searched under the exact input
              j.kmin[ch] = kNoHit;
              j.work[atomicAdd(&s_count, 1)] = ch;
            }
            ++scanned;
          }
        } else if (q == stop_at) {               // undecided: searched under its input, which is exact
          j.xused[ch] = last >= 0 ? j.m[j.perm[last]] : x0;
          j.k[ch] = -1;
          j.kmin[ch] = kNoHit;
          j.work[atomicAdd(&s_count, 1)] = ch;
        } else if (kc < 0) {
          j.work[atomicAdd(&s_count, 1)] = ch;   // stopped early: chains still waiting for a search keep their inputs
        }
      });
  if (scanned) atomicAdd(&s_scanned, scanned);
  __syncthreads();
  if (t == 0) {
    j.stats[kStatPending] = s_count;
    j.stats[kStatScanned] += s_scanned;
    j.stats[kStatNoHit] = 0;
    j.stats[kStatQueueA] = 0;
    j.stats[kStatQueueB] = 0;
  }
}

__global__ void __launch_bounds__(1024) height_value_kernel(const DevJob j) {
  after_previous();
  if (j.stats[kStatPending]) height_values(j, blockIdx.x, gridDim.x);
}
__global__ void height_next_kernel(const DevJob j) {
  after_previous();
  if (j.stats[kStatPending]) height_successors(j, blockIdx.x * blockDim.x + threadIdx.x, gridDim.x * blockDim.x);
}
__global__ void __launch_bounds__(1024) height_path_kernel(const DevJob j) {
  after_previous();
  if (j.stats[kStatPending]) height_path(j);
}
// the three in one launch
__device__ __forceinline__ void height_scan_body(const DevJob& j) {
  if (j.stats[kStatPending] == 0) return;
  height_values(j, 0, 1);
  __syncthreads();
  height_successors(j, threadIdx.x, blockDim.x);
  __syncthreads();
  height_path(j);
}
__global__ void __launch_bounds__(1024) height_scan_kernel(const DevJob j) {
  after_previous();
  height_scan_body(j);
}
__global__ void __launch_bounds__(1024) kept_mark_scan_kernel(const DevJob j, const int64_t M, const int flags) {
  after_previous();
  kept_mark_body(j, M, flags);
  __syncthreads();
  height_scan_body(j);
}

__global__ void tj_list_kernel(const DevJob j) {
  const long long total = j.stats[kStatPending] * static_cast<long long>(j.np1);
  for (long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; idx < total;
       idx += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = j.work[idx / j.np1], m = static_cast<int>(idx % j.np1);
    const int x = j.xused[i];
    j.tj[static_cast<size_t>(i) * j.np1 + m] = (x < 0) ? 0xFFFFFFFFu : threshold_det(__dsub_rn(j.W[m], j.W[x]));
  }
}

// Chains of the list (all, or work[]) that found no accepted sample in
// their first segment go to work2 -- only they need their later segments
// searched (one block).
__global__ void __launch_bounds__(1024) nohit_kernel(const DevJob j, const int list_mode) {
  __shared__ int s_count;
  if (threadIdx.x == 0) s_count = 0;
  __syncthreads();
  const int n = list_mode ? static_cast<int>(j.stats[kStatPending]) : j.p;
  const unsigned long long segN = static_cast<unsigned long long>(j.seg_len);
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const int i = list_mode ? j.work[q] : q;
    if (j.kmin[i] > segN) j.work2[atomicAdd(&s_count, 1)] = i;
  }
  __syncthreads();
  if (threadIdx.x == 0) j.stats[kStatNoHit] = s_count;
}

// ------------------------------------------------------------------ rounds of any length
// Rounds that do not start or end on a sweep (Fig. 2's M_node = 100 < N):
// attempt t of a chain visits site t mod N and draws word t&3 of Philox
// block t>>2, with the thresholds and the acceptance rule of the sweep
// kernels, so the chains are the same whichever kernel runs them.  Meant for
// short rounds: one thread per chain works straight on its bit-packed
// lattice in global memory and counts every sample into hgen.
__device__ __forceinline__ int site_spin(const uint32_t* lat, int wd, int L, int x, int y) {
  x = (x + L) % L;
  y = (y + L) % L;
  return static_cast<int>((lat[y * wd + (x >> 5)] >> (x & 31)) & 1u);
}

// one attempt: returns the new level; flips the site in lat if accepted
__device__ __forceinline__ int attempt_one(const DevJob& j, uint32_t* lat, int m, uint64_t t, uint32_t chain,
                                           uint4& r, uint64_t& blk) {
  const int site = static_cast<int>(t % static_cast<uint64_t>(j.N));
  const int x = site % j.L, y = site / j.L;
  const int sv = site_spin(lat, j.wd, j.L, x, y);
  const int a = (site_spin(lat, j.wd, j.L, x - 1, y) == sv) + (site_spin(lat, j.wd, j.L, x + 1, y) == sv) +
                (site_spin(lat, j.wd, j.L, x, y - 1) == sv) + (site_spin(lat, j.wd, j.L, x, y + 1) == sv);
  if ((t >> 2) != blk) {
    blk = t >> 2;
    r = philox4x32_10(make_uint4(static_cast<uint32_t>(blk), static_cast<uint32_t>(blk >> 32), chain, kTagFlip),
                      j.key0, j.key1);
  }
  const uint32_t u = uint4_word(r, static_cast<uint32_t>(t & 3u));
  if (u <= j.T[a * j.np1 + m]) {
    lat[y * j.wd + (x >> 5)] ^= 1u << (x & 31);
    m += a - 2;
  }
  return m;
}

// A warp of chains a block: the lattices in shared memory (a column a chain),
// the threshold table beside them where it fits, the site counted up.  What
// bounds it is one chain's serial path, two shared-memory loads and the
// arithmetic around them: 100 attempts of 32 chains at L = 20 take 24 us (60
// with the lattice and the table in global memory and the site divided out
// of the attempt's number).
template <bool TSMEM>
__global__ void __launch_bounds__(32) attempts_kernel(const DevJob j, const uint64_t t0, const int64_t n,
                                                      int32_t* __restrict__ rec) {
  extern __shared__ __align__(16) uint32_t smem[];
  const int lane = threadIdx.x, c = blockIdx.x * 32 + lane, L = j.L, wd = j.wd, np1 = j.np1;
  const uint32_t* T = j.T;
  uint32_t* lat = smem + (TSMEM ? ((5 * np1 + 3) & ~3) : 0) + lane;   // word q of the chain at lat[32 q]
  if (TSMEM) {
    for (int i = lane; i < 5 * np1; i += 32) smem[i] = j.T[i];
    T = smem;
  }
  const bool active = c < j.p;
  uint32_t* g = j.spins + static_cast<size_t>(active ? c : 0) * L * wd;
  const int site = static_cast<int>(t0 % static_cast<uint64_t>(j.N));
  int x = site % L, y = site / L;
  // only the rows swept, and one on either side (the whole lattice of 3000 chains at L = 128 for 50 attempts
  // each: 72 us, 60 with the lattices in global memory, 47 now)
  const int y0 = y, rows = static_cast<int>(min(static_cast<int64_t>(L), (x + n + L - 1) / L));
  const auto each_row = [&](int first, int count, const auto& move) {
    for (int i = 0, yy = first; i < count; ++i) {
      for (int w = 0; w < wd; ++w) move(yy * wd + w);
      if (++yy == L) yy = 0;
    }
  };
  if (active) each_row(y0 ? y0 - 1 : L - 1, min(L, rows + 2), [&](int q) { lat[32 * q] = g[q]; });
  __syncwarp();
  if (!active) return;
  int m = j.m[c];
  uint4 r = make_uint4(0u, 0u, 0u, 0u);
  int32_t* lv = rec ? rec + static_cast<size_t>(c) * n : nullptr;
  const auto spin = [&](int xx, int yy) { return (lat[32 * (yy * wd + (xx >> 5))] >> (xx & 31)) & 1u; };
  for (int64_t k = 0; k < n; ++k) {
    const uint64_t t = t0 + static_cast<uint64_t>(k);
    if ((t & 3u) == 0u || k == 0)
      r = philox4x32_10(make_uint4(static_cast<uint32_t>(t >> 2), static_cast<uint32_t>(t >> 34),
                                   static_cast<uint32_t>(c), kTagFlip),
                        j.key0, j.key1);
    const uint32_t sv = spin(x, y);
    const int a = (spin(x ? x - 1 : L - 1, y) == sv) + (spin(x + 1 == L ? 0 : x + 1, y) == sv) +
                  (spin(x, y ? y - 1 : L - 1) == sv) + (spin(x, y + 1 == L ? 0 : y + 1) == sv);
    const uint32_t u = uint4_word(r, static_cast<uint32_t>(t & 3u));
    if (u <= T[a * np1 + m]) {
      lat[32 * (y * wd + (x >> 5))] ^= 1u << (x & 31);
      m += a - 2;
    }
    atomicAdd(&j.hgen[m], 1ull);
    if (lv) lv[k] = m;
    if (++x == L) {
      x = 0;
      if (++y == L) y = 0;
    }
  }
  each_row(y0, rows, [&](int q) { g[q] = lat[32 * q]; });
  j.m[c] = m;
}

// The joint of such a round (Sec. 2 steps 3-5) from the recorded levels, by
// heights (mc_height.cuh): every chain's height from all its samples, a warp
// a chain; the scan that settles every input; then, a warp a chain again, the
// first passing sample of the chains that keep some and the count of the
// discarded ones.  A round of 32 chains of 100 samples takes 31 us (63 one
// chain after another), the whole of 4096 chains of 500 attempts
// 0.52 ms instead of 23.2.  An input the heights cannot settle leaves the whole
// round to partial_joint_kernel.
__global__ void __launch_bounds__(128) partial_height_kernel(const DevJob j, const int64_t M, const uint32_t r) {
  after_previous();
  const float* wl = level_weights(j);
  const int lane = threadIdx.x & 31, nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < j.p; q += nwarps) {
    const int c = j.perm[q];
    const int32_t* lv = j.plv + static_cast<size_t>(c) * M;
    Height h = height_none();
    for (int64_t k = lane; k < M; k += 32) {
      const uint4 v = philox4x32_10(make_uint4(static_cast<uint32_t>(k >> 2), r, static_cast<uint32_t>(c), kTagJoint),
                                    j.key0, j.key1);
      Height one = height_none();
      one.m = static_cast<uint32_t>(lv[k]);
      one.u = uint4_word(v, static_cast<uint32_t>(k & 3));
      one.best = one.u ? wl[one.m] + height_draw(one.u) : CUDART_INF_F;
      if (one.best == one.best) h = height_merge(h, one);   // (no number: passes no test)
    }
    for (int o = 16; o > 0; o >>= 1) {
      Height b;
      b.m = __shfl_xor_sync(0xFFFFFFFFu, h.m, o);
      b.u = __shfl_xor_sync(0xFFFFFFFFu, h.u, o);
      b.best = __shfl_xor_sync(0xFFFFFFFFu, h.best, o);
      b.second = __shfl_xor_sync(0xFFFFFFFFu, h.second, o);
      h = height_merge(h, b);
    }
    if (lane == 0) {
      heights(j)[c] = h;
      // the whole joint is the scan's: nothing known, from the first position on
      j.k[c] = -1;
      j.lastacc[q] = -1;
      if (q == 0) {
        j.stats[kStatPending] = j.p;
        j.stats[kStatFirstPending] = 0;
      }
    }
  }
}

__global__ void __launch_bounds__(128) partial_finish_kernel(const DevJob j, const int64_t M, const uint32_t r) {
  after_previous();
  if (j.stats[kStatScanned] < j.p) return;   // undecided somewhere: partial_joint_kernel
  const int lane = threadIdx.x & 31, nwarps = (gridDim.x * blockDim.x) >> 5;
  for (int c = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < j.p; c += nwarps) {
    const int32_t* lv = j.plv + static_cast<size_t>(c) * M;
    int64_t kf = j.k[c];   // 0 or 1 are final
    __syncwarp();
    if (kf < 0) {
      const double wx = j.W[j.xused[c]];
      for (int64_t base = 0; base < M; base += 32) {
        const int64_t k = base + lane;
        bool hit = false;
        if (k < M) {
          const uint4 v = philox4x32_10(
              make_uint4(static_cast<uint32_t>(k >> 2), r, static_cast<uint32_t>(c), kTagJoint), j.key0, j.key1);
          hit = uint4_word(v, static_cast<uint32_t>(k & 3)) <= threshold_det(__dsub_rn(j.W[lv[k]], wx));
        }
        const unsigned hits = __ballot_sync(0xFFFFFFFFu, hit);
        if (hits) {
          kf = base + __ffs(hits);
          break;
        }
      }
      if (lane == 0) j.k[c] = kf;
    }
    const int64_t nd = kf > 0 ? kf - 1 : M;   // discarded samples
    for (int64_t k = lane; k < nd; k += 32) atomicAdd(&j.dpre[lv[k]], 1ull);
  }
}

// The same joint by the serial rule: the chains in joint order, one at a time
// (the input of each is the level passed on by those before it), the samples
// of a chain tested in parallel -- sample k passes iff its joint uniform
// Philox((k-1)>>2, r, chain, 1) word (k-1)&3 is at most thr(W[m_k] - W[x]) --
// in blocks of the block's threads, stopping at the first block with a pass;
// k_i is the smallest passing k.  The samples before it (all M when none
// passes) go to dpre.  Where the heights have settled the round it only
// fixes the carry.
__global__ void __launch_bounds__(1024) partial_joint_kernel(const DevJob j, const int64_t M, const uint32_t r) {
  after_previous();
  __shared__ unsigned long long s_k;
  __shared__ int s_carry, s_valid;
  const int t = threadIdx.x, nt = blockDim.x;
  if (j.stats[kStatScanned] == j.p) {
    if (t == 0) s_carry = -1;
    __syncthreads();
    for (int q = t; q < j.p; q += nt)
      if (j.k[j.perm[q]] > 0) atomicMax(&s_carry, q);
    __syncthreads();
    if (t == 0) {
      if (s_carry >= 0) {
        j.stats[kStatCarry] = j.m[j.perm[s_carry]];
        j.stats[kStatCarryValid] = 1;
      }
      j.stats[kStatSearched] = static_cast<long long>(j.p) * M;
      j.stats[kStatScanned] = 0;
    }
    return;
  }
  if (t == 0) {
    s_valid = static_cast<int>(j.stats[kStatCarryValid]);
    s_carry = static_cast<int>(j.stats[kStatCarry]);
  }
  __syncthreads();
  long long searched = 0;
  for (int q = 0; q < j.p; ++q) {
    const int c = j.perm[q];
    const int valid = s_valid, carry = s_carry;
    const int32_t* lv = j.plv + static_cast<size_t>(c) * M;
    __syncthreads();   // everyone has read s_valid / s_carry of this chain
    if (t == 0) {
      s_k = kNoHit;
      j.xused[c] = valid ? carry : -1;
    }
    __syncthreads();
    int64_t kf = 1;   // nothing passed on yet: the chain is kept whole
    if (valid) {
      const double wx = j.W[carry];
      for (int64_t base = 0; base < M; base += nt) {
        const int64_t k0 = base + t;   // sample k0 + 1
        bool hit = false;
        if (k0 < M) {
          const uint4 v = philox4x32_10(make_uint4(static_cast<uint32_t>(k0 >> 2), r, static_cast<uint32_t>(c), kTagJoint),
                                        j.key0, j.key1);
          hit = uint4_word(v, static_cast<uint32_t>(k0 & 3)) <= threshold_det(__dsub_rn(j.W[lv[k0]], wx));
          ++searched;
        }
        if (hit) atomicMin(&s_k, static_cast<unsigned long long>(k0 + 1));
        if (__syncthreads_or(hit)) break;
      }
      kf = s_k == kNoHit ? 0 : static_cast<int64_t>(s_k);
    }
    const int64_t nd = kf > 0 ? kf - 1 : M;   // discarded samples
    for (int64_t k0 = t; k0 < nd; k0 += nt) atomicAdd(&j.dpre[lv[k0]], 1ull);
    if (t == 0) {
      j.k[c] = kf;
      if (kf > 0) {
        s_carry = j.m[c];
        s_valid = 1;
      }
    }
    __syncthreads();
  }
  if (searched) atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatSearched]),
                          static_cast<unsigned long long>(searched));
  if (t == 0) {
    j.stats[kStatCarry] = s_carry;
    j.stats[kStatCarryValid] = s_valid;
    j.stats[kStatMismatch] = 0;
    j.stats[kStatPasses] = 0;
    j.stats[kStatScanned] = 0;
  }
}

// The joint of such a round by the serial rule itself (Sec. 2 steps 3-5),
// one thread: each chain, in joint order, is regenerated from its round
// start until its first sample that passes the test against the level
// passed on; the samples before it go to dpre.
constexpr int kMaxLatWords = 128 * 4;
__global__ void serial_joint_kernel(const DevJob j, const uint64_t t0, const int64_t M, const uint32_t r) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  int carry_valid = static_cast<int>(j.stats[kStatCarryValid]);
  int carry = static_cast<int>(j.stats[kStatCarry]);
  uint32_t lat[kMaxLatWords];
  long long searched = 0;
  for (int q = 0; q < j.p; ++q) {
    const int c = j.perm[q];
    int64_t kf = 0;
    j.xused[c] = carry_valid ? carry : -1;
    if (!carry_valid) {
      kf = 1;
    } else {
      const uint32_t* src = j.spins0 + static_cast<size_t>(c) * j.L * j.wd;
      for (int w = 0; w < j.L * j.wd; ++w) lat[w] = src[w];
      int m = j.m0[c];
      uint4 fr = make_uint4(0u, 0u, 0u, 0u), jr = fr;
      uint64_t blk = ~0ull;
      const double wx = j.W[carry];
      for (int64_t k = 1; k <= M; ++k) {
        m = attempt_one(j, lat, m, t0 + static_cast<uint64_t>(k - 1), static_cast<uint32_t>(c), fr, blk);
        const uint64_t qk = static_cast<uint64_t>(k - 1);
        if ((qk & 3u) == 0u || k == 1)
          jr = philox4x32_10(make_uint4(static_cast<uint32_t>(qk >> 2), r, static_cast<uint32_t>(c), kTagJoint),
                             j.key0, j.key1);
        ++searched;
        if (uint4_word(jr, static_cast<uint32_t>(qk & 3u)) <= threshold_det(__dsub_rn(j.W[m], wx))) {
          kf = k;
          break;
        }
        j.dpre[m] += 1ull;   // a discarded sample
      }
    }
    j.k[c] = kf;
    if (kf > 0) {
      carry = j.m[c];
      carry_valid = 1;
    }
  }
  j.stats[kStatCarry] = carry;
  j.stats[kStatCarryValid] = carry_valid;
  j.stats[kStatMismatch] = 0;
  j.stats[kStatPasses] = 0;
  j.stats[kStatScanned] = 0;
  j.stats[kStatSearched] = searched;
}

cudaError_t k_generate_attempts(const DevJob& j, uint64_t t0, int64_t n, bool record, cudaStream_t st) {
  const size_t lat = 128ull * j.L * j.wd, table = 4ull * ((5 * j.np1 + 3) & ~3);
  const bool ts = lat + table <= kMaxSmem;
  auto kern = ts ? attempts_kernel<true> : attempts_kernel<false>;
  const size_t bytes = lat + (ts ? table : 0);
  const cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  kern<<<blocks_for(j.p, 32), 32, bytes, st>>>(j, t0, n, record ? j.plv : nullptr);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t k_join_attempts(const DevJob& j, uint64_t t0, int64_t M, uint32_t r, bool naive, bool recorded,
                            cudaStream_t st) {
  if (!naive && recorded) {
    cudaError_t e = kept_prelude(j, st);
    if (e != cudaSuccess) return e;
    const unsigned warps = std::min(2432u, blocks_for(j.p, 4));
    launch_next(partial_height_kernel, warps, 128, 0, st, j, M, r);
    if ((e = kept_scan(j, st)) != cudaSuccess) return e;
    launch_next(partial_finish_kernel, warps, 128, 0, st, j, M, r);
    launch_next(partial_joint_kernel, 1, 1024, 0, st, j, M, r);
    launch_finalize(j, M, false, st);
    launches_add(4);
    return cudaGetLastError();
  }
  order_kernel<<<1, 1024, 0, st>>>(j);
  if (naive) naive_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j);
  else serial_joint_kernel<<<1, 32, 0, st>>>(j, t0, M, r);
  launch_finalize(j, M, false, st);
  launches_add(3);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ host side
size_t gen_smem_bytes(int L, const LaunchShape& s, bool* table_in_smem) {
  const bool ts = table_fits(L, s, true);
  if (table_in_smem) *table_in_smem = ts;
  return plan_bytes(L, s, ts, true);
}

bool shape_supported(int L, const LaunchShape& s) {
  if (L < 4 || L > 128 || (L % 4) != 0) return false;
  if (s.cpw < 1 || s.cpw > 32 || s.wpb < 1 || s.wpb > 4) return false;
  if (s.placement == kPlaceReg && L > 32) return false;
  if (s.placement == kPlaceGlobal && L != 96 && L != 100 && L != 128) return false;
  if (s.placement != kPlaceReg && s.placement != kPlaceSmem && s.placement != kPlaceGlobal) return false;
  return plan_bytes(L, s, false, true) <= kMaxSmem;
}

// One chain a lane: the shape when there are too many chains for one a warp.
static LaunchShape lane_shape(int L, int p, int num_sms) {
  LaunchShape s;
  // lattice rows in registers for L <= 32, except L = 24 and 32, whose
  // compile-time shared-memory bodies measured faster (L = 32, 16384 chains:
  // generation 6 % shorter, no rotation of 32 row registers per row)
  s.placement = (L <= 32 && L != 24 && L != 32) ? kPlaceReg : kPlaceSmem;
  s.wpb = 4;
  const int warps = std::max(1, num_sms) * 4;  // one warp per SM sub-partition
  s.cpw = std::min(32, std::max(1, (p + warps - 1) / warps));
  // lattices in global memory: at L = 96 so that the threshold table fits in
  // shared memory (generation 2.2x faster at 1024 and 2048 chains, 20
  // sweeps); at L = 100, 128 (table in global memory either way) only with
  // full warps, where they leave a block's shared memory to the histogram --
  // lane groups ran 6-9 % faster with the lattices in shared memory
  if (L == 96 || ((L == 100 || L == 128) && s.cpw > 8)) s.placement = kPlaceGlobal;
  while (s.wpb > 1 && !shape_supported(L, s)) s.wpb >>= 1;
  while (s.cpw > 1 && !shape_supported(L, s)) s.cpw >>= 1;
  return s;
}

LaunchShape default_shape(int L, int p, int num_sms) {
  if (warp_chain_better(L, p, num_sms)) return LaunchShape{kPlaceSmem, 1, 4};   // one chain a warp
  return lane_shape(L, p, num_sms);
}

// Shape of a job that shares the GPU with others (the server's).  One chain a
// warp where that is the faster form alone: its rounds are so much shorter
// that it also serves more (the 20-jobs-a-second stream of 400 jobs through 16
// slots: 3.06e10 kept samples/s against 2.70e10 with full warps of one chain
// a lane, latency p50 3.2 against 4.2 s).  Else as many chains a warp as there
// are (up to 32), keeping the threshold table in shared memory if the default
// shape has it there: the time of a round is set by the latency of one chain,
// which a fuller warp does not change (measured: within 5 % for L <= 64 and
// 128), so the job takes the same time on far fewer warps.
static LaunchShape full_lane_shape(int L, int p, int num_sms);
LaunchShape dense_shape(int L, int p, int num_sms) {
  return warp_chain_better(L, p, num_sms) ? default_shape(L, p, num_sms) : full_lane_shape(L, p, num_sms);
}

static LaunchShape full_lane_shape(int L, int p, int num_sms) {
  LaunchShape def = lane_shape(L, p, num_sms);
  // full warps at L = 100, 128 keep their lattices in global memory: a block
  // of 128 chains then needs only the histogram's shared memory, so blocks
  // of other jobs fit beside it
  if (L == 100 || L == 128) def.placement = kPlaceGlobal;
  const bool ts = table_fits(L, def, true);
  for (int cpw = std::min(32, std::max(1, p)); cpw >= 1; --cpw)
    for (int w = 4; w >= 1; --w) {
      LaunchShape s{def.placement, cpw, w};
      if (w > 1 && (w - 1) * cpw >= p) continue;  // no empty warps
      if (shape_supported(L, s) && (!ts || table_fits(L, s, true))) return s;
    }
  return def;
}

// Time of one attempt of every chain, ns, by launch form: one chain a lane
// (a chain's serial path, whatever the chains), one a warp (the larger of a
// window's latency and the schedulers' share of instructions).  Measured alone
// on 152 SMs; used to compare forms, not to predict times.
static double lane_ns(int L) {
  if (L <= 32) return L == 24 || L == 32 ? 29.0 : 33.0;
  if (L == 48) return 43.0;
  if (L == 64) return 29.0;
  if (L == 96) return 45.0;
  if (L == 128) return 60.0;
  return 75.0;
}
static double warp_ns(int L, int p, int num_sms) {
  const int wd = (L + 31) / 32, loads = (p + 4 * num_sms - 1) / (4 * num_sms);
  const double windows = warp_pairs(L, p, num_sms) ? 440.0 * ((L + 63) / 64) : 290.0 * wd;   // ns a row
  return std::max(windows / L, 2.9 * loads * 32.0 * wd / L);
}

// Jobs side by side take as long as the longest, so only the jobs that would
// be longer than that one's faster form with a chain a lane take a warp a
// chain: a full warp of lanes issues a third of the instructions a site.
// (The uneven batch, young weights: 90 us a sweep with L = 48 and 64 a warp a
// chain and the others a lane, 120 with L = 32 a warp too, 166 with all a lane;
// L = 48 and 64 alone 48 each, together 76: the schedulers are then full.)
void batch_branch_shapes(int n, const int* L, const int* p, int num_sms, LaunchShape* out) {
  double longest = 0.0;
  for (int i = 0; i < n; ++i)
    longest = std::max(longest, L[i] * L[i] * std::min(lane_ns(L[i]), warp_ns(L[i], p[i], num_sms)));
  for (int i = 0; i < n; ++i) {
    if (L[i] * L[i] * lane_ns(L[i]) <= longest || !warp_chain_better(L[i], p[i], num_sms)) {
      out[i] = full_lane_shape(L[i], p[i], num_sms);
    } else {
      out[i] = LaunchShape{kPlaceSmem, 1, 4};
    }
  }
}

// The joint's replay kernels take their own launch shape (their work items
// are (chain, segment) pairs, not chains): as many lanes a block as the
// lattices leave room for, preferring shapes whose threshold table (and the
// prefix pass's histogram) still fit in shared memory.  The prefix pass, which
// also needs the histogram there, narrows the warps further if it must
// (launch_join_t).  L = 128: 28 lanes x 4 warps instead of 32 x 2 -- the
// lattices, 2 KB a lane, fill shared memory either way, and four warps keep
// all four sub-partitions issuing.
static bool replay_fits(int L, const LaunchShape& s) {
  if (s.cpw < 1 || s.cpw > 32 || s.wpb < 1 || s.wpb > 4) return false;
  if (s.placement == kPlaceReg && L > 32) return false;
  return plan_bytes(L, s, false, false) <= kMaxSmem;
}

static LaunchShape join_shape(int L, const LaunchShape& gen_shape) {
  LaunchShape gen = gen_shape;
  if (gen.placement == kPlaceGlobal) gen.placement = kPlaceSmem;   // replays restore into shared memory
  if (gen.cpw == 1 && L <= 32 && L != 24 && L != 32) gen.placement = kPlaceReg;   // (one chain a warp)
  LaunchShape best = gen;
  int best_lanes = 0;
  bool best_ts = false;
  for (int w = 4; w >= 1; --w) {
    int cpw = 32;
    while (cpw > 1 && !replay_fits(L, LaunchShape{gen.placement, cpw, w})) --cpw;
    const LaunchShape s{gen.placement, cpw, w};
    if (!replay_fits(L, s)) continue;
    int c2 = cpw;  // most chains per warp that leave the table and histogram in shared memory
    while (c2 >= 1 && !table_fits(L, LaunchShape{gen.placement, c2, w}, true)) --c2;
    if (c2 >= 16) {
      if (!best_ts || c2 * w > best_lanes) best = LaunchShape{gen.placement, c2, w}, best_lanes = c2 * w, best_ts = true;
    } else if (!best_ts && cpw * w > best_lanes) {
      best = s, best_lanes = cpw * w;
    }
  }
  return best;
}

cudaError_t join_prelude(const DevJob& j, cudaStream_t st) {
  order_kernel<<<1, 1024, 0, st>>>(j);
  spec_inputs_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j);
  clear_stats_kernel<<<256, 256, 0, st>>>(j);
  tj_kernel<<<blocks_for(static_cast<long long>(j.p) * j.np1, 256), 256, 0, st>>>(j, nullptr, j.p);
  launches_add(4);
  return cudaGetLastError();
}

// k_i = the earliest accepted sample the search found (0: none).
__global__ void select_kernel(const DevJob j, const int listed) {
  const int n = listed ? static_cast<int>(j.stats[kStatPending]) : j.p;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const int i = listed ? j.work[q] : q;
  const unsigned long long k = j.kmin[i];
  j.k[i] = k == kNoHit ? 0 : static_cast<int64_t>(k);
}

// Work list of the prefix pass: for every chain, its whole segments before
// the one holding k_i (all segments if nothing is kept) and, if k_i is not
// the first sample of its segment, that segment as a partial item.  Whole
// segments are counted first, then placed at the front of the list.
__global__ void prefix_count_kernel(const DevJob j, const int64_t S) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= j.p) return;
  const int64_t segN = j.seg_len;
  const int64_t k = j.k[i];
  const int whole = (k > 0) ? static_cast<int>((k - 1) / segN) : j.ck_K;
  atomicAdd(reinterpret_cast<unsigned long long*>(&j.stats[kStatQueuePrefix]), static_cast<unsigned long long>(whole));
  (void)S;
}

__global__ void prefix_fill_kernel(const DevJob j, const int64_t S) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= j.p) return;
  const int64_t segN = j.seg_len;
  const int64_t k = j.k[i];
  const int whole = (k > 0) ? static_cast<int>((k - 1) / segN) : j.ck_K;
  unsigned long long* w = reinterpret_cast<unsigned long long*>(&j.stats[kStatWholeFill]);
  unsigned long long* pcount = reinterpret_cast<unsigned long long*>(&j.stats[kStatPartial]);
  if (whole > 0) {
    const unsigned long long pos = atomicAdd(w, static_cast<unsigned long long>(whole));
    for (int s = 0; s < whole; ++s) j.plist[pos + s] = make_int2(i, s);
  }
  if (k > 0 && (k - 1) % segN != 0) {
    const unsigned long long total_whole = static_cast<unsigned long long>(j.stats[kStatQueuePrefix]);
    const unsigned long long pos = total_whole + atomicAdd(pcount, 1ull);
    j.plist[pos] = make_int2(i, whole);
  }
  (void)S;
}

__global__ void prefix_total_kernel(const DevJob j) {
  if (threadIdx.x == 0) j.stats[kStatQueuePrefix] += j.stats[kStatPartial];
}

__global__ void reset_queue_kernel(const DevJob j) {
  if (threadIdx.x == 0) j.stats[kStatQueueSearch] = 0;
}

cudaError_t join_summary_init(const DevJob& j, cudaStream_t st) {
  summary_init_kernel<<<1024, 256, 0, st>>>(j);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t join_scan(const DevJob& j, cudaStream_t st) {
  // one warp per (chain, candidate input), grid-stride
  cand_kernel<<<std::min(1024u, blocks_for(static_cast<long long>(j.p) * kScanCand * 32, 256)), 256, 0, st>>>(j);
  scan_kernel<<<1, 1024, 0, st>>>(j);
  launches_add(2);
  return cudaGetLastError();
}

cudaError_t kept_prelude(const DevJob& j, cudaStream_t st) {
  if (j.ordered) launch_next(order_kernel, 1, 1024, 0, st, j);
  launch_next(kept_prelude_kernel, std::min(304u, blocks_for(std::max(j.p, j.np1), 256)), 256, 0, st, j);
  launches_add(j.ordered ? 2 : 1);
  return cudaGetLastError();
}

cudaError_t kept_mark(const DevJob& j, int64_t S, int flags, cudaStream_t st) {
  launch_next(kept_mark_kernel, 1, 1024, 0, st, j, S * j.N, flags);
  launches_add(1);
  return cudaGetLastError();
}

// (one block does the whole scan where its three parts are short: two launches saved)
constexpr int kScanOneBlock = 4096;
cudaError_t kept_mark_scan(const DevJob& j, int64_t S, int flags, cudaStream_t st) {
  if (j.p <= kScanOneBlock) {
    launch_next(kept_mark_scan_kernel, 1, 1024, 0, st, j, S * j.N, flags);
    launches_add(1);
    return cudaGetLastError();
  }
  const cudaError_t e = kept_mark(j, S, flags, st);
  return e == cudaSuccess ? kept_scan(j, st) : e;
}

cudaError_t kept_scan(const DevJob& j, cudaStream_t st) {
  if (j.p <= kScanOneBlock) {
    launch_next(height_scan_kernel, 1, 1024, 0, st, j);
    launches_add(1);
    return cudaGetLastError();
  }
  launch_next(height_value_kernel, std::min(152u, blocks_for(j.p, 1024)), 1024, 0, st, j);
  launch_next(height_next_kernel, std::min(1024u, blocks_for(j.p + 1, 128)), 128, 0, st, j);
  launch_next(height_path_kernel, 1, 1024, 0, st, j);
  launches_add(3);
  return cudaGetLastError();
}

cudaError_t join_reset_queue(const DevJob& j, cudaStream_t st) {
  reset_queue_kernel<<<1, 32, 0, st>>>(j);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t join_prefix_list(const DevJob& j, cudaStream_t st) {
  prefix_count_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j, 0);
  prefix_fill_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j, 0);
  prefix_total_kernel<<<1, 32, 0, st>>>(j);
  launches_add(3);
  return cudaGetLastError();
}

cudaError_t join_select(const DevJob& j, bool listed, cudaStream_t st) {
  select_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j, listed ? 1 : 0);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t join_mark(const DevJob& j, cudaStream_t st, bool thresholds, bool defer) {
  mark_kernel<<<1, 1024, 0, st>>>(j, defer ? 1 : 0);
  launches_add(1);
  return thresholds ? join_tj_list(j, st) : cudaGetLastError();
}

cudaError_t join_nohit(const DevJob& j, int list_mode, cudaStream_t st) {
  nohit_kernel<<<1, 1024, 0, st>>>(j, list_mode);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t join_tj_list(const DevJob& j, cudaStream_t st) {
  tj_list_kernel<<<256, 256, 0, st>>>(j);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t join_finalize(const DevJob& j, int64_t S, cudaStream_t st) {
  launch_finalize(j, S * j.N, j.rec || j.flips, st);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t chain_kernels_warp(const DevJob& j, uint64_t t0, int64_t S, bool trace, cudaStream_t st) {
  int dev = 0, sms = 1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int warps = 1;
  bool ts = false;
  warp_chain_shape(j.L, j.p, sms, &warps, &ts);
  const bool pairs = warp_pairs(j.L, j.p, sms);
  if (j.wd == 1) return chain_kernels_warp_1(j, warps, ts, pairs, t0, S, trace, st);
  if (j.wd == 2) return (j.L <= 48 ? chain_kernels_warp_2a : chain_kernels_warp_2b)(j, warps, ts, pairs, t0, S, trace, st);
  if (j.wd == 3) return (j.L <= 80 ? chain_kernels_warp_3a : chain_kernels_warp_3b)(j, warps, ts, pairs, t0, S, trace, st);
  return (j.L <= 112 ? chain_kernels_warp_4a : chain_kernels_warp_4b)(j, warps, ts, pairs, t0, S, trace, st);
}

static cudaError_t dispatch(const DevJob& j, const LaunchShape& s, bool gen, uint64_t t0, int64_t S, bool trace,
                            uint32_t r, cudaStream_t st) {
  if (gen && s.placement == kPlaceSmem && s.cpw == 1) return chain_kernels_warp(j, t0, S, trace, st);
  if (s.placement == kPlaceReg) {
    if (j.L <= 16) return chain_kernels_reg_a(j, s, gen, t0, S, trace, r, st);
    if (j.L <= 28) return chain_kernels_reg_b(j, s, gen, t0, S, trace, r, st);
    return chain_kernels_reg_c(j, s, gen, t0, S, trace, r, st);
  }
  switch (j.L) {
    case 16:
    case 24: return chain_kernels_smem_L16_24(j, s, gen, t0, S, trace, r, st);
    case 32: return chain_kernels_smem_L32(j, s, gen, t0, S, trace, r, st);
    case 48: return chain_kernels_smem_L48(j, s, gen, t0, S, trace, r, st);
    case 64: return chain_kernels_smem_L64(j, s, gen, t0, S, trace, r, st);
    case 96: return chain_kernels_smem_L96(j, s, gen, t0, S, trace, r, st);
    case 100: return chain_kernels_smem_L100(j, s, gen, t0, S, trace, r, st);
    case 128: return chain_kernels_smem_L128(j, s, gen, t0, S, trace, r, st);
    default: break;
  }
  switch (j.wd) {
    case 1: return chain_kernels_smem_1(j, s, gen, t0, S, trace, r, st);
    case 2: return chain_kernels_smem_2(j, s, gen, t0, S, trace, r, st);
    case 3: return chain_kernels_smem_3(j, s, gen, t0, S, trace, r, st);
    case 4: return chain_kernels_smem_4(j, s, gen, t0, S, trace, r, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t k_generate(const DevJob& j, const LaunchShape& s, uint64_t t0, int64_t S, bool trace, cudaStream_t st) {
  if (j.rec) {   // a recorded round is never replayed: no checkpoints
    DevJob g = j;
    g.ckpt = nullptr;
    return dispatch(g, s, true, t0, S, trace, 0u, st);
  }
  return dispatch(j, s, true, t0, S, trace, 0u, st);
}

cudaError_t k_join(const DevJob& j, const LaunchShape& s, uint64_t t0, int64_t S, uint32_t r, bool naive,
                   cudaStream_t st) {
  if (naive) {
    order_kernel<<<1, 1024, 0, st>>>(j);
    naive_kernel<<<blocks_for(j.p, 256), 256, 0, st>>>(j);
    launch_finalize(j, S * j.N, false, st);
    launches_add(3);
    return cudaGetLastError();
  }
  if (j.rec) return chain_kernels_record(j, S, r, st);   // levels recorded: no replays
  if (j.flips) return chain_kernels_flips(j, S, r, st);   // nor where the flips are
  return dispatch(j, join_shape(j.L, s), false, t0, S, false, r, st);
}

cudaError_t k_order(const DevJob& j, cudaStream_t st) {
  order_kernel<<<1, 1024, 0, st>>>(j);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t k_init_lattice(const DevJob& j, int start, cudaStream_t st) {
  const long long n = static_cast<long long>(j.p) * j.L * j.wd;
  init_lattice_kernel<<<blocks_for(n, 256), 256, 0, st>>>(j, start);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t k_levels(const DevJob& j, cudaStream_t st) {
  levels_kernel<<<blocks_for(32ll * j.p, 128), 128, 0, st>>>(j);
  launches_add(1);
  return cudaGetLastError();
}

cudaError_t k_build_table(const DevJob& j, cudaStream_t st) {
  launch_next(table_kernel, blocks_for(5ll * j.np1, 256), 256, 0, st, j);
  launches_add(1);
  return cudaGetLastError();
}

size_t thermo_doubles(int np1, int n) { return 5ull * n + 2 * kThermoParts + (np1 + 1) / 2; }

// buf: thermo_doubles() doubles -- betas, then the results, then scratch.
cudaError_t k_thermo(const DevJob& j, int n, double* buf, cudaStream_t st) {
  double* norm = buf + 5ull * n;
  float* neg = reinterpret_cast<float*>(norm + 2 * kThermoParts);
  // L <= 32, up to two blocks an SM: 1025 exponentials a block, 4 a thread, against a launch (L = 16, 10
  // betas 47 against 51 us a call; L = 32, 10000 betas 1.28 against 0.85 ms)
  const bool own = j.np1 <= 1025 && n <= 304;
  const int bytes = (own ? 12 : 8) * j.np1;
  auto kern = own ? thermo_kernel<true> : thermo_kernel<false>;
  const cudaError_t e = allow_smem(kern);
  if (e != cudaSuccess) return e;
  if (!own) thermo_norm_kernel<<<kThermoParts, kThermoThreads, 0, st>>>(j, norm, neg);
  kern<<<n, kThermoThreads, bytes, st>>>(j, buf, norm, neg, buf + n);
  launches_add(own ? 1 : 2);
  return cudaGetLastError();
}

cudaError_t k_update_weights(const DevJob& j, cudaStream_t st) {
  launch_next(weights_kernel, blocks_for(j.np1, 256), 256, 0, st, j);
  launches_add(1);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return k_build_table(j, st);
}

}  // namespace mcgpu
