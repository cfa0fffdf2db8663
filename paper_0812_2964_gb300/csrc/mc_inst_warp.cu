// Instantiation unit: generation with one chain per warp, rows of up to 32, 64 and 128 sites, L read at run time.
#include "mc_warp_chain.cuh"

namespace mcgpu {

template <class Rows, bool TSMEM, int KEEP>
__global__ void __launch_bounds__(32 * kWarpChainBlock, 1)
    warp_gen_kernel(const DevJob j, const uint64_t t0, const int64_t S, const int64_t flushF, const int do_trace) {
  warp_gen_body<Rows, TSMEM, KEEP>(j, t0, S, flushF, do_trace, blockIdx.x);
}

template <class Rows>
static cudaError_t launch_rows(const DevJob& j, int warps, bool ts, uint64_t t0, int64_t S, bool trace,
                               cudaStream_t st) {
  auto kern = ts ? warp_gen_kernel<Rows, true, kKeepNone> : warp_gen_kernel<Rows, false, kKeepNone>;
  if (j.rec) kern = ts ? warp_gen_kernel<Rows, true, kKeepLevels> : warp_gen_kernel<Rows, false, kKeepLevels>;
  else if (j.flips) kern = ts ? warp_gen_kernel<Rows, true, kKeepFlips> : warp_gen_kernel<Rows, false, kKeepFlips>;
  const size_t bytes = 4ull * warp_plan(j.L, warps, ts).total;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  if (e != cudaSuccess) return e;
  kern<<<blocks_for(j.p, warps), 32 * warps, bytes, st>>>(j, t0, S, warp_flush_sweeps(warps, j.N, S), trace ? 1 : 0);
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
  if (j.wd == 1) return launch_rows<Words<1>>(j, warps, ts, t0, S, trace, st);
  if (j.wd == 2) return launch_rows<TwoWords<1>>(j, warps, ts, t0, S, trace, st);
  if (j.wd == 3) return launch_rows<Words<3>>(j, warps, ts, t0, S, trace, st);
  if (warp_pairs(j.L, j.p, sms)) return launch_rows<TwoWords<2>>(j, warps, ts, t0, S, trace, st);
  return launch_rows<Words<4>>(j, warps, ts, t0, S, trace, st);
}

}  // namespace mcgpu
