// Instantiation unit: generation with one chain per warp, 1 to 4 words per row, L read at run time.
#include "mc_chain_kernels.cuh"
#include "mc_warp_chain.cuh"

namespace mcgpu {

template <int WD, bool TSMEM, bool REC>
__global__ void __launch_bounds__(32 * kWarpChainBlock, 1) warp_gen_kernel(const DevJob j, const uint64_t t0,
                                                                        const int64_t S, const int64_t flushF,
                                                                        const int do_trace) {
  warp_gen_body<WD, TSMEM, REC>(j, t0, S, flushF, do_trace, blockIdx.x);
}

template <int WD>
static cudaError_t launch_wd(const DevJob& j, int warps, bool ts, uint64_t t0, int64_t S, bool trace, cudaStream_t st) {
  const bool rec = j.rec != nullptr;
  auto kern = ts ? (rec ? warp_gen_kernel<WD, true, true> : warp_gen_kernel<WD, true, false>)
                 : (rec ? warp_gen_kernel<WD, false, true> : warp_gen_kernel<WD, false, false>);
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
  switch (j.wd) {
    case 1: return launch_wd<1>(j, warps, ts, t0, S, trace, st);
    case 2: return launch_wd<2>(j, warps, ts, t0, S, trace, st);
    case 3: return launch_wd<3>(j, warps, ts, t0, S, trace, st);
    case 4: return launch_wd<4>(j, warps, ts, t0, S, trace, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mcgpu
