// Launcher of the multi-scale strip kernels and their float4 instantiations.
#include <algorithm>
#include <atomic>

#include "nrm_multiscale_strip.cuh"

namespace nrm {

template const void* ms_strip::by_form<NRM_OUT_F32X4>(int, bool, int);

using namespace ms_strip;

int ms_strip_tile_y() { return kRows * kWarps; }

cudaError_t launch_multiscale_strip(const MsConsts& ms, const Globals& g, int out_dtype, int form, int total_tiles,
                                    bool u16, cudaStream_t stream, void* param_block) {
  if (out_dtype < 0 || out_dtype > 2 || (form != NRM_MS_PAIR && form != NRM_MS_QUAD)) return cudaErrorInvalidValue;
  const bool secant = g.mask_mode == NRM_MASK_SECANT;
  const void* fn = out_dtype == NRM_OUT_F32X4   ? by_form<NRM_OUT_F32X4>(form, secant, ms.K)
                   : out_dtype == NRM_OUT_F16X4 ? by_form<NRM_OUT_F16X4>(form, secant, ms.K)
                                                : by_form<NRM_OUT_OCT16>(form, secant, ms.K);
  if (!fn) return cudaErrorInvalidValue;
  const int eb = u16 ? 2 : 4;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  // Shared memory granted and SMs looked up once per kernel and device.
  static std::atomic<int> sm_count[3][2][2][kMsStripMaxScales + 1][64];
  std::atomic<int>& known = sm_count[out_dtype][form][secant][ms.K][dev];
  if (known.load() == 0) {
    int sms = 0;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)strip_smem_bytes(kRows * kWarps, ms.K, 4, kStages));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    known.store(sms);
  }
  BatchArgs a = {};
  a.stages = kStages;
  a.stage_bytes = strip_stage_bytes(kRows * kWarps, ms.K, eb);
  Globals gg = g;
  void* pargs[3] = {param_block, &a, &gg};
  return cudaLaunchKernel(fn, dim3(std::min(total_tiles, known.load())), dim3((kWarps + 1) * 32), pargs,
                          strip_smem_bytes(kRows * kWarps, ms.K, eb, kStages), stream);
}

}  // namespace nrm
