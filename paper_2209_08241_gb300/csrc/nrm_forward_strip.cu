// Registry and launcher of the strip kernels (nrm_forward_strip.cuh).
//
// Launch shape. For float4 and half4 outputs the kernel would be held by HBM,
// and there more warps and deeper read-ahead make it slower: with the memory
// system saturated, reads that arrive all the time between the writes cost
// DRAM throughput (64 x 1920x1080 uint16 -> float4: 437-450 us = 84 % of the
// measured copy for every shape with more than about 100 staged rows per SM,
// whatever the store width or cache policy; an L2 prefetch further ahead:
// 480 us). One CTA per SM, with just enough compute warps, and a ring of about
// 72 staged rows (float4) or 144 (half4) lets the loads hold back the stores:
//   float4: 6 warps x 4 rows, 3 stages   375-380 us (98 %), float32 input 429 us
//           (96 %), alpha 3 / 4 392 / 379 us; 256 mixed float32 frames 1.05 ms
//           (98 %)  [8 warps x 8 rows, 3 stages 440; 4 x 4, 4 stages, 409]
//   half4:  12 warps x 4 rows, 3 stages  226 us (95 %), float32 input 259 us
//           (98 %)  [10 warps, 4 stages 222 / 292; 8 x 8, 3 stages 221 / 294]
// The tiled kernel in its default geometry (128x16, 256 threads) takes 441,
// 348 and 1283 us on the float4, half4 and mixed batches.
// The octahedral output is bound by instruction issue (about 40 instructions a
// pixel), so as many warps as fit run: 4 warps x 8 rows, 192 us (71 %; tiled
// 341 us); float32 input with 2 stages, 4 CTAs, 198 us (3 stages, 3 CTAs: 205).
// Batches of few tiles take all the CTAs that fit: there the ramp counts, not the
// steady state (16 x 640x480 float32: 18.8 us with 3 CTAs per SM, 20.9 with one;
// 2 x 1080p 15.2 against 16.0, 4 x 1080p 30.7 against 29.6 us).
#include <algorithm>
#include <atomic>

#include "nrm_forward_strip.cuh"

namespace nrm {

namespace {

constexpr int kStripFewTiles = 12;  // tiles per SM

int strip_stages(int out_dtype, bool u16) { return out_dtype == NRM_OUT_OCT16 ? (u16 ? 4 : 2) : 3; }

template <int OUT, bool SECANT>
const void* strip_kernel_for(int alpha, bool param) {
  switch (alpha) {
    case 1: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 1> : (const void*)fwd_strip_kernel<OUT, SECANT, 1>;
    case 2: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 2> : (const void*)fwd_strip_kernel<OUT, SECANT, 2>;
    case 3: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 3> : (const void*)fwd_strip_kernel<OUT, SECANT, 3>;
    case 4: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 4> : (const void*)fwd_strip_kernel<OUT, SECANT, 4>;
    default: return nullptr;
  }
}

const void* strip_kernel(int out_dtype, bool secant, int alpha, bool param) {
  switch (out_dtype) {
    case NRM_OUT_F32X4: return secant ? strip_kernel_for<NRM_OUT_F32X4, true>(alpha, param) : strip_kernel_for<NRM_OUT_F32X4, false>(alpha, param);
    case NRM_OUT_F16X4: return secant ? strip_kernel_for<NRM_OUT_F16X4, true>(alpha, param) : strip_kernel_for<NRM_OUT_F16X4, false>(alpha, param);
    case NRM_OUT_OCT16: return secant ? strip_kernel_for<NRM_OUT_OCT16, true>(alpha, param) : strip_kernel_for<NRM_OUT_OCT16, false>(alpha, param);
    default: return nullptr;
  }
}

}  // namespace

cudaError_t launch_forward_strip(const BatchArgs& args, const Globals& g, int out_dtype, int total_tiles, bool u16,
                                 cudaStream_t stream, const void* param_block) {
  const bool param = param_block != nullptr;
  const bool secant = g.mask_mode == NRM_MASK_SECANT;
  const void* fn = strip_kernel(out_dtype, secant, g.alpha, param);
  if (!fn) return cudaErrorInvalidValue;
  const int eb = u16 ? 2 : 4;
  const int stages = strip_stages(out_dtype, u16);
  const unsigned smem = strip_smem_bytes(strip_tile_y(out_dtype), g.alpha, eb, stages);
  const int threads = strip_threads(out_dtype);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  // CTAs of this kernel and staging size that fit an SM, found once, and the SMs.
  static std::atomic<int> fit[3][2][kStripMaxAlpha + 1][2][2][64];
  static std::atomic<int> sm_count[64];
  std::atomic<int>& occ = fit[out_dtype][secant][g.alpha][param][u16][dev];
  if (occ.load() == 0) {
    int sms = 0, n = 0;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)strip_smem_bytes(strip_tile_y(out_dtype), kStripMaxAlpha, 4, 3));
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) return cudaErrorInvalidConfiguration;
    sm_count[dev].store(sms);
    occ.store(n);
  }
  const int sms = sm_count[dev].load();
  // One CTA per SM once an SM has more than kStripFewTiles tiles (float4 and
  // half4; see the file comment), else as many as fit.
  const int per_sm = out_dtype != NRM_OUT_OCT16 && total_tiles > kStripFewTiles * sms ? 1 : occ.load();
  const int ctas = per_sm * sms;
  BatchArgs a = args;
  a.stages = stages;
  a.stage_bytes = strip_stage_bytes(strip_tile_y(out_dtype), g.alpha, eb);
  Globals gg = g;
  const dim3 grid(std::min(total_tiles, ctas)), block(threads);
  if (param) {
    void* pargs[3] = {const_cast<void*>(param_block), &a, &gg};
    return cudaLaunchKernel(fn, grid, block, pargs, smem, stream);
  }
  void* kargs[2] = {&a, &gg};
  return cudaLaunchKernel(fn, grid, block, kargs, smem, stream);
}

}  // namespace nrm
