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
// The octahedral output is bound by instruction issue (37.5 warp instructions per 32
// pixels, issue slots 65 % busy), so as many warps as fit run: 4 warps x 8 rows, 192 us
// (71 %; tiled 341 us); float32 input with 2 stages, 4 CTAs, 198 us (3 stages, 3 CTAs:
// 205).
// Batches of few tiles take all the CTAs that fit: there the ramp counts, not the
// steady state (16 x 640x480 float32: 18.8 us with 3 CTAs per SM, 20.9 with one;
// 2 x 1080p 15.2 against 16.0, 4 x 1080p 30.7 against 29.6 us).
//
// Frames of any alignment (loader warps instead of TMA; nothing comes near
// saturating HBM): as many CTAs as fit, 6 compute and 4 loader warps (octahedral
// 4 and 2). 64 x 1921x1081: uint16 -> float4 487 us (76 %; the tiled kernel's plain
// loads 1080), float32 -> float4 503 (1160), uint16 -> half4 485 (812), octahedral
// 439 (831); two 3001x2001 uint16 frames 44 us (75). [float4 from uint16 and float32,
// half4: 6 loader warps 521 / 520 / 539; 4 compute warps, 3 CTAs 488 / 504 / 515; 12
// and 16 compute warps, 1 CTA 650 / 685 / 566.] Which calls take which kernel:
// forward_plan in nrm_api.cpp.
#include <algorithm>
#include <atomic>

#include "nrm_forward_strip.cuh"

namespace nrm {

namespace {

constexpr int kStripFewTiles = 12;  // tiles per SM

int strip_stages(int out_dtype, bool u16) { return out_dtype == NRM_OUT_OCT16 ? (u16 ? 4 : 2) : 3; }

}  // namespace

template const void* strip_kernel<true>(int, bool, int, bool);

cudaError_t launch_forward_strip(const BatchArgs& args, const Globals& g, int out_dtype, int total_tiles, bool u16,
                                 bool aligned, cudaStream_t stream, const void* param_block) {
  const bool param = param_block != nullptr;
  const bool secant = g.mask_mode == NRM_MASK_SECANT;
  const void* fn = aligned ? strip_kernel<true>(out_dtype, secant, g.alpha, param)
                           : strip_kernel<false>(out_dtype, secant, g.alpha, param);
  if (!fn) return cudaErrorInvalidValue;
  const int eb = u16 ? 2 : 4;
  const int stages = strip_stages(out_dtype, u16);
  const unsigned rowbuf = aligned ? 0 : strip_warps(out_dtype, aligned) * strip_rowbuf(out_dtype);
  const unsigned smem = strip_smem_bytes(strip_tile_y(out_dtype, aligned), g.alpha, eb, stages) + rowbuf;
  const int threads = strip_block(out_dtype, aligned);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  // CTAs of this kernel and staging size that fit an SM, found once, and the SMs.
  static std::atomic<int> fit[2][3][2][kStripMaxAlpha + 1][2][2][64];
  static std::atomic<int> sm_count[64];
  std::atomic<int>& occ = fit[aligned][out_dtype][secant][g.alpha][param][u16][dev];
  if (occ.load() == 0) {
    int sms = 0, n = 0;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(strip_smem_bytes(strip_tile_y(out_dtype, aligned), kStripMaxAlpha, 4, 3) + rowbuf));
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
  const int per_sm = aligned && out_dtype != NRM_OUT_OCT16 && total_tiles > kStripFewTiles * sms ? 1 : occ.load();
  const int ctas = per_sm * sms;
  BatchArgs a = args;
  a.stages = stages;
  a.stage_bytes = strip_stage_bytes(strip_tile_y(out_dtype, aligned), g.alpha, eb);
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
