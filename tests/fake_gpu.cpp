// A stand-in for the GPU under the host side of the library (nrm_api.cpp): the
// CUDA runtime calls that it makes, on host memory, and the kernel launchers,
// which append one line per launch to a log instead of launching. With it the
// choice of kernels, the launch counts, the cache keys and the error paths of
// the C ABI are tested without a GPU (tests/fake_gpu.py builds and loads it).
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "nrm_internal.h"

namespace {

std::string g_log;
int g_capture = 0;      // what cudaStreamIsCapturing reports
int g_fail_at = -1;     // the launch that fails (0 = the next), or none
int g_timing = 0;       // elapsed-time queries answered so far
int g_fastest = -1;     // the query that gets the shortest time
int g_event_syncs = 0;
bool g_no_memory = false;  // allocations fail

cudaError_t launched(const std::string& line) {
  if (g_fail_at == 0) {
    g_fail_at = -1;
    return cudaErrorLaunchFailure;
  }
  if (g_fail_at > 0) --g_fail_at;
  const bool none = g_no_memory;  // (the log itself may grow)
  g_no_memory = false;
  g_log += line + "\n";
  g_no_memory = none;
  return cudaSuccess;
}

std::string describe(const char* name, const nrm::BatchHeader* hdr) {
  return std::string(name) + " frames=" + std::to_string(hdr->n_frames) + " tiles=" + std::to_string(hdr->total_tiles);
}

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void* base, const cuuint64_t*, const cuuint64_t* strides,
                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                CUtensorMapFloatOOBfill) {
  return reinterpret_cast<uintptr_t>(base) % 16 || strides[0] % 16 ? CUDA_ERROR_INVALID_VALUE : CUDA_SUCCESS;
}

// Kernel addresses: one byte each.
char k_plain[3], k_persistent[3], k_points[2], k_param;
const nrm::FwdKernelSet kSets[2] = {
    {128, 16, 256, {&k_plain[0], &k_plain[1], &k_plain[2]}, {&k_persistent[0], &k_persistent[1], &k_persistent[2]}},
    {128, 8, 128, {&k_plain[0], &k_plain[1], &k_plain[2]}, {&k_persistent[0], &k_persistent[1], &k_persistent[2]}}};

const char* kernel_name(const void* fn) {
  if (fn >= k_plain && fn < k_plain + 3) return "plain";
  if (fn >= k_persistent && fn < k_persistent + 3) return "tiled_ring";
  if (fn == &k_points[0]) return "plain_points";
  if (fn == &k_points[1]) return "tiled_points";
  return fn == &k_param ? "tiled" : "unknown";
}

}  // namespace

void* operator new(size_t n) {
  void* p = g_no_memory ? nullptr : malloc(n ? n : 1);
  if (!p) throw std::bad_alloc();
  return p;
}
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

#define FAKE extern "C" __attribute__((visibility("default")))

FAKE const char* fake_log() { return g_log.c_str(); }
FAKE void fake_reset() {
  g_log.clear();
  g_capture = 0;
  g_fail_at = -1;
  g_timing = 0;
  g_fastest = -1;
  g_event_syncs = 0;
}
FAKE void fake_capture(int on) { g_capture = on; }
FAKE void fake_fail_launch(int k) { g_fail_at = k; }
FAKE void fake_fastest(int k) { g_fastest = k; }
FAKE int fake_timings() { return g_timing; }
FAKE void fake_no_memory(int on) { g_no_memory = on != 0; }
FAKE int fake_event_syncs() { return g_event_syncs; }

extern "C" {

cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  std::strcpy(p->name, "FAKE");
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaMalloc(void** p, size_t n) { return *p = aligned_alloc(256, (n + 255) / 256 * 256), cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaMemset(void* p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  g_log += "upload\n";
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void*, size_t, const void*, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = reinterpret_cast<cudaEvent_t>(&g_log), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return ++g_event_syncs, cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = g_timing == g_fastest ? 0.5f : 1.0f + g_timing;
  ++g_timing;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = nullptr, cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  return *s = g_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone, cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  return *n = 3, cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernel(const void* fn, dim3, dim3, void** args, size_t, cudaStream_t) {
  return launched(fn == &k_param ? describe("tiled", static_cast<const nrm::BatchHeader*>(args[0])) : kernel_name(fn));
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return *g = reinterpret_cast<cudaGraph_t>(&g_log), cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphAddMemcpyNode1D(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, void*, const void*,
                                     size_t, cudaMemcpyKind) {
  return *n = nullptr, cudaSuccess;
}
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t,
                                   const cudaKernelNodeParams*) {
  return *n = nullptr, cudaSuccess;
}
cudaError_t cudaGraphAddEventRecordNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, cudaEvent_t) {
  return *n = nullptr, cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return *e = reinterpret_cast<cudaGraphExec_t>(&g_log), cudaSuccess;
}
cudaError_t cudaGraphExecMemcpyNodeSetParams1D(cudaGraphExec_t, cudaGraphNode_t, void*, const void*, size_t,
                                               cudaMemcpyKind) {
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return launched("tiled_graph"); }

}  // extern "C"

namespace nrm {

int fwd_kernel_count() { return 2; }
const FwdKernelSet* fwd_kernel(int i) { return &kSets[i]; }
const FwdKernelSet* fwd_kernel_find(int tx, int ty, int threads) {
  for (const auto& s : kSets)
    if (s.tile_x == tx && s.tile_y == ty && s.threads == threads) return &s;
  return nullptr;
}
const void* fwd_points_kernel(int, int, int, int, bool persistent) { return &k_points[persistent]; }
const void* fwd_param_kernel(int, int, int, int) { return &k_param; }
size_t param_batch_bytes() { return sizeof(BatchHeader) + sizeof(FrameDesc) * kParamMaxFrames; }
void pack_param_batch(void* dst, const BatchHeader& hdr, const int* tb, const FrameDesc* frames, int n) {
  if (n > kParamMaxFrames || tb[n] != hdr.total_tiles) abort();
  std::memcpy(dst, &hdr, sizeof(hdr));
  std::memcpy(static_cast<char*>(dst) + sizeof(hdr), frames, sizeof(FrameDesc) * (size_t)n);
}
cudaError_t launch_forward_strip(const BatchArgs& a, const Globals&, int, int tiles, bool, bool aligned, cudaStream_t,
                                 const void* pb) {
  const BatchHeader* hdr = pb ? static_cast<const BatchHeader*>(pb) : a.hdr;
  if (hdr->total_tiles != tiles) abort();
  return launched(describe(aligned ? "strip" : "strip_any", hdr));
}
cudaError_t launch_multiscale(const FrameDesc&, const MsConsts&, const Globals&, int, int, cudaStream_t) {
  return launched("ms_plain");
}
cudaError_t launch_multiscale_batched(const BatchArgs& a, const MsConsts&, const Globals&, int, int, int tiles, bool,
                                      cudaStream_t, const void* pb) {
  const BatchHeader* hdr = pb ? static_cast<const BatchHeader*>(pb) : a.hdr;
  if (hdr->total_tiles != tiles) abort();
  return launched(describe("ms_tiled", hdr));
}
cudaError_t launch_multiscale_strip(const MsConsts&, const Globals&, int, int, int tiles, bool, cudaStream_t, void* pb) {
  const BatchHeader* hdr = static_cast<const BatchHeader*>(pb);
  if (hdr->total_tiles != tiles) abort();
  return launched(describe("ms_strip", hdr));
}
int ms_strip_tile_y() { return 64; }
cudaError_t launch_backward(const FrameDesc& d, const BwdMaps&, const Globals& g, bool walk, cudaStream_t,
                            const float*) {
  return launched("bwd walk=" + std::to_string(walk) + " tma=" + std::to_string(d.use_tma));
}
cudaError_t launch_backward_batched(const BwdBatchArgs&, int n, int, const Globals&, bool walk, cudaStream_t,
                                    const float*) {
  return launched("bwd_ring walk=" + std::to_string(walk) + " frames=" + std::to_string(n));
}
cudaError_t launch_backward_batched_param(const FrameDesc*, const BwdMaps*, int n, int, const Globals&, bool walk,
                                          cudaStream_t, const float*) {
  return launched("bwd_batch walk=" + std::to_string(walk) + " frames=" + std::to_string(n));
}
cudaError_t launch_loss_scale(const LossCountFrame*, int, unsigned*, unsigned*, float*, cudaStream_t) {
  return launched("loss_scale");
}
cudaError_t launch_spherical(const float*, const uint8_t*, int, int, long long, float*, float*, cudaStream_t) {
  return launched("spherical");
}
cudaError_t launch_angle_mse(const float*, const uint8_t*, const float*, const uint8_t*, int, int, long long, double*,
                             unsigned*, double*, int*, unsigned long long, cudaStream_t) {
  return launched("mse");
}
cudaError_t launch_wait_expiry(unsigned long long, int*, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t launch_bounds_selftest(int*, int*, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t launch_plane_fit(const FrameDesc&, int, float, int, cudaStream_t) { return launched("plane_fit"); }

}  // namespace nrm
