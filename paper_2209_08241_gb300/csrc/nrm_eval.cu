// Evaluation kernels (arXiv 2209.08241, Section 4): the spherical angle images
// I_phi, I_theta of a normal map and the mean squared error of those images
// between an estimate and a reference (Tables 2-5).
//
//   phi   = atan2(n_y, n_x), taken into [0, 2 pi)
//   theta = atan2(sqrt(n_x^2 + n_y^2), n_z), in [0, pi]
//
// over valid pixels (masked pixels get 0). The MSE is the mean, over pixels
// valid in both maps, of the squared plain differences of the angle images.
// It is reduced deterministically: a fixed grid of kMseBlocks blocks, each
// summing a fixed set of row pieces (per thread in FP32 over at most 32 pixels,
// beyond that in FP64) in a fixed order; the last block to finish sums the
// blocks' partials in a fixed order.
#include <atomic>

#include "nrm_device.cuh"

namespace nrm {

namespace {

constexpr int kThreads = 256;

// atan2(y, x) for the angle images: the quotient of the smaller by the larger
// magnitude, t in [0, 1], gives atan(t) from a polynomial in t^2 (our own
// near-minimax fit, atan_fit.py beside this file: 3.8e-8 rad, 1.1e-7 rad as
// evaluated in FP32), then the octant is restored: pi/2 - r where |y| > |x|,
// pi - r where x is negative (its sign bit set, so that -0 counts as
// negative, as in IEEE atan2), and the sign of y is copied onto the result
// (y = +-0 then gives +-0 or +-pi). Both zero gives +-0 or +-pi the same way.
// Accurate to about 3e-7 rad over the whole plane (tests/test_atan_fit.py).
__device__ __forceinline__ float atan2_fit(float y, float x) {
  const float ax = fabsf(x), ay = fabsf(y);
  const float hi = fmaxf(ax, ay), lo = fminf(ax, ay);
  const float t = lo * dev::rcp_ftz(fmaxf(hi, 1.17549435e-38f));
  const float s = t * t;
  float p = -4.054556135e-03f;
  p = fmaf(p, s, 2.186293714e-02f);
  p = fmaf(p, s, -5.591233820e-02f);
  p = fmaf(p, s, 9.642202407e-02f);
  p = fmaf(p, s, -1.390863359e-01f);
  p = fmaf(p, s, 1.994656771e-01f);
  p = fmaf(p, s, -3.332986236e-01f);
  p = fmaf(p, s, 9.999993443e-01f);
  float r = t * p;
  r = ay > ax ? 1.57079632679489662f - r : r;
  r = signbit(x) ? 3.14159265358979324f - r : r;
  return copysignf(r, y);
}

__device__ __forceinline__ void angles(float4 n, float& phi, float& theta) {
  phi = atan2_fit(n.y, n.x);
  phi = phi < 0.0f ? phi + 6.28318530717958647692f : phi;
  theta = atan2_fit(sqrtf(fmaf(n.x, n.x, n.y * n.y)), n.z);
}

// atan2_fit of two directions, operation for operation, with the quotient and the
// polynomial in paired FP32.
__device__ __forceinline__ float2 atan2_fit2(float2 y, float2 x) {
  using dev::f2;
  const float2 hi = f2(fmaxf(fmaxf(fabsf(x.x), fabsf(y.x)), 1.17549435e-38f),
                       fmaxf(fmaxf(fabsf(x.y), fabsf(y.y)), 1.17549435e-38f));
  const float2 lo = f2(fminf(fabsf(x.x), fabsf(y.x)), fminf(fabsf(x.y), fabsf(y.y)));
  const float2 t = __fmul2_rn(lo, f2(dev::rcp_ftz(hi.x), dev::rcp_ftz(hi.y)));
  const float2 s = __fmul2_rn(t, t);
  auto c = [](float v) { return f2(v, v); };
  float2 p = __ffma2_rn(c(-4.054556135e-03f), s, c(2.186293714e-02f));
  p = __ffma2_rn(p, s, c(-5.591233820e-02f));
  p = __ffma2_rn(p, s, c(9.642202407e-02f));
  p = __ffma2_rn(p, s, c(-1.390863359e-01f));
  p = __ffma2_rn(p, s, c(1.994656771e-01f));
  p = __ffma2_rn(p, s, c(-3.332986236e-01f));
  p = __ffma2_rn(p, s, c(9.999993443e-01f));
  float2 r = __fmul2_rn(t, p);
  r.x = fabsf(y.x) > fabsf(x.x) ? 1.57079632679489662f - r.x : r.x;
  r.y = fabsf(y.y) > fabsf(x.y) ? 1.57079632679489662f - r.y : r.y;
  r.x = signbit(x.x) ? 3.14159265358979324f - r.x : r.x;
  r.y = signbit(x.y) ? 3.14159265358979324f - r.y : r.y;
  return f2(copysignf(r.x, y.x), copysignf(r.y, y.y));
}

// Square roots of two values: the hardware's reciprocal square root y, then one Newton
// step for s^2 = x from s = x y, s + (x - s^2) y / 2, whose residual one FMA gives exactly.
// The same bits as sqrtf for 0 and for every float from 2^-100 to the largest
// (compared one by one); below that the angle is off by at most 1.1e-19 rad, and
// infinity counts as the largest float (the angle is pi / 2 either way). So the MSE is
// that of the angle images as spherical_kernel forms them, without sqrtf's branch per
// value: the MSE kernel at 4096 x 3072 takes 77.4 us, with sqrtf 94, with the hardware's
// approximate square root (other bits for one float in six) 72.8.
__device__ __forceinline__ float2 sqrt2(float2 x) {
  using dev::f2;
  const float kFltMin = 1.17549435e-38f, kFltMax = 3.402823466e38f;
  x = f2(fminf(x.x, kFltMax), fminf(x.y, kFltMax));
  const float2 y = f2(dev::rsqrt_ftz(fmaxf(x.x, kFltMin)), dev::rsqrt_ftz(fmaxf(x.y, kFltMin)));
  const float2 s = __fmul2_rn(x, y), ns = __fmul2_rn(s, f2(-1.0f, -1.0f)), h = __fmul2_rn(y, f2(0.5f, 0.5f));
  return __ffma2_rn(__ffma2_rn(ns, s, x), h, s);
}

// The angles of two normals (the lanes of phi and theta), operation for operation those
// of angles().
__device__ __forceinline__ void angles2(float4 a, float4 b, float2& phi, float2& theta) {
  phi = atan2_fit2(dev::f2(a.y, b.y), dev::f2(a.x, b.x));
  phi.x = phi.x < 0.0f ? phi.x + 6.28318530717958647692f : phi.x;
  phi.y = phi.y < 0.0f ? phi.y + 6.28318530717958647692f : phi.y;
  theta = atan2_fit2(sqrt2(dev::f2(fmaf(a.x, a.x, a.y * a.y), fmaf(b.x, b.x, b.y * b.y))), dev::f2(a.z, b.z));
}

constexpr int kSphRows = 4;  // rows per thread of the angle-image kernel

__global__ void __launch_bounds__(kThreads)
    spherical_kernel(const float4* __restrict__ n, const uint8_t* __restrict__ valid, int H, int W,
                     long long pitch, float* __restrict__ phi, float* __restrict__ theta) {
  NRM_DEBUG_ENTRY(nullptr);
  const int x = blockIdx.x * kThreads + threadIdx.x;
  if (x >= W) return;
  // Each thread takes kSphRows rows of its column per step and issues all
  // their loads (mask byte and normal, independent of the mask) before the
  // first angle, so that several memory latencies overlap; a masked pixel's
  // stored normal is (0, 0, 0, 0).
  for (int y0 = blockIdx.y * kSphRows; y0 < H; y0 += gridDim.y * kSphRows) {
    uint8_t v[kSphRows];
    float4 nn[kSphRows];
#pragma unroll
    for (int r = 0; r < kSphRows; ++r) {
      v[r] = 0;
      nn[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (y0 + r < H) {
        const long long o = (long long)(y0 + r) * pitch + x;
        v[r] = __ldg(valid + o);
        nn[r] = __ldg(n + o);
      }
    }
#pragma unroll
    for (int r = 0; r < kSphRows; ++r) {
      if (y0 + r >= H) break;
      const long long o = (long long)(y0 + r) * pitch + x;
      float p = 0.0f, t = 0.0f;
      if (v[r]) angles(nn[r], p, t);
      if (NRM_GOK(phi + o, phi, dev::dbg_span(H, W, pitch, 4))) __stcs(phi + o, p);
      if (NRM_GOK(theta + o, theta, dev::dbg_span(H, W, pitch, 4))) __stcs(theta + o, t);
    }
  }
}

__device__ __forceinline__ double warp_sum(double v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  return v;
}

// Sums three values over the block in a fixed order; thread 0 gets the totals.
__device__ __forceinline__ void block_sum3(double& a, double& b, double& c) {
  __shared__ double s[3][kThreads / 32];
  a = warp_sum(a);
  b = warp_sum(b);
  c = warp_sum(c);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    s[0][warp] = a;
    s[1][warp] = b;
    s[2][warp] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    a = b = c = 0.0;
    for (int w = 0; w < kThreads / 32; ++w) {
      a += s[0][w];
      b += s[1][w];
      c += s[2][w];
    }
  }
}

// MSE kernel. A warp takes pieces of kMsePiece pixels of a row (piece w, w + W, ...
// of the W warps of the grid): both maps' normals come by bulk copies into a ring
// of kMseStages stages of the warp's own, so that the copies of the next pieces
// are under way while it evaluates four arctangents a pixel (paired: the estimate
// and the reference in one instruction), and the mask bytes of the next piece are
// loaded a piece ahead. Three CTAs fill an SM; the grid is one wave, so no SM
// waits for a last partial one. The pieces are taken from the maps' end: what a
// call before this one read last (the angle images of the same map) is still in
// L2 (both calls on 4096 x 3072: 127.5 us; from the maps' start 9 us more).
//
// Bound by issue, HBM (34 B/px) close behind. 4096 x 3072: 77.4 us (81 % of the
// measured copy); before, with a step's loads issued together from global memory,
// 2048 blocks of rows (3.4 waves), sqrtf and a second kernel for the sums, 84.6 us and
// 29 us for any small map (now 12). Two CTAs of 3 stages 3 us more, four pixels
// unrolled 5, sqrtf 17.
constexpr int kMsePiece = 128, kMseStages = 2, kMseWarps = kThreads / 32;
constexpr unsigned kMseStageBytes = 2 * kMsePiece * 16;
constexpr unsigned kMseSmem = kMseWarps * kMseStages * (kMseStageBytes + 8);

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

__global__ void __launch_bounds__(kThreads, 3)
    mse_kernel(const float4* __restrict__ na, const uint8_t* __restrict__ va, const float4* __restrict__ nb,
               const uint8_t* __restrict__ vb, int H, int W, long long pitch, double* __restrict__ partials,
               unsigned* __restrict__ ticket, double* __restrict__ out, int* status, unsigned long long timeout_ns) {
  extern __shared__ __align__(128) unsigned char smem[];
  NRM_DEBUG_ENTRY(status);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* ring = smem + warp * kMseStages * kMseStageBytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + kMseWarps * kMseStages * kMseStageBytes) + warp * kMseStages;
  if (lane == 0) {
    for (int s = 0; s < kMseStages; ++s) dev::mbar_init(dev::smem_u32(&full[s]), 1);
    dev::fence_barrier_init();
  }
  __syncwarp();
  const long long per_row = (W + kMsePiece - 1) / kMsePiece;
  const long long total = per_row * H;
  const long long first = (long long)blockIdx.x * kMseWarps + warp, step = (long long)gridDim.x * kMseWarps;
  const long long mine = first < total ? (total - 1 - first) / step + 1 : 0;
  // Offset of piece i of this warp and its pixels.
  auto piece = [&](long long i, int& n) {
    const long long u = total - 1 - (first + i * step);
    const long long y = u / per_row;
    const int x = (int)(u - y * per_row) * kMsePiece;
    n = min(kMsePiece, W - x);
    return y * pitch + x;
  };
  auto issue = [&](long long i, int s) {
    int n;
    const long long o = piece(i, n);
    const uint32_t bar = dev::smem_u32(&full[s]), dst = dev::smem_u32(ring + s * kMseStageBytes);
    dev::mbar_arrive_expect_tx(bar, 32u * (uint32_t)n);
    bulk_load(dst, na + o, 16u * (uint32_t)n, bar);
    bulk_load(dst + kMsePiece * 16, nb + o, 16u * (uint32_t)n, bar);
  };
  uint8_t ma[4], mb[4];
  auto load_masks = [&](long long i) {
    int n = 0;
    const long long o = i < mine ? piece(i, n) : 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int x = lane + 32 * k;
      ma[k] = mb[k] = 0;
      if (x < n) {
        ma[k] = __ldg(va + o + x);
        mb[k] = __ldg(vb + o + x);
      }
    }
  };
  if (lane == 0)
    for (int s = 0; s < kMseStages && s < mine; ++s) issue(s, s);
  load_masks(0);
  double dst = 0.0, dsp = 0.0;
  float st = 0.0f, sp = 0.0f;
  int cnt = 0, s = 0;
  uint32_t parity = 0;
  for (long long i = 0; i < mine; ++i) {
    if (!__all_sync(0xffffffffu, dev::mbar_wait_bounded(dev::smem_u32(&full[s]), parity, timeout_ns))) {
      if (lane == 0) {
        dev::record_error(status, NRM_ERR_TIMEOUT);
        // Let the copies in flight land before the block can exit.
        for (int k = 0; k < kMseStages && i + k < mine; ++k)
          dev::mbar_wait_bounded(dev::smem_u32(&full[(s + k) % kMseStages]), parity ^ (s + k >= kMseStages), timeout_ns);
      }
      break;
    }
    unsigned on = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) on |= ma[k] && mb[k] ? 1u << k : 0u;
    load_masks(i + 1);
    const float4* a = reinterpret_cast<const float4*>(ring + s * kMseStageBytes) + lane;
#pragma unroll 2
    for (int k = 0; k < 4; ++k) {
      float2 phi, theta;
      angles2(NRM_LDS(float4, a + 32 * k), NRM_LDS(float4, a + kMsePiece + 32 * k), phi, theta);
      const bool v = (on >> k) & 1;  // (beyond a piece's end the stage holds anything)
      const float dt = v ? theta.x - theta.y : 0.0f, dp = v ? phi.x - phi.y : 0.0f;
      st = fmaf(dt, dt, st);
      sp = fmaf(dp, dp, sp);
    }
    cnt += __popc(on);
    __syncwarp();
    if (lane == 0 && i + kMseStages < mine) issue(i + kMseStages, s);
    if ((i & 7) == 7) {
      dst += st;
      dsp += sp;
      st = sp = 0.0f;
    }
    if (++s == kMseStages) {
      s = 0;
      parity ^= 1;
    }
  }
  dst += st;
  dsp += sp;
  double dcnt = cnt;
  block_sum3(dst, dsp, dcnt);
  __shared__ bool last;
  if (threadIdx.x == 0) {
    if (NRM_IOK(3 * (long long)blockIdx.x + 2, 3LL * kMseBlocks)) {
      partials[3 * blockIdx.x + 0] = dst;
      partials[3 * blockIdx.x + 1] = dsp;
      partials[3 * blockIdx.x + 2] = dcnt;
    }
    __threadfence();
    // Counts up to the grid and wraps to 0 for the next call.
    last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double et = 0.0, ep = 0.0, ec = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x && NRM_IOK(3LL * i + 2, 3LL * kMseBlocks); i += kThreads) {
    et += __ldcg(partials + 3 * i + 0);
    ep += __ldcg(partials + 3 * i + 1);
    ec += __ldcg(partials + 3 * i + 2);
  }
  block_sum3(et, ep, ec);
  if (threadIdx.x == 0) {
    out[0] = ec > 0.0 ? et / ec : 0.0;
    out[1] = ec > 0.0 ? ep / ec : 0.0;
    out[2] = ec;
  }
}

}  // namespace

cudaError_t launch_spherical(const float* normals, const uint8_t* valid, int H, int W, long long pitch, float* phi,
                             float* theta, cudaStream_t stream) {
  const int row_steps = (H + kSphRows - 1) / kSphRows;
  dim3 grid((W + kThreads - 1) / kThreads, row_steps < 65535 ? row_steps : 65535);
  const float4* n4 = reinterpret_cast<const float4*>(normals);
  void* args[7] = {&n4, &valid, &H, &W, &pitch, &phi, &theta};
  return cudaLaunchKernel((const void*)spherical_kernel, grid, dim3(kThreads), args, 0, stream);
}

cudaError_t launch_angle_mse(const float* na, const uint8_t* va, const float* nb, const uint8_t* vb, int H, int W,
                             long long pitch, double* partials, unsigned* ticket, double* out, int* status,
                             unsigned long long timeout_ns, cudaStream_t stream) {
  static std::atomic<bool> granted[64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  if (!granted[dev].load()) {
    e = cudaFuncSetAttribute((const void*)mse_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMseSmem);
    if (e != cudaSuccess) return e;
    granted[dev].store(true);
  }
  const float4* a4 = reinterpret_cast<const float4*>(na);
  const float4* b4 = reinterpret_cast<const float4*>(nb);
  void* args[12] = {&a4, &va, &b4, &vb, &H, &W, &pitch, &partials, &ticket, &out, &status, &timeout_ns};
  return cudaLaunchKernel((const void*)mse_kernel, dim3(kMseBlocks), dim3(kThreads), args, kMseSmem, stream);
}

}  // namespace nrm
