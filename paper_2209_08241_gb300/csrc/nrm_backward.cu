// Adjoint of the forward normal map with respect to float32 depth, mask held
// fixed (arXiv 2209.08241: derivatives of Eq. 4-6 and of the normalisation).
//
// For a valid pixel p with unit normal n_hat = s n / ||n|| (s = +-1) and upstream
// gradient g_p = dL/d(n_hat_p):
//   h_p = s (g_p - (g_p . n_hat) n_hat) / ||n||            (d n_hat / d n)^T g_p
// and, with e_x = h_x - u1 h_z, e_y = h_y - v1 h_z (the n_z row of Eq. 6 folded in),
// the four depth weights w_k(p) = h_p . dn/dd_k are
//   w2 = -e_x a S35 - e_y b D35 + h_z c S35
//   w4 = +e_x a S35 - e_y b D35 + h_z c S35
//   w3 = -e_x a D24 - e_y b S24 + h_z c S24
//   w5 = -e_x a D24 + e_y b S24 + h_z c S24
// (a, b, c the Eq. 4-6 constants). dn/dd1 = 0. Each depth pixel q then gathers
//   dL/dd_q = w2(q - alpha x) + w4(q + alpha x) + w3(q - alpha y) + w5(q + alpha y),
// a deterministic gather with no atomics.
//
// One CTA per output tile. Three TMA loads on one mbarrier stage the tile's
// inputs in shared memory: the depth halo, the upstream gradient of the
// extended region (a 2-D box of 8-byte elements, two per pixel, i.e. float4 per
// pixel) and the mask of the same region (bwd_shape, nrm_internal.h). Frames
// whose buffers cannot be TMA-mapped use plain loads into the same shared-memory
// layout. bwd_kernel covers one frame (grid = its tiles); bwd_batched_kernel
// covers a batch (grid = max tiles of a frame x frames).
//
// Two forms. The walk (bwd_tile, alpha = 2..4): a warp owns kRows rows of a 64 x 32
// extended region, two columns (x, x + 32) per lane as the pairs of the paired FP32
// instructions, and keeps the weights in registers: the horizontal sums take w2 and w4
// from other lanes by shuffles, the vertical ones w3 and w5 from the lane's own
// registers or, across bands, from a row exchange in shared memory. The gather
// (bwd_tile_gather, any alpha) stores the four weights of each pixel in shared memory
// and gathers them: at 4096 x 3072 and alpha 1 36 shared-memory wavefronts and 127 warp
// instructions per 32 pixels, against 20 and 102 of the walk at alpha 2.
// alpha 2: 4096 x 3072 walk 60.1 us (77 % of the measured copy), gather 68.1; loss
// step of 8 x 1920x1080 201 against 205 us, of 32 x 640x480, which the walk's 60 x 28
// tiles overhang by 8 %, 101 against 99.7: hence the rule on extended pixels
// (BwdChoice). alpha 3 and 4, 32 x 640x480 and 8 x 1080p: 116 / 205 and 124 / 220
// against 125 / 223 and 126 / 226; alpha 1, where the gather has the smallest halo,
// 114 against 112. (Walk with 3 CTAs per SM in place of 4: 69.1 us; 9, 10 or 12
// warps: 66.9, 64.4, 75.7.)
#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <utility>
#include <vector>

#include "nrm_device.cuh"

namespace nrm {

using namespace dev;

namespace {

constexpr int NT = kBwdThreads;
constexpr int NW = NT / 32;
constexpr int MW = kBwdMaskBoxW;   // mask tile pitch (bytes)
constexpr int kMinCtas = 4;        // CTAs per SM (as shared memory allows)
constexpr int kRows = 4;           // rows of the extended region per warp (bwd_tile)

__host__ __device__ constexpr unsigned round128(unsigned b) { return (b + 127) / 128 * 128; }
__host__ __device__ constexpr unsigned depth_tile_bytes(BwdShape s) {
  return round128((unsigned)(s.dep_w * s.dep_h * 4));
}
__host__ __device__ constexpr unsigned weight_tile_bytes(BwdShape s) {
  return round128((unsigned)(s.ex_w * s.ex_h * 16));
}
__host__ __device__ constexpr unsigned mask_tile_bytes(BwdShape s) { return round128((unsigned)(MW * s.ex_h)); }
// Ray coordinates: per row (-v1, -v1, v1, v1) (bwd_tile), or u1 per column and v1
// per row (bwd_tile_gather).
__host__ __device__ constexpr unsigned coord_table_bytes(BwdShape s) {
  return round128((unsigned)(s.ex_h * 16 + s.ex_w * 4));
}

// Stages the tile's inputs; false if the bounded wait for the copies ran out
// (thread 0 has then recorded NRM_ERR_TIMEOUT). All threads; ends with a barrier.
__device__ __forceinline__ bool stage_inputs(const FrameDesc& fd, const BwdShape& sh, int alpha, const void* tmap_d,
                                             const void* tmap_g, const void* tmap_m, int gx0, int gy0, const Globals& g,
                                             float* dep, float4* gw, uint8_t* msk, uint64_t* bar) {
  const int xd = gx0 - sh.dep_x, yd = gy0 - 2 * alpha, xe = gx0 - sh.ex_x, ye = gy0 - alpha, xm = xe & ~15;
  if (fd.use_tma) {
    const uint32_t b = smem_u32(bar);
    if (threadIdx.x == 0) {
      mbar_init(b, 1);
      fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      mbar_arrive_expect_tx(b, (uint32_t)(sh.dep_w * sh.dep_h * 4 + sh.ex_w * sh.ex_h * 16 + MW * sh.ex_h));
      tma_load_2d(smem_u32(dep), tmap_d, xd, yd, b);
      tma_load_2d(smem_u32(gw), tmap_g, 2 * xe, ye, b);  // x in 8-byte units: even
      tma_load_2d(smem_u32(msk), tmap_m, xm, ye, b);
    }
    const bool ok = mbar_wait_warp(b, 0, g.timeout_ns);
    if (__syncthreads_or(!ok)) {
      if (threadIdx.x == 0) {
        record_error(g.status, NRM_ERR_TIMEOUT);
        mbar_wait_bounded(b, 0, g.timeout_ns);
      }
      return false;
    }
    return true;
  }
  load_tile_plain(dep, sh.dep_w, sh.dep_h, fd, xd, yd);
  const float4* gn = reinterpret_cast<const float4*>(fd.normals);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // (In registers: read from the descriptor in the loop, 8 x 641x481 at alpha 1 takes
  // 36.9 us instead of 33.1, at alpha 5 55.6 instead of 50.2.)
  const int W = fd.W, H = fd.H, w = sh.ex_w, h = sh.ex_h;
  for (int ey = warp; ey < h; ey += NW) {
    const int py = ye + ey;
    for (int ex = lane; ex < w; ex += 32) {
      const int px = xe + ex;
      const bool in = px >= 0 && py >= 0 && px < W && py < H;
      const long long o = (long long)py * fd.out_pitch + px;
      NRM_STS(gw + ey * w + ex, in ? __ldg(gn + o) : make_float4(0.f, 0.f, 0.f, 0.f));
      NRM_STS(msk + ey * MW + ex + xe - xm, in ? __ldg(fd.valid + o) : (uint8_t)0);
    }
  }
  __syncthreads();
  return true;
}

// The depth weights w2..w5 of a pixel pair (Eq. 4-6 differentiated; the file
// comment) from its stencil and upstream gradient, each operation that of
// bwd_tile_gather. mx = -n_x and my = -n_y are formed, with -1/||n|| beside 1/||n||,
// since the paired instructions take no negated operands.
struct PairWeights {
  float2 w2, w3, w4, w5;
};
__device__ __forceinline__ PairWeights pair_weights(float2 d2, float2 d3, float2 d4, float2 d5, float2 gx, float2 gy,
                                                    float2 gz, float2 KA, float2 KB, float2 KC, float2 u1, float2 nu1,
                                                    float2 v1, float2 nv1, float2 sign) {
  const float2 M1 = f2(-1.0f, -1.0f);
  const float2 S24 = __fadd2_rn(d2, d4), D24 = __ffma2_rn(M1, d4, d2);
  const float2 S35 = __fadd2_rn(d3, d5), D35 = __ffma2_rn(M1, d5, d3);
  const float2 A35 = __fmul2_rn(KA, S35), B35 = __fmul2_rn(KB, D35), C35 = __fmul2_rn(KC, S35);
  const float2 A24 = __fmul2_rn(KA, D24), B24 = __fmul2_rn(KB, S24), C24 = __fmul2_rn(KC, S24);
  const float2 mx = __fmul2_rn(A35, D24), my = __fmul2_rn(B24, D35), P = __fmul2_rn(C24, S35);
  const float2 nz = __ffma2_rn(u1, mx, __ffma2_rn(v1, my, P));
  const float2 q = __ffma2_rn(mx, mx, __ffma2_rn(my, my, __fmul2_rn(nz, nz)));
  const float2 inv = f2(rsqrt_ftz(fmaxf(q.x, 1.17549435e-38f)), rsqrt_ftz(fmaxf(q.y, 1.17549435e-38f)));
  const float2 ninv = __fmul2_rn(M1, inv);
  const float2 hx0 = __fmul2_rn(mx, ninv), hy0 = __fmul2_rn(my, ninv), hz0 = __fmul2_rn(nz, inv);
  const float2 ngd = __fmul2_rn(M1, __ffma2_rn(gx, hx0, __ffma2_rn(gy, hy0, __fmul2_rn(gz, hz0))));
  const float2 si = __fmul2_rn(sign, inv);
  const float2 hx = __fmul2_rn(__ffma2_rn(ngd, hx0, gx), si);
  const float2 hy = __fmul2_rn(__ffma2_rn(ngd, hy0, gy), si);
  const float2 hz = __fmul2_rn(__ffma2_rn(ngd, hz0, gz), si);
  const float2 ex = __ffma2_rn(nu1, hz, hx), ey = __ffma2_rn(nv1, hz, hy);
  const float2 nex = __fmul2_rn(M1, ex), ney = __fmul2_rn(M1, ey);
  const float2 c35 = __ffma2_rn(hz, C35, __fmul2_rn(ney, B35));
  const float2 c24 = __ffma2_rn(hz, C24, __fmul2_rn(nex, A24));
  return {__ffma2_rn(nex, A35, c35), __ffma2_rn(ney, B24, c24), __ffma2_rn(ex, A35, c35), __ffma2_rn(ey, B24, c24)};
}

// One output tile (gx0, gy0) of frame fd for a pixel distance 2..4. scale: the
// upstream gradient is scale[frame] times the staged float4.
template <int ALPHA>
__device__ __forceinline__ void bwd_tile(const FrameDesc& fd, const void* tmap_d, const void* tmap_g,
                                         const void* tmap_m, int gx0, int gy0, const Globals& g,
                                         unsigned char* smem, const float* __restrict__ scale, int frame) {
  constexpr BwdShape SH = bwd_shape(ALPHA, true);
  static_assert(SH.ex_w == 64 && SH.ex_h == kRows * NW && ALPHA <= kRows && ALPHA <= SH.ex_x, "one band per warp");
  float* dep = reinterpret_cast<float*>(smem);
  float4* gw = reinterpret_cast<float4*>(smem + depth_tile_bytes(SH));
  uint8_t* msk = smem + depth_tile_bytes(SH) + weight_tile_bytes(SH);
  float4* vtab = reinterpret_cast<float4*>(msk + mask_tile_bytes(SH));
  uint64_t* bar = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(vtab) + coord_table_bytes(SH));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < SH.ex_h) {
    const float v1 = ((float)(gy0 - ALPHA + (int)threadIdx.x) - fd.cy) * fd.inv_fy;
    NRM_STS(vtab + threadIdx.x, make_float4(-v1, -v1, v1, v1));
  }
  if (!stage_inputs(fd, SH, ALPHA, tmap_d, tmap_g, tmap_m, gx0, gy0, g, dep, gw, msk, bar)) return;

  const int xe = gx0 - SH.ex_x;
  const float ua = ((float)(xe + lane) - fd.cx) * fd.inv_fx, ub = ((float)(xe + lane + 32) - fd.cx) * fd.inv_fx;
  const float2 u1 = f2(ua, ub), nu1 = f2(-ua, -ub);
  const float2 KA = f2(fd.a, fd.a), KB = f2(fd.b, fd.b), KC = f2(fd.c, fd.c), sign = f2(g.sign, g.sign);
  const float sc = scale ? __ldg(scale + frame) : 1.0f;
  const int row0 = warp * kRows;  // the band's first row in the extended region
  // Centre column depths of the band's rows and ALPHA rows above and below.
  const float* pc = dep + row0 * SH.dep_w + SH.dep_x - SH.ex_x + lane;
  float2 R[kRows + 2 * ALPHA];
#pragma unroll
  for (int i = 0; i < 2 * ALPHA; ++i)
    R[i] = f2(NRM_LDS(float, pc + i * SH.dep_w), NRM_LDS(float, pc + i * SH.dep_w + 32));
  const uint8_t* pm = msk + row0 * MW + (xe & 15) + lane;
  float2 t[kRows], w3[kRows], w5[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const float* p = pc + (r + ALPHA) * SH.dep_w;
    R[r + 2 * ALPHA] = f2(NRM_LDS(float, p + ALPHA * SH.dep_w), NRM_LDS(float, p + ALPHA * SH.dep_w + 32));
    const float2 d2 = f2(NRM_LDS(float, p + ALPHA), NRM_LDS(float, p + ALPHA + 32));
    const float2 d4 = f2(NRM_LDS(float, p - ALPHA), NRM_LDS(float, p - ALPHA + 32));
    const float4* pg = gw + (row0 + r) * 64 + lane;
    const float4 ga = NRM_LDS(float4, pg), gb = NRM_LDS(float4, pg + 32);
    float2 gx = f2(ga.x, gb.x), gy = f2(ga.y, gb.y), gz = f2(ga.z, gb.z);
    if (scale) {
      const float2 s2 = f2(sc, sc);
      gx = __fmul2_rn(gx, s2);
      gy = __fmul2_rn(gy, s2);
      gz = __fmul2_rn(gz, s2);
    }
    const float4 vv = NRM_LDS(float4, vtab + row0 + r);
    PairWeights w = pair_weights(d2, R[r + 2 * ALPHA], d4, R[r], gx, gy, gz, KA, KB, KC, u1, nu1, f2(vv.z, vv.w),
                                 f2(vv.x, vv.y), sign);
    // Only valid pixels have weights (elsewhere depth and gradient can be anything).
    const bool ka = NRM_LDS(uint8_t, pm + r * MW) != 0, kb = NRM_LDS(uint8_t, pm + r * MW + 32) != 0;
    const float w2a = ka ? w.w2.x : 0.0f, w2b = kb ? w.w2.y : 0.0f;
    const float w4a = ka ? w.w4.x : 0.0f, w4b = kb ? w.w4.y : 0.0f;
    w3[r] = f2(ka ? w.w3.x : 0.0f, kb ? w.w3.y : 0.0f);
    w5[r] = f2(ka ? w.w5.x : 0.0f, kb ? w.w5.y : 0.0f);
    // w2 from ALPHA columns to the left, w4 from ALPHA to the right (the columns
    // whose source lies outside the extended region are not in the tile).
    const float la = __shfl_sync(0xffffffffu, w2a, lane - ALPHA), lb = __shfl_sync(0xffffffffu, w2b, lane - ALPHA);
    const float ra = __shfl_sync(0xffffffffu, w4a, lane + ALPHA), rb = __shfl_sync(0xffffffffu, w4b, lane + ALPHA);
    t[r] = __fadd2_rn(f2(la, lane < ALPHA ? la : lb), f2(lane >= 32 - ALPHA ? rb : ra, rb));
  }
  // Rows that a neighbouring band needs, in this warp's own part of the gradient
  // tile (which only it has read): w5 of the first ALPHA rows, then w3 of the last.
  __syncwarp();
  float* xch = reinterpret_cast<float*>(gw + row0 * 64);
#pragma unroll
  for (int i = 0; i < ALPHA; ++i) {
    NRM_STS(xch + i * 64 + lane, w5[i].x);
    NRM_STS(xch + i * 64 + lane + 32, w5[i].y);
    NRM_STS(xch + (ALPHA + i) * 64 + lane, w3[kRows - ALPHA + i].x);
    NRM_STS(xch + (ALPHA + i) * 64 + lane + 32, w3[kRows - ALPHA + i].y);
  }
  __syncthreads();
  const float* up = xch - kRows * 64 * 4 + ALPHA * 64 + lane;  // w3 of the band above
  const float* down = xch + kRows * 64 * 4 + lane;             // w5 of the band below
  const int xa = xe + lane, xb = xa + 32;
  const bool oka = lane >= SH.ex_x && xa < fd.W, okb = lane < 32 - SH.ex_x && xb < fd.W;
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int er = row0 + r;
    const int gy = gy0 - ALPHA + er;
    if (er < ALPHA || er >= SH.ex_h - ALPHA || gy >= fd.H) continue;
    const float2 a = r >= ALPHA ? w3[r >= ALPHA ? r - ALPHA : 0]
                                : f2(NRM_LDS(float, up + r * 64), NRM_LDS(float, up + r * 64 + 32));
    const float* pd = down + (r + ALPHA - kRows) * 64;
    const float2 b = r + ALPHA < kRows ? w5[r + ALPHA < kRows ? r + ALPHA : 0]
                                       : f2(NRM_LDS(float, pd), NRM_LDS(float, pd + 32));
    const float2 v = __fadd2_rn(__fadd2_rn(t[r], a), b);
    float* q = fd.grad_depth + (long long)gy * fd.depth_pitch + xa;
    [[maybe_unused]] const long long len = dbg_span(fd.H, fd.W, fd.depth_pitch, 4);
    if (oka && NRM_GOK(q, fd.grad_depth, len)) *q = v.x;
    if (okb && NRM_GOK(q + 32, fd.grad_depth, len)) q[32] = v.y;
  }
}

// One output tile (gx0, gy0) of frame fd. tmap_d/tmap_g/tmap_m: its depth,
// gradient and mask tensor maps (param or global memory; used only when
// fd.use_tma), for the pixel distance ALPHA or, if that is 0, g.alpha. If the bounded wait for the
// copies runs out, the tile records NRM_ERR_TIMEOUT in the status word and writes
// nothing.
template <int ALPHA>
__device__ __forceinline__ void bwd_tile_gather(const FrameDesc& fd, const void* tmap_d, const void* tmap_g,
                                         const void* tmap_m, int gx0, int gy0, const Globals& g,
                                         unsigned char* smem, const float* __restrict__ scale, int frame) {
  // Upstream gradient = scale[frame] x the staged float4 when scale is given
  // (the fused loss entry: the staged values are then target normals).
  const float sc = scale ? __ldg(scale + frame) : 1.0f;
  const int alpha = ALPHA > 0 ? ALPHA : g.alpha;
  const BwdShape sh = bwd_shape(alpha, false);
  const int bw = sh.dep_w;     // depth tile pitch
  const int ex_w = sh.ex_w;    // extended region (gradient / weight / mask)
  const int ex_h = sh.ex_h;
  const int TX = sh.tx, TY = sh.ty;
  float* dep = reinterpret_cast<float*>(smem);
  float4* gw = reinterpret_cast<float4*>(smem + depth_tile_bytes(sh));
  uint8_t* msk = smem + depth_tile_bytes(sh) + weight_tile_bytes(sh);
  float* ucol = reinterpret_cast<float*>(msk + mask_tile_bytes(sh));  // u1 of extended column ex
  float* vrow = ucol + ex_w;                                          // v1 of extended row ey
  uint64_t* bar = reinterpret_cast<uint64_t*>(reinterpret_cast<unsigned char*>(ucol) + coord_table_bytes(sh));
  const int H = fd.H, W = fd.W;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // The ray coordinates of the extended region, formed before the copies are
  // waited for (the barrier that follows them publishes these too).
  for (int t = threadIdx.x; t < ex_w + ex_h; t += NT) {
    if (t < ex_w)
      NRM_STS(ucol + t, ((float)(gx0 - alpha + t) - fd.cx) * fd.inv_fx);
    else
      NRM_STS(vrow + t - ex_w, ((float)(gy0 - alpha + t - ex_w) - fd.cy) * fd.inv_fy);
  }
  if (!stage_inputs(fd, sh, alpha, tmap_d, tmap_g, tmap_m, gx0, gy0, g, dep, gw, msk, bar)) return;

  // Phase 1: the weights of every pixel p of the extended tile, in place of
  // its staged gradient. Threads walk the ex_w x ex_h elements in row-major
  // order with stride NT, advancing (ey, ex) by increments (no division).
  // A pixel the forward marked valid has a positive finite five-point stencil
  // (that is what made it valid), so only the mask is consulted here.
  // With A35 = a S35, B35 = b D35, C35 = c S35 and A24 = a D24, B24 = b S24,
  // C24 = c S24, Eq. 4-6 read n_x = -A35 D24, n_y = -B24 D35, P = C24 S35, and
  // the weights (e_x = h_x - u1 h_z, e_y = h_y - v1 h_z) are
  //   w2 = -e_x A35 - e_y B35 + h_z C35,  w4 = e_x A35 - e_y B35 + h_z C35,
  //   w3 = -e_x A24 - e_y B24 + h_z C24,  w5 = -e_x A24 + e_y B24 + h_z C24.
  const float ka = fd.a, kb = fd.b, kc = fd.c;
  const int n_ext = ex_w * ex_h;
  const int step_rows = NT / ex_w, step_cols = NT - step_rows * ex_w;
  int ey = threadIdx.x / ex_w;
  int ex = threadIdx.x - ey * ex_w;
  const float* dep_c = dep + alpha * bw + sh.dep_x - alpha;  // depth-tile position of (ey, ex) = (0, 0)
  const uint8_t* msk_c = msk + ((gx0 - alpha) & 15);
  for (int i = threadIdx.x; i < n_ext; i += NT) {
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (NRM_LDS(uint8_t, msk_c + ey * MW + ex)) {
      const float* pc = dep_c + ey * bw + ex;
      const float d2 = NRM_LDS(float, pc + alpha), d4 = NRM_LDS(float, pc - alpha);
      const float d3 = NRM_LDS(float, pc + alpha * bw), d5 = NRM_LDS(float, pc - alpha * bw);
      const float S24 = d2 + d4, D24 = d2 - d4, S35 = d3 + d5, D35 = d3 - d5;
      const float u1 = NRM_LDS(float, ucol + ex), v1 = NRM_LDS(float, vrow + ey);
      const float A35 = ka * S35, B35 = kb * D35, C35 = kc * S35;
      const float A24 = ka * D24, B24 = kb * S24, C24 = kc * S24;
      const float nx = -A35 * D24, ny = -B24 * D35, P = C24 * S35;
      const float nz = fmaf(-u1, nx, fmaf(-v1, ny, P));
      const float q = fmaf(nx, nx, fmaf(ny, ny, nz * nz));
      const float inv = rsqrt_ftz(fmaxf(q, 1.17549435e-38f));
      const float hx0 = nx * inv, hy0 = ny * inv, hz0 = nz * inv;
      float4 gv = NRM_LDS(float4, gw + i);
      if (scale) {
        gv.x *= sc;
        gv.y *= sc;
        gv.z *= sc;
      }
      const float gd = fmaf(gv.x, hx0, fmaf(gv.y, hy0, gv.z * hz0));
      const float si = g.sign * inv;
      const float hx = fmaf(-gd, hx0, gv.x) * si;
      const float hy = fmaf(-gd, hy0, gv.y) * si;
      const float hz = fmaf(-gd, hz0, gv.z) * si;
      const float e_x = fmaf(-u1, hz, hx);
      const float e_y = fmaf(-v1, hz, hy);
      const float c35 = fmaf(hz, C35, -e_y * B35);
      const float c24 = fmaf(hz, C24, -e_x * A24);
      w.x = fmaf(-e_x, A35, c35);  // w2
      w.y = fmaf(-e_y, B24, c24);  // w3
      w.z = fmaf(e_x, A35, c35);   // w4
      w.w = fmaf(e_y, B24, c24);   // w5
    }
    NRM_STS(gw + i, w);
    ey += step_rows;
    ex += step_cols;
    if (ex >= ex_w) {
      ex -= ex_w;
      ++ey;
    }
  }
  __syncthreads();
  // Phase 2: gather.
  float* __restrict__ grad = fd.grad_depth;
  for (int ly = warp; ly < TY; ly += NW) {
    const int qy = gy0 + ly;
    if (qy >= H) break;
    for (int lx = lane; lx < TX; lx += 32) {
      const int qx = gx0 + lx;
      if (qx >= W) break;
      const int c = (ly + alpha) * ex_w + (lx + alpha);
      const float v = NRM_LDS(float4, gw + c - alpha).x + NRM_LDS(float4, gw + c + alpha).z +
                      NRM_LDS(float4, gw + c - alpha * ex_w).y + NRM_LDS(float4, gw + c + alpha * ex_w).w;
      float* q = grad + (long long)qy * fd.depth_pitch + qx;
      if (NRM_GOK(q, grad, dbg_span(H, W, fd.depth_pitch, 4))) *q = v;
    }
  }
}

template <int ALPHA, bool WALK>
__device__ __forceinline__ void bwd_any_tile(const FrameDesc& fd, const void* tmap_d, const void* tmap_g,
                                             const void* tmap_m, int gx0, int gy0, const Globals& g,
                                             unsigned char* smem, const float* __restrict__ scale, int frame) {
  if constexpr (WALK)
    bwd_tile<ALPHA>(fd, tmap_d, tmap_g, tmap_m, gx0, gy0, g, smem, scale, frame);
  else
    bwd_tile_gather<ALPHA>(fd, tmap_d, tmap_g, tmap_m, gx0, gy0, g, smem, scale, frame);
}

template <int ALPHA, bool WALK>
__global__ void __launch_bounds__(NT, kMinCtas)
    bwd_kernel(const __grid_constant__ FrameDesc fd, const __grid_constant__ BwdMaps maps, const Globals g,
               const float* scale) {
  extern __shared__ __align__(128) unsigned char smem[];
  NRM_DEBUG_ENTRY(g.status);
  const BwdShape sh = bwd_shape(ALPHA > 0 ? ALPHA : g.alpha, WALK);
  bwd_any_tile<ALPHA, WALK>(fd, &fd.tmap, &maps.grad, &maps.mask, blockIdx.x * sh.tx, blockIdx.y * sh.ty, g, smem,
                            scale, 0);
}

// Grid (max tiles of a frame, frames): block (x, f) is tile x of frame f; frames
// with fewer tiles leave their extra blocks idle.
template <int ALPHA, bool WALK>
__global__ void __launch_bounds__(NT, kMinCtas)
    bwd_batched_kernel(const BwdBatchArgs args, const Globals g, const float* scale) {
  extern __shared__ __align__(128) unsigned char smem[];
  NRM_DEBUG_ENTRY(g.status);
  const int f = (int)blockIdx.y;
  const FrameDesc& fd = args.frames[f];
  const int tiles_x = fd.tiles_x;
  const int local = (int)blockIdx.x;
  const BwdShape sh = bwd_shape(ALPHA > 0 ? ALPHA : g.alpha, WALK);
  if (tiles_x == 0 || local >= tiles_x * ((fd.H + sh.ty - 1) / sh.ty)) return;
  if (threadIdx.x == 0 && fd.use_tma) {
    fence_tensormap_acquire(&fd.tmap);
    fence_tensormap_acquire(&args.maps[f].grad);
    fence_tensormap_acquire(&args.maps[f].mask);
  }
  const int ty = local / tiles_x;
  const int tx = local - ty * tiles_x;
  bwd_any_tile<ALPHA, WALK>(fd, &fd.tmap, &args.maps[f].grad, &args.maps[f].mask, tx * sh.tx, ty * sh.ty, g, smem,
                            scale, f);
}

// A batch of at most kBwdParamMaxFrames frames with its records and tensor
// maps in kernel-parameter space: no descriptor upload and no tensor-map fence
// (each CTA of the global-memory form fences three maps for its one tile).
struct alignas(128) BwdParamBatch {
  FrameDesc frames[kBwdParamMaxFrames];
  BwdMaps maps[kBwdParamMaxFrames];
};
static_assert(sizeof(BwdParamBatch) <= 32764, "the descriptor block must fit the kernel parameter limit");

// Grid (max tiles of a frame, frames), as bwd_batched_kernel.
template <int ALPHA, bool WALK>
__global__ void __launch_bounds__(NT, kMinCtas)
    bwd_batched_param_kernel(const __grid_constant__ BwdParamBatch pb, const Globals g, const float* scale) {
  extern __shared__ __align__(128) unsigned char smem[];
  NRM_DEBUG_ENTRY(g.status);
  const int f = (int)blockIdx.y;
  const FrameDesc& fd = pb.frames[f];
  const int tiles_x = fd.tiles_x;
  const int local = (int)blockIdx.x;
  const BwdShape sh = bwd_shape(ALPHA > 0 ? ALPHA : g.alpha, WALK);
  if (tiles_x == 0 || local >= tiles_x * ((fd.H + sh.ty - 1) / sh.ty)) return;
  const int ty = local / tiles_x;
  const int tx = local - ty * tiles_x;
  bwd_any_tile<ALPHA, WALK>(fd, &fd.tmap, &pb.maps[f].grad, &pb.maps[f].mask, tx * sh.tx, ty * sh.ty, g, smem, scale,
                            f);
}

// The kernel of a launch kind for a distance and form: compiled for alpha = 1..4
// (constant offsets and loop steps), generic above.
enum { kOneFrame, kBatch, kBatchParam };
template <int ALPHA, bool WALK>
const void* bwd_kernel_of(int kind) {
  return kind == kOneFrame ? (const void*)bwd_kernel<ALPHA, WALK>
         : kind == kBatch  ? (const void*)bwd_batched_kernel<ALPHA, WALK>
                           : (const void*)bwd_batched_param_kernel<ALPHA, WALK>;
}
const void* bwd_kernel_for(int alpha, bool walk, int kind) {
  if (walk)
    return alpha == 2 ? bwd_kernel_of<2, true>(kind) : alpha == 3 ? bwd_kernel_of<3, true>(kind)
                                                                  : bwd_kernel_of<4, true>(kind);
  return alpha == 1 ? bwd_kernel_of<1, false>(kind) : alpha == 2 ? bwd_kernel_of<2, false>(kind)
                                                                 : bwd_kernel_of<0, false>(kind);
}

// Grants the dynamic shared memory a kernel needs, once per (kernel, device)
// and size.
cudaError_t set_smem(const void* fn, unsigned bytes) {
  static std::map<std::pair<const void*, int>, unsigned> granted;
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);
  int dev = 0;
  cudaGetDevice(&dev);
  auto key = std::make_pair(fn, dev);
  auto it = granted.find(key);
  if (it != granted.end() && it->second >= bytes) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) granted[key] = bytes;
  return e;
}

// The per-frame factor of the cosine loss, scale = -1 / max(N_valid, 1), with
// N_valid the number of nonzero mask bytes of the frame: kCountBlocks blocks
// per frame count 16 bytes per load, of the whole frame where its rows are
// contiguous (at 640x480 every thread's two or three loads are then in flight
// together), else a warp per row, or several warps per row where the rows are fewer
// than the warps (one 1,000,000-pixel row with a gap behind it: 4.3 us, with one warp
// for it 184, one byte per load 92; four rows of 100,000: 4.2, 22.2 and 12.5).
// Bound by latency: the loss step of 32 x 640x480 takes 99.7 us with
// it (one byte per load, a block per row: 112.5). Each block adds its count to the
// frame's counter, and the last block of the frame to finish (the ordering of a
// fence and an atomic ticket) writes the scale and returns both counters to zero
// for the next call. Integer sums: the result does not depend on the order.
constexpr int kCountBlocks = 32;
constexpr int kCountThreads = 256;
constexpr int kCountWarps = kCountBlocks * kCountThreads / 32;
constexpr int kCountSegment = 512;  // a row's parts hold at least about this many bytes: one load per lane

// Nonzero bytes among those of p[0, n) that are worker i's of `workers` (>= 16).
__device__ __forceinline__ unsigned count_nonzero(const uint8_t* __restrict__ p, long long n, int i, int workers) {
  const long long head = min(n, (long long)(-reinterpret_cast<intptr_t>(p) & 15));
  const long long units = (n - head) / 16;
  unsigned c = i < head && __ldg(p + i) != 0 ? 1u : 0u;
  const uint4* q = reinterpret_cast<const uint4*>(p + head);
#pragma unroll 4
  for (long long u = i; u < units; u += workers) {
    const uint4 w = __ldg(q + u);
    const uint32_t v[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int k = 0; k < 4; ++k)  // bit 7 of each byte: the byte is not 0
      c += __popc((((v[k] & 0x7f7f7f7fu) + 0x7f7f7f7fu) | v[k]) & 0x80808080u);
  }
  const long long tail = head + 16 * units + i;
  return c + (tail < n && __ldg(p + tail) != 0 ? 1u : 0u);
}

// The parts that a row is counted in, a warp each: as many as there are warps for,
// of kCountSegment bytes or more. Rows without gaps are counted as one row.
__host__ __device__ inline int count_segments(const LossCountFrame& f) {
  if (f.pitch == f.W || f.H <= 0 || f.H >= kCountWarps) return 1;
  const int fit = kCountWarps / f.H, of = f.W / kCountSegment;
  return fit < of ? fit : of > 1 ? of : 1;
}

struct CountArgs {
  LossCountFrame f[kLossCountMaxFrames];
};

// LONG_ROWS: a batch with frames of fewer rows than warps.
template <bool LONG_ROWS>
__global__ void __launch_bounds__(kCountThreads)
    loss_scale_kernel(const __grid_constant__ CountArgs a, unsigned* __restrict__ counts,
                      unsigned* __restrict__ tickets, float* __restrict__ scale) {
  NRM_DEBUG_ENTRY(nullptr);
  const int f = (int)blockIdx.y;
  const LossCountFrame fr = a.f[f];
  unsigned c = 0;
  if (fr.pitch == fr.W) {
    c = count_nonzero(fr.valid, (long long)fr.H * fr.W, (int)(blockIdx.x * kCountThreads + threadIdx.x),
                      kCountBlocks * kCountThreads);
  } else {
    const int first = blockIdx.x * (kCountThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if constexpr (!LONG_ROWS) {
      for (int y = first; y < fr.H; y += kCountWarps)
        c += count_nonzero(fr.valid + (long long)y * fr.pitch, fr.W, lane, 32);
    } else {
      const int segs = count_segments(fr);
      const long long len = ((long long)fr.W + 16 * segs - 1) / (16 * segs) * 16;  // (whole 16-byte units)
      for (long long u = first; u < (long long)fr.H * segs; u += kCountWarps) {
        const long long y = u / segs, x = (u - y * segs) * len;
        c += count_nonzero(fr.valid + y * fr.pitch + x, max(0LL, min(len, fr.W - x)), lane, 32);
      }
    }
  }
  c = __reduce_add_sync(0xffffffffu, c);
  __shared__ unsigned part[kCountThreads / 32];
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned t = 0;
    for (int w = 0; w < kCountThreads / 32; ++w) t += part[w];
    atomicAdd(counts + f, t);
    __threadfence();
    if (atomicAdd(tickets + f, 1u) == gridDim.x - 1) {
      const unsigned total = atomicExch(counts + f, 0u);
      atomicExch(tickets + f, 0u);
      scale[f] = -1.0f / (float)(total > 0 ? total : 1u);
    }
  }
}

}  // namespace

cudaError_t launch_loss_scale(const LossCountFrame* frames, int n, unsigned* counts, unsigned* tickets, float* scale,
                              cudaStream_t stream) {
  for (int first = 0; first < n; first += kLossCountMaxFrames) {
    const int m = std::min(kLossCountMaxFrames, n - first);
    CountArgs a;
    std::memset(&a, 0, sizeof(a));
    std::memcpy(a.f, frames + first, sizeof(LossCountFrame) * (size_t)m);
    unsigned* c = counts + first;
    unsigned* t = tickets + first;
    float* sc = scale + first;
    void* args[4] = {&a, &c, &t, &sc};
    bool long_rows = false;
    for (int i = 0; i < m; ++i) long_rows = long_rows || count_segments(a.f[i]) > 1;
    const void* fn = long_rows ? (const void*)loss_scale_kernel<true> : (const void*)loss_scale_kernel<false>;
    cudaError_t e = cudaLaunchKernel(fn, dim3(kCountBlocks, m), dim3(kCountThreads), args, 0, stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

unsigned bwd_smem_bytes(int alpha, bool walk) {
  const BwdShape s = bwd_shape(alpha, walk);
  return depth_tile_bytes(s) + weight_tile_bytes(s) + mask_tile_bytes(s) + coord_table_bytes(s) + 16;
}

cudaError_t launch_backward(const FrameDesc& fd, const BwdMaps& maps, const Globals& g, bool walk,
                            cudaStream_t stream, const float* scale) {
  const unsigned smem = bwd_smem_bytes(g.alpha, walk);
  const void* fn = bwd_kernel_for(g.alpha, walk, kOneFrame);
  cudaError_t e = set_smem(fn, smem);
  if (e != cudaSuccess) return e;
  const BwdShape s = bwd_shape(g.alpha, walk);
  dim3 grid((fd.W + s.tx - 1) / s.tx, (fd.H + s.ty - 1) / s.ty);
  FrameDesc d = fd;
  BwdMaps m = maps;
  Globals gg = g;
  const float* sc = scale;
  void* args[4] = {&d, &m, &gg, &sc};
  e = cudaLaunchKernel(fn, grid, dim3(NT), args, smem, stream);
  return e;
}

cudaError_t launch_backward_batched(const BwdBatchArgs& args, int n_frames, int max_tiles, const Globals& g,
                                    bool walk, cudaStream_t stream, const float* scale) {
  const unsigned smem = bwd_smem_bytes(g.alpha, walk);
  const void* fn = bwd_kernel_for(g.alpha, walk, kBatch);
  cudaError_t e = set_smem(fn, smem);
  if (e != cudaSuccess) return e;
  BwdBatchArgs a = args;
  Globals gg = g;
  const float* sc = scale;
  void* kargs[3] = {&a, &gg, &sc};
  e = cudaLaunchKernel(fn, dim3(max_tiles, n_frames), dim3(NT), kargs, smem, stream);
  return e;
}

cudaError_t launch_backward_batched_param(const FrameDesc* frames, const BwdMaps* maps, int n_frames, int max_tiles,
                                          const Globals& g, bool walk, cudaStream_t stream,
                                          const float* scale) {
  if (n_frames < 1 || n_frames > kBwdParamMaxFrames) return cudaErrorInvalidValue;
  const unsigned smem = bwd_smem_bytes(g.alpha, walk);
  const void* fn = bwd_kernel_for(g.alpha, walk, kBatchParam);
  cudaError_t e = set_smem(fn, smem);
  if (e != cudaSuccess) return e;
  std::vector<unsigned char> raw(sizeof(BwdParamBatch) + 128);
  void* aligned = raw.data() + (128 - reinterpret_cast<uintptr_t>(raw.data()) % 128) % 128;
  BwdParamBatch* pb = static_cast<BwdParamBatch*>(aligned);
  std::memset(pb, 0, sizeof(BwdParamBatch));
  std::memcpy(pb->frames, frames, sizeof(FrameDesc) * (size_t)n_frames);
  std::memcpy(pb->maps, maps, sizeof(BwdMaps) * (size_t)n_frames);
  Globals gg = g;
  const float* sc = scale;
  void* kargs[3] = {pb, &gg, &sc};
  return cudaLaunchKernel(fn, dim3(max_tiles, n_frames), dim3(NT), kargs, smem, stream);
}

}  // namespace nrm
