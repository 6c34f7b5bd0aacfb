// Local plane fitting ("plane-PCA"), the ground truth the paper compares
// against (arXiv 2209.08241: Section 1 describes it; Section 4 uses it with 25
// neighbouring points): for each pixel, the unit eigenvector of the scatter
// matrix of the back-projected points of its (2R+1) x (2R+1) window for the
// smallest eigenvalue, oriented away from the camera (n . P > 0).
//
// FP32 with care for cancellation: points are taken relative to the window's
// centre point P0 = z0 (u0, v0, 1) as
//   q = ((z - z0) u + z0 dcol/fx,  (z - z0) v + z0 drow/fy,  z - z0),
// whose terms are all small, so each has a relative error of a few ulp. The
// scatter matrix is then sum q q^T - (sum q)(sum q)^T / n: relative to P0 the
// window's mean is small (it is zero for the in-plane offsets of a symmetric
// window), so the subtraction loses little. The symmetric 3 x 3 eigenproblem is
// solved by cyclic Jacobi rotations until the off-diagonal part is below 1e-7
// of the diagonal (at most 6 sweeps; quadratic convergence makes 3-4 usual).
// The normal direction does not depend on the depth unit, so uint16 depth is
// used in its raw integer units (exact in FP32) without the depth scale.
// A pixel is valid iff every depth of its window is inside the image and
// positive and finite (the decoded tile holds NaN elsewhere, which propagates).
//
// The kernel is bound by FP32 issue (at R = 2 about 300 operations a pixel for the
// window sums and 400 for the rotations), so a thread takes two adjacent pixels
// as the lanes of the paired FP32 instructions, operation for operation those of
// one pixel, and the rotations are free of branches: a pixel that is done rotates by
// zero, which leaves its bits. 1920x1080 float32, R = 2: 49.8 us (one pixel per
// thread with branching rotations: 68.1); ~31 us is the FMA pipe's time for
// these operations. Frames that do not fill the GPU are bound by the chain of one
// thread, which is shorter with one pixel per thread (launch_plane_fit):
// 160x120 at R = 1 / 2 / 3 / 4 3.7 / 3.7 / 4.2 / 4.5 us with one, 4.8 / 5.0 / 5.4 / 6.2 with two;
// 320x240 5.0 / 5.6 / 6.0 / 7.0 and 4.8 / 5.5 / 5.8 / 6.6.
#include <type_traits>

#include "nrm_device.cuh"

namespace nrm {

namespace {

constexpr int PY = 8, PT = 32 * PY;  // rows and threads of a CTA

using dev::f2;
using dev::rsqrt_ftz;

// The values of a thread's N pixels, and the operations on them.
template <int N>
using Px = std::conditional_t<N == 2, float2, float>;
template <int N>
__device__ __forceinline__ Px<N> all(float x) {
  if constexpr (N == 2)
    return f2(x, x);
  else
    return x;
}
__device__ __forceinline__ float2 add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float2 neg(float2 x) { return __fmul2_rn(x, f2(-1.0f, -1.0f)); }
__device__ __forceinline__ float neg(float x) { return -x; }
__device__ __forceinline__ float& px(float2& v, int i) { return i ? v.y : v.x; }
__device__ __forceinline__ float px(const float2& v, int i) { return i ? v.y : v.x; }
__device__ __forceinline__ float& px(float& v, int) { return v; }
__device__ __forceinline__ float px(const float& v, int) { return v; }

// One Jacobi rotation zeroing a[p][q] of the symmetric matrices a of a thread's
// pixels, accumulated into the eigenvector columns of v. A pixel that is done
// (!on) or whose a[p][q] is nothing takes t = 0, which leaves it bit for bit as it
// is. Approximate reciprocal and square root suffice: c and s are formed from t
// so that c^2 + s^2 = 1 to rounding whatever t's last bits, and an error of a few
// ulp in t only leaves an off-diagonal residue of a few ulp of |a_pq|, the size
// of the rounding already in S. (|theta| is capped at 1e18, where theta^2 would
// come near overflow and t is nothing beside 1.)
template <int p, int q, int N>
__device__ __forceinline__ void jacobi_rotate(Px<N> (&a)[3][3], Px<N> (&v)[3][3], const bool (&on)[N]) {
  using V = Px<N>;
  const V apq = a[p][q], one = all<N>(1.0f);
  // t = tan of the rotation angle, the smaller root of t^2 + 2 theta t - 1 = 0.
  const V den = add(apq, apq);
  const V num = fma(all<N>(-1.0f), a[p][p], a[q][q]);
  V r, at, t;
#pragma unroll
  for (int i = 0; i < N; ++i) px(r, i) = dev::rcp_ftz(px(den, i));
  const V theta = mul(num, r);
#pragma unroll
  for (int i = 0; i < N; ++i) px(at, i) = fminf(fabsf(px(theta, i)), 1e18f);
  const V h = fma(at, at, one);
#pragma unroll
  for (int i = 0; i < N; ++i) px(r, i) = rsqrt_ftz(px(h, i));
  const V d = fma(h, r, at);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    px(t, i) = copysignf(dev::rcp_ftz(px(d, i)), px(theta, i));
    px(t, i) = on[i] && fabsf(px(apq, i)) >= 1e-35f ? px(t, i) : 0.0f;
  }
  const V g = fma(t, t, one);
  V c;
#pragma unroll
  for (int i = 0; i < N; ++i) px(c, i) = rsqrt_ftz(px(g, i));
  const V s = mul(t, c), ns = neg(s);
  a[p][p] = fma(neg(t), apq, a[p][p]);
  a[q][q] = fma(t, apq, a[q][q]);
  a[p][q] = a[q][p] = all<N>(0.0f);
  constexpr int o = 3 - p - q;
  const V aop = a[o][p], aoq = a[o][q];
  a[o][p] = a[p][o] = fma(c, aop, mul(ns, aoq));
  a[o][q] = a[q][o] = fma(c, aoq, mul(s, aop));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const V vkp = v[k][p], vkq = v[k][q];
    v[k][p] = fma(c, vkp, mul(ns, vkq));
    v[k][q] = fma(s, vkp, mul(c, vkq));
  }
}

// The unit eigenvector of one pixel's smallest diagonal entry, oriented away from
// the camera (n . (u0, v0, 1) > 0), then the caller's orientation; 0 if invalid.
__device__ __forceinline__ float4 smallest(const float (&d)[3], const float (&v)[3][3], float u0, float v0, float sign,
                                           bool valid) {
  float nx = v[0][0], ny = v[1][0], nz = v[2][0], lmin = d[0];
  if (d[1] < lmin) {
    lmin = d[1];
    nx = v[0][1];
    ny = v[1][1];
    nz = v[2][1];
  }
  if (d[2] < lmin) {
    nx = v[0][2];
    ny = v[1][2];
    nz = v[2][2];
  }
  const float inv = rsqrt_ftz(fmaf(nx, nx, fmaf(ny, ny, nz * nz)));
  const float o = (fmaf(nx, u0, fmaf(ny, v0, nz)) < 0.0f ? -inv : inv) * sign;
  return valid ? make_float4(nx * o, ny * o, nz * o, 0.0f) : make_float4(0.f, 0.f, 0.f, 0.f);
}

// N adjacent pixels per thread.
template <int R, int N>
__global__ void __launch_bounds__(PT)
    plane_fit_kernel(const __grid_constant__ FrameDesc fd, float sign) {
  using V = Px<N>;
  constexpr int PX = 32 * N;
  // The decoded halo tile and, for two pixels, the same shifted by one column: a
  // thread's two depths at any offset are one aligned 8-byte load of one of the two.
  constexpr int tw = PX + 2 * R, th = PY + 2 * R;
  __shared__ __align__(16) float tile[N][th * tw];
  NRM_DEBUG_ENTRY(nullptr);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * PX - R, y0 = blockIdx.y * PY - R;
  const bool u16 = fd.in_dtype == NRM_IN_U16_MM;
  for (int ly = warp; ly < th; ly += PT / 32) {
    const int y = y0 + ly;
    const bool row = y >= 0 && y < fd.H;
    const long long o = (long long)y * fd.depth_pitch + x0;
#pragma unroll
    for (int lx = lane; lx < tw; lx += 32) {
      const int x = x0 + lx;
      float z = __int_as_float(0x7fc00000);
      if (row && x >= 0 && x < fd.W)
        z = u16 ? dev::decode_depth_u16(__ldg(reinterpret_cast<const uint16_t*>(fd.depth) + o + lx))
                : dev::decode_depth(__ldg(reinterpret_cast<const float*>(fd.depth) + o + lx));
      if (NRM_IOK(ly * tw + lx, tw * th)) {
        tile[0][ly * tw + lx] = z;
        if (N == 2 && lx > 0) tile[N - 1][ly * tw + lx - 1] = z;
      }
    }
  }
  __syncthreads();
  const int col = blockIdx.x * PX + N * lane, py = blockIdx.y * PY + warp;
  if (col >= fd.W || py >= fd.H) return;
  // Depths of the thread's pixels at window offset (dx, dy).
  auto at = [&](int dx, int dy) {
    const int c = R + dx, odd = N == 2 ? c & 1 : 0;
    const int i = (warp + R + dy) * tw + N * lane + c - odd;
    if (!NRM_IOK(i + N - 1, tw * th)) return all<N>(0.0f);
    return *reinterpret_cast<const V*>(&tile[odd][i]);
  };
  const V z0 = at(0, 0), nz0 = neg(z0);
  V u0;
#pragma unroll
  for (int i = 0; i < N; ++i) px(u0, i) = ((float)(col + i) - fd.cx) * fd.inv_fx;
  const float v0 = ((float)py - fd.cy) * fd.inv_fy;
  V sx = all<N>(0.f), sy = sx, sz = sx;
  V a00 = sx, a01 = sx, a02 = sx, a11 = sx, a12 = sx, a22 = sx;
#pragma unroll
  for (int dy = -R; dy <= R; ++dy) {
    const float e1 = (float)dy * fd.inv_fy, v1 = __fadd_rn(v0, e1);
    const V v = all<N>(v1), ey = mul(z0, all<N>(e1));
#pragma unroll
    for (int dx = -R; dx <= R; ++dx) {
      const V e = all<N>((float)dx * fd.inv_fx);
      const V u = add(u0, e);
      const V dz = add(at(dx, dy), nz0);
      const V qx = fma(dz, u, mul(z0, e));
      const V qy = fma(dz, v, ey);
      sx = add(sx, qx);
      sy = add(sy, qy);
      sz = add(sz, dz);
      a00 = fma(qx, qx, a00);
      a01 = fma(qx, qy, a01);
      a02 = fma(qx, dz, a02);
      a11 = fma(qy, qy, a11);
      a12 = fma(qy, dz, a12);
      a22 = fma(dz, dz, a22);
    }
  }
  // A NaN depth in the window leaves a NaN in the sums.
  bool ok[N], on[N], any = false;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    ok[i] = on[i] = fabsf(px(sx, i)) + fabsf(px(sy, i)) + fabsf(px(sz, i)) <= 3.402823466e38f;
    any = any || on[i];
  }
  constexpr float kInvN = 1.0f / (float)((2 * R + 1) * (2 * R + 1));
  const V inv_n = all<N>(-kInvN);
  const V mx = mul(sx, inv_n), my = mul(sy, inv_n), mz = mul(sz, inv_n);
  V a[3][3];
  a[0][0] = fma(mx, sx, a00);
  a[0][1] = a[1][0] = fma(mx, sy, a01);
  a[0][2] = a[2][0] = fma(mx, sz, a02);
  a[1][1] = fma(my, sy, a11);
  a[1][2] = a[2][1] = fma(my, sz, a12);
  a[2][2] = fma(mz, sz, a22);
  V vec[3][3];
#pragma unroll
  for (int k = 0; k < 9; ++k) vec[k / 3][k % 3] = all<N>(k % 4 ? 0.f : 1.f);
#pragma unroll 1
  for (int sweep = 0; sweep < 6 && any; ++sweep) {
    jacobi_rotate<0, 1, N>(a, vec, on);
    jacobi_rotate<0, 2, N>(a, vec, on);
    jacobi_rotate<1, 2, N>(a, vec, on);
    const V off = fma(a[0][1], a[0][1], fma(a[0][2], a[0][2], mul(a[1][2], a[1][2])));
    const V diag = fma(a[0][0], a[0][0], fma(a[1][1], a[1][1], mul(a[2][2], a[2][2])));
    any = false;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      on[i] = on[i] && !(px(off, i) <= 1e-14f * px(diag, i));
      any = any || on[i];
    }
  }
  const long long oo = (long long)py * fd.out_pitch + col;
  float4* out = reinterpret_cast<float4*>(fd.normals) + oo;
  uint8_t* mask = fd.valid + oo;
  [[maybe_unused]] const long long nlen = dev::dbg_span(fd.H, fd.W, fd.out_pitch, 16);
  [[maybe_unused]] const long long mlen = dev::dbg_span(fd.H, fd.W, fd.out_pitch, 1);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    if (col + i >= fd.W) break;
    const float d[3] = {px(a[0][0], i), px(a[1][1], i), px(a[2][2], i)};
    float w[3][3];
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k / 3][k % 3] = px(vec[k / 3][k % 3], i);
    if (NRM_GOK(out + i, fd.normals, nlen)) out[i] = smallest(d, w, px(u0, i), v0, sign, ok[i]);
    if (NRM_GOK(mask + i, fd.valid, mlen)) mask[i] = ok[i];
  }
}

template <int N>
const void* kernel_for(int radius) {
  switch (radius) {
    case 1: return (const void*)plane_fit_kernel<1, N>;
    case 2: return (const void*)plane_fit_kernel<2, N>;
    case 3: return (const void*)plane_fit_kernel<3, N>;
    case 4: return (const void*)plane_fit_kernel<4, N>;
    default: return nullptr;
  }
}

}  // namespace

cudaError_t launch_plane_fit(const FrameDesc& fd, int radius, float sign, int sms, cudaStream_t stream) {
  const int rows = (fd.H + PY - 1) / PY;
  // One pixel per thread while its CTAs are at most one per SM (see the file comment).
  const int n = (long long)((fd.W + 31) / 32) * rows <= sms ? 1 : 2;
  const void* fn = n == 1 ? kernel_for<1>(radius) : kernel_for<2>(radius);
  if (!fn) return cudaErrorInvalidValue;
  dim3 grid((fd.W + 32 * n - 1) / (32 * n), rows);
  FrameDesc d = fd;
  float sg = sign;
  void* args[2] = {&d, &sg};
  return cudaLaunchKernel(fn, grid, dim3(PT), args, 0, stream);
}

}  // namespace nrm
