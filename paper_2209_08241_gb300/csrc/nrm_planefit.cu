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
// these operations.
#include "nrm_device.cuh"

namespace nrm {

namespace {

constexpr int PX = 64, PY = 8, PT = PX / 2 * PY;

using dev::f2;

using dev::rsqrt_ftz;
__device__ __forceinline__ float2 neg(float2 x) { return __fmul2_rn(x, f2(-1.0f, -1.0f)); }

// One Jacobi rotation zeroing a[p][q] of the symmetric matrices a of a pixel
// pair, accumulated into the eigenvector columns of v. A pixel that is done
// (!on) or whose a[p][q] is nothing takes t = 0, which leaves it bit for bit as it
// is. Approximate reciprocal and square root suffice: c and s are formed from t
// so that c^2 + s^2 = 1 to rounding whatever t's last bits, and an error of a few
// ulp in t only leaves an off-diagonal residue of a few ulp of |a_pq|, the size
// of the rounding already in S. (|theta| is capped at 1e18, where theta^2 would
// come near overflow and t is nothing beside 1.)
template <int p, int q>
__device__ __forceinline__ void jacobi_rotate(float2 (&a)[3][3], float2 (&v)[3][3], bool on0, bool on1) {
  const float2 apq = a[p][q];
  // t = tan of the rotation angle, the smaller root of t^2 + 2 theta t - 1 = 0.
  const float2 den = __fadd2_rn(apq, apq);
  const float2 num = __ffma2_rn(f2(-1.0f, -1.0f), a[p][p], a[q][q]);
  const float2 theta = __fmul2_rn(num, f2(dev::rcp_ftz(den.x), dev::rcp_ftz(den.y)));
  const float2 at = f2(fminf(fabsf(theta.x), 1e18f), fminf(fabsf(theta.y), 1e18f));
  const float2 h = __ffma2_rn(at, at, f2(1.0f, 1.0f));
  const float2 d = __ffma2_rn(h, f2(rsqrt_ftz(h.x), rsqrt_ftz(h.y)), at);
  float2 t = f2(copysignf(dev::rcp_ftz(d.x), theta.x), copysignf(dev::rcp_ftz(d.y), theta.y));
  t.x = on0 && fabsf(apq.x) >= 1e-35f ? t.x : 0.0f;
  t.y = on1 && fabsf(apq.y) >= 1e-35f ? t.y : 0.0f;
  const float2 g = __ffma2_rn(t, t, f2(1.0f, 1.0f));
  const float2 c = f2(rsqrt_ftz(g.x), rsqrt_ftz(g.y));
  const float2 s = __fmul2_rn(t, c), ns = neg(s);
  a[p][p] = __ffma2_rn(neg(t), apq, a[p][p]);
  a[q][q] = __ffma2_rn(t, apq, a[q][q]);
  a[p][q] = a[q][p] = f2(0.0f, 0.0f);
  constexpr int r = 3 - p - q;
  const float2 arp = a[r][p], arq = a[r][q];
  a[r][p] = a[p][r] = __ffma2_rn(c, arp, __fmul2_rn(ns, arq));
  a[r][q] = a[q][r] = __ffma2_rn(c, arq, __fmul2_rn(s, arp));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float2 vkp = v[k][p], vkq = v[k][q];
    v[k][p] = __ffma2_rn(c, vkp, __fmul2_rn(ns, vkq));
    v[k][q] = __ffma2_rn(s, vkp, __fmul2_rn(c, vkq));
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

template <int R>
__global__ void __launch_bounds__(PT)
    plane_fit_kernel(const __grid_constant__ FrameDesc fd, float sign) {
  // The decoded halo tile, and the same shifted by one column: a thread's two
  // depths at any offset are one aligned 8-byte load of one of the two.
  constexpr int tw = PX + 2 * R, th = PY + 2 * R;
  __shared__ __align__(16) float tile[2][th * tw];
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
        if (lx > 0) tile[1][ly * tw + lx - 1] = z;
      }
    }
  }
  __syncthreads();
  const int px = blockIdx.x * PX + 2 * lane, py = blockIdx.y * PY + warp;
  if (px >= fd.W || py >= fd.H) return;
  // Depths of the pixel pair at window offset (dx, dy).
  auto at = [&](int dx, int dy) {
    const int c = R + dx, odd = c & 1;
    const int i = (warp + R + dy) * tw + 2 * lane + c - odd;
    if (!NRM_IOK(i + 1, tw * th)) return f2(0.0f, 0.0f);
    return *reinterpret_cast<const float2*>(&tile[odd][i]);
  };
  const float2 z0 = at(0, 0), nz0 = neg(z0);
  const float2 u0 = f2(((float)px - fd.cx) * fd.inv_fx, ((float)(px + 1) - fd.cx) * fd.inv_fx);
  const float v0 = ((float)py - fd.cy) * fd.inv_fy;
  float2 sx = f2(0.f, 0.f), sy = sx, sz = sx;
  float2 a00 = sx, a01 = sx, a02 = sx, a11 = sx, a12 = sx, a22 = sx;
#pragma unroll
  for (int dy = -R; dy <= R; ++dy) {
    const float e1 = (float)dy * fd.inv_fy, v1 = __fadd_rn(v0, e1);
    const float2 v = f2(v1, v1), ey = __fmul2_rn(z0, f2(e1, e1));
#pragma unroll
    for (int dx = -R; dx <= R; ++dx) {
      const float e = (float)dx * fd.inv_fx;
      const float2 u = __fadd2_rn(u0, f2(e, e));
      const float2 dz = __fadd2_rn(at(dx, dy), nz0);
      const float2 qx = __ffma2_rn(dz, u, __fmul2_rn(z0, f2(e, e)));
      const float2 qy = __ffma2_rn(dz, v, ey);
      sx = __fadd2_rn(sx, qx);
      sy = __fadd2_rn(sy, qy);
      sz = __fadd2_rn(sz, dz);
      a00 = __ffma2_rn(qx, qx, a00);
      a01 = __ffma2_rn(qx, qy, a01);
      a02 = __ffma2_rn(qx, dz, a02);
      a11 = __ffma2_rn(qy, qy, a11);
      a12 = __ffma2_rn(qy, dz, a12);
      a22 = __ffma2_rn(dz, dz, a22);
    }
  }
  // A NaN depth in the window leaves a NaN in the sums.
  const bool ok0 = fabsf(sx.x) + fabsf(sy.x) + fabsf(sz.x) <= 3.402823466e38f;
  const bool ok1 = fabsf(sx.y) + fabsf(sy.y) + fabsf(sz.y) <= 3.402823466e38f;
  constexpr float kInvN = 1.0f / (float)((2 * R + 1) * (2 * R + 1));
  const float2 inv_n = f2(-kInvN, -kInvN);
  const float2 mx = __fmul2_rn(sx, inv_n), my = __fmul2_rn(sy, inv_n), mz = __fmul2_rn(sz, inv_n);
  float2 a[3][3];
  a[0][0] = __ffma2_rn(mx, sx, a00);
  a[0][1] = a[1][0] = __ffma2_rn(mx, sy, a01);
  a[0][2] = a[2][0] = __ffma2_rn(mx, sz, a02);
  a[1][1] = __ffma2_rn(my, sy, a11);
  a[1][2] = a[2][1] = __ffma2_rn(my, sz, a12);
  a[2][2] = __ffma2_rn(mz, sz, a22);
  float2 vec[3][3];
#pragma unroll
  for (int k = 0; k < 9; ++k) vec[k / 3][k % 3] = k % 4 ? f2(0.f, 0.f) : f2(1.f, 1.f);
  bool on0 = ok0, on1 = ok1;
#pragma unroll 1
  for (int sweep = 0; sweep < 6 && (on0 || on1); ++sweep) {
    jacobi_rotate<0, 1>(a, vec, on0, on1);
    jacobi_rotate<0, 2>(a, vec, on0, on1);
    jacobi_rotate<1, 2>(a, vec, on0, on1);
    const float2 off = __ffma2_rn(a[0][1], a[0][1], __ffma2_rn(a[0][2], a[0][2], __fmul2_rn(a[1][2], a[1][2])));
    const float2 diag = __ffma2_rn(a[0][0], a[0][0], __ffma2_rn(a[1][1], a[1][1], __fmul2_rn(a[2][2], a[2][2])));
    on0 = on0 && !(off.x <= 1e-14f * diag.x);
    on1 = on1 && !(off.y <= 1e-14f * diag.y);
  }
  const float d0[3] = {a[0][0].x, a[1][1].x, a[2][2].x}, d1[3] = {a[0][0].y, a[1][1].y, a[2][2].y};
  float w0[3][3], w1[3][3];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    w0[k / 3][k % 3] = vec[k / 3][k % 3].x;
    w1[k / 3][k % 3] = vec[k / 3][k % 3].y;
  }
  const long long oo = (long long)py * fd.out_pitch + px;
  float4* out = reinterpret_cast<float4*>(fd.normals) + oo;
  uint8_t* mask = fd.valid + oo;
  [[maybe_unused]] const long long nlen = dev::dbg_span(fd.H, fd.W, fd.out_pitch, 16);
  [[maybe_unused]] const long long mlen = dev::dbg_span(fd.H, fd.W, fd.out_pitch, 1);
  if (NRM_GOK(out, fd.normals, nlen)) *out = smallest(d0, w0, u0.x, v0, sign, ok0);
  if (NRM_GOK(mask, fd.valid, mlen)) *mask = ok0;
  if (px + 1 < fd.W) {
    if (NRM_GOK(out + 1, fd.normals, nlen)) out[1] = smallest(d1, w1, u0.y, v0, sign, ok1);
    if (NRM_GOK(mask + 1, fd.valid, mlen)) mask[1] = ok1;
  }
}

}  // namespace

cudaError_t launch_plane_fit(const FrameDesc& fd, int radius, float sign, cudaStream_t stream) {
  dim3 grid((fd.W + PX - 1) / PX, (fd.H + PY - 1) / PY);
  const void* fn = nullptr;
  switch (radius) {
    case 1: fn = (const void*)plane_fit_kernel<1>; break;
    case 2: fn = (const void*)plane_fit_kernel<2>; break;
    case 3: fn = (const void*)plane_fit_kernel<3>; break;
    case 4: fn = (const void*)plane_fit_kernel<4>; break;
    default: return cudaErrorInvalidValue;
  }
  FrameDesc d = fd;
  float sg = sign;
  void* args[2] = {&d, &sg};
  return cudaLaunchKernel(fn, grid, dim3(PT), args, 0, stream);
}

}  // namespace nrm
