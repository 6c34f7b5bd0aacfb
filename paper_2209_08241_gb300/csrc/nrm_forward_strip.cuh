// The strip kernels: batched forward pass (arXiv 2209.08241, Section 3.1
// Eq. 4-6 and the Section 3.2 mask) for frames whose rows TMA can load and
// whose outputs take whole-vector stores (ALIGNED), or for frames of any pitch
// and alignment, for pixel distance ALPHA = 1..4.
//
// One CTA is strip_warps compute warps and a producer warp. The producer walks
// the CTA's tiles (128 x strip_tile_y pixels) of the batch's work list and, per
// tile, issues one TMA box of raw depth into an S-stage ring and writes the
// tile's record, its column table and its row table next to it. A compute warp
// takes a band of strip_rows rows, four consecutive columns per lane, and walks
// down the band in steps of ALPHA rows, so that a row's four depths are
// converted to float once and serve as lower, centre and upper neighbour in
// turn from registers; only the left and right neighbours are read a second
// time. No decoded copy of the tile is kept in shared memory and no barrier
// joins the warps of a CTA: a warp waits for its stage's TMA copy and frees the
// stage when it is done with it. Warp instructions per 32 pixels (uint16 input,
// alpha 2): float4 37.7, half4 36.8, octahedral 37.5 (the tiled kernel's vector loops
// about 50 a pixel).
//
// Invalid depths are found per pixel from the smallest of the five depths
// (three-operand minimum, NaN propagating) instead of coding each of them as
// NaN: uint16 0 and float32 values <= 0 fail "> 0"; float32 infinities become
// NaN when they are loaded (0 x inf + inf) and then fail the minimum as NaNs do. For
// valid pixels every operation is that of emit_pair (nrm_device.cuh), in its
// order, so both give the same bits. (uint16 frames come here only if q >= FLT_MIN
// holds for every valid pixel, so that test is left out for them.)
#pragma once

#include "nrm_forward_kernels.cuh"

namespace nrm {

using namespace dev;

// Per-stage record of the producer.
struct alignas(16) StripInfo {
  float a, b, c;  // Eq. 4-6 constants with the sign folded in
  int u16;
  unsigned char* normals;  // of the tile's first pixel
  uint8_t* valid;
  long long out_pitch;
  int cols, rows;  // pixels of the tile inside the frame
#ifdef NRM_DEBUG_CHECKS
  const void *normals0, *valid0;  // the frame's outputs and their extents
  long long nlen, mlen;
#endif
};
constexpr unsigned kStripInfoBytes = 128;
static_assert(sizeof(StripInfo) <= kStripInfoBytes, "StripInfo must fit its slot");

// Shared memory of a stage: raw depth box, record, column table (two float4
// per lane), row table.
NRM_HD constexpr unsigned strip_table_bytes(int tile_y) {
  return (kStripInfoBytes + (kStripX / 2 + tile_y) * 16u + 127) / 128 * 128;
}
NRM_HD inline unsigned strip_stage_bytes(int tile_y, int halo, int eb) {
  return stage_bytes_for(kStripX, tile_y, halo, eb) + strip_table_bytes(tile_y);
}
NRM_HD inline unsigned strip_smem_bytes(int tile_y, int halo, int eb, int stages) {
  return (strip_stage_bytes(tile_y, halo, eb) + 16) * stages;
}

__device__ __forceinline__ float min3_nan(float a, float b, float c) {
  float d;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// 32-byte streaming store (the address is a multiple of 32): every store writes
// whole 32-byte sectors although a lane's four float4 normals are 64 bytes apart
// from the next lane's.
__device__ __forceinline__ void store32(void* p, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e,
                                        uint32_t f, uint32_t g, uint32_t h) {
  asm volatile("st.global.cs.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a), "r"(b), "r"(c),
               "r"(d), "r"(e), "r"(f), "r"(g), "r"(h)
               : "memory");
}

// Two raw depths as floats. uint16: 0x4B00uuuu is the float 2^23 + u, and
// subtracting 2^23 is exact (0 stays 0). float32: 0 x d + d is d for finite d
// and NaN for infinities.
__device__ __forceinline__ float2 depth_pair(uint32_t w) {
  const float2 k = f2(-8388608.0f, -8388608.0f);
  return __fadd2_rn(f2(__uint_as_float(__byte_perm(w, 0x4B000000u, 0x7410)),
                       __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7432))), k);
}
__device__ __forceinline__ float2 depth_pair(float2 d) { return __ffma2_rn(d, f2(0.0f, 0.0f), d); }

// The lane's four depths of a staged row.
__device__ __forceinline__ void load_run(const uint16_t* p, float2& a, float2& b) {
  const uint2 w = NRM_LDS(uint2, reinterpret_cast<const uint2*>(p));
  a = depth_pair(w.x);
  b = depth_pair(w.y);
}
__device__ __forceinline__ void load_run(const float* p, float2& a, float2& b) {
  const float4 w = NRM_LDS(float4, reinterpret_cast<const float4*>(p));
  a = depth_pair(f2(w.x, w.y));
  b = depth_pair(f2(w.z, w.w));
}
__device__ __forceinline__ float2 load_two(const uint16_t* p) {
  return depth_pair(NRM_LDS(uint32_t, reinterpret_cast<const uint32_t*>(p)));
}
__device__ __forceinline__ float2 load_two(const float* p) {
  return depth_pair(NRM_LDS(float2, reinterpret_cast<const float2*>(p)));
}

// Section 3.2 for one pixel pair, in the operation order of emit_pair: n_z, q and
// the mask decisions. mn: the smallest of all depths each pixel uses.
template <bool SECANT, bool U16>
__device__ __forceinline__ void strip_decide(float2 mn, float2 nx, float2 ny, float2 P, float2 T, float tau2,
                                             float2 nu1, float2 ku, float2 nv1, float2 kv, float2& nz, float2& q,
                                             bool& ka, bool& kb) {
  const float kFltMin = 1.17549435e-38f;
  nz = __ffma2_rn(nu1, nx, __ffma2_rn(nv1, ny, P));
  q = __ffma2_rn(nx, nx, __ffma2_rn(ny, ny, __fmul2_rn(nz, nz)));
  ka = mn.x > 0.0f;
  kb = mn.y > 0.0f;
  if (!U16) {
    ka = ka & (q.x >= kFltMin);
    kb = kb & (q.y >= kFltMin);
  }
  if (SECANT) {
    const float2 lhs = __fmul2_rn(q, __fadd2_rn(ku, kv));
    const float2 rhs = __fmul2_rn(T, __fmul2_rn(P, P));
    ka = ka & (lhs.x <= rhs.x);
    kb = kb & (lhs.y <= rhs.y);
  } else {
    ka = ka & (q.x <= tau2);
    kb = kb & (q.y <= tau2);
  }
}

// The stencil of Eq. 4-6 of one pixel pair, in the operation order of
// QuadStencil, then strip_decide.
template <bool SECANT, bool U16>
__device__ __forceinline__ void strip_pair(float2 d1, float2 d2, float2 d3, float2 d4, float2 d5, float2 A, float2 B,
                                           float2 C, float2 T, float tau2, float2 nu1, float2 ku, float2 nv1,
                                           float2 kv, float2& nx, float2& ny, float2& nz, float2& q, bool& ka,
                                           bool& kb) {
  const float2 M1 = f2(-1.0f, -1.0f);
  const float2 S24 = __fadd2_rn(d2, d4), D24 = __ffma2_rn(M1, d4, d2);
  const float2 S35 = __fadd2_rn(d3, d5), D35 = __ffma2_rn(M1, d5, d3);
  nx = __fmul2_rn(__fmul2_rn(A, S35), D24);
  ny = __fmul2_rn(__fmul2_rn(B, S24), D35);
  const float2 P = __fmul2_rn(__fmul2_rn(C, S24), S35);
  const float2 mn = f2(min3_nan(min3_nan(d1.x, d2.x, d3.x), d4.x, d5.x),
                       min3_nan(min3_nan(d1.y, d2.y, d3.y), d4.y, d5.y));
  strip_decide<SECANT, U16>(mn, nx, ny, P, T, tau2, nu1, ku, nv1, kv, nz, q, ka, kb);
}

// The octahedral codes of a pixel pair (oct16_code, operation for operation,
// with the additions, the scale and the rounding steps paired).
__device__ __forceinline__ void strip_codes(float2 nx, float2 ny, float2 nz, uint32_t& ca, uint32_t& cb) {
  const float2 r = f2(rcp_ftz(fabsf(nx.x) + fabsf(ny.x) + fabsf(nz.x)), rcp_ftz(fabsf(nx.y) + fabsf(ny.y) + fabsf(nz.y)));
  const float2 s = __fmul2_rn(f2(32767.0f, 32767.0f), r);
  const float2 m = f2(fmaxf(-nz.x, 0.0f), fmaxf(-nz.y, 0.0f));
  const float2 tx = __fadd2_rn(nx, f2(copysignf(m.x, nx.x), copysignf(m.y, nx.y)));
  const float2 ty = __fadd2_rn(ny, f2(copysignf(m.x, ny.x), copysignf(m.y, ny.y)));
  const float2 k = f2(12582912.0f, 12582912.0f);  // 1.5 * 2^23
  const float2 x = __ffma2_rn(tx, s, k), y = __ffma2_rn(ty, s, k);
  ca = __byte_perm(__float_as_uint(x.x), __float_as_uint(y.x), 0x5410);
  cb = __byte_perm(__float_as_uint(x.y), __float_as_uint(y.y), 0x5410);
}

// A row of one band written at any alignment (float4, half4): the lanes' results go to the warp's
// row buffer at the offset that the row has in memory modulo 16 bytes (mask:
// modulo 4), and the warp then copies whole 16-byte (4-byte) units with
// consecutive lanes, the ragged units at the ends element by element. (One store
// per pixel straight from the lanes, 4 pixels apart, writes part of a 32-byte
// sector at a time: 64 x 1921x1081 uint16 -> float4 745 us, half4 755 us with one
// CTA per SM; through the buffer 646 and 492 us, with two CTAs 487 and 484. The
// octahedral codes, whose ragged ends would be three of four elements, go straight
// from the lanes, 439 us; through a buffer they took half as long again.) float4: units
// are pixels, stored with their index's low bits XORed by bits 3-5, so that neither
// side has bank conflicts.
constexpr int kRowBufMask = 160;  // the mask's part of a row buffer
NRM_HD constexpr int strip_rowbuf(int out_dtype) {
  return out_dtype == NRM_OUT_OCT16 ? 0 : kRowBufMask + (out_dtype == NRM_OUT_F32X4 ? 2048 : 1040);
}

// Copies bytes [m, m + len) of buf to the same offsets from base, units of U
// bytes by consecutive lanes, elements of E bytes at the ragged ends.
template <int U, int E, int BYTES, typename Unit, typename Elem>
__device__ __forceinline__ void copy_out(const unsigned char* buf, unsigned char* base, int m, int len) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < (BYTES / U + 1 + 31) / 32; ++k) {
    const int b = (lane + 32 * k) * U;
    if (b >= m && b + U <= m + len) {
      __stcs(reinterpret_cast<Unit*>(base + b), NRM_LDS(Unit, reinterpret_cast<const Unit*>(buf + b)));
    } else if (b + U > m && b < m + len) {
#pragma unroll
      for (int e = 0; e < U; e += E)
        if (b + e >= m && b + e < m + len)
          __stcs(reinterpret_cast<Elem*>(base + b + e), NRM_LDS(Elem, reinterpret_cast<const Elem*>(buf + b + e)));
    }
  }
}

template <int OUT>
__device__ __forceinline__ void store_row(const uint32_t* w, uint32_t mbits, unsigned char* np, uint8_t* mp,
                                          unsigned char* buf, [[maybe_unused]] const StripInfo& f) {
  static_assert(OUT == NRM_OUT_F32X4 || OUT == NRM_OUT_F16X4, "octahedral codes are stored from the lanes");
  constexpr int BPP = OUT == NRM_OUT_F32X4 ? 16 : 8;
  const int lane = threadIdx.x & 31;
  unsigned char* row = np - 4 * lane * BPP;  // the row's first pixel in this tile
  uint8_t* mrow = mp - 4 * lane;
  const int count = min(f.cols, kStripX);
#ifdef NRM_DEBUG_CHECKS
  if (!(dbg_gmem_ok(row, count * BPP, f.normals0, f.nlen, "strip normals", __LINE__) &&
        dbg_gmem_ok(mrow, count, f.valid0, f.mlen, "strip mask", __LINE__)))
    return;
#endif
  unsigned char* nbuf = buf + kRowBufMask;
  const int mm = (int)(reinterpret_cast<uintptr_t>(mrow) & 3);
  __syncwarp();  // the previous row has left the buffer
  if (mm == 0) {
    NRM_STS(reinterpret_cast<uint32_t*>(buf) + lane, mbits);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) NRM_STS(buf + mm + 4 * lane + i, (unsigned char)(mbits >> (8 * i)));
  }
  if constexpr (OUT == NRM_OUT_F32X4) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 4 * lane + i;
      NRM_STS(reinterpret_cast<uint4*>(nbuf) + (c ^ ((c >> 3) & 7)),
              make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]));
    }
    __syncwarp();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = lane + 32 * k;
      if (c < count)
        __stcs(reinterpret_cast<uint4*>(row) + c, NRM_LDS(uint4, reinterpret_cast<const uint4*>(nbuf) + (c ^ ((c >> 3) & 7))));
    }
  } else {
    const int m = (int)(reinterpret_cast<uintptr_t>(row) & 15);
#pragma unroll
    for (int i = 0; i < 4; ++i) NRM_STS(reinterpret_cast<uint2*>(nbuf + m) + 4 * lane + i, make_uint2(w[2 * i], w[2 * i + 1]));
    __syncwarp();
    copy_out<16, 8, 1024, uint4, uint2>(nbuf, row - m, m, count * BPP);
  }
  copy_out<4, 1, 128, uint32_t, uint8_t>(buf, mrow - mm, mm, count);
}

// The normals (or codes) and mask bytes of a lane's four pixels: np, mp point at
// the first one's; k[i] says whether pixel i is valid; n > 0 of them lie in the
// frame. ALIGNED: whole vectors, straight to memory (n >= 4); else float4 and half4
// through the warp's row buffer (store_row), octahedral codes one by one.
template <int OUT, bool ALIGNED>
__device__ __forceinline__ void strip_store(const float2 (&nx)[2], const float2 (&ny)[2], const float2 (&nz)[2],
                                            const float2 (&q)[2], const bool (&k)[4], unsigned char* np, uint8_t* mp,
                                            int n, [[maybe_unused]] unsigned char* buf,
                                            [[maybe_unused]] const StripInfo& f) {
  [[maybe_unused]] constexpr int BPP = OUT == NRM_OUT_F32X4 ? 16 : OUT == NRM_OUT_F16X4 ? 8 : 4;
  const uint32_t mbits =
      (k[0] ? 1u : 0u) | (k[1] ? 0x100u : 0u) | (k[2] ? 0x10000u : 0u) | (k[3] ? 0x1000000u : 0u);
  uint32_t w[4 * BPP / 4];
  if constexpr (OUT == NRM_OUT_OCT16) {
    strip_codes(nx[0], ny[0], nz[0], w[0], w[1]);
    strip_codes(nx[1], ny[1], nz[1], w[2], w[3]);
    w[0] = k[0] ? w[0] : 0u;
    w[1] = k[1] ? w[1] : 0u;
    w[2] = k[2] ? w[2] : 0u;
    w[3] = k[3] ? w[3] : 0u;
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const bool ka = k[2 * j], kb = k[2 * j + 1];
      const float2 inv = f2(rsqrt_ftz(q[j].x), rsqrt_ftz(q[j].y));
      const float2 ox = __fmul2_rn(nx[j], inv), oy = __fmul2_rn(ny[j], inv), oz = __fmul2_rn(nz[j], inv);
      if constexpr (OUT == NRM_OUT_F16X4) {
        w[4 * j] = ka ? h2_bits(__floats2half2_rn(ox.x, oy.x)) : 0u;
        w[4 * j + 1] = ka ? h2_bits(__floats2half2_rn(oz.x, 0.0f)) : 0u;
        w[4 * j + 2] = kb ? h2_bits(__floats2half2_rn(ox.y, oy.y)) : 0u;
        w[4 * j + 3] = kb ? h2_bits(__floats2half2_rn(oz.y, 0.0f)) : 0u;
      } else {
        w[8 * j] = __float_as_uint(ka ? ox.x : 0.0f);
        w[8 * j + 1] = __float_as_uint(ka ? oy.x : 0.0f);
        w[8 * j + 2] = __float_as_uint(ka ? oz.x : 0.0f);
        w[8 * j + 3] = 0u;
        w[8 * j + 4] = __float_as_uint(kb ? ox.y : 0.0f);
        w[8 * j + 5] = __float_as_uint(kb ? oy.y : 0.0f);
        w[8 * j + 6] = __float_as_uint(kb ? oz.y : 0.0f);
        w[8 * j + 7] = 0u;
      }
    }
  }
  if constexpr (ALIGNED) {
#ifdef NRM_DEBUG_CHECKS
    if (n > 0 && !(dbg_gmem_ok(np, 4 * BPP, f.normals0, f.nlen, "strip normals", __LINE__) &&
                   dbg_gmem_ok(mp, 4, f.valid0, f.mlen, "strip mask", __LINE__)))
      return;
#endif
    if (n > 0) {
      if constexpr (OUT == NRM_OUT_F32X4) {
        store32(np, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
        store32(np + 32, w[8], w[9], w[10], w[11], w[12], w[13], w[14], w[15]);
      } else if constexpr (OUT == NRM_OUT_F16X4) {
        store32(np, w[0], w[1], w[2], w[3], w[4], w[5], w[6], w[7]);
      } else {
        __stcs(reinterpret_cast<uint4*>(np), make_uint4(w[0], w[1], w[2], w[3]));
      }
      __stcs(reinterpret_cast<unsigned int*>(mp), mbits);
    }
  } else if constexpr (OUT == NRM_OUT_OCT16) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i >= n) break;
#ifdef NRM_DEBUG_CHECKS
      if (!(dbg_gmem_ok(np + i * BPP, BPP, f.normals0, f.nlen, "strip normals", __LINE__) &&
            dbg_gmem_ok(mp + i, 1, f.valid0, f.mlen, "strip mask", __LINE__)))
        return;
#endif
      __stcs(reinterpret_cast<uint32_t*>(np) + i, w[i]);
      __stcs(mp + i, (uint8_t)(mbits >> (8 * i)));
    }
  } else {
    store_row<OUT>(w, mbits, np, mp, buf, f);
  }
}

// One band: strip_rows(OUT) rows of 128 columns from the staged box S (its first
// row is ALPHA above the band's, its column PAD the tile's first).
template <int OUT, bool SECANT, int ALPHA, bool ALIGNED, typename InT>
__device__ __forceinline__ void strip_band(const InT* __restrict__ S, const float4* __restrict__ ctab,
                                           const float4* __restrict__ rtab, const StripInfo& f, int band, float tau2,
                                           [[maybe_unused]] unsigned char* buf) {
  constexpr int EB = (int)sizeof(InT);
  constexpr int PAD = EB == 2 ? 8 : 4;        // pad_x(ALPHA, EB) for ALPHA <= 4
  constexpr int SP = kStripX + 2 * PAD;       // staged row pitch
  constexpr int BPP = OUT == NRM_OUT_F32X4 ? 16 : OUT == NRM_OUT_F16X4 ? 8 : 4;
  constexpr int ROWS = strip_rows(OUT);
  constexpr int STEPS = (ROWS + ALPHA - 1) / ALPHA;
  const int lane = threadIdx.x & 31;
  const float4 c0 = NRM_LDS(float4, ctab + 2 * lane), c1 = NRM_LDS(float4, ctab + 2 * lane + 1);
  const float2 nu1[2] = {f2(c0.x, c0.y), f2(c1.x, c1.y)};
  const float2 ku[2] = {f2(c0.z, c0.w), f2(c1.z, c1.w)};
  const float2 A = f2(f.a, f.a), B = f2(f.b, f.b), C = f2(f.c, f.c), T = f2(tau2, tau2);
  const int row0 = band * ROWS;
  const int rows = min(ROWS, f.rows - row0);
  const int n = f.cols - 4 * lane;  // of the lane's pixels, those in the frame
  const InT* base = S + row0 * SP + PAD + 4 * lane;
#pragma unroll 1
  for (int c = 0; c < ALPHA; ++c) {
    if (c >= rows) break;
    const InT* p = base + c * SP;  // staged row of the pixels ALPHA above row c
    float2 u0, u1, m0, m1;
    load_run(p, u0, u1);
    load_run(p + ALPHA * SP, m0, m1);
    unsigned char* np = f.normals + ((long long)(row0 + c) * f.out_pitch + 4 * lane) * BPP;
    uint8_t* mp = f.valid + (long long)(row0 + c) * f.out_pitch + 4 * lane;
#pragma unroll
    for (int k = 0; k < STEPS; ++k) {
      const int r = c + k * ALPHA;
      if (r >= rows) break;
      float2 b0, b1;
      load_run(p + (k + 2) * ALPHA * SP, b0, b1);
      const InT* pc = p + (k + 1) * ALPHA * SP;
      float2 l0, l1, r0, r1;  // left and right neighbours of the two pairs
      if (ALPHA == 1) {
        const float2 l = load_two(pc - 2), e = load_two(pc + 4);
        l0 = f2(l.y, m0.x);
        r0 = l1 = f2(m0.y, m1.x);
        r1 = f2(m1.y, e.x);
      } else if (ALPHA == 2) {
        l0 = load_two(pc - 2);
        l1 = m0;
        r0 = m1;
        r1 = load_two(pc + 4);
      } else {
        float2 la, lb, ra, rb;  // columns -4..-1 and 4..7
        load_run(pc - 4, la, lb);
        load_run(pc + 4, ra, rb);
        l0 = ALPHA == 4 ? la : f2(la.y, lb.x);
        l1 = ALPHA == 4 ? lb : f2(lb.y, m0.x);
        r0 = ALPHA == 4 ? ra : f2(m1.y, ra.x);
        r1 = ALPHA == 4 ? rb : f2(ra.y, rb.x);
      }
      const float4 rr = NRM_LDS(float4, rtab + row0 + r);
      const float2 nv1 = f2(rr.x, rr.y), kv = f2(rr.z, rr.w);
      float2 nx[2], ny[2], nz[2], q[2];
      bool keep[4];
      strip_pair<SECANT, EB == 2>(m0, r0, b0, l0, u0, A, B, C, T, tau2, nu1[0], ku[0], nv1, kv, nx[0], ny[0], nz[0],
                                  q[0], keep[0], keep[1]);
      strip_pair<SECANT, EB == 2>(m1, r1, b1, l1, u1, A, B, C, T, tau2, nu1[1], ku[1], nv1, kv, nx[1], ny[1], nz[1],
                                  q[1], keep[2], keep[3]);
      strip_store<OUT, ALIGNED>(nx, ny, nz, q, keep, np, mp, n, buf, f);
      np += ALPHA * f.out_pitch * BPP;
      mp += ALPHA * f.out_pitch;
      u0 = m0;
      u1 = m1;
      m0 = b0;
      m1 = b1;
    }
  }
}

// The record of the tile at (gx0, gy0) of frame fd.
template <int BPP>
__device__ __forceinline__ void write_record(StripInfo* dst, const FrameDesc& fd, float sign, int gx0, int gy0) {
  StripInfo si;
  si.a = -sign * fd.a;
  si.b = -sign * fd.b;
  si.c = sign * fd.c;
  si.u16 = fd.in_dtype == NRM_IN_U16_MM;
  si.out_pitch = fd.out_pitch;
  si.normals = reinterpret_cast<unsigned char*>(fd.normals) + ((long long)gy0 * fd.out_pitch + gx0) * BPP;
  si.valid = fd.valid + (long long)gy0 * fd.out_pitch + gx0;
  si.cols = fd.W - gx0;
  si.rows = fd.H - gy0;
#ifdef NRM_DEBUG_CHECKS
  si.normals0 = fd.normals;
  si.valid0 = fd.valid;
  si.nlen = dbg_span(fd.H, fd.W, fd.out_pitch, BPP);
  si.mlen = dbg_span(fd.H, fd.W, fd.out_pitch, 1);
#endif
  NRM_STS(dst, si);
}

// The tile's column table, two float4 per lane, and row table (the terms of
// emit_pair), by one warp.
template <int TY>
__device__ __forceinline__ void write_tables(float4* ctab, const FrameDesc& fd, int gx0, int gy0) {
  const int lane = threadIdx.x & 31;
  const float cx = fd.cx, cy = fd.cy, ifx = fd.inv_fx, ify = fd.inv_fy;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float ua = ((float)(gx0 + 4 * lane + 2 * h) - cx) * ifx;
    const float ub = ((float)(gx0 + 4 * lane + 2 * h + 1) - cx) * ifx;
    NRM_STS(ctab + 2 * lane + h, make_float4(-ua, -ub, fmaf(ua, ua, 1.0f), fmaf(ub, ub, 1.0f)));
  }
  for (int r = lane; r < TY; r += 32) {
    const float v1 = ((float)(gy0 + r) - cy) * ify;
    NRM_STS(ctab + kStripX / 2 + r, make_float4(-v1, -v1, v1 * v1, v1 * v1));
  }
}

// Loads the rows warp, warp + LOADERS, ... of the halo box of a frame without a
// usable tensor map into its staged layout, in plain loads of one depth per lane
// (a row may start on any element); 0 outside the frame. These loads are bound by
// latency, so up to BATCH rows, five loads each (128 columns, then the halo
// columns), are in flight before the first is stored.
template <int HALO, int TY, int LOADERS, typename InT>
__device__ __forceinline__ void load_box(InT* __restrict__ st, const FrameDesc& fd, int gx0, int gy0, int warp) {
  constexpr int PAD = sizeof(InT) == 2 ? 8 : (HALO + 3) / 4 * 4;
  constexpr int SP = kStripX + 2 * PAD;
  constexpr int ROWS = TY + 2 * HALO;
  constexpr int PER_WARP = (ROWS + LOADERS - 1) / LOADERS;
  constexpr int BATCH = PER_WARP < 8 ? PER_WARP : 8;
  const int lane = threadIdx.x & 31;
  const InT* src = reinterpret_cast<const InT*>(fd.depth);
  const int H = fd.H, W = fd.W;
  const long long pitch = fd.depth_pitch;
  // The lane's five columns of a row; the last is a halo column (lanes < 2 HALO).
  int col[5];
  bool in[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) {
    col[k] = k < 4 ? lane + 32 * k : lane < HALO ? lane - HALO : kStripX + lane - HALO;
    in[k] = (k < 4 || lane < 2 * HALO) && gx0 + col[k] >= 0 && gx0 + col[k] < W;
  }
#pragma unroll 1
  for (int r0 = warp; r0 < ROWS; r0 += BATCH * LOADERS) {
    InT v[BATCH][5];
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      const int y = gy0 - HALO + r0 + b * LOADERS;
      const bool row = r0 + b * LOADERS < ROWS && y >= 0 && y < H;
      const InT* p = src + y * pitch + gx0;
#pragma unroll
      for (int k = 0; k < 5; ++k) v[b][k] = row && in[k] ? __ldg(p + col[k]) : InT(0);
    }
#pragma unroll
    for (int b = 0; b < BATCH; ++b) {
      const int r = r0 + b * LOADERS;
      if (r >= ROWS) break;
      InT* q = st + r * SP + PAD;
#pragma unroll
      for (int k = 0; k < 5; ++k)
        if (k < 4 || lane < 2 * HALO) NRM_STS(q + col[k], v[b][k]);
    }
  }
}

// The pipeline of a strip kernel: tiles of kStripX x (ROWS x WARPS) pixels with a halo
// of HALO; band(stage, column table, row table, record, warp) computes one
// band, its stage pointer typed by the frame's depth type. RING: the descriptors
// are in global memory written by the host (each tensor map is fenced before
// its first use), else in kernel-parameter space. LOADERS = 0: one producer warp
// and TMA; LOADERS > 0: that many warps fill the stages with load_box (any pitch
// and alignment).
template <int OUT, int HALO, int ROWS, int WARPS, int LOADERS, bool RING, class Band>
__device__ __forceinline__ void strip_pipeline(const BatchArgs& args, const Globals& g, const Band& band) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int BPP = OUT == NRM_OUT_F32X4 ? 16 : OUT == NRM_OUT_F16X4 ? 8 : 4;
  const int S = args.stages;
  const unsigned SB = args.stage_bytes;
  constexpr int TY = ROWS * WARPS;
  constexpr unsigned TB = strip_table_bytes(TY);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + (size_t)S * SB);
  uint64_t* empty = full + S;
  const int total = args.hdr->total_tiles;
  const int nf = args.hdr->n_frames;
  const int G = (int)gridDim.x;
  const int my = (int)blockIdx.x < total ? (total - 1 - (int)blockIdx.x) / G + 1 : 0;
  if (my == 0) return;
  NRM_DEBUG_ENTRY(g.status);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&full[s]), LOADERS ? LOADERS : 2);
      mbar_init(smem_u32(&empty[s]), WARPS);
    }
    fence_barrier_init();
  }
  __syncthreads();

  if (warp >= WARPS) {
    // ------------------------------------------------------------ producer
    int cur = 0, fenced = -1, s = 0;
    uint32_t parity = 1;
    // Waits (bounded) for the copies of the last tiles before the j-th, the only ones
    // that can be under way, so that none lands after the CTA has ended, also when a
    // compute warp gave a late one up.
    auto land = [&](int j) {
      if (LOADERS == 0 && lane == 0)
        for (int k = j > S ? j - S : 0; k < j; ++k)
          mbar_wait_bounded(smem_u32(&full[k % S]), (uint32_t)((k / S) & 1), g.timeout_ns);
    };
    for (int j = 0; j < my; ++j) {
      if (j >= S && !mbar_wait_warp(smem_u32(&empty[s]), parity, g.timeout_ns)) {
        if (lane == 0) record_error(g.status, NRM_ERR_TIMEOUT);
        land(j);
        return;
      }
      const int t = (int)blockIdx.x + j * G;
      while (cur + 1 < nf && load_index<RING>(args.tile_begin + cur + 1) <= t) ++cur;
      const FrameDesc* fd = args.frames + cur;
      const int local = t - load_index<RING>(args.tile_begin + cur);
      const int tiles_x = fd->tiles_x;
      const int ty = local / tiles_x;
      const int gx0 = (local - ty * tiles_x) * kStripX, gy0 = ty * TY;
      const int eb = fd->in_dtype == NRM_IN_U16_MM ? 2 : 4;
      unsigned char* st = smem + (size_t)s * SB;
      if constexpr (LOADERS > 0) {
        const int w = warp - WARPS;
        if (eb == 2)
          load_box<HALO, TY, LOADERS>(reinterpret_cast<uint16_t*>(st), *fd, gx0, gy0, w);
        else
          load_box<HALO, TY, LOADERS>(reinterpret_cast<float*>(st), *fd, gx0, gy0, w);
        if (w == 0) {
          if (lane == 0) write_record<BPP>(reinterpret_cast<StripInfo*>(st + SB - TB), *fd, g.sign, gx0, gy0);
          write_tables<TY>(reinterpret_cast<float4*>(st + SB - TB + kStripInfoBytes), *fd, gx0, gy0);
        }
      } else {
        if (lane == 0) {
          if (RING && cur != fenced) {
            fence_tensormap_acquire(&fd->tmap);
            fenced = cur;
          }
          const int padx = pad_x(HALO, eb);
          const uint32_t bar = smem_u32(&full[s]);
          mbar_arrive_expect_tx(bar, (uint32_t)((kStripX + 2 * padx) * (TY + 2 * HALO) * eb));
          tma_load_2d(smem_u32(st), &fd->tmap, gx0 - padx, gy0 - HALO, bar);
          write_record<BPP>(reinterpret_cast<StripInfo*>(st + SB - TB), *fd, g.sign, gx0, gy0);
        }
        write_tables<TY>(reinterpret_cast<float4*>(st + SB - TB + kStripInfoBytes), *fd, gx0, gy0);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&full[s]));
      if (++s == S) {
        s = 0;
        parity ^= 1;
      }
    }
    land(my);
    return;
  }

  // -------------------------------------------------------------- compute
  int s = 0;
  uint32_t parity = 0;
  for (int i = 0; i < my; ++i) {
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(smem_u32(&full[s]), parity, g.timeout_ns))) {
      if (lane == 0) record_error(g.status, NRM_ERR_TIMEOUT);
      return;
    }
    const unsigned char* st = smem + (size_t)s * SB;
    const StripInfo f = NRM_LDS(StripInfo, reinterpret_cast<const StripInfo*>(st + SB - TB));
    const float4* ctab = reinterpret_cast<const float4*>(st + SB - TB + kStripInfoBytes);
    if (f.u16)
      band(reinterpret_cast<const uint16_t*>(st), ctab, ctab + kStripX / 2, f, warp);
    else
      band(reinterpret_cast<const float*>(st), ctab, ctab + kStripX / 2, f, warp);
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&empty[s]));
    if (++s == S) {
      s = 0;
      parity ^= 1;
    }
  }
}

// Loader warps of the kernels for frames of any alignment.
NRM_HD constexpr int strip_loaders(int out_dtype) { return out_dtype == NRM_OUT_OCT16 ? 2 : 4; }

template <int OUT, bool SECANT, int ALPHA, bool ALIGNED, bool RING>
__device__ __forceinline__ void strip_forward(const BatchArgs& args, const Globals& g) {
  strip_pipeline<OUT, ALPHA, strip_rows(OUT), strip_warps(OUT, ALIGNED), ALIGNED ? 0 : strip_loaders(OUT), RING>(
      args, g, [&](const auto* S, const float4* ctab, const float4* rtab, const StripInfo& f, int warp) {
        extern __shared__ __align__(128) unsigned char smem[];
        unsigned char* buf = smem + args.stages * (args.stage_bytes + 16) + warp * strip_rowbuf(OUT);
        strip_band<OUT, SECANT, ALPHA, ALIGNED>(S, ctab, rtab, f, warp, g.tau2, buf);
      });
}

NRM_HD constexpr int strip_block(int out_dtype, bool aligned) {
  return (strip_warps(out_dtype, aligned) + (aligned ? 1 : strip_loaders(out_dtype))) * 32;
}

NRM_HD constexpr int strip_min_ctas(int out_dtype, bool aligned) {
  return out_dtype == NRM_OUT_OCT16 ? (aligned ? 4 : 3) : aligned ? 1 : 2;
}

template <int OUT, bool SECANT, int ALPHA, bool ALIGNED>
__global__ void __launch_bounds__(strip_block(OUT, ALIGNED), strip_min_ctas(OUT, ALIGNED))
    fwd_strip_param_kernel(const __grid_constant__ ParamBatch pb, const BatchArgs ring, const Globals g) {
  BatchArgs args = ring;
  args.hdr = &pb.hdr;
  args.tile_begin = pb.tile_begin;
  args.frames = pb.frames;
  strip_forward<OUT, SECANT, ALPHA, ALIGNED, false>(args, g);
}

template <int OUT, bool SECANT, int ALPHA, bool ALIGNED>
__global__ void __launch_bounds__(strip_block(OUT, ALIGNED), strip_min_ctas(OUT, ALIGNED))
    fwd_strip_kernel(const BatchArgs args, const Globals g) {
  strip_forward<OUT, SECANT, ALPHA, ALIGNED, true>(args, g);
}

// The kernel of one output type, or NULL (instantiated in a file per ALIGNED).
template <int OUT, bool SECANT, bool ALIGNED>
const void* strip_by_alpha(int alpha, bool param) {
  switch (alpha) {
    case 1: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 1, ALIGNED>
                         : (const void*)fwd_strip_kernel<OUT, SECANT, 1, ALIGNED>;
    case 2: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 2, ALIGNED>
                         : (const void*)fwd_strip_kernel<OUT, SECANT, 2, ALIGNED>;
    case 3: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 3, ALIGNED>
                         : (const void*)fwd_strip_kernel<OUT, SECANT, 3, ALIGNED>;
    case 4: return param ? (const void*)fwd_strip_param_kernel<OUT, SECANT, 4, ALIGNED>
                         : (const void*)fwd_strip_kernel<OUT, SECANT, 4, ALIGNED>;
    default: return nullptr;
  }
}

template <bool ALIGNED>
const void* strip_kernel(int out_dtype, bool secant, int alpha, bool param) {
  switch (out_dtype) {
    case NRM_OUT_F32X4:
      return secant ? strip_by_alpha<NRM_OUT_F32X4, true, ALIGNED>(alpha, param)
                    : strip_by_alpha<NRM_OUT_F32X4, false, ALIGNED>(alpha, param);
    case NRM_OUT_F16X4:
      return secant ? strip_by_alpha<NRM_OUT_F16X4, true, ALIGNED>(alpha, param)
                    : strip_by_alpha<NRM_OUT_F16X4, false, ALIGNED>(alpha, param);
    case NRM_OUT_OCT16:
      return secant ? strip_by_alpha<NRM_OUT_OCT16, true, ALIGNED>(alpha, param)
                    : strip_by_alpha<NRM_OUT_OCT16, false, ALIGNED>(alpha, param);
    default: return nullptr;
  }
}
extern template const void* strip_kernel<true>(int, bool, int, bool);
extern template const void* strip_kernel<false>(int, bool, int, bool);

}  // namespace nrm
