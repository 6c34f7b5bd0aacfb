// Strip kernels of the batched multi-scale variant (nrm_multiscale.cu) for
// consecutive distances alpha_i = i, i = 1..K (K = 2..kMsStripMaxScales), on the
// pipeline of the single-scale strip kernels (nrm_forward_strip.cuh) and with
// their conditions on the frames.
//
// A lane owns four consecutive columns and walks down its warp's band; the
// decoded rows the vertical neighbours come from stay in registers (fully
// unrolled, so a row is converted once for all scales), and the horizontal ones
// come from one decoded window of the row, 4 (K <= 4) or 8 columns to the left and
// right. (Each K is twelve kernels, unrolled over rows and scales. 7 and 8 scales are
// not compiled and not measured here; they take the run-time kernel.) With the distances compiled in, a scale costs its 8 (pair) or 10
// (quad) paired FP32 instructions per two pixels and no loads or indexing.
//
// Every operation on valid pixels is that of ms_compute (nrm_multiscale.cu) in its
// order: the same bits.
//
// One CTA of 8 x 8 rows per SM and two stages, for the reason given in
// nrm_forward_strip.cu (a shallow ring keeps HBM off saturation). Measured, alpha
// 1..4: 16 x 1920x1080 uint16 -> float4 pair 100.3 us (93 % of the measured copy;
// the run-time-distance kernel 163.9), quad 100.7; one 4096x3072 float32 frame
// quad 47.8 us (81 %; 65.6); 16 x 1080p pair -> half4 79, quad -> octahedral 101.
// (6 warps 107-111 / 124 / 50.5; 3 stages 113 / 105 / 49.2; 2 CTAs of 4 warps
// 116 / 107 / 48.9; bands of 4 rows 100.2 / 101.5 / 46.7, float32 input 120
// against 118.)
#pragma once

#include "nrm_forward_strip.cuh"

namespace nrm {

namespace ms_strip {

constexpr int kRows = 8;  // per warp
constexpr int kWarps = 8;
constexpr int kStages = 2;

template <int OUT, int FORM, bool SECANT, int K, typename InT>
__device__ __forceinline__ void ms_band(const InT* __restrict__ S, const float4* __restrict__ ctab,
                                        const float4* __restrict__ rtab, const StripInfo& f, int band, float tau2) {
  constexpr int EB = (int)sizeof(InT);
  constexpr bool QUAD = FORM == NRM_MS_QUAD;
  constexpr int PAD = EB == 2 ? 8 : (K + 3) / 4 * 4;  // pad_x(K, EB) for K <= 8
  constexpr int SP = kStripX + 2 * PAD;
  constexpr int KW = (K + 3) / 4 * 4;     // columns of the window on each side
  constexpr int L = QUAD ? KW : 0;        // the pair form has no left and upper neighbours
  constexpr int UP = QUAD ? K : 0;
  constexpr int BPP = OUT == NRM_OUT_F32X4 ? 16 : OUT == NRM_OUT_F16X4 ? 8 : 4;
  const int lane = threadIdx.x & 31;
  const float4 c0 = NRM_LDS(float4, ctab + 2 * lane), c1 = NRM_LDS(float4, ctab + 2 * lane + 1);
  const float2 nu1[2] = {f2(c0.x, c0.y), f2(c1.x, c1.y)};
  const float2 ku[2] = {f2(c0.z, c0.w), f2(c1.z, c1.w)};
  const float2 T = f2(tau2, tau2), M1 = f2(-1.0f, -1.0f);
  const int row0 = band * kRows;
  const int rows = min(kRows, f.rows - row0);
  if (rows <= 0) return;
  const int n = f.cols - 4 * lane;
  const InT* p = S + (row0 + K) * SP + PAD + 4 * lane;  // the band's first row
  unsigned char* np = f.normals + ((long long)row0 * f.out_pitch + 4 * lane) * BPP;
  uint8_t* mp = f.valid + (long long)row0 * f.out_pitch + 4 * lane;
  // R[i]: band row i - UP.
  float2 R[kRows + K + UP][2];
#pragma unroll
  for (int i = 0; i < K + UP; ++i) load_run(p + (i - UP) * SP, R[i][0], R[i][1]);
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    if (r >= rows) break;
    load_run(p + (r + K) * SP, R[r + K + UP][0], R[r + K + UP][1]);
    // The row's window: columns -L .. 3 + KW of the lane.
    float w[L + 4 + KW];
    const InT* pc = p + r * SP;
#pragma unroll
    for (int c = 0; c < L + 4 + KW; c += 4) {
      float2 a, b;
      if (c == L) {
        a = R[r + UP][0];
        b = R[r + UP][1];
      } else {
        load_run(pc - L + c, a, b);
      }
      w[c] = a.x, w[c + 1] = a.y, w[c + 2] = b.x, w[c + 3] = b.y;
    }
    const float4 rr = NRM_LDS(float4, rtab + row0 + r);
    const float2 nv1 = f2(rr.x, rr.y), kv = f2(rr.z, rr.w);
    float2 nx[2], ny[2], nz[2], q[2];
    bool keep[4];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float2 d1 = R[r + UP][j];
      float2 ax = f2(-0.f, -0.f), ay = ax, ap = ax, mn = d1;
#pragma unroll
      for (int al = 1; al <= K; ++al) {
        const float fa = (float)al;
        const float sa = fa * f.a, sb = fa * f.b, sc = fa * fa * f.c;
        const float2 A = f2(sa, sa), B = f2(sb, sb), C = f2(sc, sc);
        const float2 d2 = f2(w[L + 2 * j + al], w[L + 2 * j + al + 1]);
        const float2 d3 = R[r + UP + al][j];
        if (QUAD) {
          const float2 d4 = f2(w[L + 2 * j - (QUAD ? al : 0)], w[L + 2 * j + 1 - (QUAD ? al : 0)]);
          const float2 d5 = R[r + UP - (QUAD ? al : 0)][j];
          const float2 S24 = __fadd2_rn(d2, d4), D24 = __ffma2_rn(M1, d4, d2);
          const float2 S35 = __fadd2_rn(d3, d5), D35 = __ffma2_rn(M1, d5, d3);
          ax = __ffma2_rn(__fmul2_rn(A, S35), D24, ax);
          ay = __ffma2_rn(__fmul2_rn(B, S24), D35, ay);
          ap = __ffma2_rn(__fmul2_rn(C, S24), S35, ap);
          mn = f2(min3_nan(mn.x, d4.x, d5.x), min3_nan(mn.y, d4.y, d5.y));
        } else {
          const float2 D21 = __ffma2_rn(M1, d1, d2), D31 = __ffma2_rn(M1, d1, d3);
          ax = __ffma2_rn(__fmul2_rn(A, d3), D21, ax);
          ay = __ffma2_rn(__fmul2_rn(B, d2), D31, ay);
          ap = __ffma2_rn(__fmul2_rn(C, d2), d3, ap);
        }
        mn = f2(min3_nan(mn.x, d2.x, d3.x), min3_nan(mn.y, d2.y, d3.y));
      }
      nx[j] = ax;
      ny[j] = ay;
      strip_decide<SECANT, EB == 2>(mn, ax, ay, ap, T, tau2, nu1[j], ku[j], nv1, kv, nz[j], q[j], keep[2 * j],
                                    keep[2 * j + 1]);
    }
    strip_store<OUT, true>(nx, ny, nz, q, keep, np, mp, n, nullptr, f);
    np += f.out_pitch * BPP;
    mp += f.out_pitch;
  }
}

template <int OUT, int FORM, bool SECANT, int K>
__global__ void __launch_bounds__((kWarps + 1) * 32, 1)
    fwd_ms_strip_kernel(const __grid_constant__ ParamBatch pb, const BatchArgs ring, const Globals g) {
  BatchArgs args = ring;
  args.hdr = &pb.hdr;
  args.tile_begin = pb.tile_begin;
  args.frames = pb.frames;
  strip_pipeline<OUT, K, kRows, kWarps, 0, false>(
      args, g, [&](const auto* S, const float4* ctab, const float4* rtab, const StripInfo& f, int warp) {
        ms_band<OUT, FORM, SECANT, K>(S, ctab, rtab, f, warp, g.tau2);
      });
}

template <int OUT, int FORM, bool SECANT>
const void* by_scales(int K) {
  switch (K) {
    case 2: return (const void*)fwd_ms_strip_kernel<OUT, FORM, SECANT, 2>;
    case 3: return (const void*)fwd_ms_strip_kernel<OUT, FORM, SECANT, 3>;
    case 4: return (const void*)fwd_ms_strip_kernel<OUT, FORM, SECANT, 4>;
    case 5: return (const void*)fwd_ms_strip_kernel<OUT, FORM, SECANT, 5>;
    case 6: return (const void*)fwd_ms_strip_kernel<OUT, FORM, SECANT, 6>;
    default: return nullptr;
  }
}

// The kernel of one output type (instantiated in a file each, so that they
// compile side by side), or NULL.
template <int OUT>
const void* by_form(int form, bool secant, int K) {
  if (form == NRM_MS_PAIR) return secant ? by_scales<OUT, NRM_MS_PAIR, true>(K) : by_scales<OUT, NRM_MS_PAIR, false>(K);
  return secant ? by_scales<OUT, NRM_MS_QUAD, true>(K) : by_scales<OUT, NRM_MS_QUAD, false>(K);
}
extern template const void* by_form<NRM_OUT_F32X4>(int, bool, int);
extern template const void* by_form<NRM_OUT_F16X4>(int, bool, int);
extern template const void* by_form<NRM_OUT_OCT16>(int, bool, int);

}  // namespace ms_strip

}  // namespace nrm
