// stage.cuh -- layout-D staging shared by the group encoders (Sec. IV-B, Fig. SetupD): a warp turns two groups of
// 16 slots into 32 blocks of 16 texels.
//
// Slot t of a group is the Gaussian perm[slot] (a padding slot repeats the group's last valid slot before it; none:
// texel 128); its 48 floats are quantised (Sec. V-A) and coefficient k goes to texel t of block (group, k), packed
// r | g << 8 | b << 16 at tex[t][block].
//
// The rows lie anywhere in memory, so the time is that of the reads: twelve neighbouring lanes read one row of 192
// bytes in 16-byte pieces, whole sectors at a time. One lane per row instead read half a sector per request and
// found the other half gone from L1: 3M Gaussians in 390 us, against 170 us. The quantised bytes cross over
// in shared memory; the odd row strides keep every access but the pieces' own free of conflicts.
#pragma once
#include "gsc_internal.cuh"

#define STAGE_RAW (32 * 13)  // words of crossing space per warp

// The scales spread over a row's 48 floats, and their reciprocals.
struct StageScale {
  float4 s[12], r[12];
  int fast;  // every scale is in [2^-60, 2^60]
};

// by one warp
__device__ __forceinline__ void stage_scales(StageScale& T, const float* __restrict__ scales) {
  const int lane = threadIdx.x & 31;
  const float s = scales[lane & 15], r = __frcp_rn(s);
  const bool fast = __all_sync(0xFFFFFFFFu, s >= 0x1p-60f && s <= 0x1p60f);
  if (lane < 16)
    for (int c = 0; c < 3; c++) {
      reinterpret_cast<float*>(T.s)[3 * lane + c] = s;
      reinterpret_cast<float*>(T.r)[3 * lane + c] = r;
    }
  if (lane == 0) T.fast = fast;
}

// gsc_quant1 without the divide, r = RN(1 / s): the code is the low byte of the result. Beyond +-0.503 s and 0.499 s
// the code is 0 or 255 (x / s * 255 is past -128.2 or 127.2 and rounds to -128 or 127 at least), so x is clamped there
// (NaN to the lower end, as there). The quotient is rounded correctly by Markstein's correction (IBM J. Res. Dev. 34,
// 1990): q0 = RN(x r) is off by at most 1.5 ulp; a first residual step brings that below one, where the second residual
// is exact and RN(q + r e) = RN(x / s). Residuals that underflow belong to |x| < 2^-78, whose code is 128 in any
// case. Adding 1.5 * 2^23 + 128 rounds to an integer, ties to even, as rint does.
__device__ __forceinline__ uint32_t stage_quant(float x, float s, float r) {
  x = fminf(fmaxf(x, s * -0.503f), s * 0.499f);
  float q = __fmul_rn(x, r);
  q = __fmaf_rn(__fmaf_rn(-q, s, x), r, q);
  q = __fmaf_rn(__fmaf_rn(-q, s, x), r, q);
  return __float_as_uint(__fadd_rn(__fmul_rn(q, 255.0f), 12583040.0f));
}
__device__ __forceinline__ uint32_t stage_quant4(float4 x, float4 s, float4 r) {
  const uint32_t lo = __byte_perm(stage_quant(x.x, s.x, r.x), stage_quant(x.y, s.y, r.y), 0x0040);
  const uint32_t hi = __byte_perm(stage_quant(x.z, s.z, r.z), stage_quant(x.w, s.w, r.w), 0x0040);
  return __byte_perm(lo, hi, 0x5410);
}

// Four texels of three bytes from three words, STEP words apart.
template <int STEP>
__device__ __forceinline__ void stage_unpack(uint32_t a, uint32_t b, uint32_t c, uint32_t* to) {
  to[0] = a & 0xFFFFFFu;
  to[STEP] = __funnelshift_r(a, b, 24) & 0xFFFFFFu;
  to[2 * STEP] = __funnelshift_r(b, c, 16) & 0xFFFFFFu;
  to[3 * STEP] = c >> 8;
}

// By one warp: groups g0 and g0 + 1 (those below n_groups) into the 32 columns of tex. STRIDE: words between texel
// rows, one more than a multiple of 32. raw: STAGE_RAW words. STEPS: eighths of rows read ahead, times 8 rows
// (4: all in flight together; 1: a quarter of the code).
template <int STRIDE, int STEPS = 4>
__device__ __forceinline__ void stage_groups(const float* __restrict__ sh, const int32_t* __restrict__ perm,
                                             const StageScale& T, int64_t g0, int64_t n_groups,
                                             uint32_t (*tex)[STRIDE], uint32_t* raw) {
  int lane = threadIdx.x & 31;
  asm volatile("" : "+r"(lane));  // what derives from it is not kept in registers between calls
  const int t = lane & 15;
  const int64_t g = g0 + (lane >> 4);
  const int32_t o = g < n_groups ? __ldg(perm + g * 16 + t) : -1;
  // last valid slot at or before t inside this half-warp's group
  const unsigned upto = __ballot_sync(0xFFFFFFFFu, o >= 0) & (0xFFFFu << (lane & 16)) & (0xFFFFFFFFu >> (31 - lane));
  const int32_t got = __shfl_sync(0xFFFFFFFFu, o, upto ? 31 - __clz(upto) : lane);
  const int32_t src = upto ? got : -1;
  if (T.fast) {
    // piece 32 b + lane of the eight rows 8 a .. 8 a + 7
    const int p0 = lane % 12, p1 = (lane + 8) % 12, p2 = (lane + 4) % 12;
    const int r0 = lane / 12, r1 = (lane + 32) / 12, r2 = (lane + 64) / 12;
#pragma unroll 1
    for (int a0 = 0; a0 < 4; a0 += STEPS) {
      float4 x[STEPS][3];
#pragma unroll
      for (int a = 0; a < STEPS; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
          const int p = b == 0 ? p0 : b == 1 ? p1 : p2, row = 8 * (a0 + a) + (b == 0 ? r0 : b == 1 ? r1 : r2);
          const int32_t from = __shfl_sync(0xFFFFFFFFu, src, row);
          x[a][b] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (from >= 0) x[a][b] = __ldg(reinterpret_cast<const float4*>(sh + (int64_t)from * 48) + p);
        }
#pragma unroll
      for (int b = 0; b < 3; b++) {
        const int p = b == 0 ? p0 : b == 1 ? p1 : p2, row = 8 * a0 + (b == 0 ? r0 : b == 1 ? r1 : r2);
        const float4 s = T.s[p], r = T.r[p];
#pragma unroll
        for (int a = 0; a < STEPS; a++) raw[(row + 8 * a) * 13 + p] = stage_quant4(x[a][b], s, r);
      }
    }
  } else {
    uint8_t* q = reinterpret_cast<uint8_t*>(raw + lane * 13);
#pragma unroll 1
    for (int e = 0; e < 48; e++)
      q[e] = src < 0 ? (uint8_t)128
                     : (uint8_t)gsc_quant1(__ldg(sh + (int64_t)src * 48 + e), reinterpret_cast<const float*>(T.s)[e]);
  }
  __syncwarp();
  const uint32_t* q = raw + lane * 13;
#pragma unroll
  for (int j = 0; j < 4; j++) stage_unpack<1>(q[3 * j], q[3 * j + 1], q[3 * j + 2], &tex[t][(lane & 16) + 4 * j]);
  __syncwarp();
}

// A block's 48 bytes of texels into column `col` of a tile (its first row's word; STRIDE words between rows). wide: the
// array starts on a 16-byte boundary.
template <int STRIDE>
__device__ __forceinline__ void stage_texels(const uint8_t* __restrict__ p, bool wide, uint32_t* col) {
  if (wide) {
    const uint4* q = reinterpret_cast<const uint4*>(p);
    const uint4 a = __ldg(q), b = __ldg(q + 1), c = __ldg(q + 2);
    stage_unpack<STRIDE>(a.x, a.y, a.z, col);
    stage_unpack<STRIDE>(a.w, b.x, b.y, col + 4 * STRIDE);
    stage_unpack<STRIDE>(b.z, b.w, c.x, col + 8 * STRIDE);
    stage_unpack<STRIDE>(c.y, c.z, c.w, col + 12 * STRIDE);
  } else {
#pragma unroll 1
    for (int t = 0; t < 16; t++)
      col[t * STRIDE] = (uint32_t)p[3 * t] | ((uint32_t)p[3 * t + 1] << 8) | ((uint32_t)p[3 * t + 2] << 16);
  }
}
