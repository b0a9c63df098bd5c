// decode_dev.cuh -- device code shared by the software decoders and the fused evaluations:
// the BC1 interpolation rule, the BC7 mode descriptors, decode tables, whole-block
// decoders and the SH basis polynomials (Sec. III-B: BC1 / BC7 formats; Sec. II: c(f) = H w(f - p)).
// The constant tables are per translation unit (static); each unit that launches a kernel using
// them uploads its own copy with dec_tables_upload() when a context is created.
#pragma once
#include "bc7_tables.h"
#include "gsc_internal.cuh"

static __constant__ uint32_t d_part2[64];
static __constant__ uint32_t d_part3[64];
static __constant__ uint8_t d_anc2[64];
static __constant__ uint8_t d_anc3a[64];
static __constant__ uint8_t d_anc3b[64];

// ---- BC1 -----------------------------------------------------------------------------
__device__ __forceinline__ int dx5(int x) { return (x << 3) | (x >> 2); }
__device__ __forceinline__ int dx6(int x) { return (x << 2) | (x >> 4); }
// interior entries: the GB300 texture unit's rule (5-bit on codes, 6-bit on expansions)
__device__ __forceinline__ int d_third5(int a, int b) { return ((2 * a + b) * 11) >> 2; }
__device__ __forceinline__ int d_third6(int a, int b) { int A = dx6(a), B = dx6(b); return A + (((B - A) * 321 + 512) >> 10); }
__device__ __forceinline__ int d_half5(int a, int b) { return ((a + b) * 33) >> 3; }
__device__ __forceinline__ int d_half6(int a, int b) { int A = dx6(a), B = dx6(b); return A + (((B - A) * 257 + 256) >> 9); }

// ---- BC7 -----------------------------------------------------------------------------
struct DModeInfo { int ns, pb, rb, isb, cb, ab, epb, spb, ib, ib2; };
__host__ __device__ constexpr DModeInfo d_mode_info(int m) {
  switch (m) {
    case 0: return {3, 4, 0, 0, 4, 0, 1, 0, 3, 0};
    case 1: return {2, 6, 0, 0, 6, 0, 0, 1, 3, 0};
    case 2: return {3, 6, 0, 0, 5, 0, 0, 0, 2, 0};
    case 3: return {2, 6, 0, 0, 7, 0, 1, 0, 2, 0};
    case 4: return {1, 0, 2, 1, 5, 6, 0, 0, 2, 3};
    case 5: return {1, 0, 2, 0, 7, 8, 0, 0, 2, 2};
    case 6: return {1, 0, 0, 0, 7, 7, 1, 0, 4, 0};
    default: return {2, 6, 0, 0, 5, 5, 1, 0, 2, 0};
  }
}

__host__ __device__ __forceinline__ int d_wgt(int ib, int j) {
  if (ib == 2) return (0x402B1500u >> (8 * j)) & 255;
  if (ib == 3) return (int)((0x40372E251B120900ull >> (8 * j)) & 255);
  return j < 8 ? (int)((0x1E1A15110D090400ull >> (8 * j)) & 255) : (int)((0x403C37332F2B2622ull >> (8 * (j - 8))) & 255);
}

#define SH_C0 0.28209479177387814f   /* sqrt(1/(4 pi)) */
#define SH_C1 0.4886025119029199f    /* sqrt(3/(4 pi)) */
#define SH_C2A 1.0925484305920792f   /* sqrt(15/(4 pi)) */
#define SH_C2B 0.31539156525252005f  /* sqrt(5/(16 pi)) */
#define SH_C2C 0.5462742152960396f   /* sqrt(15/(16 pi)) */
#define SH_C3A 0.5900435899266435f   /* sqrt(35/(32 pi)) */
#define SH_C3B 2.890611442640554f    /* sqrt(105/(4 pi)) */
#define SH_C3C 0.4570457994644658f   /* sqrt(21/(32 pi)) */
#define SH_C3D 0.3731763325901154f   /* sqrt(7/(16 pi)) */
#define SH_C3E 1.445305721320277f    /* sqrt(105/(16 pi)) */

// ---- whole-block BC7 decode -----------------------------------------------------------------
// Every mode takes the same code; what differs between them is a row of constants. A row is a mode, with the rotation
// and the index selection for modes 4 and 5: rows 0-3, 6 and 7 their modes, 8 + rotation + 4 selection mode 4, 16 +
// rotation mode 5, 20 the reserved mode. A rotation puts the alpha values in the place of one channel: the row names
// two channels x1, x2 that take the colour index and one, y, that takes its own, and how they go back.
// A window is a position in the block: its word in bits 7-9 (as an offset of the words' rows), its bit in bits 0-4.
struct DecTables {
  // 0: windows of the endpoint fields of x1, x2, y and of the p-bits
  // 1: windows of the indices of x and of y, one bit early; shift and mask of the partition
  // 2: first partition entry; of an endpoint code of x1 and x2: mask, 16 - bits, 2 bits
  // 3: expansion of a pair of codes c, c' << 16, with p-bits p, p' << 16: (c * [0] + p * [1]) >> [2]; [3] p-bit mask
  //    (top bit: one p-bit for both endpoints)
  // 4: of y: code mask, 16 - bits, expansion [0] and [2]
  // 5: index widths of x and of y, their first weights
  // 6: index masks of x and of y, byte selector of the texel, whether y takes the index of x
  uint4 row[7][24];
  uint2 part[130];     // subset of each texel, two bits each; the anchors after texel 0, plus one, in ascending bytes
  uint64_t above[66];  // [q]: bits q - 1 and up; [0] none
  uint32_t wt[48];     // [width - 2][index]: 256 - 4 w | 4 w << 16
};
static __device__ DecTables g_dec;

static uint32_t dec_window(int pos) { return (uint32_t)((pos >> 5) << 7 | (pos & 31)); }

static void dec_row(DecTables& T, int row, int mode, int rot, int isbv) {
  const DModeInfo M = d_mode_info(mode);
  const int cstart = mode + 1 + M.pb + M.rb + M.isb, astart = cstart + 6 * M.ns * M.cb, pstart = astart + 2 * M.ns * M.ab;
  const int istart = pstart + (M.epb ? 2 * M.ns : (M.spb ? M.ns : 0)), second = istart + 16 * M.ib - 1;
  const int chan[4] = {cstart, cstart + 2 * M.ns * M.cb, cstart + 4 * M.ns * M.cb, astart};
  const int hp = M.epb | M.spb, n = M.cb + hp, ycb = rot ? M.ab : M.cb, yn = rot ? M.ab : n, yhp = rot ? 0 : hp;
  const int cbits = isbv ? M.ib2 : M.ib, ybits = rot ? (isbv ? M.ib : M.ib2) : cbits;
  const int cpos = isbv ? second : istart, ypos = rot ? (isbv ? istart : second) : cpos;
  static const uint32_t out[4] = {0x4510u, 0x4105u, 0x4150u, 0x4510u};
  const uint32_t mul = (1u << n) + 1u, ymul = (1u << yn) + 1u, cm = (1u << M.cb) - 1u, ycm = (1u << ycb) - 1u;
  T.row[0][row] = make_uint4(dec_window(chan[rot == 1 ? 1 : 0]), dec_window(chan[rot == 1 || rot == 2 ? 2 : 1]),
                             dec_window(chan[rot ? 3 : 2]), dec_window(pstart));
  T.row[1][row] = make_uint4(dec_window(cpos - 1), dec_window(ypos - 1), (uint32_t)mode + 1, (1u << M.pb) - 1u);
  T.row[2][row] = make_uint4(M.ns == 1 ? 0 : (M.ns == 2 ? 1 : 65), cm, 16 - M.cb, 2 * M.cb);
  T.row[3][row] = make_uint4(mul << hp, mul, 2 * n - 8, M.epb ? (1u << (2 * M.ns)) - 1u : (M.spb ? 0x80000000u : 0u));
  T.row[4][row] = make_uint4(ycm, 16 - ycb, ymul << yhp, 2 * yn - 8);
  T.row[5][row] = make_uint4(cbits, ybits, 16 * (cbits - 2), 16 * (ybits - 2));
  T.row[6][row] = make_uint4((1u << cbits) - 1u, (1u << ybits) - 1u, out[rot], rot == 0);
}

static void dec_tables_build(DecTables& T) {
  memset(&T, 0, sizeof(T));
  for (int m = 0; m < 8; m++)
    if (m != 4 && m != 5) dec_row(T, m, m, 0, 0);
  for (int r = 0; r < 4; r++) {
    dec_row(T, 8 + r, 4, r, 0);
    dec_row(T, 12 + r, 4, r, 1);
    dec_row(T, 16 + r, 5, r, 0);
  }
  // the reserved mode: endpoints expand to 0, and so every texel is 0
  dec_row(T, 20, 6, 0, 0);
  T.row[3][20] = make_uint4(0, 0, 0, 0);
  T.row[4][20].z = 0;
  for (int p = 0; p < 64; p++) {
    const uint32_t a = kBC7Anchor3a[p] + 1u, b = kBC7Anchor3b[p] + 1u;
    T.part[1 + p] = make_uint2(bc7_pack_part2(p), kBC7Anchor2[p] + 1u);
    T.part[65 + p] = make_uint2(bc7_pack_part3(p), a < b ? a | b << 8 : b | a << 8);
  }
  for (int q = 1; q < 66; q++) T.above[q] = q > 64 ? 0ull : ~0ull << (q - 1);
  for (int ib = 2; ib <= 4; ib++)
    for (int j = 0; j < 1 << ib; j++) {
      const uint32_t w = (uint32_t)d_wgt(ib, j);
      T.wt[16 * (ib - 2) + j] = (256u - 4u * w) | (4u * w << 16);
    }
}

static cudaError_t dec_tables_upload() {
  uint32_t p2[64], p3[64];
  for (int p = 0; p < 64; p++) { p2[p] = bc7_pack_part2(p); p3[p] = bc7_pack_part3(p); }
  static DecTables T;
  dec_tables_build(T);
  cudaError_t e;
  if ((e = cudaMemcpyToSymbol(g_dec, &T, sizeof(T))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(d_part2, p2, sizeof(p2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(d_part3, p3, sizeof(p3))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(d_anc2, kBC7Anchor2, 64)) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(d_anc3a, kBC7Anchor3a, 64)) != cudaSuccess) return e;
  return cudaMemcpyToSymbol(d_anc3b, kBC7Anchor3b, 64);
}

__device__ __forceinline__ void load_tables(DecTables* s) {
  for (int i = threadIdx.x; i < (int)(sizeof(DecTables) / 16); i += blockDim.x)
    reinterpret_cast<uint4*>(s)[i] = reinterpret_cast<const uint4*>(&g_dec)[i];
}

// A warp's scratch, aligned to 1024 bytes: the endpoints of subset s of lane l's block at 256 s + 8 l, word r of the
// block at 1024 + 128 r + 4 l (words 4 and 5 are zero). A lane uses its own columns only.
#define DEC_AREA 2048
__device__ __forceinline__ uint32_t dec_ld(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint2 dec_ld2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ void dec_st(uint32_t a, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void dec_st2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ uint32_t dec_area(void* area) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(area), l = 4 * (threadIdx.x & 31);
  dec_st(a + 1024 + 4 * 128 + l, 0u);
  dec_st(a + 1024 + 5 * 128 + l, 0u);
  return a;
}
__device__ __forceinline__ uint32_t dec_win(uint32_t words, uint32_t at) {
  const uint32_t a = (at & 0x380u) | words;
  return __funnelshift_r(dec_ld(a), dec_ld(a + 128), at);
}
// 16 indices of `bits` bits from a window one bit early: texel 0's index is one bit short (its top bit is 0)
__device__ __forceinline__ uint64_t dec_indices(uint32_t words, uint32_t at, uint32_t mask) {
  const uint32_t a = (at & 0x380u) | words, w1 = dec_ld(a + 128);
  const uint32_t lo = __funnelshift_r(dec_ld(a), w1, at), hi = __funnelshift_r(w1, dec_ld(a + 256), at);
  return (uint64_t)hi << 32 | ((lo & ~mask) | ((lo >> 1) & (mask >> 1)));
}
// c + a.lo * b.byte[0] + a.hi * b.byte[1], or of bytes 2 and 3
__device__ __forceinline__ uint32_t dec_dp_lo(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("dp2a.lo.u32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(128u));
  return d;
}
__device__ __forceinline__ uint32_t dec_dp_hi(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("dp2a.hi.u32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(128u));
  return d;
}

// Texel t of the block comes out as r | g << 8 | b << 16 (the top byte is unspecified). An interpolation
// ((64 - w) e0 + w e1 + 32) >> 6 is byte 1 of a two-term product with the weights scaled by 4.
// 551 instructions per block with its rows' stores, against 976 with the fields located by arithmetic on 64-bit halves
// and alpha interpolated beside every texel. Weights computed instead of looked up cost 62 instructions more and take
// as long.
__device__ __forceinline__ void bc7_block(uint4 w, uint32_t (&tx)[16], const DecTables& S, uint32_t area) {
  const uint32_t lane = threadIdx.x & 31, words = area + 1024 + 4 * lane, ep = area + 8 * lane;
  dec_st(words, w.x);
  dec_st(words + 128, w.y);
  dec_st(words + 256, w.z);
  dec_st(words + 384, w.w);
  const int mode = __ffs((int)((w.x & 255u) | 256u)) - 1;
  const int row = mode == 4 ? 8 + (int)((w.x >> 5) & 7u) : mode == 5 ? 16 + (int)((w.x >> 6) & 3u) : mode == 8 ? 20 : mode;
  const uint4 R0 = S.row[0][row], R1 = S.row[1][row], R2 = S.row[2][row], R3 = S.row[3][row], R4 = S.row[4][row];
  const uint4 R5 = S.row[5][row], R6 = S.row[6][row];
  const uint2 part = S.part[R2.x + ((w.x >> R1.z) & R1.w)];
  // endpoints
  const uint32_t f1 = dec_win(words, R0.x), f2 = dec_win(words, R0.y), fy = dec_win(words, R0.z);
  uint32_t pb = dec_win(words, R0.w);
  pb = (R3.w >> 31) ? (0xFC30u >> (4 * (pb & 3u))) & 15u : pb & R3.w;
  const uint32_t ch = R2.y << 16, yh = R4.x << 16;
#pragma unroll
  for (int s = 0; s < 3; s++) {
    const uint32_t pp = (((pb >> (2 * s)) & 1u) | ((pb << (15 - 2 * s)) & 0x10000u)) * R3.y;
    const uint32_t a = f1 >> (s * R2.w), b = f2 >> (s * R2.w), y = fy >> (s * R2.w);
    const uint32_t za = (((a & R2.y) | ((a << R2.z) & ch)) * R3.x + pp) >> R3.z;
    const uint32_t zb = (((b & R2.y) | ((b << R2.z) & ch)) * R3.x + pp) >> R3.z;
    const uint32_t zy = (((y & R4.x) | ((y << R4.y) & yh)) * R4.z + pp) >> R4.w;
    dec_st2(ep + 256 * s, __byte_perm(za, zb, 0x6420), __byte_perm(zy, zy, 0x2020));
  }
  // indices at a fixed width per texel: a zero bit goes in at the top of each anchor's
  uint64_t c = dec_indices(words, R1.x, R6.x);
  c += c & S.above[(part.y & 255u) * R5.x];
  c += c & S.above[(part.y >> 8) * R5.x];
  uint64_t v = dec_indices(words, R1.y, R6.y);
  if (R6.w) v = c;
  uint32_t cw = (uint32_t)c, vw = (uint32_t)v;
  const uint32_t c8 = __funnelshift_rc(cw, (uint32_t)(c >> 32), 8 * R5.x), v8 = __funnelshift_rc(vw, (uint32_t)(v >> 32), 8 * R5.y);
#pragma unroll
  for (int t = 0; t < 16; t++) {
    if (t == 8) { cw = c8; vw = v8; }
    const uint32_t wc = S.wt[(cw & R6.x) | R5.z], wy = S.wt[(vw & R6.y) | R5.w];
    cw >>= R5.x;
    vw >>= R5.y;
    const uint2 e = dec_ld2(((t < 4 ? part.x << (8 - 2 * t) : part.x >> (2 * t - 8)) & 0x300u) + ep);
    tx[t] = __byte_perm(__byte_perm(dec_dp_lo(wc, e.x), dec_dp_hi(wc, e.x), 0x0051u), dec_dp_lo(wy, e.y), R6.z);
  }
}

__device__ __forceinline__ void bc1_block(uint2 w, uint32_t (&tx)[16]) {
  const uint32_t c0 = w.x & 0xFFFF, c1 = w.x >> 16;
  const int r0 = c0 >> 11, g0 = (c0 >> 5) & 63, b0 = c0 & 31;
  const int r1 = c1 >> 11, g1 = (c1 >> 5) & 63, b1 = c1 & 31;
  const uint32_t p0 = dx5(r0) | (dx6(g0) << 8) | (dx5(b0) << 16) | 0xFF000000u;
  const uint32_t p1 = dx5(r1) | (dx6(g1) << 8) | (dx5(b1) << 16) | 0xFF000000u;
  uint32_t p2, p3;
  if (c0 > c1) {
    p2 = d_third5(r0, r1) | (d_third6(g0, g1) << 8) | (d_third5(b0, b1) << 16) | 0xFF000000u;
    p3 = d_third5(r1, r0) | (d_third6(g1, g0) << 8) | (d_third5(b1, b0) << 16) | 0xFF000000u;
  } else {
    p2 = d_half5(r0, r1) | (d_half6(g0, g1) << 8) | (d_half5(b0, b1) << 16) | 0xFF000000u;
    p3 = 0u;
  }
#pragma unroll
  for (int t = 0; t < 16; t++) {
    const uint32_t j = (w.y >> (2 * t)) & 3;
    tx[t] = (j & 2) ? ((j & 1) ? p3 : p2) : ((j & 1) ? p1 : p0);
  }
}

// 2^23 + q as float for byte c of v (0x4B0000qq)
__device__ __forceinline__ float u23(uint32_t v, int c) {
  return __uint_as_float(__byte_perm(v, 0x4B000000u, 0x7650u | (uint32_t)c));
}

// SH basis polynomials without their constants (the constants, with their signs, are folded
// into the per-coefficient dequantisation factors s_k / 255 * C_k), for two directions at once.
// The directions are unit vectors, so x^2 + y^2 + z^2 = 1 shortens the band-2 and band-3 terms:
// 2zz - xx - yy = 3zz - 1, 4zz - xx - yy = 5zz - 1, 2zz - 3xx - 3yy = 5zz - 3.
__device__ __forceinline__ void sh_poly2(float2 x, float2 y, float2 z, float2 (&P)[16]) {
  const float2 xx = __fmul2_rn(x, x), yy = __fmul2_rn(y, y), zz = __fmul2_rn(z, z);
  const float2 xy = __fmul2_rn(x, y), yz = __fmul2_rn(y, z), xz = __fmul2_rn(x, z);
  const float2 m1 = make_float2(-1.f, -1.f), five = make_float2(5.f, 5.f);
  const float2 xmy = __ffma2_rn(yy, m1, xx);                                        // xx - yy
  const float2 t5 = __ffma2_rn(five, zz, m1);                                        // 5zz - 1
  P[0] = make_float2(1.f, 1.f);
  P[1] = y; P[2] = z; P[3] = x;
  P[4] = xy; P[5] = yz; P[6] = __ffma2_rn(make_float2(3.f, 3.f), zz, m1); P[7] = xz; P[8] = xmy;  // 3zz - 1
  P[9] = __fmul2_rn(y, __ffma2_rn(make_float2(3.f, 3.f), xx, make_float2(-yy.x, -yy.y)));      // y (3xx - yy)
  P[10] = __fmul2_rn(xy, z);
  P[11] = __fmul2_rn(y, t5);
  P[12] = __fmul2_rn(z, __ffma2_rn(five, zz, make_float2(-3.f, -3.f)));                 // z (5zz - 3)
  P[13] = __fmul2_rn(x, t5);
  P[14] = __fmul2_rn(z, xmy);
  P[15] = __fmul2_rn(x, __ffma2_rn(make_float2(-3.f, -3.f), yy, xx));                  // x (xx - 3yy)
}

static __constant__ float c_shc[16] = {SH_C0, -SH_C1, SH_C1, -SH_C1, SH_C2A, -SH_C2A, SH_C2B, -SH_C2A, SH_C2C,
                                -SH_C3A, SH_C3B, -SH_C3C, SH_C3D, -SH_C3C, SH_C3E, -SH_C3A};

