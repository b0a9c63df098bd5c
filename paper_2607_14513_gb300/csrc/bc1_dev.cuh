// bc1_dev.cuh -- BC1 encoder device code (Sec. III-A with P = 16, Q = 2; Sec. III-B), shared
// by the single-scene kernels (bc1.cu) and the persistent multi-scene kernel (bc7.cu).
#pragma once
#include "gsc_internal.cuh"
#include "stage.cuh"

// Per channel value: best (a, b) code pair for a constant block, packed a | b << 8. Each
// translation unit that includes this header has its own copy, filled at context creation
// from bc1_const_tables().
static __constant__ uint16_t c_const5[256];
static __constant__ uint16_t c_const6[256];
void bc1_const_tables(uint16_t* t5, uint16_t* t6);

__device__ __forceinline__ int ex5(int x) { return (x << 3) | (x >> 2); }
__device__ __forceinline__ int ex6(int x) { return (x << 2) | (x >> 4); }
// Interior entries: measured GB300 texture-unit rule (5-bit on codes, 6-bit on expansions).
__device__ __forceinline__ int third5(int a, int b) { return ((2 * a + b) * 11) >> 2; }
__device__ __forceinline__ int third6(int a, int b) {
  int A = ex6(a), B = ex6(b);
  return A + (((B - A) * 321 + 512) >> 10);
}

struct Bc1Res {
  uint32_t sse;
  uint32_t idx;   // 2 bits per texel
  uint16_t c0, c1;
};

// An entry P gives a texel the error |v|^2 - 510 (v_r + v_g + v_b) + |P|^2 + 2 v.(255 - P): base is the sum of the
// first two terms over a block, which no entry changes.
//
// Indices and error of a pair: keys 4 (|p_j|^2 + 2 v.(255 - p_j)) + j, whose minimum gives the first entry of least
// error (j = key & 3).
__device__ __forceinline__ Bc1Res bc1_eval_k(const uint32_t (&tx)[16], int base, uint32_t a, uint32_t b) {
  Bc1Res r;
  r.c0 = (uint16_t)max(a, b);
  r.c1 = (uint16_t)min(a, b);
  r.idx = 0;
  const int ra = r.c0 >> 11, ga = (r.c0 >> 5) & 63, ba = r.c0 & 31;
  const int rb = r.c1 >> 11, gb = (r.c1 >> 5) & 63, bb = r.c1 & 31;
  const uint32_t P0 = (uint32_t)ex5(ra) | ((uint32_t)ex6(ga) << 8) | ((uint32_t)ex5(ba) << 16);
  const int q0 = 4 * (int)__dp4a(P0, P0, 0u);
  int s = 0;
  if (r.c0 == r.c1) {
#pragma unroll
    for (int t = 0; t < 16; t++) s += (int)__dp4a(tx[t], ~P0, 0u);
    r.sse = (uint32_t)(base + 4 * q0 + 2 * s);
    return r;
  }
  const uint32_t P1 = (uint32_t)ex5(rb) | ((uint32_t)ex6(gb) << 8) | ((uint32_t)ex5(bb) << 16);
  const uint32_t P2 = (uint32_t)third5(ra, rb) | ((uint32_t)third6(ga, gb) << 8) | ((uint32_t)third5(ba, bb) << 16);
  const uint32_t P3 = (uint32_t)third5(rb, ra) | ((uint32_t)third6(gb, ga) << 8) | ((uint32_t)third5(bb, ba) << 16);
  const int q1 = 4 * (int)__dp4a(P1, P1, 0u) + 1, q2 = 4 * (int)__dp4a(P2, P2, 0u) + 2, q3 = 4 * (int)__dp4a(P3, P3, 0u) + 3;
#pragma unroll
  for (int t = 0; t < 16; t++) {
    const uint32_t v = tx[t];
    const int e0 = q0 + 8 * (int)__dp4a(v, ~P0, 0u), e1 = q1 + 8 * (int)__dp4a(v, ~P1, 0u);
    const int e2 = q2 + 8 * (int)__dp4a(v, ~P2, 0u), e3 = q3 + 8 * (int)__dp4a(v, ~P3, 0u);
    const int key = min(__vimin3_s32(e0, e1, e2), e3);
    s += key;  // below 16 * 4 * (2^18 + 2^19)
    r.idx = __funnelshift_r(r.idx, (uint32_t)key, 2);
  }
  s -= __popc(r.idx & 0x55555555u) + 2 * __popc(r.idx & 0xAAAAAAAAu);
  r.sse = (uint32_t)(base + (s >> 2));
  return r;
}

// clamp(round_div(num, den), 0, 255), half away from zero, for |num| < 2^23 and 0 < den < 2^15; rcp: 1 / (2 den),
// rounded. A negative numerator clamps to 0; the float quotient of floor((2 num + den) / (2 den)) is off by at most
// one, and one exact step each way lands on it.
__device__ __forceinline__ int bc1_ratio(int num, int den, float rcp) {
  if (num < 0) return 0;
  const int D = 2 * den, N = 2 * num + den;
  if (N >= 256 * D) return 255;
  int q = min((int)((float)N * rcp), 255);
  if (q * D > N) q--;
  if ((q + 1) * D <= N) q++;
  return min(q, 255);
}

__device__ __forceinline__ int q5(int v) { return (v * 31 + 127) / 255; }
__device__ __forceinline__ int q6(int v) { return (v * 63 + 127) / 255; }
__device__ __forceinline__ uint32_t pack565(int r, int g, int b) { return (q5(r) << 11) | (q6(g) << 5) | q5(b); }

// A warp's blocks: texel t of block b at tex[t][b], packed r | g << 8 | b << 16 (top byte 0).
template <int BPW>
struct Bc1Warp {
  uint32_t tex[16][BPW + 1];
  union {
    uint32_t raw[STAGE_RAW];  // while the texels are staged
    struct {
      uint32_t pair[BPW];   // best endpoint pair so far, c0 | c1 << 16 (c0 >= c1)
      uint32_t err[BPW];    // its error
      int base[BPW];        // sum over the texels of |v|^2 - 510 (v_r + v_g + v_b)
      uint16_t stack[BPW];  // blocks with a neighbourhood step to do: block | steps done << 8
    };
  };
};

// The channels of four texels apart, a byte each.
__device__ __forceinline__ void bc1_planes(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t (&p)[3]) {
  const uint32_t x = __byte_perm(a, b, 0x5140), y = __byte_perm(c, d, 0x5140);
  p[0] = __byte_perm(x, y, 0x5410);
  p[1] = __byte_perm(x, y, 0x7632);
  p[2] = __byte_perm(__byte_perm(a, b, 0x0062), __byte_perm(c, d, 0x0062), 0x5410);
}

// Of a block: the pair before the neighbourhood search (constant blocks: the final one), its error, base, and the
// error against mid-grey; whether there is a search. Sums over the texels are byte dot products of the planes.
__device__ __forceinline__ bool bc1_start(const uint32_t (&tx)[16], uint32_t& pair, uint32_t& err, int& base, uint32_t& grey) {
  uint32_t pl[4][3];
  int s1[3] = {0, 0, 0}, sq = 0;
#pragma unroll
  for (int w = 0; w < 4; w++) {
    bc1_planes(tx[4 * w], tx[4 * w + 1], tx[4 * w + 2], tx[4 * w + 3], pl[w]);
#pragma unroll
    for (int c = 0; c < 3; c++) {
      s1[c] = (int)__dp4a(pl[w][c], 0x01010101u, (uint32_t)s1[c]);
      sq = (int)__dp4a(pl[w][c], pl[w][c], (uint32_t)sq);
    }
  }
  const int sum = s1[0] + s1[1] + s1[2];
  base = sq - 510 * sum;
  grey = (uint32_t)(sq - 256 * sum + 48 * 16384);
  // red and blue in 16-bit halves, green of two texels
  uint32_t lrb = 0x00FF00FFu, hrb = 0u, lg = 0x00FF00FFu, hg = 0u;
#pragma unroll
  for (int t = 0; t < 16; t += 2) {
    const uint32_t a = tx[t] & 0x00FF00FFu, b = tx[t + 1] & 0x00FF00FFu, g = __byte_perm(tx[t], tx[t + 1], 0x3531);
    lrb = __vminu2(__vminu2(lrb, a), b);
    hrb = __vmaxu2(__vmaxu2(hrb, a), b);
    lg = __vminu2(lg, g);
    hg = __vmaxu2(hg, g);
  }
  const int lo[3] = {(int)(lrb & 0xFFFFu), (int)min(lg & 0xFFFFu, lg >> 16), (int)(lrb >> 16)};
  const int hi[3] = {(int)(hrb & 0xFFFFu), (int)max(hg & 0xFFFFu, hg >> 16), (int)(hrb >> 16)};
  if (lo[0] == hi[0] && lo[1] == hi[1] && lo[2] == hi[2]) {
    const uint32_t pr = c_const5[lo[0]], pg = c_const6[lo[1]], pb = c_const5[lo[2]];
    const uint32_t c0 = ((pr & 255) << 11) | ((pg & 255) << 5) | (pb & 255);
    const uint32_t c1 = ((pr >> 8) << 11) | ((pg >> 8) << 5) | (pb >> 8);
    pair = max(c0, c1) | (min(c0, c1) << 16);
    err = 0u;
    return false;
  }
  // covariances (scaled by 16) of the channel of largest range (the first) with each other channel; its own entry
  // is positive
  int rg = 0, rb = 0, gb = 0;
#pragma unroll
  for (int w = 0; w < 4; w++) {
    rg = (int)__dp4a(pl[w][0], pl[w][1], (uint32_t)rg);
    rb = (int)__dp4a(pl[w][0], pl[w][2], (uint32_t)rb);
    gb = (int)__dp4a(pl[w][1], pl[w][2], (uint32_t)gb);
  }
  rg = 16 * rg - s1[0] * s1[1];
  rb = 16 * rb - s1[0] * s1[2];
  gb = 16 * gb - s1[1] * s1[2];
  const int dr = hi[0] - lo[0], dg = hi[1] - lo[1], db = hi[2] - lo[2];
  const bool g_ref = dg > dr, b_ref = db > max(dr, dg);
  const int cov[3] = {b_ref ? rb : g_ref ? rg : 1, b_ref ? gb : g_ref ? 1 : rg, b_ref ? 1 : g_ref ? gb : rb};
  int e0[3], e1[3];
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const int d = (hi[c] - lo[c]) >> 4, a = hi[c] - d, b = lo[c] + d;
    e0[c] = cov[c] < 0 ? b : a;
    e1[c] = cov[c] < 0 ? a : b;
  }
  // the diagonal, then two least-squares refinements: weights (3,0,2,1)/3 on c0 for indices 0..3
  Bc1Res best;
#pragma unroll 1
  for (int it = 0;; it++) {
    const Bc1Res r = bc1_eval_k(tx, base, pack565(e0[0], e0[1], e0[2]), pack565(e1[0], e1[1], e1[2]));
    if (it == 0 || r.sse < best.sse) best = r; else break;
    if (it == 2 || best.c0 == best.c1) break;
    int sa = 0, saa = 0, sav[3] = {0, 0, 0};
#pragma unroll
    for (int w = 0; w < 4; w++) {
      uint32_t j = (best.idx >> (8 * w)) & 255u;
      j = (j | (j << 4)) & 0x0F0Fu;
      j = (j | (j << 2)) & 0x3333u;
      const uint32_t a = __byte_perm(0x01020003u, 0u, j);
      sa = (int)__dp4a(a, 0x01010101u, (uint32_t)sa);
      saa = (int)__dp4a(a, a, (uint32_t)saa);
#pragma unroll
      for (int c = 0; c < 3; c++) sav[c] = (int)__dp4a(a, pl[w][c], (uint32_t)sav[c]);
    }
    const int sbb = 144 - 6 * sa + saa, sab = 3 * sa - saa, det = saa * sbb - sab * sab;  // weights a and 3 - a
    if (det == 0) break;
    const float rcp = __frcp_rn((float)(2 * det));
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const int sbv = 3 * s1[c] - sav[c];
      e0[c] = bc1_ratio(3 * (sbb * sav[c] - sab * sbv), det, rcp);
      e1[c] = bc1_ratio(3 * (saa * sbv - sab * sav[c]), det, rcp);
    }
  }
  pair = (uint32_t)best.c0 | ((uint32_t)best.c1 << 16);
  err = best.sse;
  return true;
}

// c + a.lo * b.byte[0] + a.hi * b.byte[1], or of bytes 2 and 3: signed halves, unsigned bytes
__device__ __forceinline__ int bc1_dp2_lo(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp2a.lo.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ int bc1_dp2_hi(uint32_t a, uint32_t b, int c) {
  int d;
  asm("dp2a.hi.s32.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// A channel of an entry from x to y: the entry's error changes by (y - x) (x + y) - 2 (y - x) v, as halves for
// bc1_dp2 with the bytes v, 1 (both below 2^13 in size).
__device__ __forceinline__ uint32_t bc1_move(int x, int y) {
  const int d = y - x;
  return __byte_perm((uint32_t)(-2 * d), (uint32_t)(d * (x + y)), 0x5410);
}

// One neighbourhood step: the best of the pairs a step of one code away in one channel of one endpoint (order: c0,
// c1; channel R, G, B; +1, -1; first on ties) replaces the pair if its error is less. The palette of a pair does not
// depend on its order as a set, nor does the least error, and equal endpoints give four equal entries: every
// candidate takes the same code. A step past the end of a code's range leaves the pair as it is, which never has
// the lesser error. A candidate moves three entries in one channel: the errors of the pair's own entries are
// computed once, and each candidate's follow by one two-term product.
template <int STRIDE>
__device__ __forceinline__ bool bc1_step(const uint32_t* tex, int base, uint32_t& pair, uint32_t& err) {
  const uint32_t c0 = pair & 0xFFFFu, c1 = pair >> 16;
  const int ra = c0 >> 11, ga = (c0 >> 5) & 63, ba = c0 & 31, rb = c1 >> 11, gb = (c1 >> 5) & 63, bb = c1 & 31;
  const uint32_t P0 = (uint32_t)ex5(ra) | ((uint32_t)ex6(ga) << 8) | ((uint32_t)ex5(ba) << 16);
  const uint32_t P1 = (uint32_t)ex5(rb) | ((uint32_t)ex6(gb) << 8) | ((uint32_t)ex5(bb) << 16);
  const uint32_t P2 = (uint32_t)third5(ra, rb) | ((uint32_t)third6(ga, gb) << 8) | ((uint32_t)third5(ba, bb) << 16);
  const uint32_t P3 = (uint32_t)third5(rb, ra) | ((uint32_t)third6(gb, ga) << 8) | ((uint32_t)third5(bb, ba) << 16);
  int em[16], es[16], e2[16], e3[16];  // of the entries: moving endpoint, staying endpoint, interior
  {
    const int k0 = (int)__dp4a(P0, P0, 0u), k1 = (int)__dp4a(P1, P1, 0u), k2 = (int)__dp4a(P2, P2, 0u), k3 = (int)__dp4a(P3, P3, 0u);
#pragma unroll
    for (int t = 0; t < 16; t++) {
      const uint32_t v = tex[t * STRIDE];
      em[t] = k0 + 2 * (int)__dp4a(v, ~P0, 0u);
      es[t] = k1 + 2 * (int)__dp4a(v, ~P1, 0u);
      e2[t] = k2 + 2 * (int)__dp4a(v, ~P2, 0u);
      e3[t] = k3 + 2 * (int)__dp4a(v, ~P3, 0u);
    }
  }
  int least = (int)err - base, pick = -1;
#pragma unroll
  for (int ep = 0; ep < 2; ep++) {
#pragma unroll 1
    for (int c = 0; c < 3; c++) {
      uint32_t w[8];  // the channel of two texels, each followed by a byte 1
#pragma unroll
      for (int t = 0; t < 8; t++)
        w[t] = __byte_perm(tex[2 * t * STRIDE], tex[(2 * t + 1) * STRIDE], 0x7430 + 0x0101 * c) | 0x01000100u;
      const int sh = c == 0 ? 11 : c == 1 ? 5 : 0, lim = c == 1 ? 63 : 31;
      const int m = (int)((ep ? c1 : c0) >> sh) & lim, f = (int)((ep ? c0 : c1) >> sh) & lim;
      const int x0 = (int)((ep ? P1 : P0) >> (8 * c)) & 255, x2 = (int)(P2 >> (8 * c)) & 255, x3 = (int)(P3 >> (8 * c)) & 255;
#pragma unroll 1
      for (int d = 1; d >= -1; d -= 2) {
        const int n = max(min(m + d, lim), 0);
        const int y0 = c == 1 ? ex6(n) : ex5(n), ya = c == 1 ? third6(n, f) : third5(n, f), yb = c == 1 ? third6(f, n) : third5(f, n);
        const uint32_t m0 = bc1_move(x0, y0), m2 = bc1_move(x2, ep ? yb : ya), m3 = bc1_move(x3, ep ? ya : yb);
        int s = 0;
#pragma unroll
        for (int t = 0; t < 16; t += 2) {
          s += min(__vimin3_s32(bc1_dp2_lo(m0, w[t / 2], em[t]), bc1_dp2_lo(m2, w[t / 2], e2[t]), bc1_dp2_lo(m3, w[t / 2], e3[t])), es[t]);
          s += min(__vimin3_s32(bc1_dp2_hi(m0, w[t / 2], em[t + 1]), bc1_dp2_hi(m2, w[t / 2], e2[t + 1]), bc1_dp2_hi(m3, w[t / 2], e3[t + 1])),
                   es[t + 1]);
        }
        if (s < least) {
          least = s;
          pick = 6 * ep + 2 * c + (d < 0);
        }
      }
    }
#pragma unroll
    for (int t = 0; t < 16; t++) {
      const int x = em[t];
      em[t] = es[t];
      es[t] = x;
    }
  }
  if (pick < 0) return false;
  const int ep = pick >= 6, c = (ep ? pick - 6 : pick) >> 1;
  const int one = c == 0 ? 1 << 11 : c == 1 ? 1 << 5 : 1;
  const uint32_t moved = (ep ? c1 : c0) + (pick & 1 ? -one : one), fixed = ep ? c0 : c1;
  pair = max(moved, fixed) | (min(moved, fixed) << 16);
  err = (uint32_t)(least + base);
  return true;
}

__device__ __forceinline__ uint2 bc1_bits(const Bc1Res& r) {
  return make_uint2((uint32_t)r.c0 | ((uint32_t)r.c1 << 16), r.idx);
}

// Encodes the warp's staged blocks blk0 .. blk0 + BPW - 1 (those below total). The neighbourhood search takes one to
// four steps, 2.4 on average on the scene-scale distribution, but four for some lane of nearly every warp: blocks
// with a step to do are kept on a stack in shared memory and stepped 32 at a time.
template <int BPW>
__device__ __forceinline__ void bc1_encode_warp(Bc1Warp<BPW>& W, int64_t blk0, int64_t total, uint2* __restrict__ blocks,
                                                uint32_t* __restrict__ sse1, uint32_t* __restrict__ sse0,
                                                uint64_t* __restrict__ sse64) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  int cnt = 0;
#pragma unroll 1
  for (int b = lane; b < BPW; b += 32) {
    const bool live = blk0 + b < total;
    bool step = false;
    if (live) {
      uint32_t tx[16], pair, err, grey;
      int base;
#pragma unroll
      for (int t = 0; t < 16; t++) tx[t] = W.tex[t][b];
      step = bc1_start(tx, pair, err, base, grey);
      W.base[b] = base;
      W.pair[b] = pair;
      W.err[b] = err;
      if (sse0) sse0[blk0 + b] = grey;
    }
    const unsigned m = __ballot_sync(0xFFFFFFFFu, step);
    if (step) W.stack[cnt + __popc(m & below)] = (uint16_t)b;
    cnt += __popc(m);
  }
  __syncwarp();
  while (cnt > 0) {
    const int take = min(cnt, 32);
    cnt -= take;
    bool again = false;
    uint32_t e = 0u;
    if (lane < take) {
      e = W.stack[cnt + lane];
      const int b = (int)(e & 255u);
      uint32_t pair = W.pair[b], err = W.err[b];
      if (bc1_step<BPW + 1>(&W.tex[0][b], W.base[b], pair, err)) {
        W.pair[b] = pair;
        W.err[b] = err;
        e += 256u;
        again = e < 4u * 256u;
      }
    }
    __syncwarp();
    const unsigned m = __ballot_sync(0xFFFFFFFFu, again);
    if (again) W.stack[cnt + __popc(m & below)] = (uint16_t)e;
    cnt += __popc(m);
    __syncwarp();
  }
#pragma unroll 1
  for (int b = lane; b < BPW; b += 32) {
    if (blk0 + b >= total) continue;
    uint32_t tx[16];
#pragma unroll
    for (int t = 0; t < 16; t++) tx[t] = W.tex[t][b];
    const Bc1Res r = bc1_eval_k(tx, W.base[b], W.pair[b] & 0xFFFFu, W.pair[b] >> 16);
    blocks[blk0 + b] = bc1_bits(r);
    if (sse1) sse1[blk0 + b] = r.sse;
    if (sse64) sse64[blk0 + b] = r.sse;
  }
}
