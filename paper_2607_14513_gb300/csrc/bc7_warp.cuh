// bc7_warp.cuh -- the BC7 encoder of one warp: candidate search, solve and pack (included by bc7.cu only).
//
// A warp owns 32 blocks (8 where there are few). The search is the exhaustive one (285 candidates, the first of least
// error), but a candidate is fitted only where an exact lower bound of its error allows it to win:
//
//  * every palette entry lies within sqrt(3)/2 of a point on the line through its two endpoints
//    (each channel is the interpolated value rounded to the nearest integer), so for a subset of
//    texels v the error of any fit is at least the squared distance of the v to their best line, and
//    over a whole block  sqrt(error) >= sqrt(R) - sqrt(16 * 3/4)  with R the sum over the subsets of
//    (trace - largest eigenvalue) of the subset's scatter matrix;
//  * R comes from exact integer moments (byte dot products of the texels with the subset's mask) and
//    an upper bound of the largest eigenvalue: the closed form (t + 2 sqrt(t^2 - 3 c2)) / 3 (t, c2, c3:
//    the characteristic polynomial's coefficients), then one Newton step, which from above stays
//    above. All float roundings are covered by margins on the safe side;
//  * a candidate is dropped when that bound exceeds the best error so far strictly, so ties still
//    go to the lowest enumeration index and the result is the exhaustive search's, bit for bit.
//
// Survivors differ from block to block, so (block, partition) pairs are collected in a stack in
// shared memory, partition after partition, and fitted 32 at a time, a subset per lane, the largest
// subsets first; a pair goes back on the stack for its next subset only if its errors so far and the
// bound of what is left do not exceed the best. Neighbouring pairs share a partition or one of the
// same subset sizes, so the lanes' texel loops have nearly the same length, and no lane idles for a
// block that has nothing left to fit. A lane reads any of the warp's 32 blocks from shared memory.
#pragma once

#define BC7_STRIDE 33  // words between a block's consecutive texels in a warp's tile

struct Bc7Warp {
  uint32_t tex[16][BC7_STRIDE];  // texel t of block b at [t][b], r | g << 8 | b << 16
  uint32_t best[32];             // least error so far << 9 | enumeration index
  uint16_t r[64][32];            // the bound R of the phase's partition p, block b (bound_pack)
  // fits to do: block | partition << 5 | part << 11 | texels of the parts from this one on << 13,
  // the errors so far of the (up to three) candidates, and a bound R of the parts from this one on
  uint32_t stack[64];
  int err[3][64];
  float rest[64];
};

// subset masks, a byte of ones per member texel (texel 4 w + i in byte i of word w): subset 1 of the
// two-subset partitions, subsets 1 and 2 of the three-subset partitions; and the subsets' sizes
__constant__ uint4 c_msk2[64];
__constant__ uint4 c_msk3[64][2];
__constant__ uint8_t c_cnt2[64];
__constant__ uint8_t c_cnt3[64][2];
__constant__ float c_inv[17];  // 1 / n rounded down
// the order in which a phase offers its partitions: by the size of their largest subset (three subsets; the
// first 16 of them; two subsets; identity for the rotations)
__constant__ uint8_t c_order[4][64];
// member texels of each subset: texel indices in increasing order, four bits each from bit 0, and the
// member count in bits 60-63. g_mem*: the largest subset first (the search adds the subsets' errors in
// any order), g_org*: in the format's order. Read per lane, so in global memory.
__device__ uint64_t g_mem2[64][2], g_org2[64][2];
__device__ uint64_t g_mem3[64][3], g_org3[64][3];

// ---- moments and the line bound -------------------------------------------------------------
// The block's texels as signed bytes v - 128, four texels of one channel per word.
struct Planes {
  int c[3][4];
};
// sums over a subset of the centred channels and of their products
struct Moments {
  int s[3], q[6];  // q: rr, gg, bb, rg, rb, gb
};

__device__ __forceinline__ Planes planes_of(const uint32_t* tex) {
  Planes P;
#pragma unroll
  for (int w = 0; w < 4; w++) {
    const uint32_t a0 = tex[(4 * w) * BC7_STRIDE], a1 = tex[(4 * w + 1) * BC7_STRIDE];
    const uint32_t a2 = tex[(4 * w + 2) * BC7_STRIDE], a3 = tex[(4 * w + 3) * BC7_STRIDE];
    const uint32_t t0 = __byte_perm(a0, a1, 0x5140u), t1 = __byte_perm(a2, a3, 0x5140u);
    const uint32_t u0 = __byte_perm(a0, a1, 0x0062u), u1 = __byte_perm(a2, a3, 0x0062u);
    P.c[0][w] = (int)(__byte_perm(t0, t1, 0x5410u) ^ 0x80808080u);
    P.c[1][w] = (int)(__byte_perm(t0, t1, 0x7632u) ^ 0x80808080u);
    P.c[2][w] = (int)(__byte_perm(u0, u1, 0x5410u) ^ 0x80808080u);
  }
  return P;
}

__device__ __forceinline__ Moments moments_of(const Planes& P, const uint4& mask) {
  Moments m;
#pragma unroll
  for (int i = 0; i < 3; i++) m.s[i] = 0;
#pragma unroll
  for (int i = 0; i < 6; i++) m.q[i] = 0;
  const uint32_t mw[4] = {mask.x, mask.y, mask.z, mask.w};
#pragma unroll
  for (int w = 0; w < 4; w++) {
    const int r = P.c[0][w] & (int)mw[w], g = P.c[1][w] & (int)mw[w], b = P.c[2][w] & (int)mw[w];
    m.s[0] = __dp4a(r, 0x01010101, m.s[0]);
    m.s[1] = __dp4a(g, 0x01010101, m.s[1]);
    m.s[2] = __dp4a(b, 0x01010101, m.s[2]);
    m.q[0] = __dp4a(r, P.c[0][w], m.q[0]);
    m.q[1] = __dp4a(g, P.c[1][w], m.q[1]);
    m.q[2] = __dp4a(b, P.c[2][w], m.q[2]);
    m.q[3] = __dp4a(r, P.c[1][w], m.q[3]);
    m.q[4] = __dp4a(r, P.c[2][w], m.q[4]);
    m.q[5] = __dp4a(g, P.c[2][w], m.q[5]);
  }
  return m;
}

__device__ __forceinline__ Moments minus(const Moments& a, const Moments& b) {
  Moments m;
#pragma unroll
  for (int i = 0; i < 3; i++) m.s[i] = a.s[i] - b.s[i];
#pragma unroll
  for (int i = 0; i < 6; i++) m.q[i] = a.q[i] - b.q[i];
  return m;
}

// An integer of [-2^22, 2^22) as a float: added to the bits of 1.5 * 2^23 it gives that float plus it.
__device__ __forceinline__ float small_float(int v) { return __int_as_float(v + 0x4B400000) - 12582912.0f; }
// n q - s s' as a float, exact: the same for centred and plain texels, at most 4,161,600 for 16 of them
__device__ __forceinline__ float scatter(int n, int q, int sa, int sb) { return small_float(n * q - sa * sb); }

__device__ __forceinline__ float approx_sqrt(float x) {  // PTX sqrt.approx: relative error below 2^-22
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float approx_rcp(float x) {  // PTX rcp.approx: relative error below 2^-22
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// A lower bound of the squared distance of a subset's n texels to their best line: (trace - an
// upper bound of the largest eigenvalue) of n times the scatter matrix, over n. The matrix's
// entries and the trace t are exact; c2 and the discriminant are off by less than 6e-7 t^2, the
// polynomial and its derivative below by less than 2e-6 t^3 and 1e-6 t^2, so the margins leave a
// factor of two.
__device__ __forceinline__ float line_bound(const Moments& m, int n) {
  const float rr = scatter(n, m.q[0], m.s[0], m.s[0]), gg = scatter(n, m.q[1], m.s[1], m.s[1]);
  const float bb = scatter(n, m.q[2], m.s[2], m.s[2]), rg = scatter(n, m.q[3], m.s[0], m.s[1]);
  const float rb = scatter(n, m.q[4], m.s[0], m.s[2]), gb = scatter(n, m.q[5], m.s[1], m.s[2]);
  const float t = rr + gg + bb, tt = t * t;
  const float m0 = fmaf(gg, bb, -gb * gb), m1 = fmaf(rr, bb, -rb * rb), m2 = fmaf(rr, gg, -rg * rg);
  const float c2 = m0 + m1 + m2;
  const float c3 = fmaf(rr, m0, fmaf(-rg, fmaf(rg, bb, -rb * gb), rb * fmaf(rg, gb, -rb * gg)));
  const float disc = fmaf(2e-6f, tt, fmaxf(fmaf(-3.0f, c2, tt), 0.0f));
  const float x0 = fmaf(approx_sqrt(disc), 0.666668f, t * 0.333334f);  // above (t + 2 sqrt(disc)) / 3
  const float p = fmaf(fmaf(x0 - t, x0, c2), x0, -c3);
  const float dp = fmaf(fmaf(3.0f, x0, -2.0f * t), x0, c2);
  const float step = fmaxf(fmaf(-4e-6f * t, tt, p), 0.0f) * approx_rcp(fmaxf(fmaf(2e-6f, tt, dp), 1e-30f));
  const float r = fmaf(step, 0.999999f, t - x0);
  return fmaxf(fmaf(-1e-6f, t, r), 0.0f) * c_inv[n];
}

// The same for two of the channels (the rotated forms): the smaller eigenvalue is det / larger one.
__device__ __forceinline__ float line_bound2(float aa, float bb, float ab) {
  const float t = aa + bb, d = aa - bb;
  const float hi = 0.5000005f * (t + approx_sqrt(fmaf(d, d, 4.0f * ab * ab)) * 1.000001f);
  const float det = fmaf(-1e-6f * aa, bb, fmaf(aa, bb, -ab * ab));
  return hi > 0.0f ? fmaxf(det, 0.0f) * approx_rcp(hi) * 0.999999f * c_inv[16] : 0.0f;
}

// A candidate with bound R can still win against the best key while R <= the threshold:
// sqrt(R) <= sqrt(E) + slack, slack the root of the palettes' greatest summed rounding (16 texels,
// 1/4 per coded channel), rounded up.
#define BC7_SLACK3 3.46411f  // sqrt(12)
#define BC7_SLACK2 2.82844f  // sqrt(8)
__device__ __forceinline__ float prune_limit(uint32_t key) {
  const float s = fmaf(approx_sqrt((float)(key >> 9)), 1.000001f, BC7_SLACK3);
  return s * s * 1.00001f;
}

// ---- fits ---------------------------------------------------------------------------------------
// A fit works on the member texels of one subset, their bytes permuted by `sel` on load (identity for
// the partitioned modes); a channel permuted to zero behaves as uncoded: its range, its endpoints and
// its products are zero.
struct Mem {
  uint64_t list;
  int n;
};
__device__ __forceinline__ Mem mem_at(const uint64_t* p) {
  const uint64_t v = __ldg(reinterpret_cast<const unsigned long long*>(p));
  return {v, (int)(v >> 60)};
}
// all 16 texels, with a length the compiler does not unroll by
__device__ __forceinline__ Mem mem_whole() {
  Mem M = {0xFEDCBA9876543210ull, 16};
  asm("" : "+r"(M.n));
  return M;
}
#define BC7_ID 0x3210u

// Calls f(texel, its index) for every member, one copy of f in a rolled loop: the search is bound by
// instruction fetch as much as by issue (two members per step, with a tail, made it a tenth slower).
template <class F>
__device__ __forceinline__ void each_member(const uint32_t* __restrict__ tex, Mem M, uint32_t sel, F f) {
  uint64_t L = M.list;
#pragma unroll 1
  for (int i = 0; i < M.n; i++) {
    const int t = (int)(L & 15);
    L >>= 4;
    f(__byte_perm(tex[t * BC7_STRIDE], 0u, sel), t);
  }
}

// Palette of 2^IB entries between endpoints a and b with BC7 weights. Two channels share one
// multiply-add in 16-bit lanes scaled by 4, so byte 1 of each lane is ((64 - w) a + w b + 32) >> 6
// exactly. Keys pk: KEY = 0 |entry|^2 (when only the least error matters), 16: 16 |entry|^2 + index,
// 128: 128 |entry|^2 + weight; the low bits pick the first of equal errors.
template <int IB, int KEY>
__device__ __forceinline__ void build_pal(const int (&a)[3], const int (&b)[3], uint32_t (&pal)[1 << IB],
                                          int (&pk)[1 << IB]) {
  const uint32_t A = ((uint32_t)a[0] | ((uint32_t)a[1] << 16)) << 2, B = ((uint32_t)b[0] | ((uint32_t)b[1] << 16)) << 2;
  const uint32_t Ab = (uint32_t)a[2] << 2, Bb = (uint32_t)b[2] << 2;
  // (64 - w) A + w B = 64 A + w (B - A): with B - A formed in 32-bit arithmetic a lane may be
  // negative, but each lane's result lies in [0, 2^16), so the packed sum is exact
  const uint32_t rg0 = 64u * A + 0x00800080u, drg = B - A, bb0 = 64u * Ab + 0x80u, dbb = Bb - Ab;
#pragma unroll
  for (int j = 0; j < (1 << IB); j++) {
    const uint32_t w = (uint32_t)wgt<IB>(j);
    const uint32_t rg = rg0 + w * drg, bb = bb0 + w * dbb;
    pal[j] = __byte_perm(rg, bb, 0x7531u);
    const int n2 = (int)__dp4a(pal[j], pal[j], 0u);
    pk[j] = KEY == 128 ? 128 * n2 + (int)w : (KEY == 16 ? 16 * n2 + j : n2);
  }
}

// min_j (pk_j - SCALE dot(v, pal_j)): with SCALE twice the keys' factor this is the least of
// factor (|v - pal_j|^2 - |v|^2) + low bits, an exact palette search
template <int F, int SCALE>
__device__ __forceinline__ int best_key(uint32_t v, const uint32_t (&pal)[F], const int (&pk)[F]) {
  int k = __vimin3_s32(pk[0] - SCALE * (int)__dp4a(v, pal[0], 0u), pk[1] - SCALE * (int)__dp4a(v, pal[1], 0u),
                       pk[2] - SCALE * (int)__dp4a(v, pal[2], 0u));
#pragma unroll
  for (int j = 3; j + 1 < F; j += 2)
    k = __vimin3_s32(k, pk[j] - SCALE * (int)__dp4a(v, pal[j], 0u), pk[j + 1] - SCALE * (int)__dp4a(v, pal[j + 1], 0u));
  return min(k, pk[F - 1] - SCALE * (int)__dp4a(v, pal[F - 1], 0u));
}

struct Box {
  int e0[3], e1[3], s1[3], q[6], n;  // q: sums of products rr, gg, bb, rg, rb, gb
};

// bounding-box diagonal oriented by covariance signs, and the members' moments
__device__ __forceinline__ Box box_axis(const uint32_t* __restrict__ tex, Mem M, uint32_t sel) {
  // channels r and b in the 16-bit halves of one word
  uint32_t lo_rb = 0x00FF00FFu, hi_rb = 0u, s_rb = 0u;
  int lo_g = 255, hi_g = 0, s_g = 0;
  Box B;
#pragma unroll
  for (int i = 0; i < 6; i++) B.q[i] = 0;
  each_member(tex, M, sel, [&](uint32_t v, int) {
    const uint32_t rb = v & 0x00FF00FFu;
    const int r = (int)(v & 255u), g = (int)((v >> 8) & 255u), b = (int)(v >> 16);
    lo_rb = __vminu2(lo_rb, rb); hi_rb = __vmaxu2(hi_rb, rb); s_rb += rb;
    lo_g = min(lo_g, g); hi_g = max(hi_g, g); s_g += g;
    B.q[0] += r * r; B.q[1] += g * g; B.q[2] += b * b;
    B.q[3] += r * g; B.q[4] += r * b; B.q[5] += g * b;
  });
  B.n = M.n;
  B.s1[0] = (int)(s_rb & 0xFFFFu); B.s1[1] = s_g; B.s1[2] = (int)(s_rb >> 16);
  const int lo[3] = {(int)(lo_rb & 0xFFFFu), lo_g, (int)(lo_rb >> 16)};
  const int hi[3] = {(int)(hi_rb & 0xFFFFu), hi_g, (int)(hi_rb >> 16)};
  // reference channel = widest range (first on ties)
  int ref = 0, rw = hi[0] - lo[0], s1r = B.s1[0];
  if (hi[1] - lo[1] > rw) { rw = hi[1] - lo[1]; ref = 1; s1r = B.s1[1]; }
  if (hi[2] - lo[2] > rw) { ref = 2; s1r = B.s1[2]; }
  const int cross[3] = {ref == 1 ? B.q[3] : B.q[4], ref == 0 ? B.q[3] : B.q[5], ref == 0 ? B.q[4] : B.q[5]};
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const bool flip = i != ref && M.n * cross[i] - s1r * B.s1[i] < 0;
    B.e0[i] = flip ? lo[i] : hi[i];
    B.e1[i] = flip ? hi[i] : lo[i];
  }
  return B;
}

// clamp(floor(N / D), 0, 255) for 0 < D < 2^20 and |N| < 2^31: quotient estimated in float from below (below: a
// reciprocal at most 1 / D, short of it by less than 2^-19 of it, so that quotients up to 255 are off by at most
// one) and corrected exactly
__device__ __forceinline__ int ratio255(int N, int D, float below) {
  N = max(N, 0);
  int q = (int)((float)N * below);
  if (N - q * D >= D) q++;
  return min(q, 255);
}

// One least-squares refinement of the box diagonal: every member takes its entry (weight w) of the
// diagonal's palette, and the endpoints become the values at w = 0 and w = 64 of each channel's
// regression line over w, rounded. With V = n sum w^2 - (sum w)^2:
//   e0 = (sum w^2 sum c - sum w sum wc) / V,  e1 = ((64 n - sum w) sum wc - (64 sum w - sum w^2) sum c) / V,
// the normal equations of weights 64 - w and w reduced by their common factor 4096, rounded half away from
// zero: floor((2 num + V) / (2 V)) where that is not negative. Every term fits 32 bits (sum w^2 <= 2^16,
// sum c < 2^12, sum wc < 2^18, V <= 2^18).
template <int IB>
__device__ __forceinline__ void refine(const uint32_t* __restrict__ tex, Mem M, const Box& B, uint32_t sel,
                                       int (&e0)[3], int (&e1)[3]) {
  constexpr int F = 1 << IB;
  uint32_t pal[F];
  int pk[F];
  build_pal<IB, 128>(B.e0, B.e1, pal, pk);
  int sw = 0, sww = 0, swc[3] = {0, 0, 0};
  each_member(tex, M, sel, [&](uint32_t v, int) {
    const int w = best_key<F, 256>(v, pal, pk) & 127;
    sw += w; sww += w * w;
    swc[0] += w * (int)(v & 255u); swc[1] += w * (int)((v >> 8) & 255u); swc[2] += w * (int)(v >> 16);
  });
  const int V = B.n * sww - sw * sw, D = 2 * V;
  const int a0 = 2 * sww, b0 = -2 * sw, a1 = 2 * (sww - 64 * sw), b1 = 2 * (64 * B.n - sw);
  const float below = approx_rcp((float)max(D, 1)) * 0.999999f;
#pragma unroll
  for (int i = 0; i < 3; i++) {
    e0[i] = ratio255(a0 * B.s1[i] + (b0 * swc[i] + V), D, below);
    e1[i] = ratio255(a1 * B.s1[i] + (b1 * swc[i] + V), D, below);
  }
  if (V == 0) {
#pragma unroll
    for (int i = 0; i < 3; i++) { e0[i] = B.e0[i]; e1[i] = B.e1[i]; }
  }
}

// Least over U palettes of the members' summed errors, less their summed squared norms, times U, plus the
// first palette u that has it. Palette u lies between the endpoints quantised through the tables at
// q + 256 t0[u] and q + 256 t1[u] (expanded values).
template <int IB, int U>
__device__ __forceinline__ int quant_err(const uint32_t* __restrict__ tex, Mem M, const int (&e0)[3],
                                         const int (&e1)[3], const uint8_t* __restrict__ q, const int (&t0)[U],
                                         const int (&t1)[U], uint32_t sel) {
  constexpr int F = 1 << IB;
  uint32_t pal[U][F];
  int pk[U][F], err[U];
#pragma unroll
  for (int u = 0; u < U; u++) {
    int v0[3], v1[3];
#pragma unroll
    for (int i = 0; i < 3; i++) { v0[i] = q[256 * t0[u] + e0[i]]; v1[i] = q[256 * t1[u] + e1[i]]; }
    build_pal<IB, 0>(v0, v1, pal[u], pk[u]);
    err[u] = 0;
  }
  each_member(tex, M, sel, [&](uint32_t v, int) {
#pragma unroll
    for (int u = 0; u < U; u++) err[u] += best_key<F, 2>(v, pal[u], pk[u]);
  });
  int b = U * err[0];
#pragma unroll
  for (int u = 1; u < U; u++) b = min(b, U * err[u] + u);
  return b;
}

// ---- the phases of the search -------------------------------------------------------------------
// PH_MODE2: mode 2. PH_MODE0: mode 0. PH_ROT: mode 4 with 2-bit and with 3-bit colour, mode 5. PH_MODE6:
// mode 6. PH_TWO: modes 1, 3 and 7 of a two-subset partition.
enum { PH_MODE2 = 0, PH_MODE0, PH_ROT, PH_MODE6, PH_TWO };

// texel bytes of rotation rot's colour part (the rotated channel zero, the others in order) and of its
// scalar part (rotation 0 has none: all zero, error 0)
__device__ __forceinline__ uint32_t rot_colour(int rot) {
  return rot == 0 ? BC7_ID : (rot == 1 ? 0x4421u : (rot == 2 ? 0x4420u : 0x4410u));
}
__device__ __forceinline__ uint32_t rot_scalar(int rot) { return rot == 0 ? 0x4444u : (0x4440u | (uint32_t)(rot - 1)); }

// The least key of a pair's candidates, all parts fitted.
__device__ __forceinline__ uint32_t pair_key(int phase, int p, const int (&err)[3]) {
  const int ex = phase == PH_MODE2 ? 80 + p : (phase == PH_MODE0 ? p : (phase == PH_TWO ? 16 + p : (phase == PH_MODE6 ? 220 : 208 + 2 * p)));
  const uint32_t key = ((uint32_t)err[0] << 9) | (uint32_t)ex;
  const uint32_t k1 = ((uint32_t)err[1] << 9) | (uint32_t)(phase == PH_ROT ? 209 + 2 * p : 144 + p);
  const uint32_t k2 = ((uint32_t)err[2] << 9) | (uint32_t)(phase == PH_ROT ? 216 + p : 221 + p);
  return phase == PH_ROT || phase == PH_TWO ? min(key, min(k1, k2)) : key;
}

// At least the members' squared distance to their best line: trace - a lower bound of the largest
// eigenvalue, |C w| / |w| with w = C d after one step of power iteration from the fitted direction d.
__device__ __forceinline__ float line_above(const Box& B, int dx, int dy, int dz) {
  const int n = B.n;
  const float rr = scatter(n, B.q[0], B.s1[0], B.s1[0]), gg = scatter(n, B.q[1], B.s1[1], B.s1[1]);
  const float bb = scatter(n, B.q[2], B.s1[2], B.s1[2]), rg = scatter(n, B.q[3], B.s1[0], B.s1[1]);
  const float rb = scatter(n, B.q[4], B.s1[0], B.s1[2]), gb = scatter(n, B.q[5], B.s1[1], B.s1[2]);
  const float x = small_float(dx), y = small_float(dy), z = small_float(dz);
  const float u = fmaf(rr, x, fmaf(rg, y, rb * z)), v = fmaf(rg, x, fmaf(gg, y, gb * z)), w = fmaf(rb, x, fmaf(gb, y, bb * z));
  const float a = fmaf(rr, u, fmaf(rg, v, rb * w)), b = fmaf(rg, u, fmaf(gg, v, gb * w)), c = fmaf(rb, u, fmaf(gb, v, bb * w));
  const float ww = fmaf(u, u, fmaf(v, v, w * w));  // below 10^21, its product with C^2 below 10^35
  const float along = ww > 0.0f ? approx_sqrt(fmaf(a, a, fmaf(b, b, c * c)) * approx_rcp(ww)) : 0.0f;
  return fmaxf(fmaf(1.00001f, rr + gg + bb, -along), 0.0f) * (c_inv[n] * 1.000001f);
}

// Fits part i (a subset; in PH_ROT the colour or the scalar part) of partition or rotation p of the warp's
// phase and adds the errors of the pair's (up to three) candidates to err; n: the part's texels, line: at least
// their squared distance to their best line (not for the last part). One copy of every step serves all phases:
// the warps of an SM, each in its own phase, share the instruction cache.
__device__ __forceinline__ void fit_part(const uint32_t* tex, int phase, int p, int i, bool last, const uint8_t* sq,
                                         int (&err)[3], float& line, int& n) {
  Mem M;
  uint32_t sel = BC7_ID;
  if (phase <= PH_MODE0) M = mem_at(&g_mem3[p][i]);
  else if (phase == PH_TWO) M = mem_at(&g_mem2[p][i]);
  else M = mem_whole();
  if (phase == PH_ROT) sel = i == 0 ? rot_colour(p) : rot_scalar(p);
  const Box B = box_axis(tex, M, sel);
  const int norm = B.q[0] + B.q[1] + B.q[2];  // quant_err leaves the members' squared norms out
  int e0[3], e1[3];
  n = M.n;
  line = 3e38f;  // PH_ROT: nothing is known of the scalar part
  if (phase == PH_MODE2 || phase >= PH_ROT) {
    if (phase == PH_MODE6) {
      refine<4>(tex, M, B, sel, e0, e1);
      int e = 0x7FFFFFFF;
#pragma unroll 1
      for (int c = 0; c < 4; c++) {
        const int t0[1] = {qid(7, 1, 0) + (c & 1)}, t1[1] = {qid(7, 1, 0) + (c >> 1)};
        e = min(e, quant_err<4, 1>(tex, M, e0, e1, sq, t0, t1, sel));
      }
      err[0] += norm + e;
      return;
    }
    refine<2>(tex, M, B, sel, e0, e1);
    if (phase == PH_TWO) {
#pragma unroll 1
      for (int h = 0; h < 2; h++) {  // mode 3, mode 7: four p-bit combinations each
        const int t = h ? qid(5, 1, 0) : qid(7, 1, 0);
        const int t0[4] = {t, t + 1, t, t + 1}, t1[4] = {t, t, t + 1, t + 1};
        const int e = norm + (quant_err<2, 4>(tex, M, e0, e1, sq, t0, t1, sel) >> 2);
        if (h) err[2] += e; else err[1] += e;
      }
    } else {
#pragma unroll 1
      for (int h = 0; h < (phase == PH_ROT ? 2 : 1); h++) {  // mode 2 or 4, mode 5
        const int t = h == 0 ? (i == 0 || phase == PH_MODE2 ? qid(5, 0, 0) : qid(6, 0, 0)) : (i == 0 ? qid(7, 0, 0) : qid(8, 0, 0));
        const int t0[1] = {t};
        const int e = norm + quant_err<2, 1>(tex, M, e0, e1, sq, t0, t0, sel);
        if (h) err[2] += e; else if (i == 0 || phase == PH_MODE2) err[0] += e; else err[1] += e;
      }
    }
  }
  if (phase != PH_MODE2) {
    refine<3>(tex, M, B, sel, e0, e1);
    if (phase == PH_ROT) {
      const int t0[1] = {i == 0 ? qid(5, 0, 0) : qid(6, 0, 0)};
      const int e = norm + quant_err<3, 1>(tex, M, e0, e1, sq, t0, t0, sel);
      if (i == 0) err[1] += e; else err[0] += e;
    } else {
      // mode 1: p-bits 00 and 11; mode 0: 00 and 10, then 01 and 11
      const int t = phase == PH_TWO ? qid(6, 1, 0) : qid(4, 1, 0);
      int e = 0x7FFFFFFF;
#pragma unroll 1
      for (int c = 0; c < (phase == PH_TWO ? 1 : 2); c++) {
        const int t0[2] = {t, t + 1}, t1[2] = {t + c, t + (phase == PH_TWO ? 1 : c)};
        e = min(e, quant_err<3, 2>(tex, M, e0, e1, sq, t0, t1, sel) >> 1);
      }
      err[0] += norm + e;
    }
  }
  if (phase != PH_ROT && !last) line = line_above(B, e1[0] - e0[0], e1[1] - e0[1], e1[2] - e0[2]);
}

// A bound in 16 bits, rounded down: a float in [1, 2^32) with 11 bits of mantissa, 0 below 1
__device__ __forceinline__ uint16_t bound_pack(float r) {
  return r < 1.0f ? (uint16_t)0 : (uint16_t)((__float_as_uint(r) >> 12) - (127u << 11));
}
__device__ __forceinline__ float bound_unpack(uint16_t h) {
  return h == 0 ? 0.0f : __uint_as_float(((uint32_t)h + (127u << 11)) << 12);
}

// Searches the warp's BPW blocks (columns col0.. of its tile; those of the lanes with `active`); leaves each
// block's least error and its candidate in W.best. All 32 lanes call it. sq: the 12 tables of expanded endpoint
// values. With fewer than 32 blocks, 32 / BPW lanes share a block's bounds, and the stack serves fewer blocks:
// the warp is done sooner. All warps of the CTA call it, and start each phase together.
template <int BPW>
__device__ __noinline__ void bc7_search(Bc7Warp& W, int col0, bool active, const uint8_t* sq) {
  constexpr int LPB = 32 / BPW;
  const int lane = threadIdx.x & 31, own = lane % BPW, slice = lane / BPW;
  active = __shfl_sync(0xFFFFFFFFu, (int)active, own) != 0;
  W.best[lane] = 0xFFFFFFFFu;
  const unsigned below = (1u << lane) - 1u;
  int seed = 0;
#pragma unroll 1
  for (int phase = PH_MODE2; phase <= PH_TWO; phase++) {
    __syncthreads();
    // the phase's bounds, where they are not the last one's (modes 2 and 0 share theirs)
    if (phase == PH_MODE2 || phase == PH_ROT || phase == PH_TWO) {
      const Planes P = planes_of(&W.tex[0][col0 + own]);
      const Moments T = moments_of(P, make_uint4(~0u, ~0u, ~0u, ~0u));
      if (phase == PH_ROT) {
        // rotation 0 and mode 6: one line through all 16 texels; the others: in the two channels left, whose
        // smaller slack is put into the bound, sqrt(R') = sqrt(R) + sqrt(12) - sqrt(8) rounded down
        const float one = line_bound(T, 16);
        const float rr = scatter(16, T.q[0], T.s[0], T.s[0]), gg = scatter(16, T.q[1], T.s[1], T.s[1]);
        const float bb = scatter(16, T.q[2], T.s[2], T.s[2]), rg = scatter(16, T.q[3], T.s[0], T.s[1]);
        const float rb = scatter(16, T.q[4], T.s[0], T.s[2]), gb = scatter(16, T.q[5], T.s[1], T.s[2]);
        const float b2[3] = {line_bound2(gg, bb, gb), line_bound2(rr, bb, rb), line_bound2(rr, gg, rg)};
        W.r[0][own] = bound_pack(one);
#pragma unroll
        for (int i = 0; i < 3; i++) {
          const float s = fmaf(approx_sqrt(b2[i]), 0.999999f, BC7_SLACK3 - BC7_SLACK2 - 1e-5f);
          W.r[i + 1][own] = bound_pack(s * s * 0.999999f);
        }
      } else {
        float least = 3e38f;
#pragma unroll 1
        for (int p = slice; p < 64; p += LPB) {
          Moments rest = T;
          float R = 0.0f;
          int n = 16;
#pragma unroll 1
          for (int s = 0; s < (phase == PH_MODE2 ? 2 : 1); s++) {
            const Moments a = moments_of(P, phase == PH_MODE2 ? c_msk3[p][s] : c_msk2[p]);
            const int na = phase == PH_MODE2 ? c_cnt3[p][s] : c_cnt2[p];
            R += line_bound(a, na);
            rest = minus(rest, a);
            n -= na;
          }
          R += line_bound(rest, n);
          W.r[p][own] = bound_pack(R);
          if (R < least) { least = R; if (phase == PH_MODE2) seed = p; }
        }
        if (LPB > 1 && phase == PH_MODE2) {
#pragma unroll
          for (int d = BPW; d < 32; d *= 2) {
            const float r = __shfl_xor_sync(0xFFFFFFFFu, least, d);
            const int p = __shfl_xor_sync(0xFFFFFFFFu, seed, d);
            if (r < least || (r == least && p < seed)) { least = r; seed = p; }
          }
        }
      }
    }
    __syncwarp();
    const int np = phase == PH_MODE0 ? 16 : (phase == PH_ROT ? 4 : (phase == PH_MODE6 ? 1 : 64));
    const int order = phase <= PH_MODE0 ? phase : (phase == PH_TWO ? 2 : 3);
    const int parts = phase <= PH_MODE0 ? 3 : (phase == PH_MODE6 ? 1 : 2);
    // the partition of the least three-subset bound first: its error prunes all that follows
    int cnt = 0, p = phase == PH_MODE2 ? -1 : 0;
    float limit = prune_limit(W.best[own]);
    for (;;) {
      if (cnt < 32 && p < np) {
        const int q = p < 0 ? seed : (p + slice < np ? c_order[order][p + slice] : 0);
        const float R = bound_unpack(W.r[q][own]);
        const bool want = active && (p < 0 ? slice == 0 : (p + slice < np && R <= limit && !(phase == PH_MODE2 && q == seed)));
        const unsigned m = __ballot_sync(0xFFFFFFFFu, want);
        if (want) {
          const int at = cnt + __popc(m & below);
          W.stack[at] = (uint32_t)own | ((uint32_t)q << 5) | (16u << 13);
          W.err[0][at] = W.err[1][at] = W.err[2][at] = 0;
          W.rest[at] = R;
        }
        cnt += __popc(m);
        p = p < 0 ? 0 : p + LPB;
        __syncwarp();
        if (p > 0 || cnt == 0) continue;
      }
      if (cnt == 0) break;
      const int take = min(cnt, 32);
      cnt -= take;
      uint32_t fit = 0;
      int err[3] = {0, 0, 0};
      float rest = 0.0f;
      bool more = false;
      if (lane < take) {
        fit = W.stack[cnt + lane];
#pragma unroll
        for (int k = 0; k < 3; k++) err[k] = W.err[k][cnt + lane];
        rest = W.rest[cnt + lane];
        const int b = (int)(fit & 31u), q = (int)((fit >> 5) & 63u), i = (int)((fit >> 11) & 3u);
        float line;
        int n;
        fit_part(&W.tex[0][col0 + b], phase, q, i, i + 1 == parts, sq, err, line, n);
        if (i + 1 == parts) {
          atomicMin(&W.best[b], pair_key(phase, q, err));
        } else {
          // what is left costs at least (sqrt(its bound R) - sqrt(3/4 texels))^2 on top
          fit += (1u << 11) - ((uint32_t)n << 13);
          rest = fmaxf(rest - line, 0.0f);
          const float s = fmaxf(approx_sqrt(rest) * 0.999999f - approx_sqrt(0.75f * (float)(fit >> 13)) * 1.000001f, 0.0f);
          const int least = phase <= PH_MODE0 ? err[0] : min(err[0], min(err[1], err[2]));
          more = fmaf(s * s, 0.99999f, (float)least) <= (float)(W.best[b] >> 9);
        }
      }
      __syncwarp();
      const unsigned again = __ballot_sync(0xFFFFFFFFu, more);
      if (more) {
        const int at = cnt + __popc(again & below);
        W.stack[at] = fit;
#pragma unroll
        for (int k = 0; k < 3; k++) W.err[k][at] = err[k];
        W.rest[at] = rest;
      }
      cnt += __popc(again);
      __syncwarp();
      limit = prune_limit(W.best[own]);
    }
    __syncwarp();
  }
}

// ---- the winner's 128 bits --------------------------------------------------------------------------
// per mode: subsets, partition / rotation / selection bits, colour and alpha bits, p-bits per endpoint or
// per subset, index bits
struct ModeInfo { int ns, pb, rb, isb, cb, ab, epb, spb, ib, ib2; };
__device__ __forceinline__ ModeInfo mode_info(int m) {
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

// The block under construction. Fields are written at their bit offsets.
struct Bits128 {
  uint64_t lo, hi;
  __device__ __forceinline__ void put(uint64_t v, int off) {
    if (off >= 64) { hi |= v << (off - 64); return; }
    lo |= v << off;
    if (off > 0) hi |= v >> (64 - off);
  }
};

// 16 indices of four bits each, packed to ib (2, 3 or 4) bits each
__device__ __forceinline__ uint64_t pack_indices(uint64_t x, int ib) {
  if (ib == 2) {
    x = (x | (x >> 2)) & 0x0F0F0F0F0F0F0F0Full;
    x = (x | (x >> 4)) & 0x00FF00FF00FF00FFull;
    x = (x | (x >> 8)) & 0x0000FFFF0000FFFFull;
    return (x | (x >> 16)) & 0xFFFFFFFFull;
  }
  if (ib == 3) {
    x = (x & 0x0707070707070707ull) | ((x & 0x7070707070707070ull) >> 1);
    x = (x & 0x003F003F003F003Full) | ((x & 0x3F003F003F003F00ull) >> 2);
    x = (x & 0x00000FFF00000FFFull) | ((x & 0x0FFF00000FFF0000ull) >> 4);
    return (x & 0xFFFFFFull) | ((x & 0x00FFFFFF00000000ull) >> 8);
  }
  return x;
}

// drops bit p (an anchor index's top bit, 0)
__device__ __forceinline__ uint64_t drop_bit(uint64_t x, int p) {
  const uint64_t m = (1ull << p) - 1ull;
  return (x & m) | ((x >> 1) & ~m);
}

__device__ __forceinline__ int anchor_of(int ns, int p, int s) {
  return s == 0 ? 0 : (ns == 2 ? c_anc2[p] : (s == 1 ? c_anc3a[p] : c_anc3b[p]));
}


// Solves and packs one block's winner part by part: the part is fitted again, its best p-bit combination
// quantised and indexed. Anchors are fixed losslessly by swapping endpoints and inverting indices; fields are
// LSB first.
struct Packer {
  int mode, part, rot, isb;
  Bits128 w;
  uint64_t colour, scalar;  // indices, four bits per texel

  __device__ __forceinline__ bool rotated() const { return mode == 4 || mode == 5; }
  __device__ __forceinline__ int parts() const { return rotated() ? (rot ? 2 : 1) : mode_info(mode).ns; }

  __device__ __forceinline__ void start(int e) {
    part = rot = isb = 0;
    if (e < 16) { mode = 0; part = e; }
    else if (e < 208) { mode = 1 + (e - 16) / 64; part = (e - 16) % 64; }
    else if (e < 216) { mode = 4; rot = (e - 208) / 2; isb = (e - 208) % 2; }
    else if (e < 220) { mode = 5; rot = e - 216; }
    else if (e < 221) { mode = 6; }
    else { mode = 7; part = (e - 221) & 63; }
    const ModeInfo I = mode_info(mode);
    w.lo = w.hi = colour = scalar = 0ull;
    w.put(1ull << mode, 0);
    w.put((uint64_t)part, mode + 1);
    w.put((uint64_t)rot, mode + 1 + I.pb);
    w.put((uint64_t)isb, mode + 1 + I.pb + I.rb);
    // no scalar channel: alpha 255, all ones
    if (I.ab && rot == 0) w.put((1ull << (2 * I.ns * I.ab)) - 1ull, mode + 1 + I.pb + I.rb + I.isb + 6 * I.ns * I.cb);
  }

  // fits part i and packs it; lanes with winners of different modes share the box and, per index width, the rest
  __device__ __forceinline__ void solve(const uint32_t* tex, const uint8_t* sq, int i) {
    const ModeInfo I = mode_info(mode);
    const bool alpha = rotated() && i == 1;
    const Mem M = I.ns == 1 ? mem_whole() : mem_at(I.ns == 2 ? &g_org2[part][i] : &g_org3[part][i]);
    const uint32_t sel = rotated() ? (alpha ? rot_scalar(rot) : rot_colour(rot)) : BC7_ID;
    const int ib = alpha ? (isb ? I.ib : I.ib2) : (rotated() && isb ? I.ib2 : I.ib);
    const int t = qid(alpha ? I.ab : I.cb, I.epb | I.spb, 0), kind = I.epb ? 1 : (I.spb ? 2 : 0);
    const Box B = box_axis(tex, M, sel);
    if (ib == 2) solve_width<2>(tex, M, sel, B, sq, i, t, kind);
    if (ib == 3) solve_width<3>(tex, M, sel, B, sq, i, t, kind);
    if (ib == 4) solve_width<4>(tex, M, sel, B, sq, i, t, kind);
  }

  // kind: p-bits, 0 none, 1 per endpoint, 2 per subset
  template <int IB>
  __device__ __forceinline__ void solve_width(const uint32_t* tex, Mem M, uint32_t sel, const Box& B, const uint8_t* sq,
                                              int i, int t, int kind) {
    int e0[3], e1[3], least = 0x7FFFFFFF, p0 = 0, p1 = 0;
    refine<IB>(tex, M, B, sel, e0, e1);
    // least error, first on ties
#pragma unroll 1
    for (int c = 0; c < (kind == 0 ? 0 : (kind == 1 ? 4 : 2)); c++) {
      const int a = kind == 1 ? (c & 1) : c, b = kind == 1 ? (c >> 1) : c;
      const int t0[1] = {t + a}, t1[1] = {t + b};
      const int err = quant_err<IB, 1>(tex, M, e0, e1, sq, t0, t1, sel);
      if (err < least) { least = err; p0 = a; p1 = b; }
    }
    take<IB>(tex, M, sel, e0, e1, sq, i, t, p0, p1);
  }

  // part i solved: endpoints e0 and e1 quantised through tables t + p0 and t + p1, and the indices
  template <int IB>
  __device__ __forceinline__ void take(const uint32_t* tex, Mem M, uint32_t sel, const int (&e0)[3],
                                       const int (&e1)[3], const uint8_t* sq, int i, int t, int p0, int p1) {
    constexpr int F = 1 << IB;
    const ModeInfo I = mode_info(mode);
    const bool alpha = rotated() && i == 1;
    const int hp = I.epb | I.spb, drop = 8 - ((alpha ? I.ab : I.cb) + hp);
    int v0[3], v1[3];
    uint32_t c0 = 0u, c1 = 0u;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      v0[c] = sq[256 * (t + p0) + e0[c]];
      v1[c] = sq[256 * (t + p1) + e1[c]];
      // a code is the leading bits of its expanded value, without the p-bit
      c0 |= (uint32_t)((v0[c] >> drop) >> hp) << (8 * c);
      c1 |= (uint32_t)((v1[c] >> drop) >> hp) << (8 * c);
    }
    uint32_t pal[F];
    int pk[F];
    build_pal<IB, 16>(v0, v1, pal, pk);
    uint64_t idx = 0ull, members = 0ull;
    each_member(tex, M, sel, [&](uint32_t v, int at) {
      idx |= (uint64_t)(best_key<F, 32>(v, pal, pk) & 15) << (4 * at);
      members |= 1ull << (4 * at);
    });
    const int a = rotated() ? 0 : anchor_of(I.ns, part, i);
    if ((idx >> (4 * a + IB - 1)) & 1ull) {
      const uint32_t c = c0; c0 = c1; c1 = c;
      const int p = p0; p0 = p1; p1 = p;
      idx ^= members * (uint64_t)(F - 1);
    }
    put(i, alpha, idx, c0, c1, p0, p1);
  }

  __device__ __noinline__ void put(int i, bool alpha, uint64_t idx, uint32_t c0, uint32_t c1, int p0, int p1) {
    const ModeInfo I = mode_info(mode);
    const int cstart = mode + 1 + I.pb + I.rb + I.isb, astart = cstart + 6 * I.ns * I.cb, pstart = astart + 2 * I.ns * I.ab;
    if (alpha) {
      w.put(c0 & 255u, astart);
      w.put(c1 & 255u, astart + I.ab);
      scalar = idx;
      return;
    }
    colour |= idx;
    // coded channel k of the fit is channel c of the block, the rotated one (code 0) skipped
    int k = 0;
#pragma unroll
    for (int c = 0; c < 3; c++) {
      if (c == rot - 1) continue;
      w.put((c0 >> (8 * k)) & 255u, cstart + ((c * I.ns + i) * 2) * I.cb);
      w.put((c1 >> (8 * k)) & 255u, cstart + ((c * I.ns + i) * 2 + 1) * I.cb);
      k++;
    }
    if (I.epb) w.put((uint64_t)(p0 | (p1 << 1)), pstart + 2 * i);
    if (I.spb) w.put((uint64_t)p0, pstart + i);
  }

  __device__ __forceinline__ uint4 finish() {
    const ModeInfo I = mode_info(mode);
    const int istart = mode + 1 + I.pb + I.rb + I.isb + 6 * I.ns * I.cb + 2 * I.ns * I.ab + (I.epb ? 2 * I.ns : (I.spb ? I.ns : 0));
    if (I.ib2) {
      const uint64_t first = isb ? scalar : colour, second = isb ? colour : scalar;
      w.put(drop_bit(pack_indices(first, I.ib), I.ib - 1), istart);
      w.put(drop_bit(pack_indices(second, I.ib2), I.ib2 - 1), istart + 16 * I.ib - 1);
    } else {
      uint64_t x = pack_indices(colour, I.ib);
      const int a1 = I.ns >= 2 ? anchor_of(I.ns, part, 1) : 0, a2 = I.ns >= 3 ? anchor_of(I.ns, part, 2) : 0;
      if (max(a1, a2) > 0) x = drop_bit(x, max(a1, a2) * I.ib + I.ib - 1);
      if (min(a1, a2) > 0) x = drop_bit(x, min(a1, a2) * I.ib + I.ib - 1);
      w.put(drop_bit(x, I.ib - 1), istart);
    }
    return make_uint4((uint32_t)w.lo, (uint32_t)(w.lo >> 32), (uint32_t)w.hi, (uint32_t)(w.hi >> 32));
  }
};

__device__ __noinline__ uint4 solve_pack(const uint32_t* tex, int e, const uint8_t* sq) {
  Packer K;
  K.start(e);
#pragma unroll 1
  for (int i = 0; i < K.parts(); i++) K.solve(tex, sq, i);
  return K.finish();
}

// Constant blocks (Sec. III-A: a block of one colour can be coded without error; the format
// reaches every constant colour): mode 5, rotation 0, every colour index 1 (weight 21), per
// channel the code pair of c_const7, alpha codes all ones and alpha indices 0. Texel t of the
// thread's block is tex[t * BC7_STRIDE]; returns whether the block is constant.
__device__ __forceinline__ bool const_block(const uint32_t* tex, uint4* out) {
  const uint32_t c = tex[0];
  bool same = true;
#pragma unroll
  for (int t = 1; t < 16; t++) same &= tex[t * BC7_STRIDE] == c;
  if (!same) return false;
  Bits128 w = {0ull, 0ull};
  w.put(1ull << 5, 0);
#pragma unroll
  for (int ch = 0; ch < 3; ch++) {
    const uint32_t ab = c_const7[(c >> (8 * ch)) & 255u];
    w.put(ab & 255u, 8 + 14 * ch);
    w.put(ab >> 8, 15 + 14 * ch);
  }
  w.put(0xFFFFull, 50);
  w.put(0x2AAAAAABull, 66);  // texel 0: one bit, the others two bits, all 1
  *out = make_uint4((uint32_t)w.lo, (uint32_t)(w.lo >> 32), (uint32_t)w.hi, (uint32_t)(w.hi >> 32));
  return true;
}
