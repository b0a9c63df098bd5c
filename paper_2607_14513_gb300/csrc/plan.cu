// plan.cu -- per-scene scales, quantisation and the reorder plan (Sec. V-A; Sec. III-C,
// Fig. Bit4Scan). No host synchronisation: everything is queued on the caller's stream.
#include <mutex>

#include "sort.cuh"

// ---- scales of a sharded scene: exact order statistic by 4 passes of 8-bit radix select --------
struct SelState { uint32_t prefix[GSC_SH]; uint64_t rank[GSC_SH]; };

__global__ void k_sel_init(SelState* s, uint64_t r) {
  if (threadIdx.x < GSC_SH) { s->prefix[threadIdx.x] = 0; s->rank[threadIdx.x] = r; }
}

__global__ void __launch_bounds__(256) k_sel_hist(const float4* __restrict__ sh4, int64_t n4, int shift,
                                                  const uint32_t* __restrict__ prefix, uint32_t* __restrict__ hist) {
  __shared__ uint32_t h[GSC_SH * 256];
  __shared__ uint32_t pre[GSC_SH];
  for (int i = threadIdx.x; i < GSC_SH * 256; i += blockDim.x) h[i] = 0;
  if (threadIdx.x < GSC_SH) pre[threadIdx.x] = prefix[threadIdx.x];
  __syncthreads();
  const int hs = shift + 8;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    float4 f = __ldg(sh4 + i);
    const int j0 = (int)((i * 4) % 48);
    float a[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const int k = (j0 + q) / 3;
      const uint32_t u = __float_as_uint(a[q]) & 0x7FFFFFFFu;
      if (hs >= 32 || (u >> hs) == (pre[k] >> hs)) atomicAdd(&h[k * 256 + ((u >> shift) & 255)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < GSC_SH * 256; i += blockDim.x)
    if (h[i]) atomicAdd(&hist[i], h[i]);
}

// The digit of this pass: the first whose cumulative count passes the remaining rank.
__global__ void k_sel_pick(SelState* st, const int64_t* hist, int shift) {
  const int k = threadIdx.x;
  if (k >= GSC_SH) return;
  uint64_t r = st->rank[k], cum = 0;
  int d = 0;
  for (d = 0; d < 256; d++) {
    uint64_t c = (uint64_t)hist[k * 256 + d];
    if (r < cum + c) break;
    cum += c;
  }
  if (d > 255) d = 255;
  st->prefix[k] |= (uint32_t)d << shift;
  st->rank[k] = r - cum;
}

__global__ void k_sel_finish(const SelState* st, float* scales) {
  const int k = threadIdx.x;
  if (k >= GSC_SH) return;
  float s = 2.0f * __uint_as_float(st->prefix[k]);
  scales[k] = (s == 0.0f) ? 1.0f : s;
}

__global__ void k_fill_scales_one(float* scales) {
  if (threadIdx.x < GSC_SH) scales[threadIdx.x] = 1.0f;
}

// ---- quantisation kernel (Sec. V-A) ----------------------------------------------------------
__global__ void k_quantise(const float4* __restrict__ sh4, int64_t n4, const float* __restrict__ scales,
                           uchar4* __restrict__ q4) {
  __shared__ float s_scale[GSC_SH];
  if (threadIdx.x < GSC_SH) s_scale[threadIdx.x] = scales[threadIdx.x];
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += (int64_t)gridDim.x * blockDim.x) {
    float4 f = __ldg(sh4 + i);
    const int j0 = (int)((i * 4) % 48);
    uchar4 o;
    o.x = (uint8_t)gsc_quant1(f.x, s_scale[(j0 + 0) / 3]);
    o.y = (uint8_t)gsc_quant1(f.y, s_scale[(j0 + 1) / 3]);
    o.z = (uint8_t)gsc_quant1(f.z, s_scale[(j0 + 2) / 3]);
    o.w = (uint8_t)gsc_quant1(f.w, s_scale[(j0 + 3) / 3]);
    q4[i] = o;
  }
}

static int grid_stride(int64_t n, int threads, int cap = gsc_sm_count() * 8) {
  int64_t g = ceil_div64(n > 0 ? n : 1, threads);
  return (int)(g > cap ? cap : g);
}

cudaError_t launch_quantise(const float* sh, int64_t n, const float* scales, uint8_t* q, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int64_t n4 = n * 12;
  gsc_count_launch(); k_quantise<<<grid_stride(n4, 256), 256, 0, st>>>(reinterpret_cast<const float4*>(sh), n4, scales,
                                                    reinterpret_cast<uchar4*>(q));
  return cudaGetLastError();
}

// ---- bounding box, Morton keys, colour keys --------------------------------------------------
__device__ __forceinline__ uint32_t f2ord(float f) {
  uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float ord2f(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}

__global__ void k_bbox_init(uint32_t* bb) {
  if (threadIdx.x < 3) { bb[threadIdx.x] = 0xFFFFFFFFu; bb[3 + threadIdx.x] = 0u; }
}

__global__ void k_bbox(const float* __restrict__ pos, int64_t n, uint32_t* __restrict__ bb) {
  uint32_t lo[3] = {0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu}, hi[3] = {0, 0, 0};
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
      uint32_t o = f2ord(__ldg(pos + 3 * i + a));
      lo[a] = min(lo[a], o);
      hi[a] = max(hi[a], o);
    }
  }
#pragma unroll
  for (int a = 0; a < 3; a++) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      lo[a] = min(lo[a], __shfl_xor_sync(0xFFFFFFFFu, lo[a], d));
      hi[a] = max(hi[a], __shfl_xor_sync(0xFFFFFFFFu, hi[a], d));
    }
  }
  if ((threadIdx.x & 31) == 0)
#pragma unroll
    for (int a = 0; a < 3; a++) { atomicMin(&bb[a], lo[a]); atomicMax(&bb[3 + a], hi[a]); }
}

__device__ __forceinline__ uint32_t spread3(uint32_t x) {  // 10 bits -> every third bit
  x &= 0x3FFu;
  x = (x | (x << 16)) & 0x030000FFu;
  x = (x | (x << 8)) & 0x0300F00Fu;
  x = (x | (x << 4)) & 0x030C30C3u;
  x = (x | (x << 2)) & 0x09249249u;
  return x;
}

__device__ __forceinline__ uint32_t grid10(float p, float lo, float ext) {
  if (ext == 0.0f) return 0;
  float t = __fmul_rn(__fdiv_rn(__fsub_rn(p, lo), ext), 1024.0f);
  uint32_t u = (uint32_t)floorf(t);
  return u > 1023u ? 1023u : u;
}

__device__ __forceinline__ uint32_t spread8(uint32_t x) {  // 8 bits -> every third bit (24-bit result)
  x &= 0xFFu;
  x = (x | (x << 8)) & 0x00F00Fu;
  x = (x | (x << 4)) & 0x0C30C3u;
  x = (x | (x << 2)) & 0x249249u;
  return x;
}

__global__ void k_colour_keys(const float* __restrict__ sh, const float* __restrict__ scales, int64_t n,
                              int64_t group_size, uint64_t* __restrict__ keys, const uint32_t* __restrict__ vals) {
  const float s0 = scales[0];
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t i = vals[r];
    const float* dc = sh + (int64_t)i * 48;
    uint32_t q0 = gsc_quant1(__ldg(dc + 0), s0), q1 = gsc_quant1(__ldg(dc + 1), s0), q2 = gsc_quant1(__ldg(dc + 2), s0);
    uint64_t chunk = group_size ? (uint64_t)(r / group_size) : 0;
    keys[r] = (chunk << 24) | (spread8(q0) << 2) | (spread8(q1) << 1) | spread8(q2);
  }
}

__global__ void k_finish_perm(const uint32_t* __restrict__ vals, int64_t n, int64_t ns, int identity,
                              int32_t* __restrict__ perm) {
  for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < ns; s += (int64_t)gridDim.x * blockDim.x)
    perm[s] = s < n ? (identity ? (int32_t)s : (int32_t)vals[s]) : -1;
}

// ---- the whole-scene plan -----------------------------------------------------------------------
// Scales. Small scenes (up to PLAN_SMALL): one CTA per coefficient holds all its magnitudes in shared memory and
// selects the rank, ten bits at a time. Larger ones: a stratified sample of 4,096 Gaussians brackets each
// coefficient's rank (six standard deviations of the sample's rank either way), one read of the scene counts what lies
// below and at the bracket's ends and collects what lies inside, and one CTA per coefficient selects among those. The
// four full reads that a plain radix selection takes (576 MB each at 3M Gaussians, every value an atomic in shared
// memory) were 720 of 1570 us; the bracketed one is 30 + 122 + 64 us, its read at 69% of the copy bandwidth.
// At 995 permille 0.9% of the values lie inside. Towards the middle of the distribution it would be up to 5.5%, more
// than there is room for (n / 8 of a coefficient's 3 n): where it is more than SEL_WIDE the sample is three times as
// large, and 3.2% lie inside at 500 permille (71 + 152 + 190 us; 11.9 ms in all when it did not fit). The line: 3M
// Gaussians at 970 permille (2.0%) take 467 us with the large sample, 479 with the small one, 100,000 without the
// sort 111 and 77.
// Where the rank is outside its bracket or the inside overflows its buffer all the same (a sample that does not stand
// for the scene), that CTA selects over the whole scene: the result is the exact order statistic either way.
#define PLAN_SMALL 8192
#define SEL_SAMPLE 4096
#define SEL_SAMPLE_WIDE 12288
#define SEL_WIDE 0.02
#define SEL_THREADS 1024

struct SelBracket {
  uint32_t lo[GSC_SH], hi[GSC_SH];
  unsigned long long below[GSC_SH], at_lo[GSC_SH], at_hi[GSC_SH];
  uint32_t inside[GSC_SH];
};

__device__ __forceinline__ uint32_t magnitude(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }

// The value of rank `rank` (from 0) among get(0..m-1), all below 2^bits, by a CTA of SEL_THREADS threads, ten bits at a
// time. hist: 1024, pick: 34 shared words (32 bits each: a scene of 2^32 values fits no device).
template <class Get>
__device__ __forceinline__ uint32_t select_rank(int64_t m, uint64_t rank, int bits, Get get, uint32_t* hist, uint32_t* pick) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint32_t prefix = 0u, left = (uint32_t)rank;
  for (int top = bits; top > 0; top -= 10) {
    const int shift = top > 10 ? top - 10 : 0, width = top - shift;
    hist[t] = 0u;
    __syncthreads();
    for (int64_t b = 0; b < m; b += 8 * SEL_THREADS) {
      uint32_t u[8];
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const int64_t i = b + j * SEL_THREADS + t;
        u[j] = i < m ? get(i) : 0xFFFFFFFFu;
      }
#pragma unroll
      for (int j = 0; j < 8; j++) {
        const bool in = b + j * SEL_THREADS + t < m && (u[j] >> shift >> width) == prefix;
        const uint32_t d = in ? (u[j] >> shift) & ((1u << width) - 1u) : 0xFFFFu;
        // the lanes of the first live lane's digit in one addition: most of a warp, in the leading digits
        const unsigned live = __ballot_sync(0xFFFFFFFFu, in);
        if (live == 0u) continue;
        const int first = __ffs(live) - 1;
        const unsigned same = __ballot_sync(0xFFFFFFFFu, d == __shfl_sync(0xFFFFFFFFu, d, first));
        if (lane == first) atomicAdd(&hist[d], (uint32_t)__popc(same));
        else if (in && !((same >> lane) & 1u)) atomicAdd(&hist[d], 1u);
      }
    }
    __syncthreads();
    // thread t holds bin t: the one whose running count passes the rank
    const uint32_t c = hist[t];
    uint32_t x = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) pick[w] = x;
    __syncthreads();
    uint32_t before = x - c;
    for (int k = 0; k < w; k++) before += pick[k];
    if (left >= before && left - before < c) { pick[32] = (uint32_t)t; pick[33] = left - before; }
    __syncthreads();
    prefix = (prefix << width) | pick[32];
    left = pick[33];
    __syncthreads();
  }
  return prefix;
}

__device__ __forceinline__ float scale_of(uint32_t bits) {
  const float s = 2.0f * __uint_as_float(bits);
  return s == 0.0f ? 1.0f : s;
}

// half the bracket's width in ranks of a sample of m values, around quantile q
__host__ __device__ __forceinline__ double sel_half(double q, int m) { return 6.0 * sqrt((double)m * q * (1.0 - q)) + 8.0; }

// CTAs 2 k and 2 k + 1: the low and the high end of coefficient k's bracket from a sample of SAMPLE Gaussians, and cleared
// counters
template <int SAMPLE>
__global__ void __launch_bounds__(SEL_THREADS) k_sel_sample(const float* __restrict__ sh, int64_t n, unsigned long long rank,
                                                           SelBracket* __restrict__ S) {
  extern __shared__ uint32_t v[];  // 3 * SAMPLE
  __shared__ uint32_t hist[1024], pick[34];
  const int k = blockIdx.x >> 1, m = 3 * SAMPLE;
  const bool low = (blockIdx.x & 1) == 0;
#pragma unroll 12
  for (int j = 0; j < m / SEL_THREADS; j++) {
    // one Gaussian of each of SAMPLE equal strata, at a place drawn by a hash
    const int i = j * SEL_THREADS + threadIdx.x;
    const uint64_t g = (uint64_t)(i / 3);
    uint64_t h = (g + 1) * 0x9E3779B97F4A7C15ull;
    h = (h ^ (h >> 29)) * 0xBF58476D1CE4E5B9ull;
    const int64_t at = (int64_t)((g * (uint64_t)n + (h >> 16) % (uint64_t)n) / SAMPLE);
    v[i] = magnitude(__ldg(sh + at * 48 + 3 * k + i % 3));
  }
  __syncthreads();
  const double q = ((double)rank + 0.5) / (3.0 * (double)n), mid = q * m;
  const double wide = sel_half(q, m);
  const int64_t a = (int64_t)floor(mid - wide), b = (int64_t)ceil(mid + wide);
  auto get = [&](int64_t i) { return v[i]; };
  if (low) {
    const uint32_t lo = a <= 0 ? 0u : select_rank(m, (uint64_t)a, 31, get, hist, pick);
    if (threadIdx.x == 0) {
      S->lo[k] = lo;
      S->below[k] = S->at_lo[k] = S->at_hi[k] = 0ull;
      S->inside[k] = 0u;
    }
  } else {
    const uint32_t hi = b >= m - 1 ? 0x7FFFFFFFu : select_rank(m, (uint64_t)b, 31, get, hist, pick);
    if (threadIdx.x == 0) S->hi[k] = hi;
  }
}

// One read of the scene. The grid's threads are a multiple of 12, so a thread's float4s always hold the same four
// places of the 48 and its brackets stay in registers; what lies inside goes through a buffer per CTA, which is written
// out every `rounds` rounds of four loads (a value of a full buffer takes a global addition of its own: the selection
// at 900 permille and 12M Gaussians took 9.2 ms, against 1.0 ms). Four CTAs per SM: 3M Gaussians 122 us, with three
// (76 registers) 138.
#define SEL_KEEP 256
struct SelCand {
  uint32_t* half[2];  // of coefficients 0-7 and 8-15
  uint32_t cap;       // values of one coefficient
  __device__ __forceinline__ uint32_t* of(int k) const { return half[k >> 3] + (int64_t)(k & 7) * cap; }
};
__global__ void __launch_bounds__(256, 4) k_sel_scan(const float4* __restrict__ sh4, int64_t n4, int rounds,
                                                  SelBracket* __restrict__ S, SelCand cand) {
  __shared__ uint32_t s_buf[GSC_SH][SEL_KEEP];
  __shared__ uint32_t s_n[GSC_SH], s_at[GSC_SH];
  __shared__ uint32_t s_cnt[3][GSC_SH];
  if (threadIdx.x < GSC_SH) {
    s_n[threadIdx.x] = 0u;
    for (int j = 0; j < 3; j++) s_cnt[j][threadIdx.x] = 0u;
  }
  __syncthreads();
  const int64_t i0 = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
  const int j0 = (int)((i0 * 4) % 48);
  uint32_t lo[4], span[4], below[4] = {0, 0, 0, 0}, at_lo[4] = {0, 0, 0, 0}, at_hi[4] = {0, 0, 0, 0};
#pragma unroll
  for (int q = 0; q < 4; q++) { lo[q] = S->lo[(j0 + q) / 3]; span[q] = S->hi[(j0 + q) / 3] - lo[q]; }
  auto count = [&](float4 f) {
    const uint32_t u[4] = {magnitude(f.x), magnitude(f.y), magnitude(f.z), magnitude(f.w)};
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint32_t d = u[q] - lo[q];  // below the bracket: wraps above the span
      below[q] += u[q] < lo[q];
      at_lo[q] += d == 0u;
      at_hi[q] += d == span[q] && d != 0u;
      if (d - 1u < span[q] - 1u && span[q] > 1u) {
        const int k = (j0 + q) / 3;
        const uint32_t at = atomicAdd(&s_n[k], 1u);
        if (at < SEL_KEEP) {
          s_buf[k][at] = u[q];
        } else {
          const uint32_t g = atomicAdd(&S->inside[k], 1u);
          if (g < cand.cap) cand.of(k)[g] = u[q];
        }
      }
    }
  };
  const int64_t full = n4 / (4 * step);  // rounds that every thread of the grid has
  int64_t i = i0;
  for (int64_t r = 0;;) {
    const int64_t stop = min(full, r + rounds);
    for (; r < stop; r++, i += 4 * step) {
      const float4 a = __ldg(sh4 + i), b = __ldg(sh4 + i + step), c = __ldg(sh4 + i + 2 * step), d = __ldg(sh4 + i + 3 * step);
      count(a);
      count(b);
      count(c);
      count(d);
    }
    if (r == full)
      for (; i < n4; i += step) count(__ldg(sh4 + i));
    __syncthreads();
    if (threadIdx.x < GSC_SH) {
      const int k = threadIdx.x;
      const uint32_t m = min(s_n[k], (uint32_t)SEL_KEEP);
      s_n[k] = m;
      s_at[k] = m ? atomicAdd(&S->inside[k], m) : 0u;
    }
    __syncthreads();
    for (int x = threadIdx.x; x < GSC_SH * SEL_KEEP; x += 256) {
      const int k = x / SEL_KEEP, j = x % SEL_KEEP;
      if (j < (int)s_n[k] && s_at[k] + (uint32_t)j < cand.cap) cand.of(k)[s_at[k] + j] = s_buf[k][j];
    }
    if (r == full) break;
    __syncthreads();
    if (threadIdx.x < GSC_SH) s_n[threadIdx.x] = 0u;
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < 4; q++) {
    const int k = (j0 + q) / 3;
    if (below[q]) atomicAdd(&s_cnt[0][k], below[q]);
    if (at_lo[q]) atomicAdd(&s_cnt[1][k], at_lo[q]);
    if (at_hi[q]) atomicAdd(&s_cnt[2][k], at_hi[q]);
  }
  __syncthreads();
  if (threadIdx.x < GSC_SH) {
    const int k = threadIdx.x;
    if (s_cnt[0][k]) atomicAdd(&S->below[k], (unsigned long long)s_cnt[0][k]);
    if (s_cnt[1][k]) atomicAdd(&S->at_lo[k], (unsigned long long)s_cnt[1][k]);
    if (s_cnt[2][k]) atomicAdd(&S->at_hi[k], (unsigned long long)s_cnt[2][k]);
  }
}

// CTA k: the rank's value of coefficient k
__global__ void __launch_bounds__(SEL_THREADS) k_sel_final(const float* __restrict__ sh, int64_t n, unsigned long long rank,
                                                          const SelBracket* __restrict__ S, SelCand cand,
                                                          float* __restrict__ scales) {
  __shared__ uint32_t hist[1024], pick[34];
  const int k = blockIdx.x;
  const unsigned long long below = S->below[k], at_lo = S->at_lo[k], inside = S->inside[k], at_hi = S->at_hi[k];
  uint32_t v;
  if (rank >= below && rank < below + at_lo) v = S->lo[k];
  else if (inside <= cand.cap && rank >= below + at_lo && rank < below + at_lo + inside)
    // from the bracket's low end: its width has far fewer digits
    v = S->lo[k] + select_rank((int64_t)inside, rank - below - at_lo, 32 - __clz(S->hi[k] - S->lo[k]),
                               [&](int64_t i) { return __ldg(cand.of(k) + i) - S->lo[k]; }, hist, pick);
  else if (inside <= cand.cap && rank >= below + at_lo + inside && rank < below + at_lo + inside + at_hi) v = S->hi[k];
  else
    v = select_rank(3 * n, rank, 31, [&](int64_t i) { return magnitude(__ldg(sh + (i / 3) * 48 + 3 * k + i % 3)); }, hist, pick);
  if (threadIdx.x == 0) scales[k] = scale_of(v);
}

// ---- spatial order ------------------------------------------------------------------------------
// The box's codes as maxima (of the inverted code for the low corner), so that zero is the start of both. The grid's
// threads are a multiple of 3: a thread reads one axis only.
__global__ void __launch_bounds__(256) k_plan_bbox(const float* __restrict__ pos, int64_t n3, uint32_t* __restrict__ bb) {
  __shared__ uint32_t s_bb[6];
  if (threadIdx.x < 6) s_bb[threadIdx.x] = 0u;
  __syncthreads();
  const int64_t i0 = (int64_t)blockIdx.x * 256 + threadIdx.x, step = (int64_t)gridDim.x * 256;
  uint32_t lo = 0u, hi = 0u;
  int64_t i = i0;
  for (; i + 3 * step < n3; i += 4 * step) {
    const float v[4] = {__ldg(pos + i), __ldg(pos + i + step), __ldg(pos + i + 2 * step), __ldg(pos + i + 3 * step)};
#pragma unroll
    for (int q = 0; q < 4; q++) { const uint32_t o = f2ord(v[q]); lo = max(lo, ~o); hi = max(hi, o); }
  }
  for (; i < n3; i += step) { const uint32_t o = f2ord(__ldg(pos + i)); lo = max(lo, ~o); hi = max(hi, o); }
  const int a = (int)(i0 % 3);
  if (i0 < n3) { atomicMax(&s_bb[a], lo); atomicMax(&s_bb[3 + a], hi); }
  __syncthreads();
  if (threadIdx.x < 6) atomicMax(&bb[threadIdx.x], s_bb[threadIdx.x]);
}

struct Grid { float lo[3], ext[3]; };
__device__ __forceinline__ Grid grid_of_box(const uint32_t* bb) {
  Grid g;
#pragma unroll
  for (int a = 0; a < 3; a++) { g.lo[a] = ord2f(~bb[a]); g.ext[a] = __fsub_rn(ord2f(bb[3 + a]), g.lo[a]); }
  return g;
}
__device__ __forceinline__ uint32_t morton30(const Grid& g, const float* p) {
  const uint32_t x = grid10(__ldg(p), g.lo[0], g.ext[0]), y = grid10(__ldg(p + 1), g.lo[1], g.ext[1]);
  return (spread3(x) << 2) | (spread3(y) << 1) | spread3(grid10(__ldg(p + 2), g.lo[2], g.ext[2]));
}

__global__ void __launch_bounds__(256) k_plan_morton(const float* __restrict__ pos, int64_t n, const uint32_t* __restrict__ bb,
                                                    uint32_t* __restrict__ keys) {
  const Grid g = grid_of_box(bb);
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) keys[i] = morton30(g, pos + 3 * i);
}

// Stable sort of up to WARPS * ITEMS * 32 (key, value) pairs in shared memory by one CTA, `passes` 8-bit digits.
template <int WARPS, int ITEMS, class V>
__device__ __forceinline__ void block_sort(uint32_t* s_key, V* s_val, uint32_t (*s_cnt)[256], uint32_t* s_start,
                                           uint64_t* s_scan, int count, int passes) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int p = 0; p < passes; p++) {
    uint32_t key[ITEMS], rank[ITEMS];
    V val[ITEMS];
    const int first = w * (ITEMS * 32) + lane;
#pragma unroll
    for (int r = 0; r < ITEMS; r++) {
      const int i = first + 32 * r;
      key[r] = i < count ? s_key[i] : 0u;
      val[r] = i < count ? s_val[i] : (V)0;
    }
    auto digit = [&](int r) { return first + 32 * r < count ? (key[r] >> (8 * p)) & 255u : 256u; };
    const uint32_t mine = rank_digits<WARPS, ITEMS, 8>(digit, [&](int r, uint32_t x) { rank[r] = x; }, s_cnt);
    const uint64_t start = prefix256(threadIdx.x < 256 ? mine : 0u, s_scan);
    if (threadIdx.x < 256) s_start[threadIdx.x] = (uint32_t)start;
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; r++)
      if (first + 32 * r < count) {
        const uint32_t d = digit(r), at = s_start[d] + s_cnt[w][d] + rank[r];
        s_key[at] = key[r];
        s_val[at] = val[r];
      }
    __syncthreads();
  }
}

// Small scenes in one launch: CTA k < 16 selects coefficient k's rank, CTA 16 (where the scene is sorted) orders the
// Gaussians in space. Dynamic shared memory: 3n magnitudes, or PLAN_SMALL keys and values and the digit counters.
__global__ void __launch_bounds__(SEL_THREADS) k_plan_small(const float* __restrict__ pos, const float* __restrict__ sh, int n,
                                                           unsigned long long rank, float* __restrict__ scales,
                                                           uint32_t* __restrict__ order) {
  extern __shared__ uint32_t dyn[];
  __shared__ uint32_t hist[1024], pick[34];
  const int k = blockIdx.x, t = threadIdx.x;
  if (k < GSC_SH) {
    for (int i = t; i < 3 * n; i += SEL_THREADS) dyn[i] = magnitude(__ldg(sh + (int64_t)(i / 3) * 48 + 3 * k + i % 3));
    __syncthreads();
    const uint32_t v = select_rank(3 * n, rank, 31, [&](int64_t i) { return dyn[i]; }, hist, pick);
    if (t == 0) scales[k] = scale_of(v);
    return;
  }
  uint32_t* s_key = dyn;
  uint16_t* s_val = reinterpret_cast<uint16_t*>(s_key + PLAN_SMALL);
  uint32_t(*s_cnt)[256] = reinterpret_cast<uint32_t(*)[256]>(s_val + PLAN_SMALL);
  __shared__ uint64_t s_scan[8];
  uint32_t* s_bb = hist;
  if (t < 6) s_bb[t] = 0u;
  __syncthreads();
  uint32_t lo[3] = {0u, 0u, 0u}, hi[3] = {0u, 0u, 0u};
  for (int i = t; i < n; i += SEL_THREADS)
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const uint32_t o = f2ord(__ldg(pos + 3 * i + a));
      lo[a] = max(lo[a], ~o);
      hi[a] = max(hi[a], o);
    }
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const uint32_t x = __reduce_max_sync(0xFFFFFFFFu, lo[a]), y = __reduce_max_sync(0xFFFFFFFFu, hi[a]);
    if ((t & 31) == 0) { atomicMax(&s_bb[a], x); atomicMax(&s_bb[3 + a], y); }
  }
  __syncthreads();
  const Grid g = grid_of_box(s_bb);
  for (int i = t; i < n; i += SEL_THREADS) {
    s_key[i] = morton30(g, pos + 3 * i);
    s_val[i] = (uint16_t)i;
  }
  __syncthreads();
  block_sort<SEL_THREADS / 32, PLAN_SMALL / SEL_THREADS, uint16_t>(s_key, s_val, s_cnt, hist, s_scan, n, 4);
  for (int i = t; i < n; i += SEL_THREADS) order[i] = s_val[i];
}

// ---- colour order inside the chunks ---------------------------------------------------------------
// Chunks of up to CHUNK_TILE Gaussians of the spatial order are whole in a CTA's tile (several small ones share one,
// told apart by the key's top byte), so the second sort needs no pass over global memory: keys are made from the
// gathered colours and sorted in shared memory: 118 us at 3M Gaussians, against 147 us for the keys and 5 passes of
// the device-wide sort. Chunks above that (and the whole scene as one) go through the device-wide sort.
#define CHUNK_TILE 4096
#define CHUNK_THREADS 512
__global__ void __launch_bounds__(CHUNK_THREADS) k_chunk_order(const float* __restrict__ sh, const float* __restrict__ scales,
                                                              int64_t n, int64_t ns, int group, int tile_items,
                                                              const uint32_t* __restrict__ order, int32_t* __restrict__ perm) {
  __shared__ uint32_t s_key[CHUNK_TILE];
  __shared__ uint16_t s_val[CHUNK_TILE];
  __shared__ uint32_t s_cnt[CHUNK_THREADS / 32][256];
  __shared__ uint32_t s_start[256];
  __shared__ uint64_t s_scan[8];
  const int64_t base = (int64_t)blockIdx.x * tile_items;
  const int count = (int)min((int64_t)tile_items, n - base);
  const float s0 = __ldg(scales);
  // the gather's loads in flight together
  constexpr int EACH = CHUNK_TILE / CHUNK_THREADS;
  uint32_t from[EACH];
  float dc[EACH][3];
#pragma unroll
  for (int r = 0; r < EACH; r++) {
    const int i = threadIdx.x + r * CHUNK_THREADS;
    from[r] = i < count ? __ldg(order + base + i) : 0u;
  }
#pragma unroll
  for (int r = 0; r < EACH; r++)
#pragma unroll
    for (int c = 0; c < 3; c++) dc[r][c] = __ldg(sh + (int64_t)from[r] * 48 + c);
#pragma unroll
  for (int r = 0; r < EACH; r++) {
    const int i = threadIdx.x + r * CHUNK_THREADS;
    if (i >= count) break;
    const uint32_t q0 = gsc_quant1(dc[r][0], s0), q1 = gsc_quant1(dc[r][1], s0), q2 = gsc_quant1(dc[r][2], s0);
    s_key[i] = ((uint32_t)(i / group) << 24) | (spread8(q0) << 2) | (spread8(q1) << 1) | spread8(q2);
    s_val[i] = (uint16_t)i;
  }
  __syncthreads();
  block_sort<CHUNK_THREADS / 32, CHUNK_TILE / CHUNK_THREADS, uint16_t>(s_key, s_val, s_cnt, s_start, s_scan, count,
                                                                        count > group ? 4 : 3);
  for (int i = threadIdx.x; i < count; i += CHUNK_THREADS) perm[base + i] = (int32_t)order[base + s_val[i]];
  // the padding slots past the last Gaussian
  if (base + count == n && threadIdx.x < ns - n) perm[n + threadIdx.x] = -1;
}

// The sorts' arrays, shared by the phases: two of 4 bytes and two of 8 bytes per Gaussian (32-bit spatial keys in the
// lower halves beside the selection's collected values in the upper ones, then 64-bit colour keys of chunks above
// CHUNK_TILE).
struct PlanWs {
  uint32_t *va, *vb;
  uint64_t *ka, *kb;
  SelBracket* sel;
  uint32_t* bb;
  void* state;
  size_t end;
};
static PlanWs carve_plan(void* ws, int64_t n) {
  Carve c{reinterpret_cast<uint8_t*>(ws), 0, 0};
  PlanWs w;
  w.va = c.take<uint32_t>(n);
  w.vb = c.take<uint32_t>(n);
  w.ka = c.take<uint64_t>(n);
  w.kb = c.take<uint64_t>(n);
  w.sel = c.take<SelBracket>(1);
  w.bb = c.take<uint32_t>(8);
  w.state = c.take<uint8_t>((int64_t)radix_state_bytes(n));
  w.end = c.off;
  return w;
}
size_t plan_ws_bytes(int64_t n) { return carve_plan(nullptr, n).end + 256; }

#define SMALL_SORT_BYTES (PLAN_SMALL * 6 + (SEL_THREADS / 32) * 1024)
cudaError_t plan_init() {  // dynamic shared memory above 48 KB, once per device
  cudaError_t e = cudaFuncSetAttribute(k_sel_sample<SEL_SAMPLE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 12 * SEL_SAMPLE);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_sel_sample<SEL_SAMPLE_WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 12 * SEL_SAMPLE_WIDE);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_plan_small, cudaFuncAttributeMaxDynamicSharedMemorySize, 12 * PLAN_SMALL);
  return e;
}

static int bits_for(uint64_t v) { int b = 0; while (v) { b++; v >>= 1; } return b; }

// The selection of the scales and the spatial order need nothing of each other, and neither fills the chip (the one
// waits for the scene's bytes, or runs 16 CTAs; the other's passes are short): the selection goes to one of the
// context's side streams. 3M Gaussians: the plan takes 460 us, against 547 us on one stream; 20,000: 147 against
// 178 us. Plans take the side streams in turn, so that plans on up to four streams of a context (the batched form's
// lanes) don't wait for one another: 64 scenes of 50,000 to 2M Gaussians planned on four streams 5.2 ms, against 6.3 ms
// with one side stream for all and 5.8 ms with none. On a stream of another priority than the side streams' (the default)
// all stays on that stream, and so it does under capture, so that a side stream is never part of a graph that
// another call could run into. A return before join() still makes st wait for the side's work.
struct SideStream {
  gsc_ctx* c;
  cudaStream_t main, st;
  gsc_side* side = nullptr;
  bool pending = false;
  SideStream(gsc_ctx* ctx, cudaStream_t s) : c(ctx), main(s), st(s) {}
  cudaError_t fork() {
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    cudaError_t e = cudaStreamIsCapturing(main, &cap);
    if (e != cudaSuccess || cap != cudaStreamCaptureStatusNone) return e;
    gsc_side* s = &c->side[c->side_turn % GSC_SIDES];
    int mine = 0, its = 0;
    if ((e = cudaStreamGetPriority(main, &mine)) != cudaSuccess) return e;
    if ((e = cudaStreamGetPriority(s->st, &its)) != cudaSuccess || mine != its) return e;
    c->side_turn++;
    if ((e = cudaEventRecord(s->fork, main)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(s->st, s->fork, 0)) != cudaSuccess) return e;
    side = s;
    st = s->st;
    return cudaSuccess;
  }
  cudaError_t done() {
    if (!side) return cudaSuccess;
    pending = true;
    return cudaEventRecord(side->join, st);
  }
  cudaError_t join() {
    if (!pending) return cudaSuccess;
    pending = false;
    return cudaStreamWaitEvent(main, side->join, 0);
  }
  ~SideStream() { join(); }
};

gsc_status plan_run(gsc_ctx* ctx, const float* pos, const float* sh, const gsc_plan_params* pp, int32_t* perm,
                    float* scales, void* ws, size_t ws_bytes, cudaStream_t st) {
  const int64_t n = pp->n, ns = ceil_div64(n, 16) * 16;
  if (ws_bytes < plan_ws_bytes(n)) return GSC_ERR_OOM;
  const PlanWs w = carve_plan(ws, n);
  if (n == 0) {
    gsc_count_launch(); k_fill_scales_one<<<1, 32, 0, st>>>(scales);
    GSC_CUDA(cudaGetLastError());
    return GSC_OK;
  }
  const uint64_t rank = ((uint64_t)pp->quantile_permille * (3ull * (uint64_t)n) + 999) / 1000 - 1;
  const bool small = n <= PLAN_SMALL, sort = pp->sort != 0;
  if (small) {
    const size_t smem = (size_t)(12 * n) > SMALL_SORT_BYTES ? (size_t)(12 * n) : SMALL_SORT_BYTES;
    gsc_count_launch();
    k_plan_small<<<sort ? GSC_SH + 1 : GSC_SH, SEL_THREADS, smem, st>>>(pos, sh, (int)n, rank, scales, w.va);
  }
  SideStream side{ctx, st};
  if (!small) {
    if (sort) GSC_CUDA(side.fork());
    SelCand cand;
    cand.half[0] = reinterpret_cast<uint32_t*>(w.ka) + n;
    cand.half[1] = reinterpret_cast<uint32_t*>(w.kb) + n;
    cand.cap = (uint32_t)(n / 8);
    const int64_t n4 = n * 12, want = ceil_div64(n4, 256 * 4), most = (int64_t)ctx->sm_count * 8;
    const int64_t g = (want < most ? want : most) / 3 * 3;
    // the bracket's share of the values, and how many rounds (256 values of a coefficient each) leave a third of the
    // buffer to chance
    const double q = ((double)rank + 0.5) / (3.0 * (double)n);
    double share = 2.0 * sel_half(q, 3 * SEL_SAMPLE) / (3 * SEL_SAMPLE);
    const bool wide = share > SEL_WIDE;
    if (wide) share = 2.0 * sel_half(q, 3 * SEL_SAMPLE_WIDE) / (3 * SEL_SAMPLE_WIDE);
    const int rounds = (int)(0.67 * SEL_KEEP / (256.0 * share)) + 1;
    gsc_count_launch();
    if (wide) k_sel_sample<SEL_SAMPLE_WIDE><<<2 * GSC_SH, SEL_THREADS, 12 * SEL_SAMPLE_WIDE, side.st>>>(sh, n, rank, w.sel);
    else k_sel_sample<SEL_SAMPLE><<<2 * GSC_SH, SEL_THREADS, 12 * SEL_SAMPLE, side.st>>>(sh, n, rank, w.sel);
    gsc_count_launch(); k_sel_scan<<<(int)g, 256, 0, side.st>>>(reinterpret_cast<const float4*>(sh), n4, rounds, w.sel, cand);
    gsc_count_launch(); k_sel_final<<<GSC_SH, SEL_THREADS, 0, side.st>>>(sh, n, rank, w.sel, cand, scales);
    GSC_CUDA(side.done());
  }
  GSC_CUDA(cudaGetLastError());
  if (!sort) {
    gsc_count_launch(); k_finish_perm<<<grid_stride(ns, 256), 256, 0, st>>>(nullptr, n, ns, 1, perm);
    GSC_CUDA(cudaGetLastError());
    return GSC_OK;
  }
  // spatial rank: stable sort by 30-bit Morton code of the bounding-box grid
  uint32_t* order = w.va;
  if (!small) {
    GSC_CUDA(cudaMemsetAsync(w.bb, 0, 8 * sizeof(uint32_t), st));
    const int64_t want = ceil_div64(3 * n, 256 * 4), most = (int64_t)ctx->sm_count * 8;
    gsc_count_launch(); k_plan_bbox<<<(int)((want < most ? want : most) / 3 * 3), 256, 0, st>>>(pos, 3 * n, w.bb);
    uint32_t *k32 = reinterpret_cast<uint32_t*>(w.ka), *ko;
    gsc_count_launch();
    k_plan_morton<<<grid_stride(n, 256), 256, 0, st>>>(pos, n, w.bb, k32);
    GSC_CUDA(cudaGetLastError());
    GSC_CUDA(radix_sort<uint32_t>(k32, reinterpret_cast<uint32_t*>(w.kb), w.va, w.vb, n, 30, true, false, w.state, st, &ko,
                                  &order));
  }
  GSC_CUDA(side.join());
  // slot order: stable sort by (chunk, colour key) of the rank-ordered Gaussians
  if (pp->group_size > 0 && pp->group_size <= CHUNK_TILE) {
    const int group = (int)pp->group_size, tile = CHUNK_TILE / group * group;
    gsc_count_launch();
    k_chunk_order<<<(int)ceil_div64(n, tile), CHUNK_THREADS, 0, st>>>(sh, scales, n, ns, group, tile, order, perm);
    GSC_CUDA(cudaGetLastError());
    return GSC_OK;
  }
  uint64_t* ko;
  uint32_t* alt = order == w.va ? w.vb : w.va;
  gsc_count_launch(); k_colour_keys<<<grid_stride(n, 256), 256, 0, st>>>(sh, scales, n, pp->group_size, w.ka, order);
  GSC_CUDA(cudaGetLastError());
  const uint64_t max_chunk = pp->group_size ? (uint64_t)((n - 1) / pp->group_size) : 0;
  GSC_CUDA(radix_sort<uint64_t>(w.ka, w.kb, order, alt, n, 24 + bits_for(max_chunk), false, false, w.state, st, &ko, &order));
  gsc_count_launch(); k_finish_perm<<<grid_stride(ns, 256), 256, 0, st>>>(order, n, ns, 0, perm);
  GSC_CUDA(cudaGetLastError());
  return GSC_OK;
}

// ---- allocation-free variant of gsc_plan_reorder ------------------------------------------
// Scratch lives in this file-scope device array instead of a caller workspace. Every GPU
// that loads the library holds it (2 MiB) until the process exits. Its device address is
// looked up once per device, with that device current, on the first call there, and kept for
// the life of the process: a cudaDeviceReset of that device invalidates it (the module is loaded
// again, possibly elsewhere), so this entry point must not be used after such a reset.
#define GSC_PLAN_STATIC_BYTES (2u << 20)
#define GSC_MAX_DEVICES 64
static __device__ __align__(256) uint8_t g_plan_scratch[GSC_PLAN_STATIC_BYTES];
static std::mutex g_plan_scratch_mu;
static void* g_plan_scratch_ptr[GSC_MAX_DEVICES];

extern "C" gsc_status gsc_plan_reorder_static(gsc_ctx* c, const float* d_pos, const float* d_sh,
                                              const gsc_plan_params* pp, int32_t* d_perm, float* d_scales,
                                              void* stream) {
  GscRange gsc_range_("gsc_plan_reorder_static");
  if (!c || !pp || pp->n < 0 || pp->n > GSC_PLAN_STATIC_MAX_N) return GSC_ERR_INVALID_ARG;
  if (pp->group_size < 0 || pp->group_size % 16 != 0) return GSC_ERR_INVALID_ARG;
  if (pp->quantile_permille == 0 || pp->quantile_permille > 1000) return GSC_ERR_INVALID_ARG;
  if (pp->sort != 0 && pp->sort != 1) return GSC_ERR_INVALID_ARG;
  if (!d_scales || (pp->n > 0 && (!d_sh || !d_perm || (pp->sort && !d_pos)))) return GSC_ERR_INVALID_ARG;
  if (((uintptr_t)d_sh % 16) != 0) return GSC_ERR_INVALID_ARG;
  if (c->device < 0 || c->device >= GSC_MAX_DEVICES) return GSC_ERR_UNSUPPORTED;
  if (plan_ws_bytes(pp->n) > GSC_PLAN_STATIC_BYTES) return GSC_ERR_OOM;
  GSC_CUDA(cudaSetDevice(c->device));
  void* ws = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_plan_scratch_mu);
    if (!g_plan_scratch_ptr[c->device]) {
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_plan_scratch) != cudaSuccess || !p) return GSC_ERR_CUDA;
      g_plan_scratch_ptr[c->device] = p;
    }
    ws = g_plan_scratch_ptr[c->device];
  }
  GscTimed tm(c, T_PLAN, (cudaStream_t)stream);
  return plan_run(c, d_pos, d_sh, pp, d_perm, d_scales, ws, GSC_PLAN_STATIC_BYTES, (cudaStream_t)stream);
}

// ---- one scene split over shards (Sec. V-A: the scales are order statistics of the whole
// scene; Sec. III-C: the reorder works chunk by chunk once the spatial order is known) --------
// Shards hold contiguous ranges of the input. The exchanges are integer: the bounding box
// (elementwise minimum / maximum of order-preserving float codes), the Morton codes of every
// Gaussian (to fix the spatial ranks), and the selection histograms of each pass (sums). Every
// partial and every merged value is int64, so any reduction library can combine them.

__global__ void k_bbox_widen(int64_t* bb) {  // u32 codes [6] at the front of bb -> int64 [6]
  if (threadIdx.x != 0) return;
  const uint32_t* u = reinterpret_cast<const uint32_t*>(bb);
  uint32_t v[6];
  for (int a = 0; a < 6; a++) v[a] = u[a];
  for (int a = 0; a < 6; a++) bb[a] = (int64_t)v[a];
}

__global__ void k_morton_shard(const float* __restrict__ pos, int64_t n, const int64_t* __restrict__ bb,
                               uint64_t* __restrict__ keys) {
  float lo[3], ext[3];
#pragma unroll
  for (int a = 0; a < 3; a++) {
    lo[a] = ord2f((uint32_t)bb[a]);
    ext[a] = __fsub_rn(ord2f((uint32_t)bb[3 + a]), lo[a]);
  }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    uint32_t x = grid10(__ldg(pos + 3 * i + 0), lo[0], ext[0]);
    uint32_t y = grid10(__ldg(pos + 3 * i + 1), lo[1], ext[1]);
    uint32_t z = grid10(__ldg(pos + 3 * i + 2), lo[2], ext[2]);
    keys[i] = (spread3(x) << 2) | (spread3(y) << 1) | spread3(z);
  }
}

__global__ void k_iota(uint32_t* __restrict__ v, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    v[i] = (uint32_t)i;
}

__global__ void k_widen_u32(const uint32_t* __restrict__ in, int64_t* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (int64_t)in[i];
}

cudaError_t shard_bbox(const float* pos, int64_t n, int64_t* bb, int sm_count, cudaStream_t st) {
  uint32_t* u = reinterpret_cast<uint32_t*>(bb);
  gsc_count_launch(); k_bbox_init<<<1, 32, 0, st>>>(u);
  if (n > 0) { gsc_count_launch(); k_bbox<<<grid_stride(n, 256, sm_count * 2), 256, 0, st>>>(pos, n, u); }
  gsc_count_launch(); k_bbox_widen<<<1, 32, 0, st>>>(bb);
  return cudaGetLastError();
}

cudaError_t shard_morton(const float* pos, int64_t n, const int64_t* bb, uint64_t* keys, int sm_count, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  gsc_count_launch(); k_morton_shard<<<grid_stride(n, 256, sm_count * 8), 256, 0, st>>>(pos, n, bb, keys);
  return cudaGetLastError();
}

size_t shard_order_ws_bytes(int64_t n) { return radix_ws_bytes(n) + 256; }

cudaError_t shard_order(uint64_t* keys, int64_t n, int32_t* order, void* ws, int sm_count, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  uint32_t* vals = reinterpret_cast<uint32_t*>(order);
  gsc_count_launch(); k_iota<<<grid_stride(n, 256, sm_count * 8), 256, 0, st>>>(vals, n);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return radix_sort_pairs(keys, vals, n, 30, ws, st);  // stable: equal codes keep the input order
}

size_t shard_select_state_bytes() { return align_up(sizeof(SelState), 256) + sizeof(uint32_t) * GSC_SH * 256; }

cudaError_t shard_select_begin(int64_t n_total, int permille, void* state, cudaStream_t st) {
  SelState* sel = reinterpret_cast<SelState*>(state);
  const uint64_t m = 3ull * (uint64_t)n_total;
  const uint64_t r = n_total > 0 ? ((uint64_t)permille * m + 999) / 1000 - 1 : 0;
  gsc_count_launch(); k_sel_init<<<1, 32, 0, st>>>(sel, r);
  return cudaGetLastError();
}

cudaError_t shard_select_hist(const float* sh, int64_t n, int shift, void* state, int64_t* hist, int sm_count,
                              cudaStream_t st) {
  SelState* sel = reinterpret_cast<SelState*>(state);
  uint32_t* h32 = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(state) + align_up(sizeof(SelState), 256));
  cudaError_t e = cudaMemsetAsync(h32, 0, sizeof(uint32_t) * GSC_SH * 256, st);
  if (e != cudaSuccess) return e;
  if (n > 0) {
    const int64_t n4 = n * 12;
    gsc_count_launch();
    k_sel_hist<<<grid_stride(n4, 256, sm_count * 4), 256, 0, st>>>(reinterpret_cast<const float4*>(sh), n4, shift,
                                                                    sel->prefix, h32);
  }
  gsc_count_launch(); k_widen_u32<<<16, 256, 0, st>>>(h32, hist, GSC_SH * 256);
  return cudaGetLastError();
}

cudaError_t shard_select_pick(void* state, const int64_t* hist_total, int shift, cudaStream_t st) {
  gsc_count_launch();
  k_sel_pick<<<1, 32, 0, st>>>(reinterpret_cast<SelState*>(state), hist_total, shift);
  return cudaGetLastError();
}

cudaError_t shard_select_scales(const void* state, float* scales, cudaStream_t st) {
  gsc_count_launch(); k_sel_finish<<<1, 32, 0, st>>>(reinterpret_cast<const SelState*>(state), scales);
  return cudaGetLastError();
}

size_t shard_plan_ws_bytes(int64_t n) {
  return align_up(sizeof(uint64_t) * (size_t)(n > 0 ? n : 1), 256) +
         align_up(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1), 256) + radix_ws_bytes(n) + 1024;
}

// Slot order of a shard whose Gaussians are given in spatial-rank order and whose first one
// starts a chunk: the stable (chunk, colour key) sort of the whole-scene plan, on this range.
gsc_status shard_plan(const float* sh, int64_t n, const float* scales, int64_t group_size, int32_t* perm, void* ws,
                      size_t ws_bytes, int sm_count, cudaStream_t st) {
  const int64_t ns = ceil_div64(n, 16) * 16;
  if (ws_bytes < shard_plan_ws_bytes(n)) return GSC_ERR_OOM;
  if (ns == 0) return GSC_OK;
  Carve c{reinterpret_cast<uint8_t*>(ws), 0, ws_bytes};
  uint64_t* keys = c.take<uint64_t>(n);
  uint32_t* vals = c.take<uint32_t>(n);
  void* rws = c.take<uint8_t>((int64_t)radix_ws_bytes(n));
  gsc_count_launch(); k_iota<<<grid_stride(n, 256, sm_count * 8), 256, 0, st>>>(vals, n);
  gsc_count_launch(); k_colour_keys<<<grid_stride(n, 256, sm_count * 8), 256, 0, st>>>(sh, scales, n, group_size, keys, vals);
  GSC_CUDA(cudaGetLastError());
  const uint64_t max_chunk = (uint64_t)((n - 1) / group_size);
  GSC_CUDA(radix_sort_pairs(keys, vals, n, 24 + bits_for(max_chunk), rws, st));
  gsc_count_launch(); k_finish_perm<<<grid_stride(ns, 256, sm_count * 8), 256, 0, st>>>(vals, n, ns, 0, perm);
  GSC_CUDA(cudaGetLastError());
  return GSC_OK;
}
