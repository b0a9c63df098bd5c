// sort.cu -- device-wide stable LSD radix sort of (key, u32 value) pairs, 8-bit digits, and the exclusive scan.
//
// A pass is three kernels over tiles of 4096 pairs: digit counts per tile, a scan of each digit's row of counts
// (one CTA per digit), and the tiles ranked, sorted in shared memory and written out in runs: 9 + 3 + 24 us at 3M
// pairs of 32-bit keys (one GB300, each kernel alone with cold caches), against 12 + 15 + 58 us with a three-kernel
// scan and three CTA barriers per 32 items in the scatter. The scatter is bound by latency: with the values read only
// after the keys had been placed, and half the items in flight, it took 33 us, and 30M pairs of 16-bit keys 246 us
// against 149 us; three CTAs per SM (80 registers; 60 bytes spilled with 32-bit keys, 124 with 64-bit ones, none with
// 16-bit ones) were best with 32-bit keys, four take as long with 16-bit ones. No kernel waits for another CTA: chaining the tiles in
// one kernel (decoupled look-back) took 41 us per pass with two resident CTAs per SM and 470 us with four, when
// most of the machine polled. 32-bit keys where the caller's fit.
#include "sort.cuh"
#include "sort_digits.h"

// ---- scan (exclusive, 64-bit) -------------------------------------------------------------
#define SCAN_BLOCK 1024
static int64_t scan_blocks(int64_t n) { return ceil_div64(n > 0 ? n : 1, SCAN_BLOCK); }
size_t scan_ws_bytes(int64_t n) {
  int64_t nb = scan_blocks(n);
  return align_up(sizeof(uint64_t) * (size_t)nb, 256) + align_up(sizeof(uint64_t) * (size_t)scan_blocks(nb), 256) + 256;
}

template <class T>
__device__ __forceinline__ uint64_t block_excl_scan(uint64_t v, uint64_t* s_warp, uint64_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  if (w == 0) {
    uint64_t y = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      uint64_t z = __shfl_up_sync(0xFFFFFFFFu, y, d);
      if (lane >= d) y += z;
    }
    s_warp[lane] = y;  // inclusive over warps
  }
  __syncthreads();
  uint64_t before = (w > 0 ? s_warp[w - 1] : 0) + x - v;
  if (total) *total = s_warp[(blockDim.x >> 5) - 1];
  __syncthreads();
  return before;
}

template <class T>
__global__ void k_scan_reduce(const T* __restrict__ in, int64_t n, uint64_t* __restrict__ sums) {
  __shared__ uint64_t s_warp[32];
  const int64_t i = (int64_t)blockIdx.x * SCAN_BLOCK + threadIdx.x;
  uint64_t v = i < n ? (uint64_t)in[i] : 0;
  uint64_t tot;
  block_excl_scan<T>(v, s_warp, &tot);
  if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

template <class T>
__global__ void k_scan_apply(const T* __restrict__ in, int64_t n, const uint64_t* __restrict__ offs,
                             T* __restrict__ out, uint64_t* __restrict__ total) {
  __shared__ uint64_t s_warp[32];
  const int64_t i = (int64_t)blockIdx.x * SCAN_BLOCK + threadIdx.x;
  uint64_t v = i < n ? (uint64_t)in[i] : 0;
  uint64_t tot;
  uint64_t ex = block_excl_scan<T>(v, s_warp, &tot) + (offs ? offs[blockIdx.x] : 0);
  if (i < n) out[i] = (T)ex;
  if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *total = (offs ? offs[blockIdx.x] : 0) + tot;
}

// single-block scan of up to SCAN_BLOCK * k elements held in one array (sequential chunks)
__global__ void k_scan_single(uint64_t* __restrict__ a, int64_t n) {
  __shared__ uint64_t s_warp[32];
  __shared__ uint64_t carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < n; base += SCAN_BLOCK) {
    const int64_t i = base + threadIdx.x;
    uint64_t v = i < n ? a[i] : 0;
    uint64_t tot;
    uint64_t ex = block_excl_scan<uint64_t>(v, s_warp, &tot);
    if (i < n) a[i] = ex + carry;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
}

// Exclusive scan of n values of T (uint32 or uint64) into out (may alias in); total (device, optional).
template <class T>
cudaError_t scan_exclusive(const T* in, T* out, int64_t n, uint64_t* total, void* ws, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t nb = scan_blocks(n);
  uint64_t* sums = reinterpret_cast<uint64_t*>(ws);
  gsc_count_launch(); k_scan_reduce<T><<<(int)nb, SCAN_BLOCK, 0, st>>>(in, n, sums);
  gsc_count_launch(); k_scan_single<<<1, SCAN_BLOCK, 0, st>>>(sums, nb);
  gsc_count_launch(); k_scan_apply<T><<<(int)nb, SCAN_BLOCK, 0, st>>>(in, n, sums, out, total);
  return cudaGetLastError();
}
template cudaError_t scan_exclusive<uint32_t>(const uint32_t*, uint32_t*, int64_t, uint64_t*, void*, cudaStream_t);
template cudaError_t scan_exclusive<uint64_t>(const uint64_t*, uint64_t*, int64_t, uint64_t*, void*, cudaStream_t);

// ---- radix sort -------------------------------------------------------------------------------
#define RS_THREADS 256
#define RS_ITEMS 16
#define RS_WARPS (RS_THREADS / 32)
#define RS_TILE (RS_THREADS * RS_ITEMS)

static int64_t rs_tiles(int64_t n) { return ceil_div64(n > 0 ? n : 1, RS_TILE); }
// digit totals [256], then counts [256][tiles]
size_t radix_state_bytes(int64_t n) { return 1024 + sizeof(uint32_t) * 256 * (size_t)rs_tiles(n); }

size_t radix_ws_bytes(int64_t n) {
  return align_up(sizeof(uint64_t) * (size_t)(n > 0 ? n : 1), 256) + align_up(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1), 256) +
         radix_state_bytes(n);
}

template <class K>
__global__ void __launch_bounds__(RS_THREADS) k_rs_count(const K* __restrict__ keys, int64_t n, int shift, uint32_t mask,
                                                        uint32_t* __restrict__ counts) {
  __shared__ uint32_t h[256];
  const int t = threadIdx.x, lane = t & 31;
  h[t] = 0u;
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  K k[RS_ITEMS];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) k[r] = base + r * RS_THREADS + t < n ? keys[base + r * RS_THREADS + t] : (K)0;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const bool live = base + r * RS_THREADS + t < n;
    const uint32_t d = live ? (uint32_t)(k[r] >> shift) & mask : 256u;
    // lanes of one digit (all of them, where the digit is already sorted by) in one addition
    const unsigned same = __ballot_sync(0xFFFFFFFFu, d == __shfl_sync(0xFFFFFFFFu, d, 0));
    if (lane == 0) { if (live) atomicAdd(&h[d], (uint32_t)__popc(same)); }
    else if (live && !((same >> lane) & 1u)) atomicAdd(&h[d], 1u);
  }
  __syncthreads();
  counts[(int64_t)t * gridDim.x + blockIdx.x] = h[t];
}

// CTA d: the exclusive prefix of digit d's counts over the tiles, in place, and its total
__global__ void __launch_bounds__(256) k_rs_rows(uint32_t* __restrict__ counts, int64_t nt, uint32_t* __restrict__ total) {
  __shared__ uint32_t s[8];
  uint32_t* row = counts + (int64_t)blockIdx.x * nt;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint32_t carry = 0u;
  for (int64_t b = 0; b < nt; b += 1024) {
    uint32_t v[4], sum = 0u;
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int64_t i = b + 4 * t + j;
      v[j] = i < nt ? row[i] : 0u;
      sum += v[j];
    }
    uint32_t x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
      if (lane >= d) x += y;
    }
    if (lane == 31) s[w] = x;
    __syncthreads();
    uint32_t before = carry + x - sum;
    for (int k = 0; k < 8; k++) {
      if (k < w) before += s[k];
      carry += s[k];
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int64_t i = b + 4 * t + j;
      if (i < nt) row[i] = before;
      before += v[j];
    }
    __syncthreads();
  }
  if (t == 0) total[blockIdx.x] = carry;
}

// vin = nullptr: values are the input positions; kout = nullptr: the sorted keys are not wanted. digit_mask: the pass's
// digit as it was counted. From 5 bits on it is known from BITS (with the mask in a register 30M pairs of 16-bit keys
// take 154 us instead of 149).
template <class K, int BITS>
__global__ void __launch_bounds__(RS_THREADS, 3)
    k_rs_scatter(const K* __restrict__ kin, const uint32_t* __restrict__ vin, int64_t n, int shift, uint32_t digit_mask,
                 const uint32_t* __restrict__ total, const uint32_t* __restrict__ counts, K* __restrict__ kout,
                 uint32_t* __restrict__ vout) {
  __shared__ K s_key[RS_TILE];
  __shared__ uint32_t s_val[RS_TILE];
  __shared__ uint32_t s_cnt[RS_WARPS][256];
  __shared__ uint32_t s_start[256], s_base[256];
  __shared__ uint64_t s_scan[8];
  const uint32_t mask = BITS > 4 ? (1u << BITS) - 1u : digit_mask;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t base = (int64_t)blockIdx.x * RS_TILE;
  const int count = (int)min((int64_t)RS_TILE, n - base);
  constexpr bool PACK = sizeof(K) == 2;  // the key's bits above its item's rank
  K key[PACK ? 1 : RS_ITEMS];
  uint32_t val[RS_ITEMS], rank[RS_ITEMS];
  const int first = w * (RS_ITEMS * 32) + lane;  // the thread's items: first + 32 r
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const K k = first + 32 * r < count ? kin[base + first + 32 * r] : (K)0;
    if (PACK) rank[r] = (uint32_t)k << 16;
    else key[r] = k;
  }
  const uint32_t before = counts[(int64_t)t * gridDim.x + blockIdx.x], all = total[t];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++)
    val[r] = !vin ? (uint32_t)(base + first + 32 * r) : first + 32 * r < count ? __ldg(vin + base + first + 32 * r) : 0u;
  auto key_of = [&](int r) { return PACK ? (K)(rank[r] >> 16) : key[PACK ? 0 : r]; };
  auto digit = [&](int r) { return first + 32 * r < count ? (uint32_t)(key_of(r) >> shift) & mask : 256u; };
  const uint32_t mine = rank_digits<RS_WARPS, RS_ITEMS, BITS>(digit, [&](int r, uint32_t x) { rank[r] = PACK ? rank[r] | x : x; }, s_cnt);
  // where digit t starts in the output and in the tile
  const uint64_t both = prefix256(((uint64_t)all << 16) | mine, s_scan);
  const uint32_t start = (uint32_t)(both & 0xFFFFu);
  s_start[t] = start;
  s_base[t] = (uint32_t)(both >> 16) + before - start;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++)
    if (first + 32 * r < count) {
      const uint32_t d = digit(r), at = (PACK ? rank[r] & 0xFFFFu : rank[r]) + s_start[d] + s_cnt[w][d];  // the place in the sorted tile
      s_key[at] = key_of(r);
      s_val[at] = val[r];
    }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const int i = r * RS_THREADS + t;
    if (i >= count) continue;
    const K k = s_key[i];
    const uint32_t dst = s_base[(uint32_t)(k >> shift) & mask] + (uint32_t)i;
    if (kout) kout[dst] = k;
    vout[dst] = s_val[i];
  }
}

template <class K>
cudaError_t radix_sort(K* keys, K* keys2, uint32_t* vals, uint32_t* vals2, int64_t n, int key_bits, bool iota, bool want_keys,
                       void* state, cudaStream_t st, K** out_keys, uint32_t** out_vals) {
  // one pair: a frame of one Gaussian takes 90 us without the passes' launches, 163 us with them
  const int passes = n > 1 ? sort_passes(key_bits) : 0;
  if (n == 1 && iota) {
    const cudaError_t e = cudaMemsetAsync(vals, 0, sizeof(uint32_t), st);
    if (e != cudaSuccess) return e;
  }
  uint32_t* total = reinterpret_cast<uint32_t*>(state);
  uint32_t* counts = total + 256;
  const int nt = (int)rs_tiles(n);
  for (int p = 0; p < passes; p++) {
    const SortDigit d = sort_digit(key_bits, p);
    gsc_count_launch(); k_rs_count<K><<<nt, RS_THREADS, 0, st>>>(keys, n, d.shift, d.mask, counts);
    gsc_count_launch(); k_rs_rows<<<256, 256, 0, st>>>(counts, nt, total);
    gsc_count_launch();
    const uint32_t* vin = p == 0 && iota ? nullptr : vals;
    K* kout = p + 1 < passes || want_keys ? keys2 : nullptr;
    if (d.ballots == 4) k_rs_scatter<K, 4><<<nt, RS_THREADS, 0, st>>>(keys, vin, n, d.shift, d.mask, total, counts, kout, vals2);
    else if (d.ballots == 5) k_rs_scatter<K, 5><<<nt, RS_THREADS, 0, st>>>(keys, vin, n, d.shift, d.mask, total, counts, kout, vals2);
    else if (d.ballots == 6) k_rs_scatter<K, 6><<<nt, RS_THREADS, 0, st>>>(keys, vin, n, d.shift, d.mask, total, counts, kout, vals2);
    else if (d.ballots == 7) k_rs_scatter<K, 7><<<nt, RS_THREADS, 0, st>>>(keys, vin, n, d.shift, d.mask, total, counts, kout, vals2);
    else k_rs_scatter<K, 8><<<nt, RS_THREADS, 0, st>>>(keys, vin, n, d.shift, d.mask, total, counts, kout, vals2);
    K* tk = keys; keys = keys2; keys2 = tk;
    uint32_t* tv = vals; vals = vals2; vals2 = tv;
  }
  *out_keys = keys;
  *out_vals = vals;
  return cudaGetLastError();
}
template cudaError_t radix_sort<uint16_t>(uint16_t*, uint16_t*, uint32_t*, uint32_t*, int64_t, int, bool, bool, void*, cudaStream_t,
                                          uint16_t**, uint32_t**);
template cudaError_t radix_sort<uint32_t>(uint32_t*, uint32_t*, uint32_t*, uint32_t*, int64_t, int, bool, bool, void*, cudaStream_t,
                                          uint32_t**, uint32_t**);
template cudaError_t radix_sort<uint64_t>(uint64_t*, uint64_t*, uint32_t*, uint32_t*, int64_t, int, bool, bool, void*, cudaStream_t,
                                          uint64_t**, uint32_t**);

cudaError_t radix_sort_pairs(uint64_t* keys, uint32_t* vals, int64_t n, int key_bits, void* ws, cudaStream_t st) {
  if (n <= 1 || key_bits <= 0) return cudaSuccess;
  Carve c{reinterpret_cast<uint8_t*>(ws), 0, 0};
  uint64_t* k2 = c.take<uint64_t>(n);
  uint32_t* v2 = c.take<uint32_t>(n);
  void* state = c.take<uint8_t>((int64_t)radix_state_bytes(n));
  uint64_t* ko;
  uint32_t* vo;
  cudaError_t e = radix_sort<uint64_t>(keys, k2, vals, v2, n, key_bits, false, true, state, st, &ko, &vo);
  if (e == cudaSuccess && ko != keys) {
    e = cudaMemcpyAsync(keys, ko, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(vals, vo, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
  }
  return e;
}
