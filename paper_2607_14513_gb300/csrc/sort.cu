// sort.cu -- device-wide stable LSD radix sort of (key, u32 value) pairs, 8-bit digits, and the exclusive scan.
//
// One read of the keys counts every pass's digits; each pass is then one kernel: a tile of 4096 pairs is ranked
// in the CTA, its digit counts are chained through the tiles before it (decoupled look-back: a tile publishes its
// counts at once and its running totals as soon as the tiles before it have theirs), sorted in shared memory and
// written out in runs. 32-bit keys where the caller's fit. Tiles take their numbers from an atomic counter, so
// every tile a CTA waits for has been started before it and waits only for earlier ones: the wait ends; it is
// bounded all the same (a tile that gives up records GSC_ERR_TIMEOUT in the context and writes nothing).
#include "sort.cuh"

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
#define RS_PASSES 8
#define RS_SPIN (1 << 20)  // polls of one look-back step (a poll is an L2 round trip: about a second in all)

// Counters of one sort, cleared before it: digit totals per pass, tile numbers per pass, and per (tile, digit) the
// look-back word, state << 62 | pass << 58 | count (state 1: the tile's own count, 2: of all tiles up to it); a
// word of another pass reads as not there yet.
struct RsState {
  uint32_t total[RS_PASSES][256];
  uint32_t next[RS_PASSES];
  uint32_t pad[56];
};

static int64_t rs_tiles(int64_t n) { return ceil_div64(n > 0 ? n : 1, RS_TILE); }
size_t radix_state_bytes(int64_t n) { return sizeof(RsState) + sizeof(uint64_t) * 256 * (size_t)rs_tiles(n); }

size_t radix_ws_bytes(int64_t n) {
  return align_up(sizeof(uint64_t) * (size_t)(n > 0 ? n : 1), 256) + align_up(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1), 256) +
         align_up(radix_state_bytes(n), 256) + 512;
}

// digit totals of every pass
template <class K>
__global__ void __launch_bounds__(256) k_rs_totals(const K* __restrict__ keys, int64_t n, int passes, int key_bits,
                                                   RsState* __restrict__ S) {
  extern __shared__ uint32_t h[];  // [passes][256]
  for (int i = threadIdx.x; i < passes * 256; i += 256) h[i] = 0;
  __syncthreads();
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const K k = keys[i];
    for (int p = 0; p < passes; p++) {
      const uint32_t mask = key_bits - 8 * p >= 8 ? 255u : (1u << (key_bits - 8 * p)) - 1u;
      atomicAdd(&h[p * 256 + (int)((uint32_t)(k >> (8 * p)) & mask)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * 256; i += 256)
    if (h[i]) atomicAdd(&S->total[0][0] + i, h[i]);
}

__device__ __forceinline__ uint64_t ld_word(const uint64_t* p) {
  uint64_t v;
  asm volatile("ld.relaxed.gpu.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(uint64_t* p, uint64_t v) {
  asm volatile("st.relaxed.gpu.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// One pass. vin = nullptr: values are the input positions; kout = nullptr: the sorted keys are not wanted.
template <class K>
__global__ void __launch_bounds__(RS_THREADS) k_rs_pass(const K* __restrict__ kin, const uint32_t* __restrict__ vin,
                                                       int64_t n, int pass, uint32_t mask, RsState* __restrict__ S,
                                                       uint64_t* __restrict__ words, K* __restrict__ kout,
                                                       uint32_t* __restrict__ vout, int* __restrict__ err) {
  __shared__ K s_item[RS_TILE];  // the sorted keys, then the sorted values
  __shared__ uint16_t s_cnt[RS_WARPS][256];
  __shared__ uint32_t s_start[256], s_base[256];
  __shared__ uint64_t s_scan[8];
  __shared__ uint32_t s_tile;
  __shared__ int s_stop;
  const int t = threadIdx.x, lane = t & 31, w = t >> 5, shift = 8 * pass;
  if (t == 0) { s_tile = atomicAdd(&S->next[pass], 1u); s_stop = 0; }
  __syncthreads();
  const int64_t tile = s_tile, base = tile * RS_TILE;
  const int count = (int)min((int64_t)RS_TILE, n - base);
  K key[RS_ITEMS];
  uint32_t val[RS_ITEMS], digit[RS_ITEMS], rank[RS_ITEMS];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const int i = w * (RS_ITEMS * 32) + r * 32 + lane;
    const bool live = i < count;
    key[r] = live ? kin[base + i] : (K)0;
    val[r] = live ? (vin ? vin[base + i] : (uint32_t)(base + i)) : 0u;
    digit[r] = live ? (uint32_t)(key[r] >> shift) & mask : 256u;
  }
  const uint32_t mine = rank_digits<RS_WARPS, RS_ITEMS>(digit, rank, s_cnt);
  uint64_t* word = words + tile * 256 + t;
  const uint64_t tag = (uint64_t)(pass + 1) << 58;
  st_word(word, ((tile == 0 ? 2ull : 1ull) << 62) | tag | mine);
  // where digit t starts in the output and in the tile
  const uint64_t both = prefix256(((uint64_t)S->total[pass][t] << 16) | mine, s_scan);
  const uint32_t start = (uint32_t)(both & 0xFFFFu);
  s_start[t] = start;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++)
    if (digit[r] < 256u) {
      rank[r] += s_start[digit[r]] + s_cnt[w][digit[r]];  // now the place in the sorted tile
      s_item[rank[r]] = key[r];
    }
  // eight tiles back per round trip; tile 0's word holds its running total, so the walk ends there at the latest
  uint64_t before = 0;
  bool done = tile == 0;
  int64_t q = tile - 1;
  for (int polls = 0; !done && polls < RS_SPIN && !*(volatile int*)&s_stop; polls++) {
    uint64_t v[8];
#pragma unroll
    for (int j = 0; j < 8; j++) v[j] = q - j >= 0 ? ld_word(words + (q - j) * 256 + t) : 0ull;
    bool run = true;
#pragma unroll
    for (int j = 0; j < 8; j++) {
      run = run && (v[j] << 2 >> 60) == (uint64_t)(pass + 1);
      if (run) {
        before += v[j] & ((1ull << 58) - 1ull);
        q--;
        if (v[j] >> 63) { done = true; run = false; }
      }
    }
  }
  if (!done) {
    s_stop = 1;
    if (err) gsc_record(err, nullptr, (int)GSC_ERR_TIMEOUT, 0);
  } else if (tile > 0) {
    st_word(word, (2ull << 62) | tag | (before + mine));
  }
  __syncthreads();
  if (s_stop) return;
  s_base[t] = (uint32_t)(both >> 16) + (uint32_t)before - start;
  __syncthreads();
  uint32_t dst[RS_ITEMS];
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const int i = r * RS_THREADS + t;
    if (i >= count) continue;
    const K k = s_item[i];
    dst[r] = s_base[(uint32_t)(k >> shift) & mask] + (uint32_t)i;
    if (kout) kout[dst[r]] = k;
  }
  __syncthreads();
  uint32_t* s_val = reinterpret_cast<uint32_t*>(s_item);
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++)
    if (digit[r] < 256u) s_val[rank[r]] = val[r];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < RS_ITEMS; r++) {
    const int i = r * RS_THREADS + t;
    if (i < count) vout[dst[r]] = s_val[i];
  }
}

template <class K>
cudaError_t radix_sort(K* keys, K* keys2, uint32_t* vals, uint32_t* vals2, int64_t n, int key_bits, bool iota,
                       bool want_keys, void* state, int* err, cudaStream_t st, K** out_keys, uint32_t** out_vals) {
  *out_keys = keys;
  *out_vals = vals;
  const int passes = (key_bits + 7) / 8;
  if (n <= 0 || passes > RS_PASSES) return n <= 0 ? cudaSuccess : cudaErrorInvalidValue;
  RsState* S = reinterpret_cast<RsState*>(state);
  uint64_t* words = reinterpret_cast<uint64_t*>(S + 1);
  const int64_t nt = rs_tiles(n);
  cudaError_t e = cudaMemsetAsync(state, 0, radix_state_bytes(n), st);
  if (e != cudaSuccess) return e;
  const int64_t g = ceil_div64(n, 256 * 8), cap = (int64_t)gsc_sm_count() * 8;
  gsc_count_launch();
  k_rs_totals<K><<<(int)(g < cap ? g : cap), 256, passes * 1024, st>>>(keys, n, passes, key_bits, S);
  for (int p = 0; p < passes; p++) {
    const int bits = key_bits - 8 * p < 8 ? key_bits - 8 * p : 8;
    gsc_count_launch();
    k_rs_pass<K><<<(int)nt, RS_THREADS, 0, st>>>(keys, p == 0 && iota ? nullptr : vals, n, p, (1u << bits) - 1u, S, words,
                                                 p + 1 < passes || want_keys ? keys2 : nullptr, vals2, err);
    K* tk = keys; keys = keys2; keys2 = tk;
    uint32_t* tv = vals; vals = vals2; vals2 = tv;
  }
  *out_keys = keys;
  *out_vals = vals;
  return cudaGetLastError();
}
template cudaError_t radix_sort<uint32_t>(uint32_t*, uint32_t*, uint32_t*, uint32_t*, int64_t, int, bool, bool, void*, int*,
                                          cudaStream_t, uint32_t**, uint32_t**);
template cudaError_t radix_sort<uint64_t>(uint64_t*, uint64_t*, uint32_t*, uint32_t*, int64_t, int, bool, bool, void*, int*,
                                          cudaStream_t, uint64_t**, uint32_t**);

cudaError_t radix_sort_pairs(uint64_t* keys, uint32_t* vals, int64_t n, int key_bits, void* ws, int* err, cudaStream_t st) {
  if (n <= 1 || key_bits <= 0) return cudaSuccess;
  Carve c{reinterpret_cast<uint8_t*>(ws), 0, 0};
  uint64_t* k2 = c.take<uint64_t>(n);
  uint32_t* v2 = c.take<uint32_t>(n);
  void* state = c.take<uint8_t>((int64_t)radix_state_bytes(n));
  uint64_t* ko;
  uint32_t* vo;
  cudaError_t e = radix_sort<uint64_t>(keys, k2, vals, v2, n, key_bits, false, true, state, err, st, &ko, &vo);
  if (e == cudaSuccess && ko != keys) {
    e = cudaMemcpyAsync(keys, ko, sizeof(uint64_t) * n, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(vals, vo, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
  }
  return e;
}
