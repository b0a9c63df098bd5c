// sort.cuh -- block-level radix ranking shared by the device-wide sort (sort.cu) and the plan's
// one-CTA sorts (plan.cu).
#pragma once
#include "gsc_internal.cuh"

// Exclusive prefix over the 256 threads t < 256 of a CTA of at least 256 threads (all threads call it; s: 8 words).
__device__ __forceinline__ uint64_t prefix256(uint64_t v, uint64_t* s) {
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  uint64_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += y;
  }
  if (lane == 31 && w < 8) s[w] = x;
  __syncthreads();
  uint64_t before = x - v;
#pragma unroll
  for (int k = 0; k < 8; k++)
    if (k < w) before += s[k];
  __syncthreads();
  return before;
}

// Stable ranks of a CTA's items by an 8-bit digit. Warp w holds ITEMS * 32 consecutive items, item r of lane l
// being r * 32 + l of them; digit[r] = 256 for an item past the end. On return rank[r] is the item's position
// among its warp's items of the same digit, and cnt[w][d] the number of items of digit d in the warps before w;
// the total per digit is returned to thread d < 256. cnt has WARPS rows. Each round's peers are found with one
// match; the warp's counters are its own, so rounds need no CTA barrier.
template <int WARPS, int ITEMS>
__device__ __forceinline__ uint32_t rank_digits(const uint32_t (&digit)[ITEMS], uint32_t (&rank)[ITEMS],
                                                uint16_t (*cnt)[256]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
  {
    uint32_t* z = reinterpret_cast<uint32_t*>(cnt[w]);
#pragma unroll
    for (int q = 0; q < 4; q++) z[lane + 32 * q] = 0u;
  }
  __syncwarp();
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, digit[r]);
    const uint32_t before = __popc(peers & below);
    const uint32_t old = digit[r] < 256u ? cnt[w][digit[r]] : 0u;
    rank[r] = old + before;
    __syncwarp();
    if (digit[r] < 256u && before == 0u) cnt[w][digit[r]] = (uint16_t)(old + __popc(peers));
    __syncwarp();
  }
  __syncthreads();
  uint32_t sum = 0;
  if (threadIdx.x < 256) {
#pragma unroll
    for (int k = 0; k < WARPS; k++) {
      const uint32_t c = cnt[k][threadIdx.x];
      cnt[k][threadIdx.x] = (uint16_t)sum;
      sum += c;
    }
  }
  return sum;
}
