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

// Stable ranks of a CTA's items by a digit of BITS (at most 8) bits. Warp w holds ITEMS * 32 consecutive items, item r of lane l
// being r * 32 + l of them; digit(r) = 256 for an item past the end. put(r, rank) takes the item's position
// among its warp's items of the same digit; on return cnt[w][d] is the number of items of digit d in the warps before w;
// the total per digit is returned to thread d < 256. cnt has WARPS rows. A round's peers come from BITS ballots
// (a match instruction took several times as long on digits that mostly differ), and its leaders take their
// places with one shared-memory addition each: rounds wait neither for one another nor for a barrier.
template <int WARPS, int ITEMS, int BITS, class Digit, class Put>
__device__ __forceinline__ uint32_t rank_digits(Digit digit, Put put, uint32_t (*cnt)[256]) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1u;
#pragma unroll
  for (int q = 0; q < 8; q++) cnt[w][lane + 32 * q] = 0u;
  __syncwarp();
#pragma unroll
  for (int r = 0; r < ITEMS; r++) {
    const uint32_t d = digit(r);
    const bool live = d < 256u;
    uint32_t peers = __ballot_sync(0xFFFFFFFFu, live);
#pragma unroll
    for (int b = 0; b < BITS; b++) {
      const uint32_t set = __ballot_sync(0xFFFFFFFFu, (d >> b) & 1u);
      peers &= (d >> b) & 1u ? set : ~set;
    }
    const uint32_t before = __popc(peers & below);
    uint32_t old = 0u;
    if (live && before == 0u) old = atomicAdd(&cnt[w][d], (uint32_t)__popc(peers));
    put(r, __shfl_sync(0xFFFFFFFFu, old, live ? __ffs(peers) - 1 : lane) + before);
  }
  __syncthreads();
  uint32_t sum = 0;
  if (threadIdx.x < 256) {
#pragma unroll
    for (int k = 0; k < WARPS; k++) {
      const uint32_t c = cnt[k][threadIdx.x];
      cnt[k][threadIdx.x] = sum;
      sum += c;
    }
  }
  return sum;
}
