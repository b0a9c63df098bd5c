// bc7.cu -- BC7 encoder (Sec. III-B; D3D11 / Khronos BC7 format).
//
// A warp owns 32 blocks, their texels in shared memory; bounds, pruning and the fits' mapping to
// lanes are described in bc7_warp.cuh.
//
// The search is the codec's own deterministic integer encoder. Candidates, in order:
// mode 0 partitions 0..15; modes 1, 2, 3 partitions 0..63; mode 4 rotation 0..3 x
// index selection 0..1; mode 5 rotation 0..3; mode 6; mode 7 partitions 0..63. For
// each subset: bounding-box diagonal oriented by covariance signs, indices against the
// unquantised palette, one least-squares refinement, then every p-bit combination
// quantised to the nearest codes and re-indexed; the best combination (lowest squared
// error, first on ties) scores the subset. The block takes the first candidate of
// least total error; the winner is solved again, anchors are fixed losslessly by
// swapping endpoints and inverting indices, and the fields are packed LSB first.
#include <algorithm>
#include <cmath>

#include "bc1_dev.cuh"
#include "bc7_tables.h"
#include "gsc_internal.cuh"
#include "stage.cuh"

__constant__ uint8_t c_anc2[64];
__constant__ uint8_t c_anc3a[64];
__constant__ uint8_t c_anc3b[64];
// expanded value of the nearest endpoint code per 8-bit target, 12 configurations
__device__ uint8_t g_qtab[12][256];
// constant blocks: per 8-bit value the 7-bit code pair a | b << 8 of mode 5 at weight 21
__constant__ uint16_t c_const7[256];

// table ids: (bits, p-bit present, p)
__host__ __device__ constexpr int qid(int bits, int hp, int p) {
  return bits == 4 ? p : bits == 5 ? (hp ? 3 + p : 2) : bits == 6 ? (hp ? 6 + p : 5) : bits == 7 ? (hp ? 9 + p : 8) : 11;
}

template <int IB> __device__ __forceinline__ int wgt(int j) {
  if (IB == 2) return (0x402B1500u >> (8 * j)) & 255;              // 0, 21, 43, 64
  if (IB == 3) return (int)((0x40372E251B120900ull >> (8 * j)) & 255);  // 0 9 18 27 37 46 55 64
  // 0 4 9 13 17 21 26 30 34 38 43 47 51 55 60 64
  return j < 8 ? (int)((0x1E1A15110D090400ull >> (8 * j)) & 255) : (int)((0x403C37332F2B2622ull >> (8 * (j - 8))) & 255);
}
#include "bc7_warp.cuh"

static int h_expand(int v, int n) { return n >= 8 ? v : ((v << (8 - n)) | (v >> (2 * n - 8))); }

cudaError_t bc7_init_tables() {
  uint32_t p2[64], p3[64];
  uint8_t a2[64], a3a[64], a3b[64];
  for (int p = 0; p < 64; p++) {
    p2[p] = bc7_pack_part2(p);
    p3[p] = bc7_pack_part3(p);
    a2[p] = kBC7Anchor2[p];
    a3a[p] = kBC7Anchor3a[p];
    a3b[p] = kBC7Anchor3b[p];
  }
  static const int cfg[12][3] = {{4, 1, 0}, {4, 1, 1}, {5, 0, 0}, {5, 1, 0}, {5, 1, 1}, {6, 0, 0},
                                 {6, 1, 0}, {6, 1, 1}, {7, 0, 0}, {7, 1, 0}, {7, 1, 1}, {8, 0, 0}};
  static uint8_t q[12][256];
  for (int c = 0; c < 12; c++) {
    int bits = cfg[c][0], hp = cfg[c][1], pb = cfg[c][2];
    for (int e = 0; e < 256; e++) {
      int be = -1, bv = 0;
      for (int code = 0; code < (1 << bits); code++) {
        int v = h_expand(hp ? (code << 1) | pb : code, bits + hp);
        int d = abs(v - e);
        if (be < 0 || d < be) { be = d; bv = v; }
      }
      q[c][e] = (uint8_t)bv;
    }
  }
  // Constant blocks: every 8-bit value v is ((64 - 21) ex7(a) + 21 ex7(b) + 32) >> 6 for some 7-bit
  // pair; the first with a outer and b inner is taken.
  uint16_t c7[256];
  for (int v = 0; v < 256; v++) {
    c7[v] = 0;
    bool found = false;
    for (int a = 0; a < 128 && !found; a++)
      for (int b = 0; b < 128 && !found; b++)
        if (((64 - 21) * h_expand(a, 7) + 21 * h_expand(b, 7) + 32) >> 6 == v) { c7[v] = (uint16_t)(a | (b << 8)); found = true; }
  }
  uint64_t mem2[64][2], mem3[64][3];
  for (int pp = 0; pp < 64; pp++)
    for (int ns = 2; ns <= 3; ns++)
      for (int sb = 0; sb < ns; sb++) {
        const uint32_t part = ns == 2 ? p2[pp] : p3[pp];
        uint64_t list = 0;
        int cnt = 0;
        for (int t = 0; t < 16; t++)
          if (((part >> (2 * t)) & 3u) == (uint32_t)sb) list |= (uint64_t)t << (4 * cnt++);
        if (cnt > 15) return cudaErrorInvalidValue;
        list |= (uint64_t)cnt << 60;
        if (ns == 2) mem2[pp][sb] = list; else mem3[pp][sb] = list;
      }
  // the search's tables: subset masks and sizes, member lists with the largest subset first
  uint4 msk2[64], msk3[64][2];
  uint8_t cnt2[64], cnt3[64][2];
  uint64_t big2[64][2], big3[64][3];
  float inv[17];
  auto mask_of = [](uint32_t part, uint32_t sb) {
    uint32_t w[4] = {0, 0, 0, 0};
    for (int t = 0; t < 16; t++)
      if (((part >> (2 * t)) & 3u) == sb) w[t >> 2] |= 0xFFu << (8 * (t & 3));
    return make_uint4(w[0], w[1], w[2], w[3]);
  };
  auto by_size = [](uint64_t x, uint64_t y) { return (x >> 60) > (y >> 60); };
  for (int pp = 0; pp < 64; pp++) {
    msk2[pp] = mask_of(p2[pp], 1);
    cnt2[pp] = (uint8_t)(mem2[pp][1] >> 60);
    for (int sb = 0; sb < 2; sb++) {
      msk3[pp][sb] = mask_of(p3[pp], sb + 1);
      cnt3[pp][sb] = (uint8_t)(mem3[pp][sb + 1] >> 60);
      big2[pp][sb] = mem2[pp][sb];
    }
    for (int sb = 0; sb < 3; sb++) big3[pp][sb] = mem3[pp][sb];
    std::stable_sort(big2[pp], big2[pp] + 2, by_size);
    std::stable_sort(big3[pp], big3[pp] + 3, by_size);
  }
  uint8_t order[4][64];
  for (int k = 0; k < 4; k++) {
    const int np = k == 1 ? 16 : 64;
    for (int j = 0; j < 64; j++) order[k][j] = (uint8_t)j;
    if (k < 3)
      std::stable_sort(order[k], order[k] + np, [&](uint8_t x, uint8_t y) {
        return k == 2 ? by_size(big2[x][0], big2[y][0]) : by_size(big3[x][0], big3[y][0]);
      });
  }
  inv[0] = 0.0f;
  for (int k = 1; k <= 16; k++) inv[k] = std::nextafter(1.0f / (float)k, 0.0f);
  cudaError_t e;
  if ((e = cudaMemcpyToSymbol(c_msk2, msk2, sizeof(msk2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_msk3, msk3, sizeof(msk3))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_cnt2, cnt2, sizeof(cnt2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_cnt3, cnt3, sizeof(cnt3))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_order, order, sizeof(order))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_inv, inv, sizeof(inv))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(g_mem2, big2, sizeof(big2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(g_mem3, big3, sizeof(big3))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(g_org2, mem2, sizeof(mem2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(g_org3, mem3, sizeof(mem3))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_const7, c7, sizeof(c7))) != cudaSuccess) return e;
  uint16_t t5[256], t6[256];
  bc1_const_tables(t5, t6);
  if ((e = cudaMemcpyToSymbol(c_const5, t5, sizeof(t5))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_const6, t6, sizeof(t6))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_anc2, a2, sizeof(a2))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_anc3a, a3a, sizeof(a3a))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_anc3b, a3b, sizeof(a3b))) != cudaSuccess) return e;
  return cudaMemcpyToSymbol(g_qtab, q, sizeof(q));
}

// One kernel for both sources: staged layout-D groups (sh / perm / scales) or raw
// texels [nblk][16][3] (texin != nullptr), so the search is compiled once. The warps of a CTA share the
// quantisation tables, each stages and searches its own 32 blocks (two groups), and they go from phase to phase
// together: bound by instruction issue and fetch, and warps in one phase run the same code. With barriers between the
// phases and before the solve, and ten warps per CTA, 3M blocks of the scene with outliers take 28.7 ms, against 34.5 ms
// with each of four warps at its own pace and 67.0 ms for the exhaustive search; the call for 262,144 without outliers
// 1.23, 1.40 and 6.98 ms. 20 warps per SM at most 102 registers; 24 at 80 and 16 at 128 were slower.
#define BC7_WARPS 4
// Up to this many blocks per SM a warp takes 8 blocks instead of 32: the chip has warps to spare and the time is
// one warp's. Scene without outliers, 8 against 32 blocks per warp: 1,000 blocks 122 against 194 us, 4,096 138 against
// 222, 10,000 157 against 226, 17,000 205 against 229, 20,000 239 and 239, 40,000 439 against 291.
#define BC7_FEW 112
#define BC7_MIN_BLOCKS 5
// Above this many blocks per SM a CTA has ten warps instead of four: more warps share their phase's code, but a CTA of
// 320 blocks leaves a larger part of the last wave idle. The kernel with ten against four: 120,000 blocks 637 against
// 614 us, 180,000 804 against 824, 262,144 1164 and 1164, the scene of 3M with outliers 28.7 against 29.9 ms; with
// twenty 754, 777, 1141 us and 28.8 ms.
#define BC7_MANY 1280
#define BC7_WIDE 10

// the warp's staged blocks (columns col0.. of its tile): search, solve, store. blk: this lane's block, live:
// whether it exists (lanes from BPW on have none)
template <int BPW>
__device__ __forceinline__ void bc7_finish(Bc7Warp& W, int col0, bool live, int64_t blk, const uint8_t* sq,
                                           uint4* __restrict__ blocks, uint32_t* __restrict__ sse7,
                                           uint64_t* __restrict__ sse64) {
  const int lane = threadIdx.x & 31;
  const uint32_t* my = &W.tex[0][col0 + lane % BPW];
  uint4 out;
  const bool constant = const_block(my, &out);
  bc7_search<BPW>(W, col0, live && !constant, sq);
  __syncthreads();
  if (live) {
    uint32_t err = 0;
    if (!constant) {
      const uint32_t key = W.best[lane];
      err = key >> 9;
      out = solve_pack(my, (int)(key & 511u), sq);
    }
    blocks[blk] = out;
    if (sse7) sse7[blk] = err;
    if (sse64) sse64[blk] = err;
  }
}

template <int BPW, int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 20 / WARPS)
    k_bc7(const float* __restrict__ sh, const int32_t* __restrict__ perm, const float* __restrict__ scales,
          int64_t n_groups, const uint8_t* __restrict__ texin, int64_t nblk, uint4* __restrict__ blocks,
          uint32_t* __restrict__ sse7, uint64_t* __restrict__ sse64) {
  extern __shared__ __align__(16) uint8_t dyn[];
  Bc7Warp* S = reinterpret_cast<Bc7Warp*>(dyn);
  __shared__ StageScale T;
  __shared__ uint8_t sq[12 * 256];
  for (int i = threadIdx.x; i < 12 * 256; i += blockDim.x) sq[i] = (&g_qtab[0][0])[i];
  if (!texin && threadIdx.x < 32) stage_scales(T, scales);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t total = texin ? nblk : n_groups * 16;
  // every warp of the CTA goes through the phases, one without blocks too
  for (int64_t c0 = (int64_t)blockIdx.x * WARPS * BPW; c0 < total; c0 += (int64_t)gridDim.x * WARPS * BPW) {
    const int64_t b0 = c0 + w * BPW;
    const int64_t blk = b0 + lane;
    const bool live = lane < BPW && blk < total;
    int col0 = 0;
    if (!texin) {
      // two groups, or the one that holds the warp's eight blocks
      const int64_t g0 = b0 / 16;
      stage_groups<BC7_STRIDE, 1>(sh, perm, T, g0, BPW == 32 ? n_groups : min(g0 + 1, n_groups), S[w].tex,
                                  reinterpret_cast<uint32_t*>(S[w].r));
      col0 = (int)(b0 - g0 * 16);
    } else if (live) {
      stage_texels<BC7_STRIDE>(texin + blk * 48, ((uintptr_t)texin & 15) == 0, &S[w].tex[0][lane]);
    } else {
#pragma unroll
      for (int t = 0; t < 16; t++) S[w].tex[t][lane] = 0x808080u;
    }
    __syncwarp();
    bc7_finish<BPW>(S[w], col0, live, blk, sq, blocks, sse7, sse64);
    __syncwarp();
  }
}

static cudaError_t launch_bc7(const float* sh, const int32_t* perm, const float* scales, int64_t n_groups,
                              const uint8_t* tex, int64_t nblk, uint8_t* out, uint32_t* sse7, uint64_t* sse64,
                              cudaStream_t st) {
  const int64_t total = tex ? nblk : n_groups * 16;
  const bool few = total <= (int64_t)gsc_sm_count() * BC7_FEW, many = total > (int64_t)gsc_sm_count() * BC7_MANY;
  const int warps = many ? BC7_WIDE : BC7_WARPS;
  const int64_t grid = std::min<int64_t>(ceil_div64(total, (few ? 8 : 32) * warps), 0x7FFFFFFF);
  const size_t smem = warps * sizeof(Bc7Warp);
  uint4* to = reinterpret_cast<uint4*>(out);
  gsc_count_launch();
  static_assert(BC7_WARPS * sizeof(Bc7Warp) <= 48 * 1024, "more needs a raised limit");
  if (few) k_bc7<8, BC7_WARPS><<<(int)grid, 32 * warps, smem, st>>>(sh, perm, scales, n_groups, tex, nblk, to, sse7, sse64);
  else if (many) k_bc7<32, BC7_WIDE><<<(int)grid, 32 * warps, smem, st>>>(sh, perm, scales, n_groups, tex, nblk, to, sse7, sse64);
  else k_bc7<32, BC7_WARPS><<<(int)grid, 32 * warps, smem, st>>>(sh, perm, scales, n_groups, tex, nblk, to, sse7, sse64);
  return cudaGetLastError();
}

cudaError_t bc7_init_kernels() {  // dynamic shared memory above 48 KB, once per device
  return cudaFuncSetAttribute(k_bc7<32, BC7_WIDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(BC7_WIDE * sizeof(Bc7Warp)));
}

cudaError_t launch_bc7_groups(const float* sh, const int32_t* perm, const float* scales, int64_t n_groups,
                              uint8_t* blocks, uint32_t* sse7, cudaStream_t st) {
  if (n_groups <= 0) return cudaSuccess;
  return launch_bc7(sh, perm, scales, n_groups, nullptr, 0, blocks, sse7, nullptr, st);
}

cudaError_t launch_bc7_blocks(const uint8_t* tex, int64_t nblk, uint8_t* out, uint64_t* sse, cudaStream_t st) {
  if (nblk <= 0) return cudaSuccess;
  return launch_bc7(nullptr, nullptr, nullptr, 0, tex, nblk, out, nullptr, sse, st);
}

// ---- persistent multi-scene encode -----------------------------------------------------------
// One launch per coding over the tiles of every listed scene. Tiles
// are claimed round robin (schedule 0), from an atomic work queue (1, 2), or one per claiming unit
// (3, a grid of all tiles); a tile finds its scene by binary search over the list. A BC1 CTA's four
// warps claim their own tiles and walk them 8 groups at a time, a BC7 CTA claims one for its four warps. The
// bits equal the single-scene kernels'.
__device__ __forceinline__ int64_t claim_tile(int schedule, int64_t it, int w, int lane, int* counter) {
  long long ti = 0;
  if (lane == 0)
    ti = (schedule == 0 || schedule == 3) ? (long long)((blockIdx.x + it * gridDim.x) * BC7_WARPS + w)
                                          : (long long)atomicAdd(counter, 1);
  return __shfl_sync(0xFFFFFFFFu, ti, 0);
}

__device__ __forceinline__ BatchSceneDev scene_of(const BatchSceneDev* __restrict__ scenes, int n_scenes, int64_t ti) {
  int lo = 0, hi = n_scenes - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (scenes[mid].tile0 <= ti) lo = mid; else hi = mid - 1;
  }
  return scenes[lo];
}

__global__ void __launch_bounds__(32 * BC7_WARPS, 4)
    k_batch1(const BatchSceneDev* __restrict__ scenes, int n_scenes, int64_t n_tiles, int schedule,
             int* __restrict__ counter) {
  __shared__ Bc1Warp<128> W[BC7_WARPS];
  __shared__ StageScale T[BC7_WARPS];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t it = 0;; it++) {
    const int64_t ti = claim_tile(schedule, it, w, lane, counter);
    if (ti >= n_tiles) break;
    const BatchSceneDev S = scene_of(scenes, n_scenes, ti);
    const int64_t gbeg = (ti - S.tile0) * S.tile_groups, gend = min(gbeg + (int64_t)S.tile_groups, S.work_groups);
    stage_scales(T[w], S.scales);
    __syncwarp();
    for (int64_t g0 = gbeg; g0 < gend; g0 += 8) {
#pragma unroll 1
      for (int i = 0; i < 128; i += 32)
        stage_groups<129>(S.sh, S.perm, T[w], g0 + i / 16, S.n_groups,
                          reinterpret_cast<uint32_t(*)[129]>(&W[w].tex[0][i]), W[w].raw);
      bc1_encode_warp<128>(W[w], g0 * 16, gend * 16, reinterpret_cast<uint2*>(S.b1), S.sse1, S.sse0, nullptr);
      __syncwarp();
    }
  }
}

// The CTA claims a tile for its four warps, which take two groups each and search in step (as in k_bc7).
__global__ void __launch_bounds__(32 * BC7_WARPS, BC7_MIN_BLOCKS)
    k_batch7(const BatchSceneDev* __restrict__ scenes, int n_scenes, int64_t n_tiles, int schedule,
             int* __restrict__ counter) {
  __shared__ Bc7Warp W[BC7_WARPS];
  __shared__ StageScale T[BC7_WARPS];
  __shared__ long long s_tile;
  __shared__ uint8_t sq[12 * 256];
  for (int i = threadIdx.x; i < 12 * 256; i += blockDim.x) sq[i] = (&g_qtab[0][0])[i];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int64_t it = 0;; it++) {
    __syncthreads();  // the last tile's number has been read
    if (threadIdx.x == 0)
      s_tile = (schedule == 0 || schedule == 3) ? (long long)(blockIdx.x + it * gridDim.x) : (long long)atomicAdd(counter, 1);
    __syncthreads();
    const int64_t ti = s_tile;
    if (ti >= n_tiles) break;
    const BatchSceneDev S = scene_of(scenes, n_scenes, ti);
    const int64_t gbeg = (ti - S.tile0) * S.tile_groups, gend = min(gbeg + (int64_t)S.tile_groups, S.work_groups);
    stage_scales(T[w], S.scales);
    __syncwarp();
    for (int64_t c0 = gbeg; c0 < gend; c0 += 2 * BC7_WARPS) {
      const int64_t g0 = c0 + 2 * w;
      stage_groups<BC7_STRIDE, 1>(S.sh, S.perm, T[w], g0, S.n_groups, W[w].tex, reinterpret_cast<uint32_t*>(W[w].r));
      const bool live = g0 + (lane >> 4) < gend;
      bc7_finish<32>(W[w], 0, live, g0 * 16 + lane, sq, reinterpret_cast<uint4*>(S.b7), S.sse7, nullptr);
      __syncwarp();
    }
  }
}

cudaError_t launch_batch_encode(int kind, const BatchSceneDev* scenes, int n_scenes, int64_t n_tiles, int schedule,
                                int ctas_per_sm, int sm_count, int* counter, cudaStream_t st) {
  if (n_tiles <= 0 || n_scenes <= 0) return cudaSuccess;
  // schedule 3: one claiming unit (a warp for BC1, a CTA for BC7) per tile, left to the hardware block scheduler; a BC7
  // launch has BC7_MIN_BLOCKS CTAs (what one SM holds) per ctas_per_sm
  const int64_t cta_tiles = kind == 7 ? n_tiles : ceil_div64(n_tiles, BC7_WARPS);
  int64_t grid = schedule == 3 ? cta_tiles
                               : (int64_t)(sm_count > 0 ? sm_count : gsc_sm_count()) *
                                     (ctas_per_sm > 0 ? ctas_per_sm : (kind == 7 ? 1 : 4)) *
                                     (kind == 7 ? BC7_MIN_BLOCKS : 1);
  if (grid > cta_tiles) grid = cta_tiles;
  if (grid > 0x7FFFFFFF) grid = 0x7FFFFFFF;
  if (schedule == 1 || schedule == 2) {
    cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
    if (e != cudaSuccess) return e;
  }
  gsc_count_launch();
  if (kind == 7) k_batch7<<<(int)grid, 32 * BC7_WARPS, 0, st>>>(scenes, n_scenes, n_tiles, schedule, counter);
  else k_batch1<<<(int)grid, 32 * BC7_WARPS, 0, st>>>(scenes, n_scenes, n_tiles, schedule, counter);
  return cudaGetLastError();
}

// ---- one mode family searched two ways (a measurement of the search's thread mapping) --------
// Mode 1 only (64 two-subset partitions, 6-bit endpoints with a shared p-bit, 3-bit indices):
// the least-error partition of each block, ties to the lowest, with its error. Thread per block
// (as k_bc7: every lane of a warp fits the same partition, so the member loops are uniform) or
// warp per block (lane l fits partitions l and l + 32 of the warp's block, then a shuffle
// minimum over (error, partition)); the results are the same.
__device__ __forceinline__ uint32_t mode1_err(const uint32_t* tex, int p, const uint8_t* sq) {
  int s = 0;
#pragma unroll 1
  for (int sub = 0; sub < 2; sub++) {
    const Mem M = mem_at(&g_mem2[p][sub]);
    const Box B = box_axis(tex, M, BC7_ID);
    int e0[3], e1[3];
    refine<3>(tex, M, B, BC7_ID, e0, e1);
    const int t[2] = {qid(6, 1, 0), qid(6, 1, 1)};
    s += quant_err<3, 2>(tex, M, e0, e1, sq, t, t, BC7_ID) >> 1;
    each_member(tex, M, BC7_ID, [&](uint32_t v, int) { s += (int)__dp4a(v, v, 0u); });
  }
  return (uint32_t)s;
}

#define M1_THREADS 128
template <bool WARP>
__global__ void __launch_bounds__(M1_THREADS) k_bc7_mode1(const uint8_t* __restrict__ texin, int64_t nblk,
                                                             uint32_t* __restrict__ sse_out,
                                                             int32_t* __restrict__ part_out) {
  __shared__ uint32_t tex[M1_THREADS / 32][16][BC7_STRIDE];  // texel t of block 32 w + b at [w][t][b]
  __shared__ uint8_t sq[12 * 256];
  for (int i = threadIdx.x; i < 12 * 256; i += blockDim.x) sq[i] = (&g_qtab[0][0])[i];
  const int lt = threadIdx.x, w = lt >> 5, lane = lt & 31;
  for (int64_t b0 = (int64_t)blockIdx.x * M1_THREADS; b0 < nblk; b0 += (int64_t)gridDim.x * M1_THREADS) {
    __syncthreads();
    for (int i = lt; i < M1_THREADS * 16; i += M1_THREADS) {
      const int j = i / 16, t = i % 16;
      const int64_t blk = b0 + j;
      const uint8_t* p = texin + blk * 48 + 3 * t;
      tex[j >> 5][t][j & 31] = blk < nblk ? ((uint32_t)p[0] | ((uint32_t)p[1] << 8) | ((uint32_t)p[2] << 16)) : 0x808080u;
    }
    __syncthreads();
    if (WARP) {
#pragma unroll 1
      for (int i = 0; i < 32; i++) {
        const uint32_t* my = &tex[w][0][i];
        const uint32_t sa = mode1_err(my, lane, sq);
        const uint32_t sb = mode1_err(my, lane + 32, sq);
        uint32_t best = sa;
        int bp = lane;
        if (sb < best) { best = sb; bp = lane + 32; }
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) {
          const uint32_t ob = __shfl_xor_sync(0xFFFFFFFFu, best, d);
          const int op = __shfl_xor_sync(0xFFFFFFFFu, bp, d);
          if (ob < best || (ob == best && op < bp)) { best = ob; bp = op; }
        }
        const int64_t blk = b0 + 32 * w + i;
        if (lane == 0 && blk < nblk) { sse_out[blk] = best; part_out[blk] = bp; }
      }
    } else {
      const uint32_t* my = &tex[w][0][lane];
      uint32_t best = 0xFFFFFFFFu;
      int bp = 0;
#pragma unroll 1
      for (int p = 0; p < 64; p++) {
        const uint32_t s = mode1_err(my, p, sq);
        if (s < best) { best = s; bp = p; }
      }
      const int64_t blk = b0 + lt;
      if (blk < nblk) { sse_out[blk] = best; part_out[blk] = bp; }
    }
  }
}

cudaError_t launch_bc7_mode1(const uint8_t* tex, int64_t nblk, int warp, uint32_t* sse, int32_t* part, int sm_count,
                             cudaStream_t st) {
  if (nblk <= 0) return cudaSuccess;
  int64_t g = ceil_div64(nblk, M1_THREADS);
  const int64_t cap = (int64_t)sm_count * 8;
  if (g > cap) g = cap;
  gsc_count_launch();
  if (warp) k_bc7_mode1<true><<<(int)g, M1_THREADS, 0, st>>>(tex, nblk, sse, part);
  else k_bc7_mode1<false><<<(int)g, M1_THREADS, 0, st>>>(tex, nblk, sse, part);
  return cudaGetLastError();
}
