// bc1.cu -- BC1 encoder (Sec. III-A with P = 16, Q = 2 on 4x4 blocks; Sec. III-B).
//
// A warp takes 128 blocks (32 where there are few), their texels in shared memory (bc1_dev.cuh).
//
// Search (the codec's own encoder; ties go to the lowest index, candidates in a fixed order):
//  constant block: per channel the code pair whose two-thirds point is nearest (table);
//  otherwise: bounding-box diagonal oriented by covariance signs, inset by range/16,
//  565 quantisation; two least-squares refinements on the current indices; then up to
//  four rounds of the best strictly improving +-1 step on the six endpoint channels.
//  Every candidate is scored with the four-colour palette of the GB300 texture unit.
#include "bc1_dev.cuh"


static int h_ex5(int x) { return (x << 3) | (x >> 2); }
static int h_ex6(int x) { return (x << 2) | (x >> 4); }
static int h_third(int a, int b, int bits) {
  if (bits == 5) return ((2 * a + b) * 11) >> 2;
  int A = h_ex6(a), B = h_ex6(b);
  int num = (B - A) * 321 + 512;
  return A + (num >= 0 ? num / 1024 : -((-num + 1023) / 1024));
}

void bc1_const_tables(uint16_t* t5, uint16_t* t6) {
  for (int v = 0; v < 256; v++) {
    for (int bits = 5; bits <= 6; bits++) {
      int lim = 1 << bits, be = -1, ba = 0, bb = 0;
      for (int a = 0; a < lim; a++)
        for (int b = 0; b < lim; b++) {
          int e = abs(h_third(a, b, bits) - v);
          if (be < 0 || e < be) { be = e; ba = a; bb = b; }
        }
      (bits == 5 ? t5 : t6)[v] = (uint16_t)(ba | (bb << 8));
    }
  }
}

cudaError_t bc1_init_tables() {
  uint16_t t5[256], t6[256];
  bc1_const_tables(t5, t6);
  (void)h_ex5;
  cudaError_t e = cudaMemcpyToSymbol(c_const5, t5, sizeof(t5));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbol(c_const6, t6, sizeof(t6));
}

// One kernel for both sources: staged layout-D groups (sh / perm / scales) or raw texels [nblk][16][3]
// (texin != nullptr). Four independent warps per CTA. Bound by instruction issue (70% of the slots; two thirds of it
// the neighbourhood steps, whose byte products and minima share the slots evenly). 4 CTAs (16 warps, at most 128
// registers) per SM: 3M blocks of the scene-scale distribution 1.07 ms, against 1.10 ms with 3 CTAs and 1.34 ms with
// 5 (spills); one thread per block, without the queue, took 1.74 ms.
#define BC1_WARPS 4
// Up to this many blocks per SM a warp takes 32 blocks instead of 128: shorter warps fill the chip sooner, longer ones
// keep their queues full. 32 against 128 blocks per warp: 4,096 blocks 60 against 105 us, 80,000 85 against 127 us,
// 320,000 176 against 194 us, 450,000 228 against 222 us, 3M 1174 against 1069 us.
#define BC1_FEW 2560
template <int BPW>
__global__ void __launch_bounds__(32 * BC1_WARPS, 4)
    k_bc1(const float* __restrict__ sh, const int32_t* __restrict__ perm, const float* __restrict__ scales, int64_t n_groups,
          const uint8_t* __restrict__ texin, int64_t nblk, uint2* __restrict__ blocks, uint32_t* __restrict__ sse1,
          uint32_t* __restrict__ sse0, uint64_t* __restrict__ sse64) {
  __shared__ Bc1Warp<BPW> S[BC1_WARPS];
  __shared__ StageScale T;
  if (!texin && threadIdx.x < 32) stage_scales(T, scales);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t total = texin ? nblk : n_groups * 16;
  for (int64_t b0 = ((int64_t)blockIdx.x * BC1_WARPS + w) * BPW; b0 < total; b0 += (int64_t)gridDim.x * BC1_WARPS * BPW) {
#pragma unroll 1
    for (int i = 0; i < BPW; i += 32) {
      if (!texin) {
        stage_groups<BPW + 1>(sh, perm, T, (b0 + i) / 16, n_groups,
                              reinterpret_cast<uint32_t(*)[BPW + 1]>(&S[w].tex[0][i]), S[w].raw);
      } else if (b0 + i + lane < total) {
        stage_texels<BPW + 1>(texin + (b0 + i + lane) * 48, ((uintptr_t)texin & 15) == 0, &S[w].tex[0][i + lane]);
      }
    }
    __syncwarp();
    bc1_encode_warp<BPW>(S[w], b0, total, blocks, sse1, sse0, sse64);
    __syncwarp();
  }
}

static cudaError_t launch_bc1(const float* sh, const int32_t* perm, const float* scales, int64_t n_groups,
                              const uint8_t* tex, int64_t nblk, uint8_t* out, uint32_t* sse1, uint32_t* sse0,
                              uint64_t* sse64, cudaStream_t st) {
  const int64_t total = tex ? nblk : n_groups * 16;
  const bool few = total <= (int64_t)gsc_sm_count() * BC1_FEW;
  int64_t g = ceil_div64(total, (few ? 32 : 128) * BC1_WARPS);
  if (g > 0x7FFFFFFF) g = 0x7FFFFFFF;
  gsc_count_launch();
  if (few)
    k_bc1<32><<<(int)g, 32 * BC1_WARPS, 0, st>>>(sh, perm, scales, n_groups, tex, nblk, reinterpret_cast<uint2*>(out), sse1,
                                                 sse0, sse64);
  else
    k_bc1<128><<<(int)g, 32 * BC1_WARPS, 0, st>>>(sh, perm, scales, n_groups, tex, nblk, reinterpret_cast<uint2*>(out), sse1,
                                                  sse0, sse64);
  return cudaGetLastError();
}

cudaError_t launch_bc1_groups(const float* sh, const int32_t* perm, const float* scales, int64_t n_groups,
                              uint8_t* blocks, uint32_t* sse1, uint32_t* sse0, cudaStream_t st) {
  if (n_groups <= 0) return cudaSuccess;
  return launch_bc1(sh, perm, scales, n_groups, nullptr, 0, blocks, sse1, sse0, nullptr, st);
}

cudaError_t launch_bc1_blocks(const uint8_t* tex, int64_t nblk, uint8_t* out, uint64_t* sse, cudaStream_t st) {
  if (nblk <= 0) return cudaSuccess;
  return launch_bc1(nullptr, nullptr, nullptr, 0, tex, nblk, out, nullptr, nullptr, sse, st);
}
