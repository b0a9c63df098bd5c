// layout.cu -- fixed codings of any block layout (Sec. IV-B, Figs. SetupA / SetupB / SetupD;
// Table I's BC1, BC7 and "BC7 on the first block(s), BC1 on the rest" rows).
//
// Three steps on the caller's stream: the Gaussians are quantised (Sec. V-A) and their 16 texels
// go to their blocks, BC7 blocks and BC1 blocks into two dense texel
// arrays in output order; the block encoders code each array (the same search as every other
// coding); an interleave writes every group's BC7 blocks then its BC1 blocks. A coding with
// one format writes the encoder's output in place and skips the interleave.
#include "gsc_internal.cuh"
#include "layout.cuh"
#include "stage.cuh"

namespace {

// A warp stages two groups (stage.cuh: coefficient c of slot u at tile[u][c]); a lane then collects one block's texels
// and stores its 48 bytes in 16-byte pieces. 300,000 Gaussians in
// layout B: 18 us, the whole call 518 us, against 563 us with a slot per thread that read a row alone and stored bytes.
#define LAY_WARPS 4
__global__ void __launch_bounds__(32 * LAY_WARPS) k_stage_layout(const float* __restrict__ sh, const int32_t* __restrict__ perm,
                               const float* __restrict__ scales, int64_t n_groups, int layout, int j,
                               uint8_t* __restrict__ tex7, uint8_t* __restrict__ tex1) {
  __shared__ StageScale T;
  __shared__ uint32_t tile[LAY_WARPS][16][33];
  __shared__ uint32_t raw[LAY_WARPS][STAGE_RAW];
  if (threadIdx.x < 32) stage_scales(T, scales);
  __syncthreads();
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, k = lane & 15;
  const bool b7 = lay_bc7(layout, j, k);
  const int r = lay_rank(layout, j, k);
  for (int64_t g0 = ((int64_t)blockIdx.x * LAY_WARPS + w) * 2; g0 < n_groups; g0 += (int64_t)gridDim.x * LAY_WARPS * 2) {
    stage_groups<33>(sh, perm, T, g0, n_groups, tile[w], raw[w]);
    const int64_t g = g0 + (lane >> 4);
    if (g < n_groups) {
      uint32_t x[16], v[12];
#pragma unroll
      for (int t = 0; t < 16; t++) {
        int u, c;
        lay_at(layout, k, t, u, c);
        x[t] = tile[w][u][(lane & 16) + c];
      }
#pragma unroll
      for (int q = 0; q < 4; q++) {
        v[3 * q] = __byte_perm(x[4 * q], x[4 * q + 1], 0x4210);
        v[3 * q + 1] = __byte_perm(x[4 * q + 1], x[4 * q + 2], 0x5421);
        v[3 * q + 2] = __byte_perm(x[4 * q + 2], x[4 * q + 3], 0x6542);
      }
      uint4* d = reinterpret_cast<uint4*>(b7 ? tex7 + (g * j + r) * 48 : tex1 + (g * (16 - j) + r) * 48);
#pragma unroll
      for (int q = 0; q < 3; q++) d[q] = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
    __syncwarp();
  }
}

// group g's 16 + j 8-byte words: 2j from its BC7 blocks, then 16 - j from its BC1 blocks
__global__ void k_interleave(const uint2* __restrict__ lin7, const uint2* __restrict__ lin1, int64_t n_groups, int j,
                             uint2* __restrict__ out) {
  const int64_t words = 16 + j, total = n_groups * words;
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < total; w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t g = w / words;
    const int i = (int)(w - g * words);
    out[w] = i < 2 * j ? __ldg(lin7 + g * 2 * j + i) : __ldg(lin1 + g * (16 - j) + (i - 2 * j));
  }
}

int grid_of(int64_t work) {
  int64_t g = ceil_div64(work, 256);
  if (g > gsc_sm_count() * 16) g = gsc_sm_count() * 16;
  return (int)(g < 1 ? 1 : g);
}

struct LayoutWs {
  uint8_t *tex7, *tex1, *lin7, *lin1;
};

LayoutWs carve_layout(void* ws, size_t cap, int64_t ng, int j, bool* ok) {
  Carve cv{reinterpret_cast<uint8_t*>(ws), 0, cap};
  LayoutWs L;
  L.tex7 = cv.take<uint8_t>(ng * j * 48);
  L.tex1 = cv.take<uint8_t>(ng * (16 - j) * 48);
  const bool mixed = j > 0 && j < 16;
  L.lin7 = mixed ? cv.take<uint8_t>(ng * j * 16) : nullptr;
  L.lin1 = mixed ? cv.take<uint8_t>(ng * (16 - j) * 8) : nullptr;
  *ok = cv.ok();
  return L;
}

}  // namespace

size_t layout_ws_bytes(int64_t n_groups, int j) {
  size_t b = 0;
  auto add = [&](int64_t bytes) { b = align_up(b, 256) + (size_t)(bytes > 0 ? bytes : 1); };
  add(n_groups * j * 48);
  add(n_groups * (16 - j) * 48);
  if (j > 0 && j < 16) {
    add(n_groups * j * 16);
    add(n_groups * (16 - j) * 8);
  }
  return align_up(b, 256);
}

gsc_status layout_encode_run(gsc_ctx* c, const float* sh, int64_t n, const int32_t* perm, const float* scales,
                             int layout, int j, uint8_t* blocks, void* ws, size_t ws_bytes, cudaStream_t st) {
  const int64_t ng = ceil_div64(n, 16);
  if (ng == 0) return GSC_OK;
  bool ok = false;
  const LayoutWs L = carve_layout(ws, ws_bytes, ng, j, &ok);
  if (!ws || !ok) return GSC_ERR_OOM;
  gsc_count_launch();
  k_stage_layout<<<grid_of(ng * 16), 32 * LAY_WARPS, 0, st>>>(sh, perm, scales, ng, layout, j, L.tex7, L.tex1);
  GSC_CUDA(cudaGetLastError());
  if (j > 0) {
    GscTimed tm(c, T_BC7, st);
    GSC_CUDA(launch_bc7_blocks(L.tex7, ng * j, j == 16 ? blocks : L.lin7, nullptr, st));
  }
  if (j < 16) {
    GscTimed tm(c, T_BC1, st);
    GSC_CUDA(launch_bc1_blocks(L.tex1, ng * (16 - j), j == 0 ? blocks : L.lin1, nullptr, st));
  }
  if (j > 0 && j < 16) {
    gsc_count_launch();
    k_interleave<<<grid_of(ng * (16 + j)), 256, 0, st>>>(reinterpret_cast<const uint2*>(L.lin7),
                                                          reinterpret_cast<const uint2*>(L.lin1), ng, j,
                                                          reinterpret_cast<uint2*>(blocks));
    GSC_CUDA(cudaGetLastError());
  }
  return GSC_OK;
}
