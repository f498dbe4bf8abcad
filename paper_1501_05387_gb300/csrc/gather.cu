// Construction of the gather-reduce's plan (gather.cuh): five small kernels
// over the rows and the 256-entry tiles, once per graph.
#include "gather.cuh"

namespace gr {
namespace {

constexpr int kGpWords = kGpTile / 16;  // desc words (two groups of 8 entries) per tile
constexpr int kGpBlockTiles = 128;       // tiles per block of the rank scan
constexpr int kGpThreads = 256;

// The last entry of every row, as a bit of desc.
__global__ void k_gp_ends(const int32_t *R, int32_t n, uint32_t *desc2) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r1 = R[v + 1];
    if (r1 > R[v]) {
      const uint32_t e = (uint32_t)r1 - 1u;
      atomicOr(desc2 + (e >> 4), 1u << (((e >> 3) & 1u) * 16u + (e & 7u)));
    }
  }
}

// Rows that end in each block's kGpBlockTiles tiles.
__global__ void __launch_bounds__(kGpThreads) k_gp_sums(const uint32_t *desc2, int64_t words,
                                                        int32_t *part) {
  __shared__ int32_t red[33];
  int32_t local = 0;
  const int64_t w0 = (int64_t)blockIdx.x * kGpBlockTiles * kGpWords;
  for (int j = threadIdx.x; j < kGpBlockTiles * kGpWords; j += kGpThreads)
    if (w0 + j < words) local += __popc(desc2[w0 + j] & 0x00FF00FFu);
  const int32_t total = block_sum(local, red);
  if (threadIdx.x == 0) part[blockIdx.x] = total;
}

__global__ void k_gp_parts(int32_t *part, int32_t count) {
  __shared__ int32_t red[33];
  int32_t carry = 0;
  for (int32_t b = 0; b < count; b += blockDim.x) {  // block-uniform
    const int32_t i = b + threadIdx.x;
    const int32_t x = i < count ? part[i] : 0;
    int32_t total;
    const int32_t ex = block_excl_sum(x, red, &total);
    if (i < count) part[i] = carry + ex;
    carry += total;
  }
}

// rank_base and the rank bytes of desc: kGpWords lanes per tile, one word
// each, kGpThreads / kGpWords tiles at a time.
__global__ void __launch_bounds__(kGpThreads) k_gp_apply(uint32_t *desc2, int64_t words,
                                                         const int32_t *part,
                                                         uint32_t *rank_base) {
  static_assert(kGpWords == 16, "half a warp per tile");
  __shared__ int32_t red[33];
  int32_t run = part[blockIdx.x];
  const int sub = threadIdx.x % kGpWords;
  for (int j = threadIdx.x; j < kGpBlockTiles * kGpWords; j += kGpThreads) {  // block-uniform trips
    const int64_t w = (int64_t)blockIdx.x * kGpBlockTiles * kGpWords + j;
    uint32_t x = w < words ? desc2[w] & 0x00FF00FFu : 0u;
    const int32_t lo = __popc(x & 0xFFu), mine = lo + __popc(x >> 16);
    int32_t incl = mine;  // over the tile's half warp
#pragma unroll
    for (int o = 1; o < kGpWords; o <<= 1) {
      const int32_t y = __shfl_up_sync(0xffffffffu, incl, o, kGpWords);
      if (sub >= o) incl += y;
    }
    // rows that end before this tile in the block's round
    int32_t total;
    const int32_t ex = block_excl_sum(sub == kGpWords - 1 ? incl : 0, red, &total);
    if (w < words) {
      if (sub == 0) {
        // the entry before the tile ends a row: the top flag of the word
        // before, whose rank bytes may be written already (its flags stay)
        const bool opens = w == 0 || ((desc2[w - 1] >> 23) & 1u);
        rank_base[w / kGpWords] = (uint32_t)(run + ex) | (opens ? 0x80000000u : 0u);
      }
      const uint32_t before = (uint32_t)(incl - mine);
      desc2[w] = x | (before << 8) | ((before + (uint32_t)lo) << 24);
    }
    run += total;
  }
}

__global__ void k_gp_rows(const int32_t *R, int32_t n, const uint16_t *desc,
                          const uint32_t *rank_base, int32_t *rows) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r0 = R[v];
    if (R[v + 1] > r0) {
      const uint32_t d = desc[r0 >> 3];
      const uint32_t k = (rank_base[r0 / kGpTile] & 0x7FFFFFFFu) + (d >> 8) +
                         __popc(d & ((1u << (r0 & 7)) - 1u));
      rows[k] = (int32_t)v;
    }
  }
}

}  // namespace

gr_status gather_plan_build(GatherPlan *p, const int32_t *R, int32_t n, int64_t m,
                            cudaStream_t s) {
  if (p->mem.p) return GR_OK;
  // kernels that only go into a graph would leave a plan on paper
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  GR_CUDA(cudaStreamIsCapturing(s, &capture));
  if (capture != cudaStreamCaptureStatusNone)
    return fail(GR_ECUDA, "a graph's first call cannot be captured: it builds a plan");
  // a warp's tile may take two rank_base tiles: an even number of them
  const int64_t tiles = 2 * ((m + 2 * kGpTile - 1) / (2 * kGpTile));
  const int64_t words = tiles * kGpWords;
  const int64_t blocks = (tiles + kGpBlockTiles - 1) / kGpBlockTiles;
  GR_TRY(p->mem.alloc(sizeof(uint32_t) * (size_t)(words + tiles + n + blocks), "gather plan"));
  uint32_t *desc2 = p->mem.as<uint32_t>();
  uint32_t *rank_base = desc2 + words;
  int32_t *rows = (int32_t *)(rank_base + tiles);
  int32_t *part = rows + n;
  const GatherPlanArgs a = {(const uint16_t *)desc2, rank_base, rows};
  if (m > 0) {
    const int grid = (int)std::min<int64_t>(((int64_t)n + 255) / 256, 4096);
    cudaError_t e = cudaMemsetAsync(desc2, 0, sizeof(uint32_t) * (size_t)words, s);
    if (e == cudaSuccess) {
      k_gp_ends<<<grid, 256, 0, s>>>(R, n, desc2);
      k_gp_sums<<<(unsigned)blocks, kGpThreads, 0, s>>>(desc2, words, part);
      k_gp_parts<<<1, 1024, 0, s>>>(part, (int32_t)blocks);
      k_gp_apply<<<(unsigned)blocks, kGpThreads, 0, s>>>(desc2, words, part, rank_base);
      k_gp_rows<<<grid, 256, 0, s>>>(R, n, a.desc, rank_base, rows);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
      p->mem.reset();  // not a plan
      return cuda_fail(e, "gather plan");
    }
  }
  p->a = a;
  return GR_OK;
}

gr_status gather_plan_of_call(gr_graph *g, GatherPlan *p, const int32_t *R, cudaStream_t s) {
  if (p->mem.p) return GR_OK;
  GR_TRY(gather_plan_build(p, R, g->n, g->m, s));
  const gr_status st = end_call(g, s);
  if (st != GR_OK) p->mem.reset();
  return st;
}

}  // namespace gr
