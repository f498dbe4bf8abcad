// PageRank (Sec. 5.5) in pull form.
//
// The paper keeps every vertex in the frontier, accumulates with atomicAdd
// in an advance (push) and filters out converged vertices. Here each
// iteration gathers over in-neighbourhoods instead (the neighbourhood
// gather-reduce of Sec. 7), which computes the same sums without a scatter:
//
//   gather  sum[v] = sum over edges (v, u) of contrib[u], contrib[u] =
//           rank[u] / deg(u), FP32 (gather_reduce_tiles)
//   update  rank'[v] = (1 - d)/n + d * (sum[v] + D/n), D = rank mass on
//           degree-0 vertices, as FP64 rounds it; writes contrib' and
//           clears sum; the dangling mass of rank' and the L1 change
//           sum |rank' - rank| are reduced in three floats and FP64
//
// k_pr_do runs the whole iteration loop as one cooperative kernel, a grid
// barrier after each of the two; every block takes the same stop decision
// (max_iter iterations, or the L1 change below tol). GR_MODE_LAUNCH enqueues
// the two as kernels of their own, with k_pr_end deciding.
//
// In-neighbours equal out-neighbours only for a symmetric CSR; a directed
// CSR is transposed once on the device (counting sort by column) and the
// gather runs over the transpose with out-degrees from the original.
#include <algorithm>
#include <cstring>

#include "double_single.cuh"
#include "gather.cuh"

namespace gr {

// Gather: 8 entries per lane, 1536 threads per SM. R-MAT 2^21 (63.5 M
// entries): 175 us; 207 us at 2048 threads (spills), 174 at 1280, 191 with
// 16 entries per lane at 1024. The shared-memory tiles before it took 300 us.
// Two blocks of 768 keep the grid barrier's arrivals few.
constexpr int kPrThreads = 768, kPrBlocksPerSm = 2;

struct PrCtl {
  GridBarrier bar;
  float *rank;           // output ranks (set per call)
  double red[2][2];      // L1 change and dangling mass of the ranks being produced, by parity
  double dangling;       // D of the current ranks
  double tol;
  float damping;
  int32_t iter;
  int32_t max_iter;
  int32_t done;
  int32_t error;
};

struct PrWorkspace {
  DevMem contrib, sum, ctl;
  GatherPlan plan;  // of the gather structure (fixed per graph)
  int blocks = 0;  // resident blocks of k_pr_do and k_pr_gather (all SMs)
  DevMem tr_off, tr_col;  // transpose (directed graphs only)
  bool has_transpose = false;
};

void free_pr(PrWorkspace *ws) { delete ws; }

GR_GUARD_REPORTER(guard_report_pr)

namespace {

struct PrArgs {
  const int32_t *C;   // gather structure's columns (the CSR's or its transpose's)
  const int32_t *deg; // out-degrees
  int32_t n;
  float *contrib;
  float *sum;
  PrCtl *ctl;
  int32_t m;
  GatherPlanArgs plan;
};

__global__ void k_pr_init(PrArgs a, float *rank, float damping, int32_t max_iter, double tol,
                          int32_t num_dangling) {
  const float r0 = 1.0f / (float)a.n;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < a.n;
       v += (int64_t)gridDim.x * blockDim.x) {
    rank[v] = r0;
    const int32_t d = a.deg[v];
    a.contrib[v] = d ? r0 / (float)d : 0.0f;
    a.sum[v] = 0.0f;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    PrCtl *c = a.ctl;
    grid_barrier_reset(&c->bar);
    c->rank = rank;
    c->dangling = (double)num_dangling / (double)a.n;
    c->red[0][0] = c->red[0][1] = c->red[1][0] = c->red[1][1] = 0.0;
    c->tol = tol;
    c->damping = damping;
    c->iter = 0;
    c->max_iter = max_iter;
    c->done = max_iter <= 0;
    c->error = kDevOk;
  }
}

// plain loads: k_pr_do rewrites contrib between its gathers
struct ContribG {
  static constexpr bool kWeighted = false;
  const float *contrib;
  __device__ __forceinline__ float operator()(int32_t u, int32_t) const { return contrib[u]; }
};

__device__ __forceinline__ void pr_gather(const PrArgs &a) {
  const ContribG g{a.contrib};
  const StoreReduced<float, ReduceSum<float>> to{a.sum};
  gather_reduce_tiles<1, float, ReduceSum<float>>(a.plan, a.C, nullptr, 0, a.m, g, to,
                                                  spread_warp(), grid_warps());
}

// The part of an iteration's new rank that all vertices share.
__device__ __forceinline__ double pr_base(float damping, int32_t n, double dangling) {
  const double d = damping;
  return (1.0 - d) / n + d * dangling / n;
}

// New ranks from the sums, their contributions, the block's share of the L1
// change (red[0]) and of the dangling mass (red[1]): what FP64 gives or better,
// from FP32 instructions. A rank is the FP64 sum's, rounded once
// (fma_f64_to_f32); the change and the dangling mass are summed in three floats
// a thread and in FP64 from there. In FP64 throughout (two conversions and an
// FMA per vertex, two more operations for the change, and the base's divisions
// in every thread) the FP64 pipe was busy for 50 us of a 245 us iteration at
// R-MAT 2^21; so the update takes 17 us. A thread loads two vertices at once
// (three spill).
constexpr int kPrUpdateItems = 2;

__device__ __forceinline__ void pr_update(const PrArgs &a, float *rank, float damping, double base,
                                          double *smem, double *red) {
  const float bh = (float)base, bl = (float)(base - (double)bh);
  TripleSum dang{0.f, 0.f, 0.f}, delta{0.f, 0.f, 0.f};
  const int64_t step = grid_warps() * 32;
  for (int64_t v0 = spread_warp() * 32 + (threadIdx.x & 31); v0 < a.n; v0 += kPrUpdateItems * step) {
    float s[kPrUpdateItems], ro[kPrUpdateItems];
    int32_t dg[kPrUpdateItems];
#pragma unroll
    for (int j = 0; j < kPrUpdateItems; ++j) {
      const int64_t v = v0 + j * step;
      if (v < a.n) {
        s[j] = a.sum[v];
        ro[j] = rank[v];
        dg[j] = a.deg[v];
      }
    }
#pragma unroll
    for (int j = 0; j < kPrUpdateItems; ++j) {
      const int64_t v = v0 + j * step;
      if (v >= a.n) break;
      const float rn = fma_f64_to_f32(base, bh, bl, damping, s[j]);
      rank[v] = rn;
      a.contrib[v] = dg[j] ? rn / (float)dg[j] : 0.0f;
      a.sum[v] = 0.0f;
      if (!dg[j]) ts_add(dang, rn);
      const DS diff = ds_abs_diff(rn, ro[j]);
      ts_add(delta, diff.hi);
      if (diff.lo != 0.f) ts_add(delta, diff.lo);  // ranks more than a factor of two apart
    }
  }
  block_add_f64<kPrThreads>(ts_to_double(delta), smem, red);
  block_add_f64<kPrThreads>(ts_to_double(dang), smem, red + 1);
}

__device__ __forceinline__ double read_f64(const double *p) { return *(const volatile double *)p; }

__global__ void __launch_bounds__(kPrThreads, kPrBlocksPerSm) k_pr_do(PrArgs a) {
  __shared__ double smem[kPrThreads];
  __shared__ double s_base;
  PrCtl *c = a.ctl;
  float *rank = c->rank;
  const float damping = c->damping;
  const int32_t max_iter = c->max_iter;
  double dangling = c->dangling;
  int32_t it = 0, gen = 0;
  while (it < max_iter) {
    pr_gather(a);
    if (threadIdx.x == 0) s_base = pr_base(damping, a.n, dangling);
    if (!grid_sync(&c->bar, &c->error, gen)) return;
    // the other parity was read by every block before this barrier
    double *red = c->red[it & 1];
    if (blockIdx.x == 0 && threadIdx.x < 2) c->red[(it + 1) & 1][threadIdx.x] = 0.0;
    pr_update(a, rank, damping, s_base, smem, red);
    if (!grid_sync(&c->bar, &c->error, gen)) return;
    ++it;
    dangling = read_f64(red + 1);
    if (read_f64(red) < c->tol) break;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    c->iter = it;
    c->done = 1;
  }
}

// GR_MODE_LAUNCH: one iteration as three kernels.
__global__ void __launch_bounds__(kPrThreads, kPrBlocksPerSm) k_pr_gather(PrArgs a) {
  if (!a.ctl->done) pr_gather(a);
}

__global__ void __launch_bounds__(kPrThreads, kPrBlocksPerSm) k_pr_update(PrArgs a) {
  __shared__ double smem[kPrThreads];
  __shared__ double s_base;
  PrCtl *c = a.ctl;
  if (c->done) return;
  if (threadIdx.x == 0) s_base = pr_base(c->damping, a.n, c->dangling);
  __syncthreads();
  pr_update(a, c->rank, c->damping, s_base, smem, c->red[0]);
}

__global__ void k_pr_end(PrArgs a) {
  PrCtl *c = a.ctl;
  if (c->done) return;
  c->iter += 1;
  if (c->iter >= c->max_iter || c->red[0][0] < c->tol) c->done = 1;
  c->dangling = c->red[0][1];
  c->red[0][0] = c->red[0][1] = 0.0;
}

// ---- transpose for directed graphs: counting sort of (u, v) by v
__global__ void k_tr_count(const int32_t *R, const int32_t *C, int32_t n, int32_t *cnt) {
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = gw; u < n; u += nw)
    for (int32_t e = R[u] + (threadIdx.x & 31); e < R[u + 1]; e += 32) atomicAdd(cnt + C[e], 1);
}

__global__ void k_tr_fill(const int32_t *R, const int32_t *C, int32_t n, int32_t *pos,
                          int32_t *tcol) {
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = gw; u < n; u += nw)
    for (int32_t e = R[u] + (threadIdx.x & 31); e < R[u + 1]; e += 32)
      tcol[atomicAdd(pos + C[e], 1)] = (int32_t)u;
}

// single-block exclusive scan of counts into offsets (one-time setup)
__global__ void k_tr_scan(const int32_t *cnt, int32_t n, int32_t *off, int32_t *pos) {
  __shared__ int32_t s_red[33];
  __shared__ int32_t s_carry;
  if (threadIdx.x == 0) s_carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < n; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int32_t x = i < n ? cnt[i] : 0;
    int32_t tot;
    const int32_t ex = block_excl_sum(x, s_red, &tot);
    if (i < n) {
      off[i] = s_carry + ex;
      pos[i] = s_carry + ex;
    }
    __syncthreads();
    if (threadIdx.x == 0) s_carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) off[n] = s_carry;
}

}  // namespace

static gr_status ensure_pr_ws(gr_graph *g, cudaStream_t s) {
  if (!g->pr) {
    std::unique_ptr<PrWorkspace> ws(new PrWorkspace());
    GR_TRY(ws->contrib.alloc(sizeof(float) * (size_t)g->n, "PageRank contributions"));
    GR_TRY(ws->sum.alloc(sizeof(float) * (size_t)g->n, "PageRank sums"));
    GR_TRY(ws->ctl.alloc(sizeof(PrCtl), "PageRank control"));
    GR_CUDA(cudaMemsetAsync(ws->ctl.p, 0, sizeof(PrCtl), s));
    int per_sm = 1;
    GR_TRY(fit_carveout(k_pr_gather, kPrThreads, kPrBlocksPerSm, g->device, &per_sm));
    GR_TRY(fit_carveout(k_pr_do, kPrThreads, kPrBlocksPerSm, g->device, &per_sm));
    ws->blocks = per_sm * g->num_sms;
    g->pr = ws.release();
  }
  PrWorkspace *ws = g->pr;
  if (!g->symmetric && !ws->has_transpose) {
    GR_TRY(ws->tr_off.alloc(sizeof(int32_t) * ((size_t)g->n + 1), "transpose offsets"));
    GR_TRY(ws->tr_col.alloc(sizeof(int32_t) * (size_t)g->m, "transpose columns"));
    DevMem cnt, pos;
    GR_TRY(cnt.alloc(sizeof(int32_t) * (size_t)g->n, "transpose counts"));
    GR_TRY(pos.alloc(sizeof(int32_t) * (size_t)g->n, "transpose cursor"));
    GR_CUDA(cudaMemsetAsync(cnt.p, 0, cnt.bytes, s));
    const int grid = g->num_sms * 8;
    k_tr_count<<<grid, 256, 0, s>>>(g->row_off.as<int32_t>(), g->col.as<int32_t>(), g->n,
                                    cnt.as<int32_t>());
    k_tr_scan<<<1, 1024, 0, s>>>(cnt.as<int32_t>(), g->n, ws->tr_off.as<int32_t>(),
                                 pos.as<int32_t>());
    k_tr_fill<<<grid, 256, 0, s>>>(g->row_off.as<int32_t>(), g->col.as<int32_t>(), g->n,
                                   pos.as<int32_t>(), ws->tr_col.as<int32_t>());
    GR_CUDA(cudaGetLastError());
    GR_CUDA(cudaStreamSynchronize(s));
    ws->has_transpose = true;
  }
  const int32_t *R = g->symmetric ? g->row_off.as<int32_t>() : ws->tr_off.as<int32_t>();
  return gather_plan_of_call(g, &ws->plan, R, s);
}

static PrArgs pr_args(gr_graph *g) {
  PrWorkspace *ws = g->pr;
  PrArgs a;
  a.C = g->symmetric ? g->col.as<int32_t>() : ws->tr_col.as<int32_t>();
  a.deg = g->degree.as<int32_t>();
  a.n = g->n;
  a.contrib = ws->contrib.as<float>();
  a.sum = ws->sum.as<float>();
  a.ctl = ws->ctl.as<PrCtl>();
  a.m = (int32_t)g->m;
  a.plan = ws->plan.a;
  return a;
}

static gr_status pr_enqueue_iter(gr_graph *g, const PrArgs &a, cudaStream_t s) {
  k_pr_gather<<<g->pr->blocks, kPrThreads, 0, s>>>(a);
  k_pr_update<<<g->pr->blocks, kPrThreads, 0, s>>>(a);
  k_pr_end<<<1, 1, 0, s>>>(a);
  GR_CUDA(cudaGetLastError());
  return GR_OK;
}

}  // namespace gr

using namespace gr;

extern "C" {

gr_status gr_pagerank(gr_graph *g, float damping, int32_t max_iter, double tol, float *rank,
                      int32_t *iters, const gr_opts *opts, void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!(damping > 0.0f && damping < 1.0f)) return fail(GR_EINVAL, "damping must be in (0, 1)");
  if (max_iter < 0) return fail(GR_EINVAL, "max_iter must be >= 0");
  if (!(tol >= 0.0)) return fail(GR_EINVAL, "tol must be >= 0");
  if (!rank) return fail(GR_EINVAL, "rank must not be NULL");
  const gr_opts &o = opts ? *opts : default_opts();
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  GR_TRY(ensure_pr_ws(g, s));
  void *d_rank;
  bool cp_rank;
  GR_TRY(resolve_output(g, 0, rank, sizeof(float) * (size_t)g->n, &d_rank, &cp_rank));
  PrArgs a = pr_args(g);
  k_pr_init<<<g->num_sms * 8, 256, 0, s>>>(a, (float *)d_rank, damping, max_iter, tol,
                                           g->num_isolated);
  GR_CUDA(cudaGetLastError());
  if (max_iter > 0) {
    if (o.mode == GR_MODE_LAUNCH) {
      PrCtl h;
      for (int32_t it = 0; it < max_iter;) {
        const int32_t batch = std::min<int32_t>(8, max_iter - it);
        for (int32_t i = 0; i < batch; ++i) GR_TRY(pr_enqueue_iter(g, a, s));
        it += batch;
        GR_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
        GR_CUDA(cudaStreamSynchronize(s));
        if (h.done) break;
      }
    } else {
      void *args[] = {&a};
      GR_CUDA(cudaLaunchCooperativeKernel((void *)k_pr_do, g->pr->blocks, kPrThreads, args, 0, s));
    }
  }
  if (cp_rank)
    GR_CUDA(cudaMemcpyAsync(rank, d_rank, sizeof(float) * (size_t)g->n,
                            cudaMemcpyDeviceToHost, s));
  if (iters) {
    PrCtl h;
    GR_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
    GR_CUDA(cudaStreamSynchronize(s));
    if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
    *iters = h.iter;
  }
  GR_TRY(end_call(g, s));
  return GR_OK;
}

gr_status gr_pagerank_stats(gr_graph *g, int32_t *iters) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  std::lock_guard<std::mutex> lock(g->mu);
  if (!g->pr) return fail(GR_EINVAL, "no PageRank has run on this graph");
  GR_CUDA(cudaSetDevice(g->device));
  if (g->has_last) GR_CUDA(cudaEventSynchronize(g->last_done));
  PrCtl h;
  GR_CUDA(cudaMemcpy(&h, g->pr->ctl.p, sizeof(PrCtl), cudaMemcpyDeviceToHost));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (iters) *iters = h.iter;
  return GR_OK;
}

}  // extern "C"
