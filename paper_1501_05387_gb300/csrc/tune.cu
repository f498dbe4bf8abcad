// Autotuner: per-graph choice of the traversal knobs the paper leaves to
// the user (Sec. 4.4: the hybrid's threshold "can be changed easily ... for
// their own datasets"; Sec. 6: "we can predict which strategies will be most
// beneficial based only on the degree distribution").
//
// Two stages:
//   * a prior from degree statistics, set when the graph is created
//     (tune_prior): mesh-like graphs (small maximum degree) get push-only
//     traversal and a small persistent grid (cheap barriers for thousands of
//     levels); skewed graphs get direction-optimising traversal on the full
//     GPU;
//   * gr_autotune measures the graph's present settings and candidates for
//     others (tune_core.hpp) on sample sources with CUDA events and keeps the
//     fastest: BFS level-loop driver, persistent grid
//     size, push->pull / pull->push thresholds (alpha, beta), and the SSSP
//     near/far bucket width. The results are stored in the graph and used
//     whenever the caller's options leave a field at 0.
// Tuning never changes results: every candidate computes the same depths
// and distances.
#include <algorithm>
#include <cfloat>
#include <vector>

#include "gr_internal.cuh"
#include "tune_core.hpp"

namespace gr {

int32_t bfs_push_blocks(int64_t m) {
  return m < 150'000 ? 1 : m < 700'000 ? 3 : m < 1'500'000 ? 4 : 0;
}

void tune_prior(gr_graph *g) {
  // push -> pull once the frontier's edges exceed a tenth of the unexplored
  // ones: on R-MAT s22 (16 sources, 6 blocks per SM) alpha 8-10 took 0.1875
  // ms per traversal against 0.190 at 14, 0.192 at 6 and 0.210 at 4; beta
  // 16-36 made no difference
  g->tuned_alpha = 10.f;
  g->tuned_beta = 24.f;
  if (g->max_degree <= 32) {
    g->tuned_direction = GR_DIR_PUSH;  // never pull: frontiers stay thin
    g->tuned_blocks_per_sm = 1;
    // thousands of thin iterations: one kernel with a cheap grid barrier
    g->tuned_sssp_mode = GR_MODE_PERSISTENT;
    g->tuned_sssp_blocks_per_sm = 1;
    // Thin frontiers, six mean weights a bucket: one block's search
    // (k_sssp_solo) of grids of 64 to 1024 a side, weights to 16, 64 and 1000,
    // took 1.0-1.1 times its best there, 1.1-1.5 times at two mean weights,
    // 1.0-1.1 at twelve; the grid kernel at two, six and twelve: 1400 a side 41.6,
    // 29.2, 25.1 ms, 4096 a side 147, 104, 89 ms. Thick ones, and merge-path
    // chunks (degrees 17 to 32), keep two: random graphs of degree 18 to 28 and
    // 0.4 to 1.2 M entries 250-490 us at two, 4-18 % more at six.
    if (g->has_weights && g->max_degree <= kLowDegreeMax)
      g->sssp_delta = (uint32_t)std::max(1.0, std::min(6.0 * g->mean_weight, 4.0e9));
  } else {
    g->tuned_direction = GR_DIR_AUTO;
    // Small graphs are bound by the grid barrier, whose cost grows with the
    // blocks that meet at it. BFS at 1, 2, 3 and 4 blocks per SM (means of eight
    // sources): R-MAT 1.8 M entries 47, 52, 54, 57 us; 7.6 M 58, 63, 65, 68; 15 M
    // 66, 68, 71, 73; 24 M, ids at random, 91, 85, 85, 87; 31 M 98, 88, 85, 87;
    // 64 M, ids at random, 160, 120, 110, 108; 128 M 162, 116, 109, 105.
    // Directed graphs push every level, which takes more of them (three graphs
    // each at 1 to 6): 0.1 M entries 51, 55, 57, 59, 61, 64 us; 0.47 M 75, 74,
    // 72, 75, 77, 80; 1 M 99, 84, 80, 80, 81, 81; 2.2 M 149, 111, 99, 95, 94, 93;
    // 3 M 190, 136, 115, 111, 106, 108.
    if (g->symmetric)
      g->tuned_blocks_per_sm = g->m < 20'000'000 ? 1 : g->m < 48'000'000 ? 3 : 4;
    else
      g->tuned_blocks_per_sm = bfs_push_blocks(g->m);
    // SSSP at 1 to 5: 2^12 101, 115, 123, 126, 141 us; 2^14 (0.4 M) 158, 143,
    // 133, 141, 151; 2^16 195, 181, 181, 186, 198; 2^18 422, 292, 262, 243, 251;
    // 2^20 (31 M) 1552, 914, 726, 629, 607.
    g->tuned_sssp_blocks_per_sm = sssp_prior_blocks(g->m);
    // skewed graphs reach most vertices in a few dense relaxations: the
    // persistent kernel, and buckets wide enough not to repeat them (R-MAT
    // 2^21, pushed: 2.28 ms in the graph loop at two mean weights a bucket,
    // 1.60 so; 2^16: 432 and 315 us)
    g->tuned_sssp_mode = GR_MODE_PERSISTENT;
    if (g->has_weights)
      g->sssp_delta = g->sssp_delta_thick =
          (uint32_t)std::max(1.0, std::min(8.0 * g->mean_weight, 4.0e9));
  }
  // A frontier with a third of the edges is relaxed in pull form where its
  // 256-entry tiles fill the GPU: R-MAT 2^21 0.95 ms (1.60 pushed; 0.95 from
  // half of the edges, 0.96 from a sixth, 1.01 from an eighth), 300,001
  // vertices 0.42 ms (0.55), but 2^16 and 1.4 M entries 326 us (321), 2^13
  // 128 us (115).
  g->tuned_sssp_alpha = g->m >= (int64_t)g->num_sms * 10240 ? 3.f : 0.f;
  // Degrees 17 to 32 run one block per SM, with which a pull can take longer than
  // the push; at two, pushed at one and pulled at one and two: Erdos-Renyi of
  // mean degree 8 and 1 M vertices 1282, 1543, 1045 us, 3 M 3079, 3404, 2114;
  // random of degree 20, 1.5 M vertices 3899, 5277, 2952; of degree 28, 300,000
  // vertices 1547, 946, 671; a mesh of 1000 a side with hubs 16.7, 14.3, 16.1 ms.
  if (g->tuned_sssp_alpha > 0.f && g->max_degree > kLowDegreeMax && g->max_degree <= 32)
    g->tuned_sssp_blocks_per_sm = 2;
  g->tuned_mode = GR_MODE_AUTO;
}

namespace {

// Each candidate is timed this many times over the sample (after one
// untimed run); the fastest repetition counts, so one slow run (a clock
// ramp, another process) does not decide the choice.
constexpr int kTuneReps = 3;

struct Timer {
  cudaEvent_t a = nullptr, b = nullptr;
  Timer() {
    cudaEventCreate(&a);
    cudaEventCreate(&b);
  }
  ~Timer() {
    cudaEventDestroy(a);
    cudaEventDestroy(b);
  }
};

}  // namespace

}  // namespace gr

using namespace gr;

extern "C" {

gr_status gr_autotune(gr_graph *g, const int32_t *srcs, int32_t k, int32_t what,
                      void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (k < 1 || !srcs) return fail(GR_EINVAL, "need at least one sample source");
  for (int32_t i = 0; i < k; ++i)
    if (srcs[i] < 0 || srcs[i] >= g->n) return fail(GR_EINVAL, "source out of range");
  if (what & ~(GR_TUNE_BFS | GR_TUNE_SSSP)) return fail(GR_EINVAL, "unknown tuning flags");
  if ((what & GR_TUNE_SSSP) && !g->has_weights)
    return fail(GR_EINVAL, "SSSP tuning needs edge weights");
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  DevMem out, out2;
  GR_TRY(out.alloc(sizeof(int32_t) * (size_t)g->n, "tuning output"));
  Timer t;
  if (what & GR_TUNE_BFS) {
    if (!g->bfs) GR_TRY(bfs_ws_create(g, s, &g->bfs));
    const std::vector<BfsSetting> cands =
        bfs_settings({g->tuned_mode, g->tuned_blocks_per_sm, g->tuned_direction, g->tuned_alpha,
                      g->tuned_beta},
                     g->symmetric);
    float best = FLT_MAX;
    BfsSetting pick = cands[0];
    const int32_t saved_bps = g->tuned_blocks_per_sm;
    for (const BfsSetting &c : cands) {
      gr_opts o = default_opts();
      o.mode = c.mode;
      o.alpha = c.alpha;
      o.beta = c.beta;
      o.direction = c.dir;
      g->tuned_blocks_per_sm = c.bps;
      // one untimed run, then the sample kTuneReps times
      GR_TRY(bfs_run(g, g->bfs, srcs[0], out.as<int32_t>(), nullptr, o, s));
      float ms = FLT_MAX;
      for (int rep = 0; rep < kTuneReps; ++rep) {
        GR_CUDA(cudaEventRecord(t.a, s));
        for (int32_t i = 0; i < k; ++i)
          GR_TRY(bfs_run(g, g->bfs, srcs[i], out.as<int32_t>(), nullptr, o, s));
        GR_CUDA(cudaEventRecord(t.b, s));
        GR_CUDA(cudaEventSynchronize(t.b));
        GR_TRY(bfs_read_ctl_error(g->bfs, s));
        float r = 0.f;
        GR_CUDA(cudaEventElapsedTime(&r, t.a, t.b));
        ms = std::min(ms, r);
      }
      if (ms < best) {
        best = ms;
        pick = c;
      }
    }
    g->tuned_blocks_per_sm = pick.bps;
    if (pick.mode == GR_MODE_GRAPH) g->tuned_blocks_per_sm = saved_bps;
    g->tuned_mode = pick.mode;
    g->tuned_direction = pick.dir;
    g->tuned_alpha = pick.alpha;
    g->tuned_beta = pick.beta;
    g->tuned_bfs_ms = best / k;
  }
  if (what & GR_TUNE_SSSP) {
    if (!g->sssp) GR_TRY(sssp_ws_create(g, s, &g->sssp));
    const std::vector<SsspSetting> cands = sssp_settings(
        {g->tuned_sssp_mode, g->tuned_sssp_blocks_per_sm, g->sssp_delta, g->tuned_sssp_alpha},
        g->mean_weight, g->weights_symmetric && g->max_degree > kLowDegreeMax);
    float best = FLT_MAX;
    SsspSetting pick = cands[0];
    const int32_t saved_sbps = g->tuned_sssp_blocks_per_sm;
    for (const SsspSetting &c : cands) {
      gr_opts o = default_opts();
      o.delta = c.delta;
      o.mode = c.mode;
      if (c.alpha > 0.f) o.alpha = c.alpha;
      else o.direction = GR_DIR_PUSH;
      // the candidate's grid size goes through the graph's tuned value, as
      // it will be used afterwards (o.block = 0 would mean "tuned", and 0
      // here means "all resident blocks")
      g->tuned_sssp_blocks_per_sm = c.bps;
      GR_TRY(sssp_run(g, g->sssp, srcs[0], out.as<uint32_t>(), nullptr, o, s));
      float ms = FLT_MAX;
      for (int rep = 0; rep < kTuneReps; ++rep) {
        GR_CUDA(cudaEventRecord(t.a, s));
        for (int32_t i = 0; i < k; ++i)
          GR_TRY(sssp_run(g, g->sssp, srcs[i], out.as<uint32_t>(), nullptr, o, s));
        GR_CUDA(cudaEventRecord(t.b, s));
        GR_CUDA(cudaEventSynchronize(t.b));
        GR_TRY(sssp_read_ctl_error(g->sssp, s));
        float r = 0.f;
        GR_CUDA(cudaEventElapsedTime(&r, t.a, t.b));
        ms = std::min(ms, r);
      }
      if (ms < best) {
        best = ms;
        pick = c;
      }
    }
    // UINT32_MAX selects "one bucket"; it is stored as is
    g->sssp_delta = g->sssp_delta_thick = pick.delta;
    g->tuned_sssp_alpha = pick.alpha;
    g->tuned_sssp_mode = pick.mode;
    g->tuned_sssp_blocks_per_sm = pick.mode == GR_MODE_PERSISTENT ? pick.bps : saved_sbps;
    g->tuned_sssp_ms = best / k;
  }
  GR_CUDA(cudaStreamSynchronize(s));
  GR_TRY(end_call(g, s));
  return GR_OK;
}

gr_status gr_tuned_sssp(const gr_graph *g, int32_t *mode, int32_t *blocks_per_sm,
                        uint32_t *delta) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (mode) *mode = g->tuned_sssp_mode;
  if (blocks_per_sm) *blocks_per_sm = g->tuned_sssp_blocks_per_sm;
  if (delta) *delta = g->sssp_delta;
  return GR_OK;
}

gr_status gr_tuned_opts(const gr_graph *g, gr_opts *out, double *bfs_ms, double *sssp_ms) {
  clear_error();
  if (!g || !out) return fail(GR_EINVAL, "graph and out must not be NULL");
  *out = default_opts();
  out->mode = g->tuned_mode;
  out->direction = g->tuned_direction;
  out->alpha = g->tuned_alpha;
  out->beta = g->tuned_beta;
  out->block = g->tuned_blocks_per_sm;
  out->delta = g->sssp_delta;
  out->max_iters = 0;
  if (bfs_ms) *bfs_ms = g->tuned_bfs_ms;
  if (sssp_ms) *sssp_ms = g->tuned_sssp_ms;
  return GR_OK;
}

}  // extern "C"
