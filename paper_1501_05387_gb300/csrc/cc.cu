// Connected components by hooking and pointer jumping (Sec. 5.4).
//
// The paper runs hooking as a filter over an edge frontier (every edge tries
// to give the smaller component id of its ends to the other end; edges whose
// ends already agree are filtered out) until no id changes, then pointer
// jumping as a filter over vertices until every vertex points at its root.
//
// Hooking here links roots only, larger root under smaller (atomicCAS on the
// larger root's own entry, so a root is re-pointed only while it is still a
// root). A CAS that loses a race retries with the roots it now finds, so
// each edge is settled in one visit: the paper's "repeat until no id
// changes" happens per edge instead of per sweep, and a single sweep over
// the CSR's edges (the all-vertex frontier of the load-balanced advance)
// leaves one tree per component. Finding a root halves the path it walks.
// Pointer jumping then points every vertex at its root. Because a root is
// only ever hooked under a smaller id, the root of each component is its
// smallest vertex id, which is the canonical label.
//
// Symmetric graphs store each undirected edge twice, so most edges need no
// visit at all: the sampling form of the hooking sweep starts every vertex
// under the end of a short chain of first neighbours (each with a smaller id:
// no cycle, and no atomic), hooks it to the second and compresses, which on graphs
// with one giant component already places most vertices in it; the
// component that most of a fixed sample of vertices lies in is then
// skipped, and only the vertices outside it hook all their edges (an edge
// between two vertices of that component needs no visit, one leaving it is
// visited from its other end). Labels are the same as with a full sweep:
// hooking under the smaller root makes every root its component's smallest
// id whatever the order. For a directed CSR every arc hooks in one sweep,
// giving weakly connected components (an arc is not visible from its head).
#include "advance.cuh"

namespace gr {

constexpr int kCcThreads = 256, kCcItems = 8;
constexpr int kCcPicks = 1024;  // vertices whose roots choose the skipped component
constexpr int kCcFrontierCap = 1024;

struct CcWorkspace {
  DevMem counter;  // [0] components, [1] scratch; [2..3] packed frontier counter
  DevMem q, sc, skip;
};

void free_cc(CcWorkspace *ws) { delete ws; }

GR_GUARD_REPORTER(guard_report_cc)

namespace {

// first (may be null): the vertices' first neighbours, -1 where there is none.
// A vertex starts under the end of the chain of first neighbours of ever
// smaller ids, if that ends within kCcChain steps (on a skewed graph, at a hub),
// and else on its own: a mesh's chains are as long as its side, a path's as the
// graph, and trees that deep would make every later walk to the root as long
// (linked all the way, a path of 4 M vertices took 2.7 ms).
constexpr int kCcChain = 8;
__global__ void k_cc_init(int32_t *label, const int32_t *first, int32_t n) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    int32_t x = (int32_t)v;
    bool end = !first;
    for (int i = 0; i < kCcChain && !end; ++i) {
      const int32_t u = first[x];
      end = u < 0 || u >= x || !GR_IN(u, n, 404);
      if (!end) x = u;
    }
    label[v] = end ? x : (int32_t)v;
  }
}

// root of x with path halving (pointers only ever decrease)
__device__ __forceinline__ int32_t find_root(int32_t *label, int32_t x);

// Join the trees of u and v: the larger root is re-pointed to the smaller
// one with a CAS, retried from the current roots if another thread moved
// the root first.
__device__ __forceinline__ void hook(int32_t *label, int32_t u, int32_t v);

__device__ __forceinline__ int32_t find_root(int32_t *label, int32_t x) {
  int32_t p = label[x];
  while (p != x) {
    const int32_t gp = label[p];
    if (gp != p) label[x] = gp;  // halving: benign race, gp is an ancestor
    x = p;
    p = gp;
  }
  return x;
}

__device__ __forceinline__ void hook(int32_t *label, int32_t u, int32_t v) {
  int32_t a = find_root(label, u);
  int32_t b = find_root(label, v);
  while (a != b) {
    const int32_t hi = max(a, b), lo = min(a, b);
    const int32_t prev = atomicCAS(label + hi, hi, lo);
    if (prev == hi) break;  // hooked
    // hi stopped being a root: continue from the roots as they are now
    a = find_root(label, prev);
    b = find_root(label, lo);
  }
}

struct HookF {
  int32_t *label;
  int32_t only_lower;  // symmetric graph: hook each undirected edge once
  int32_t n;
  __device__ __forceinline__ int operator()(int32_t u, int32_t v, int32_t) const {
    if (!GR_IN(u, n, 401) || !GR_IN(v, n, 402)) return 0;
    if (only_lower && v >= u) return 0;
    hook(label, u, v);
    return 0;  // edge settled: filtered out of the edge frontier
  }
};

// The sampling pass's form of hook. Its walks write only the entry of the
// thread's own vertex: halving a path on the way, as find_root does, makes
// every thread below a hub's root store to the same few entries, and an entry
// read from a stale L1 line can put an older ancestor back (R-MAT with ids at
// random, 2^20 vertices: the pass alone 350 us). An own entry only ever moves
// up, and is what other walks through the vertex follow: together they double
// their steps as halving would. Lanes that meet at one root send one CAS.
__device__ __forceinline__ int32_t walk(const int32_t *label, int32_t x) {
  int32_t p = label[x];
  while (p != x) {
    x = p;
    p = label[x];
  }
  return x;
}

__device__ __forceinline__ int32_t walk_own(int32_t *label, int32_t v) {
  int32_t p = label[v];
  if (p == v) return v;
  for (;;) {
    const int32_t gp = label[p];
    if (gp == p) return p;
    label[v] = gp;  // v is no root: nobody else writes its entry
    p = gp;
  }
}

__device__ __forceinline__ void hook_own(int32_t *label, int32_t v, int32_t x) {
  int32_t a = walk_own(label, v);
  int32_t b = walk(label, x);
  while (a != b) {
    const int32_t hi = max(a, b), lo = min(a, b);
    // whichever threads are here together: each of them gets the same mask and
    // takes part in what names it, and any such group may share one CAS
    const uint32_t peers = __match_any_sync(__activemask(), hi);
    const int leader = __ffs(peers) - 1;
    int32_t prev = 0;
    if ((threadIdx.x & 31) == leader) prev = atomicCAS(label + hi, hi, lo);
    prev = __shfl_sync(peers, prev, leader);
    const int32_t under = __shfl_sync(peers, lo, leader);
    if (prev == hi) {  // hooked under the leader's root
      if (under == lo) break;
      prev = under;
    }
    a = walk(label, prev);
    b = walk(label, lo);
  }
}

// Each vertex hooks to its second neighbour, and to its first where
// k_cc_init left it on its own. The trees are shallow by then and most pairs
// share one already: R-MAT 2^22 151 us, 240 when all vertices start on their
// own; ids at random, 2^20: 130 (350 us with halving walks), 2^18 90 (570);
// grids 300 and 700 a side 125 and 145 (155 and 235).
__global__ void k_cc_sample(const int32_t *R, const int32_t *C, const int32_t *first, int32_t n,
                            int32_t *label) {
  for (int64_t vv = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; vv < n;
       vv += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = (int32_t)vv;
    const int32_t u = first[v];
    if (u < 0) continue;
    const int32_t r = R[v] + 1;
    if (label[v] == v) hook_own(label, v, u);
    if (r < R[v + 1]) {
      const int32_t x = C[r];
      if (GR_IN(x, n, 403)) hook_own(label, v, x);
    }
  }
}

// The component to skip: the root (label after compression) that most of
// kCcPicks vertices have, spread over the ids by a multiplicative hash; the
// smallest of equals. One block, a vertex per thread; the roots are counted
// warp by warp in a hash table in shared memory. Fetching them to sort them
// on the host stopped the stream for 60 us; comparing each with all took 18.
__global__ void __launch_bounds__(kCcPicks) k_cc_pick(const int32_t *label, int32_t n,
                                                      int32_t *skip) {
  constexpr uint32_t kSlots = 2 * kCcPicks;
  __shared__ int32_t s_root[kSlots];
  __shared__ uint32_t s_count[kSlots];
  __shared__ unsigned long long s_best;
  for (uint32_t i = threadIdx.x; i < kSlots; i += kCcPicks) {
    s_root[i] = -1;
    s_count[i] = 0u;
  }
  if (threadIdx.x == 0) s_best = 0ull;
  const int32_t root = label[(int32_t)(((unsigned long long)threadIdx.x * 2654435761ull) % n)];
  __syncthreads();
  const uint32_t peers = __match_any_sync(0xffffffffu, root);
  if ((threadIdx.x & 31) == (uint32_t)(__ffs(peers) - 1)) {
    uint32_t i = ((uint32_t)root * 2654435761u) % kSlots;  // at most kCcPicks roots: one is free
    for (;;) {
      const int32_t there = atomicCAS(&s_root[i], -1, root);
      if (there == -1 || there == root) break;
      i = (i + 1) % kSlots;
    }
    atomicAdd(&s_count[i], (uint32_t)__popc(peers));
  }
  __syncthreads();
  unsigned long long best = 0ull;
  for (uint32_t i = threadIdx.x; i < kSlots; i += kCcPicks)
    if (s_count[i]) {
      const unsigned long long mine =
          ((unsigned long long)s_count[i] << 32) | (0x7FFFFFFFu - (uint32_t)s_root[i]);
      best = best > mine ? best : mine;
    }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long x = __shfl_xor_sync(0xffffffffu, best, o);
    best = best > x ? best : x;
  }
  if ((threadIdx.x & 31) == 0 && best) atomicMax(&s_best, best);
  __syncthreads();
  if (threadIdx.x == 0) *skip = (int32_t)(0x7FFFFFFFu - (uint32_t)(s_best & 0xFFFFFFFFull));
}

// The vertices outside component `skip` that have edges, with their
// degrees (an exclusive scan, emitted block by block with one packed atomic):
// the frontier whose edges the last hooking pass visits.
__global__ void __launch_bounds__(kCcThreads) k_cc_rest_frontier(const int32_t *R,
                                                                  const int32_t *label, int32_t n,
                                                                  const int32_t *skip_p, int32_t *Q,
                                                                  int32_t *S,
                                                                  unsigned long long *packed) {
  __shared__ ScannedBuf<kCcFrontierCap> buf;
  const int32_t skip = *skip_p;
  if (threadIdx.x == 0) buf.cnt = 0;
  __syncthreads();
  constexpr int PER = kCcFrontierCap / kCcThreads;
  for (int64_t base = (int64_t)blockIdx.x * kCcFrontierCap; base < n;
       base += (int64_t)gridDim.x * kCcFrontierCap) {  // block-uniform
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int64_t v = base + j * kCcThreads + threadIdx.x;
      int32_t d = 0;
      bool take = false;
      if (v < n && label[v] != skip) {
        d = R[v + 1] - R[v];
        take = d > 0;
      }
      emit_scanned(buf, take, (int32_t)v, d);
    }
    flush_scanned<kCcThreads>(buf, packed, Q, S, (long long)n + 1);
  }
}

// Hook every edge of the frontier Q (size and scan from k_cc_rest_frontier).
__global__ void __launch_bounds__(kCcThreads) k_cc_hook_rest(const int32_t *R, const int32_t *C,
                                                              int32_t n, int32_t *label,
                                                              const int32_t *Q, const int32_t *S,
                                                              const unsigned long long *packed) {
  HookF f{label, 0, n};
  const unsigned long long p = *packed;
  lb_advance<kCcThreads, kCcItems, 0>(R, C, Q, (int32_t)(p & 0xFFFFFFFFull), S, (int32_t)(p >> 32),
                                      f, nullptr, nullptr, nullptr, nullptr);
}

__global__ void __launch_bounds__(kCcThreads) k_cc_hook(const int32_t *R, const int32_t *C,
                                                         int32_t n, int32_t *label,
                                                         int32_t only_lower) {
  HookF f{label, only_lower, n};
  // every edge is settled in its visit: the edge frontier it would filter
  // into stays empty, so the advance appends nothing
  lb_advance<kCcThreads, kCcItems, 0>(R, C, nullptr, n, R, R[n], f, nullptr, nullptr, nullptr,
                                      nullptr);
}

__global__ void k_cc_jump(int32_t *label, int32_t n, int32_t *num_roots) {
  int32_t roots = 0;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    // a walk that writes nothing on the way: halving another vertex's path
    // here could put an older ancestor back over the root it has been given
    int32_t r = label[v];
    while (label[r] != r) r = label[r];
    label[v] = r;
    roots += r == v;
  }
  for (int o = 16; o > 0; o >>= 1) roots += __shfl_xor_sync(0xffffffffu, roots, o);
  if ((threadIdx.x & 31) == 0 && roots) atomicAdd(num_roots, roots);
}

}  // namespace

size_t cc_ws_bytes(const gr_graph *g) {
  return sizeof(int32_t) * 4 + sizeof(int32_t) * (2 * (size_t)g->n + 3) +
         sizeof(int32_t);
}

gr_status cc_ws_create(gr_graph *g, CcWorkspace **out) {
  std::unique_ptr<CcWorkspace> ws(new CcWorkspace());
  GR_TRY(ws->counter.alloc(sizeof(int32_t) * 4, "CC counters"));
  if (g->symmetric) {
    GR_TRY(ws->q.alloc(sizeof(int32_t) * ((size_t)g->n + 1), "CC frontier"));
    GR_TRY(ws->sc.alloc(sizeof(int32_t) * ((size_t)g->n + 2), "CC frontier degree scan"));
    GR_TRY(ws->skip.alloc(sizeof(int32_t), "CC skipped component"));
  }
  *out = ws.release();
  return GR_OK;
}

// CC into a device label array with an explicit workspace; the component
// count is left in the workspace counter (cc_count reads it).
gr_status cc_run(gr_graph *g, CcWorkspace *ws, int32_t *label, cudaStream_t s) {
  int32_t *cnt = ws->counter.as<int32_t>();
  const int grid = g->num_sms * 8;
  const int32_t *R = g->row_off.as<int32_t>(), *C = g->col.as<int32_t>();
  GR_CUDA(cudaMemsetAsync(cnt, 0, sizeof(int32_t) * 4, s));
  const int32_t *first = g->symmetric ? g->first_col.as<int32_t>() : nullptr;
  k_cc_init<<<grid, 256, 0, s>>>(label, first, g->n);
  if (!g->symmetric) {
    k_cc_hook<<<g->num_sms * 4, kCcThreads, 0, s>>>(R, C, g->n, label, 0);
  } else {
    k_cc_sample<<<grid, 256, 0, s>>>(R, C, first, g->n, label);
    k_cc_jump<<<grid, 256, 0, s>>>(label, g->n, cnt + 1);  // compress (count unused)
    int32_t *skip = ws->skip.as<int32_t>();
    k_cc_pick<<<1, kCcPicks, 0, s>>>(label, g->n, skip);
    unsigned long long *packed = ws->counter.as<unsigned long long>() + 1;
    int32_t *Q = ws->q.as<int32_t>(), *S = ws->sc.as<int32_t>();
    k_cc_rest_frontier<<<grid, kCcThreads, 0, s>>>(R, label, g->n, skip, Q, S, packed);
    k_cc_hook_rest<<<g->num_sms * 4, kCcThreads, 0, s>>>(R, C, g->n, label, Q, S, packed);
  }
  k_cc_jump<<<grid, 256, 0, s>>>(label, g->n, cnt);
  GR_CUDA(cudaGetLastError());
  return GR_OK;
}

}  // namespace gr

using namespace gr;

extern "C" {

gr_status gr_cc(gr_graph *g, int32_t *label, int32_t *num_components, const gr_opts *opts,
                void *stream) {
  clear_error();
  (void)opts;
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!label) return fail(GR_EINVAL, "label must not be NULL");
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  if (!g->cc) GR_TRY(cc_ws_create(g, &g->cc));
  void *d_label;
  bool cp_label;
  GR_TRY(resolve_output(g, 0, label, sizeof(int32_t) * (size_t)g->n, &d_label, &cp_label));
  GR_TRY(cc_run(g, g->cc, (int32_t *)d_label, s));
  if (cp_label)
    GR_CUDA(cudaMemcpyAsync(label, d_label, sizeof(int32_t) * (size_t)g->n,
                            cudaMemcpyDeviceToHost, s));
  if (num_components) {
    int32_t h = 0;
    GR_CUDA(cudaMemcpyAsync(&h, g->cc->counter.p, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    GR_CUDA(cudaStreamSynchronize(s));
    *num_components = h;
  }
  GR_TRY(end_call(g, s));
  return GR_OK;
}

}  // extern "C"
