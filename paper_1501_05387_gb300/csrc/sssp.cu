// Single-source shortest paths with a near/far frontier split (Alg. 1,
// Sec. 4.5 "Priority queue", Sec. 5.2).
//
// Alg. 1 initialises labels to infinity and label[root] = 0, then loops
// advance (UpdateLabel = atomicMin relaxation), filter (RemoveRedundant, an
// output-queue stamp per vertex) and the priority-queue split until the
// frontier is empty. Here one iteration of the device-side loop is ONE
// kernel, k_sssp_iter, in one of three modes chosen on the device:
//
//   relax  load-balanced advance over the near frontier (merge-path chunks
//          over its vertex ends and edge ranks, Sec. 4.4); per edge
//          new = dist[u] + w(e), atomicMin on dist[v]; an improved v joins
//          the next near frontier if new < T (deduplicated by a
//          per-iteration stamp, the RemoveRedundant filter) and the far pile
//          otherwise (deduplicated by a per-phase stamp)
//   pull   the relaxation in pull form (direction-optimising SSSP, which
//          the paper names for future work in Sec. 4.5 and Sec. 7), for
//          near frontiers holding much of the edges on a symmetric graph:
//          every vertex takes the minimum of dist[u] + w(e) over its
//          in-edges (= its row; gather_reduce_tiles) and keeps it if lower,
//          so no atomic is needed except for rows split between tiles; a
//          sweep over the marks of the lowered vertices then sends them to
//          near / far as in relax
//   split  only when the near frontier is empty: the far pile is split by
//          the raised threshold into near and far; entries whose distance
//          fell below the old threshold were already expanded and are
//          dropped
//
// New near vertices are emitted with their degree scan (one packed atomic
// per block), so no scan pass separates two iterations. The last block of
// an iteration swaps the buffers, raises T (jumping to the bucket of the
// smallest far distance when the next bucket would be empty) and ends the
// loop when both piles are empty.
//
// T starts at delta and grows by delta per phase (delta = UINT32_MAX: one
// bucket, i.e. plain frontier relaxation); on graphs of small maximum degree
// the graph's own width is one for meshes' thin frontiers and one for others
// (sssp_delta, sssp_delta_thick). Distances do not depend on delta.
// An optional last pass fills pred[v] with the smallest u that has an edge
// (u, v) with dist[u] + w = dist[v].
//
// Batched form (gr_sssp_batch): k sources run as ONE search over k disjoint
// copies of the graph. Vertex id l*n + v stands for vertex v in copy
// (lane) l: its row is row v of the CSR, its neighbours are l*n + C[e], and
// dist / stamps / queues are indexed by the lane-major id. Copy l holds
// only source l, and no edge joins two copies, so each lane's distances are
// exactly those of a search from its own source; the lanes share the
// threshold T and the device-side loop, so k high-diameter searches cost
// about as many iterations as one.
#include <algorithm>
#include <climits>
#include <cstring>

#include "gather.cuh"

namespace gr {

// kSsspSweep: the second half of a pull, its lowered vertices to near / far
enum : int32_t { kSsspRelax = 0, kSsspSplit = 1, kSsspPull = 2, kSsspSweep = 3 };

struct SsspCtl {
  uint32_t *dist;
  int32_t *pred;
  int32_t src;
  int32_t mode;          // kSsspRelax / kSsspSplit / kSsspPull for the current iteration
  int32_t near_parity;   // which near buffer holds the current frontier
  int32_t far_parity;    // which far buffer holds the current pile
  int32_t near_len;
  int32_t far_len;        // atomic (relax appends to the current pile)
  int32_t far_next_len;   // atomic (split output)
  int32_t done;
  int32_t error;
  int32_t iter;           // iteration id, also the near-frontier stamp
  int32_t far_epoch;      // far-pile stamp
  int32_t max_iters;
  int32_t phases;         // number of splits
  int32_t pad_;
  uint32_t far_min;       // lower bound of far-pile distances (atomicMin)
  uint32_t far_min_next;  // min distance of entries kept by a split
  unsigned long long near_next_packed;  // [31:0] next near size, [63:32] its edges
  // iteration-kernel blocks finished so far in this run; the block whose
  // arrival makes it a multiple of the grid size ends the iteration
  unsigned long long arrivals;
  unsigned long long T;   // near criterion: dist < T
  unsigned long long T_old;
  unsigned long long delta;
  long long near_edges;   // edges of the current near frontier
  long long relaxations;  // edges expanded (statistics)
  // a relaxation whose near frontier has at least this many edges runs in
  // pull form (LLONG_MAX: never; pull needs a symmetric CSR and one lane)
  long long pull_min_edges;
  int32_t pulls;          // relaxations run in pull form (statistics)
  int32_t pad2_;
  // persistent kernel: bucket width while frontiers are thick (delta: thin)
  unsigned long long delta_thick;
  // persistent kernel: counter rings and grid barrier
  unsigned long long ring_near[3];
  int32_t ring_far[3];
  uint32_t ring_fmin[3];
  GridBarrier bar;
};

struct SsspArgs {
  const int32_t *R;
  const int32_t *C;
  const uint32_t *W;
  int32_t n;
  int32_t nv;  // vertex ids in use: lanes * n (lane-major copies of the graph)
  long long m;
  int32_t *nearq[2];
  int32_t *nearS[2];
  int32_t *farq[2];
  int32_t *stamp;
  int32_t *far_stamp;
  SsspCtl *ctl;
  int32_t low_degree;  // graph of small maximum degree: per-thread relaxation
  const int4 *adjw;    // four (neighbour, weight) pairs per vertex (low_adjacency)
  int32_t solo_handoff;  // frontier size up to which k_sssp_solo goes on
  GatherPlanArgs plan;  // row structure of the pull relaxation
  uint32_t *lowered;    // marks of the vertices a pull lowered (zero between pulls)
  int32_t *qcb;        // room for the chunk bounds of a dense near frontier (or null)
};

constexpr int kSsspThreads = 256, kSsspItems = 4;
constexpr int kSsspBlocksPerSm = 5;
// Items per thread of the persistent kernel that may pull: its pushes have
// the smaller frontiers, and half the shared memory leaves the pull's random
// distance loads the L1.
constexpr int kSsspPullItems = 2;
// On graphs of at most kLowDegreeMax relaxation takes one frontier vertex
// per thread; the neighbours a thread loads at once.
constexpr int kSsspTpvItems = 4;
// A persistent relaxation first finds every chunk's bounds in one pass once
// its frontier has at least this many chunks per block.
constexpr int kSsspBoundsChunksPerBlock = 4;
// Most sources one batched run takes.
constexpr int32_t kSsspMaxLanes = 64;
// k_sssp_solo: threads of the block that runs a search, frontier vertices it
// keeps in shared memory per parity, and the frontier's edges from which the
// search goes on as k_sssp_do. A block expands a vertex of four edges in 5 ns,
// so 4096 take it twice as long as a grid barrier and their expansion on all
// SMs (9 us); but the grid keeps the search once it has it, and meshes pass 2560
// for a few iterations only (700 x 700, 12 mean weights: 7.6 ms handed over
// there).
constexpr int kSoloThreads = 1024;
constexpr int32_t kSoloQueue = 4096;
constexpr int32_t kSoloHandoffEdges = 16384;
// k_sssp_do: the share of the expanded vertices below which the far pile is that
// of a mesh (bucket width).
constexpr int32_t kSsspFarShare = 2;

struct SsspWorkspace {
  int32_t lanes = 1;  // copies of the graph the buffers hold (batched form)
  DevMem nearq[2], nearS[2], farq[2], stamp, far_stamp, ctl;
  GatherPlan plan;  // of the pull relaxation (single search on a symmetric graph)
  DevMem lowered;
  DevMem qcb;  // chunk bounds of a dense near frontier (persistent driver)
  cudaGraphExec_t exec = nullptr;
  cudaGraph_t graph = nullptr;
  ~SsspWorkspace() {
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
  }
};

void free_sssp(SsspWorkspace *ws) { delete ws; }

GR_GUARD_REPORTER(guard_report_sssp)

namespace {

__device__ __forceinline__ int32_t *pick(int32_t *const *a, int p) { return p ? a[1] : a[0]; }

// First id of the graph copy that lane-major id x lies in (0 for one lane).
__device__ __forceinline__ int32_t lane_base(int32_t x, int32_t n) {
  return x >= n ? x - x % n : 0;
}

// Sources of one run: lane l starts at vertex s[l] (id l*n + s[l]).
struct SsspSources {
  int32_t k;
  int32_t s[kSsspMaxLanes];
};

// solo: k_sssp_solo runs the searches from their sources; the control block
// then starts out as what its lanes hand over: nothing. The grid's first bucket
// is of the thick width.
__global__ void k_sssp_init(SsspArgs a, SsspSources src, uint32_t *dist, int32_t *pred,
                            unsigned long long delta, unsigned long long delta_thick,
                            int32_t max_iters, long long pull_min_edges, int32_t solo) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = tid; v < a.nv; v += stride) {
    const int32_t x = (int32_t)v;
    const int32_t base = lane_base(x, a.n);
    dist[v] = x - base == src.s[base ? base / a.n : 0] ? 0u : 0xFFFFFFFFu;
    a.stamp[v] = -1;
    a.far_stamp[v] = -1;
  }
  if (a.lowered)
    for (int64_t w = tid; w < (a.n + 31) / 32; w += stride) a.lowered[w] = 0u;
  if (tid == 0) {
    SsspCtl *c = a.ctl;
    // the initial near frontier: every lane's source with its degree scan
    int32_t edges = 0;
    for (int32_t l = 0; l < src.k; ++l) {
      const int32_t u = src.s[l];
      a.nearq[0][l] = l * a.n + u;
      a.nearS[0][l] = edges;
      edges += a.R[u + 1] - a.R[u];
    }
    a.nearS[0][src.k] = edges;
    c->dist = dist;
    c->pred = pred;
    c->src = src.s[0];
    c->mode = kSsspRelax;
    c->near_parity = 0;
    c->far_parity = 0;
    c->near_len = solo ? 0 : src.k;
    c->far_len = 0;
    c->far_next_len = 0;
    c->done = 0;
    c->error = kDevOk;
    c->iter = 0;
    c->far_epoch = 0;
    c->max_iters = max_iters;
    c->phases = 0;
    c->arrivals = 0ull;
    c->far_min = 0xFFFFFFFFu;
    c->far_min_next = 0xFFFFFFFFu;
    c->near_next_packed = 0ull;
    c->delta = delta;
    c->delta_thick = delta_thick;
    c->T = delta_thick;
    c->T_old = 0;
    c->near_edges = solo ? 0 : edges;
    c->relaxations = 0;
    c->pull_min_edges = pull_min_edges;
    c->pulls = 0;
    for (int i = 0; i < 3; ++i) {
      c->ring_near[i] = 0ull;
      c->ring_far[i] = 0;
      c->ring_fmin[i] = 0xFFFFFFFFu;
    }
    grid_barrier_reset(&c->bar);
  }
}

template <int ITEMS>
struct SsspSmem {
  static constexpr int kChunk = kSsspThreads * ITEMS;
  int32_t off[kChunk + 1];
  uint32_t du[kChunk + 1];
  int32_t row[kChunk + 1];
  int32_t base[kChunk + 1];  // first id of the vertex's graph copy
  ScannedBuf<kChunk> nearb;
  AppendBuf<kChunk> farb;
  int32_t i[2];
  int32_t sred[kSsspThreads / 32];
  int32_t last;
};

// The state one iteration reads and the counters it fills; the graph-mode
// kernel takes them from the control block, the persistent kernel from
// block-private copies and a ring of counters.
struct SsspStep {
  int32_t near_parity, far_parity;
  int32_t q;              // near frontier size
  int32_t q_edges;        // its edges (S[q])
  int32_t far_len;        // current far pile size (split input)
  unsigned long long T, T_old;
  int32_t iter, far_epoch;
  unsigned long long *near_ctr;  // packed (vertices, edges) of the next near frontier
  int32_t *far_ctr;              // far appends (relax) or far-next size (split)
  int32_t *far_dest;             // where far appends land (pile start + base)
  long long far_cap;             // entries available at far_dest
  uint32_t *fmin;                // min distance sent to the far pile
};

// The merge-path chunk bounds of a near frontier (q members, exclusive
// degree scan S[0..q), s_q entries in all: S[q] itself is not stored),
// grid-stride: cb[c] = the members whose end marker S[i + 1] + i lies before
// c * CHUNK, cb[nchunks] = q.
template <int CHUNK>
__device__ void frontier_chunk_bounds(const int32_t *S, int32_t q, int32_t s_q,
                                      long long nchunks, int32_t *cb) {
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c <= nchunks;
       c += (long long)gridDim.x * blockDim.x) {
    if (c == nchunks) {
      cb[c] = q;
      continue;
    }
    const long long d = c * CHUNK;
    int32_t lo = 0, hi = q;  // first member whose end marker is not before d
    while (lo < hi) {
      const int32_t mid = (int32_t)(((long long)lo + hi) >> 1);
      const int32_t sv = mid + 1 == q ? s_q : S[mid + 1];
      if ((long long)sv + mid < d) lo = mid + 1;
      else hi = mid;
    }
    cb[c] = lo;
  }
}

// qcb (may be null): the frontier's chunk bounds, computed for this
// iteration by frontier_chunk_bounds, so a chunk needs no search.
template <int ITEMS>
__device__ void relax_body(const SsspArgs &a, uint32_t *dist, SsspSmem<ITEMS> &sm,
                           const SsspStep &st, const int32_t *qcb = nullptr) {
  constexpr int CHUNK = kSsspThreads * ITEMS;
  const int32_t np = st.near_parity;
  const int32_t *Q = pick(a.nearq, np);
  const int32_t *S = pick(a.nearS, np);
  int32_t *Qn = pick(a.nearq, np ^ 1);
  int32_t *Sn = pick(a.nearS, np ^ 1);
  const int32_t q = st.q;
  const unsigned long long T = st.T;
  const int32_t iter = st.iter, epoch = st.far_epoch;
  uint32_t local_min = 0xFFFFFFFFu;
  const long long total = (long long)q + st.q_edges;
  const long long nchunks = (total + CHUNK - 1) / CHUNK;
  for (long long chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    const long long d0 = chunk * CHUNK;
    const long long d1 = min(d0 + CHUNK, total);
    int32_t i0, i1;
    if (qcb) {
      i0 = qcb[chunk];
      i1 = qcb[chunk + 1];
    } else {
      block_chunk_bounds<kSsspThreads>(S, q, st.q_edges, d0, d1, CHUNK, sm.sred, &i0, &i1);
    }
    const long long j0 = d0 - i0, j1 = d1 - i1;
    const int32_t nv = (i0 <= q - 1) ? (min(i1, q - 1) - i0 + 1) : 0;
    // per chunk vertex: its scan offset, its row start and its distance (read
    // once here instead of once per edge)
    for (int32_t k = threadIdx.x; k < nv; k += kSsspThreads) {
      const int32_t i = i0 + k;
      const int32_t u0 = GR_IN(i, a.nv + 1, 301) ? Q[i] : 0;
      const int32_t u = GR_IN(u0, a.nv, 303) ? u0 : 0;
      const int32_t ub = lane_base(u, a.n);
      sm.off[k] = GR_IN(i, a.nv + 2, 302) ? S[i] : 0;
      sm.row[k] = a.R[u - ub];
      sm.base[k] = ub;
      sm.du[k] = dist[u];
    }
    __syncthreads();
    // each thread takes ITEMS edges (ranks tid, tid + T, ...) and issues
    // each step's loads (heads and weights, head distances, atomicMin, stamps,
    // degrees) for all of them before using any, so the latency chains of the
    // items overlap
    const int32_t ne = (int32_t)(j1 - j0);  // <= CHUNK: one pass
    int32_t e[ITEMS], v[ITEMS], vl[ITEMS], vb[ITEMS], code[ITEMS],
        dv[ITEMS];
    uint32_t wt[ITEMS], du[ITEMS], nd[ITEMS], cur[ITEMS];
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int32_t k = j * kSsspThreads + threadIdx.x;
      e[j] = -1;
      vb[j] = 0;
      du[j] = 0xFFFFFFFFu;
      if (k < ne) {
        const int32_t er = (int32_t)(j0 + k);
        int32_t lo = 0, hi = nv - 1;
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (sm.off[mid] <= er) lo = mid;
          else hi = mid - 1;
        }
        const int32_t ee = sm.row[lo] + (er - sm.off[lo]);
        if (GR_IN(ee, a.m, 304)) {
          e[j] = ee;
          vb[j] = sm.base[lo];
          du[j] = sm.du[lo];
        }
      }
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      vl[j] = e[j] >= 0 ? a.C[e[j]] : -1;
      wt[j] = e[j] >= 0 ? a.W[e[j]] : 0u;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      nd[j] = 0xFFFFFFFFu;  // not representable below 0xFFFFFFFF: no improvement
      if (vl[j] >= 0 && !GR_IN(vl[j], a.n, 305)) vl[j] = -1;
      v[j] = vl[j] >= 0 ? vb[j] + vl[j] : -1;  // the neighbour in the same copy
      if (v[j] >= 0) {
        const unsigned long long t = (unsigned long long)du[j] + wt[j];
        if (t < 0xFFFFFFFFull) nd[j] = (uint32_t)t;
      }
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      cur[j] = nd[j] != 0xFFFFFFFFu ? dist[v[j]] : 0u;  // plain-load cull
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const bool try_it = nd[j] < cur[j];
      cur[j] = try_it ? atomicMin(dist + v[j], nd[j]) : 0u;
      if (!try_it) nd[j] = 0xFFFFFFFFu;
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      code[j] = 0;
      if (nd[j] < cur[j]) {  // this thread lowered dist[v]
        if (nd[j] < T) {
          code[j] = atomicExch(a.stamp + v[j], iter) != iter ? 1 : 0;
        } else {
          local_min = min(local_min, nd[j]);
          code[j] = atomicExch(a.far_stamp + v[j], epoch) != epoch ? 2 : 0;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j)
      dv[j] = code[j] == 1 ? a.R[vl[j] + 1] - a.R[vl[j]] : 0;
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      emit_scanned(sm.nearb, code[j] == 1, v[j], dv[j]);
      emit_plain(sm.farb, code[j] == 2, v[j]);
    }
    flush_scanned<kSsspThreads>(sm.nearb, st.near_ctr, Qn, Sn, a.nv + 1);
    flush_plain<kSsspThreads>(sm.farb, st.far_ctr, st.far_dest, st.far_cap);
  }
  if (blockIdx.x < nchunks) {
    // one atomic per warp: one per far edge kept the one address busy for
    // 0.9 of 2.5 ms (R-MAT 2^21, one mean weight a bucket)
    local_min = __reduce_min_sync(0xffffffffu, local_min);
    if ((threadIdx.x & 31) == 0 && local_min != 0xFFFFFFFFu) atomicMin(st.fmin, local_min);
  }
}

// Relaxation for graphs of small maximum degree (meshes): one thread per
// near-frontier vertex relaxes its whole neighbour list (the per-thread
// expansion of Sec. 4.4, balanced when every degree is small), so no
// merge-path search is needed. Each candidate's row offsets are loaded with
// its distance, so a vertex entering the near frontier brings its degree (for
// the frontier's edge count) without an extra round trip. Near and far
// entries are appended with one atomic per warp each.
__device__ void relax_body_thread(const SsspArgs &a, uint32_t *dist, const SsspStep &st) {
  const int32_t *Q = pick(a.nearq, st.near_parity);
  int32_t *Qn = pick(a.nearq, st.near_parity ^ 1);
  const int32_t q = st.q;
  const unsigned long long T = st.T;
  const int32_t iter = st.iter, epoch = st.far_epoch;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t qr = ((int64_t)q + 31) & ~31ll;  // warp-uniform bound
  uint32_t local_min = 0xFFFFFFFFu;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < qr; i += stride) {
    int32_t u = 0, ub = 0, r0 = 0, r1 = 0;
    uint32_t du = 0xFFFFFFFFu;
    if (i < q && GR_IN(i, a.nv + 1, 320)) {
      u = Q[i];
      if (GR_IN(u, a.nv, 321)) {
        ub = lane_base(u, a.n);
        r0 = a.R[u - ub];
        r1 = a.R[u - ub + 1];
        du = dist[u];
      }
    }
    for (int32_t e0 = r0; __any_sync(0xffffffffu, e0 < r1); e0 += kSsspTpvItems) {
      int32_t v[kSsspTpvItems], d0[kSsspTpvItems], d1[kSsspTpvItems];
      uint32_t w[kSsspTpvItems], dv[kSsspTpvItems];
      int code[kSsspTpvItems];
#pragma unroll
      for (int j = 0; j < kSsspTpvItems; ++j) {
        const int32_t e = e0 + j;
        v[j] = -1;
        w[j] = 0u;
        if (e < r1 && GR_IN(e, a.m, 322)) {
          v[j] = a.C[e];
          w[j] = a.W[e];
          if (!GR_IN(v[j], a.n, 323)) v[j] = -1;
        }
      }
#pragma unroll
      for (int j = 0; j < kSsspTpvItems; ++j) {
        dv[j] = 0u;
        d0[j] = d1[j] = 0;
        if (v[j] >= 0) {
          d0[j] = a.R[v[j]];
          d1[j] = a.R[v[j] + 1];
          v[j] += ub;  // from here on: the neighbour's id in u's copy
          dv[j] = dist[v[j]];
        }
      }
      uint32_t ncnt = 0, ndeg = 0, fcnt = 0;
#pragma unroll
      for (int j = 0; j < kSsspTpvItems; ++j) {
        code[j] = 0;
        if (v[j] < 0) continue;
        const unsigned long long nd = (unsigned long long)du + w[j];
        if (nd >= 0xFFFFFFFFull) continue;  // not representable: no improvement
        const uint32_t nd32 = (uint32_t)nd;
        if (nd32 >= dv[j]) continue;  // plain-load cull
        const uint32_t old = atomicMin(dist + v[j], nd32);
        if (nd32 >= old) continue;
        if (nd < T) {
          if (atomicExch(a.stamp + v[j], iter) != iter) {
            code[j] = 1;
            ncnt += 1;
            ndeg += (uint32_t)(d1[j] - d0[j]);
          }
        } else {
          local_min = min(local_min, nd32);
          if (atomicExch(a.far_stamp + v[j], epoch) != epoch) {
            code[j] = 2;
            fcnt += 1;
          }
        }
      }
      // near: warp scan of (edges, vertices), one packed atomic
      const unsigned long long nmine = ((unsigned long long)ndeg << 32) | ncnt;
      unsigned long long nincl = nmine;
      uint32_t fincl = fcnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, nincl, o);
        const uint32_t tf = __shfl_up_sync(0xffffffffu, fincl, o);
        if (lane >= o) {
          nincl += t;
          fincl += tf;
        }
      }
      const unsigned long long ntot = __shfl_sync(0xffffffffu, nincl, 31);
      const uint32_t ftot = __shfl_sync(0xffffffffu, fincl, 31);
      unsigned long long nbase = 0;
      int32_t fbase = 0;
      if (lane == 0) {
        if (ntot) nbase = atomicAdd(st.near_ctr, ntot);
        if (ftot) fbase = atomicAdd(st.far_ctr, (int32_t)ftot);
      }
      nbase = __shfl_sync(0xffffffffu, nbase, 0);
      fbase = __shfl_sync(0xffffffffu, fbase, 0);
      int32_t kn = (int32_t)((nbase + (nincl - nmine)) & 0xFFFFFFFFull);
      long long kf = (long long)fbase + (fincl - fcnt);
#pragma unroll
      for (int j = 0; j < kSsspTpvItems; ++j) {
        if (code[j] == 1) {
          if (GR_IN(kn, a.nv + 1, 324)) Qn[kn] = v[j];
          ++kn;
        } else if (code[j] == 2) {
          if (GR_IN(kf, st.far_cap, 325)) st.far_dest[kf] = v[j];
          ++kf;
        }
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) local_min = min(local_min, __shfl_xor_sync(0xffffffffu, local_min, o));
  if (lane == 0 && local_min != 0xFFFFFFFFu) atomicMin(st.fmin, local_min);
}

// Pull form of one relaxation: for every vertex v (one graph copy), the
// smallest dist[u] + w(e) over the entries e = (v, u) of its row, which on a
// symmetric CSR are its in-edges, replaces dist[v] if smaller, and v is
// marked. Distances change under the readers' hands, downwards only: a
// reader may miss a lowering, but the vertex lowered is marked and goes on
// the next frontier. R-MAT 2^21, 63.5 M entries: 205 us with the sweep, where
// a push of that frontier takes 750.
struct PullValue {
  static constexpr bool kWeighted = true;
  const uint32_t *dist;
  __device__ __forceinline__ uint32_t operator()(int32_t u, int32_t w) const {
    const uint32_t d = dist[u], t = d + (uint32_t)w;
    return t < d ? 0xFFFFFFFFu : t;  // sums past the range: unreachable
  }
};
struct ReduceMinU32 {
  static __device__ __forceinline__ uint32_t identity() { return 0xFFFFFFFFu; }
  static __device__ __forceinline__ uint32_t op(uint32_t a, uint32_t b) { return min(a, b); }
};
struct LowerDist {
  uint32_t *dist;
  uint32_t *lowered;
  __device__ __forceinline__ void operator()(int32_t v, uint32_t nd, bool whole) const {
    if (nd >= dist[v]) return;
    if (whole) dist[v] = nd;  // nobody else writes it in this pull
    else if (nd >= atomicMin(dist + v, nd)) return;
    atomicOr(lowered + (v >> 5), 1u << (v & 31));
  }
};

__device__ __forceinline__ void pull_body(const SsspArgs &a, uint32_t *dist) {
  gather_reduce_tiles<1, uint32_t, ReduceMinU32>(
      a.plan, a.C, (const int32_t *)a.W, 0, (int32_t)a.m, PullValue{dist},
      LowerDist{dist, a.lowered}, spread_warp(), grid_warps());
}

// The marked vertices to near (below T) or far, the marks cleared.
template <int ITEMS>
__device__ void sweep_body(const SsspArgs &a, const uint32_t *dist, SsspSmem<ITEMS> &sm,
                           const SsspStep &st) {
  constexpr int CHUNK = kSsspThreads * ITEMS;
  int32_t *Qn = pick(a.nearq, st.near_parity ^ 1);
  int32_t *Sn = pick(a.nearS, st.near_parity ^ 1);
  uint32_t local_min = 0xFFFFFFFFu;
  for (int64_t b = (int64_t)blockIdx.x * CHUNK; b < a.n; b += (int64_t)gridDim.x * CHUNK) {
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const int64_t v0 = b + j * kSsspThreads + threadIdx.x;  // a warp has one word of marks
      const uint32_t word = v0 < a.n ? a.lowered[v0 >> 5] : 0u;
      int code = 0;
      int32_t d = 0;
      if ((word >> (v0 & 31)) & 1u) {
        const uint32_t nd = dist[v0];
        if (nd < st.T) {
          code = 1;
          d = a.R[v0 + 1] - a.R[v0];
        } else {
          local_min = min(local_min, nd);
          code = atomicExch(a.far_stamp + v0, st.far_epoch) != st.far_epoch ? 2 : 0;
        }
      }
      __syncwarp();
      if ((threadIdx.x & 31) == 0 && word) a.lowered[v0 >> 5] = 0u;
      emit_scanned(sm.nearb, code == 1, (int32_t)v0, d);
      emit_plain(sm.farb, code == 2, (int32_t)v0);
    }
    flush_scanned<kSsspThreads>(sm.nearb, st.near_ctr, Qn, Sn, a.nv + 1);
    flush_plain<kSsspThreads>(sm.farb, st.far_ctr, st.far_dest, st.far_cap);
  }
  for (int o = 16; o > 0; o >>= 1) local_min = min(local_min, __shfl_xor_sync(0xffffffffu, local_min, o));
  if ((threadIdx.x & 31) == 0 && local_min != 0xFFFFFFFFu) atomicMin(st.fmin, local_min);
}

template <int ITEMS>
__device__ void split_body(const SsspArgs &a, const uint32_t *dist, SsspSmem<ITEMS> &sm,
                           const SsspStep &st) {
  const int32_t *F = pick(a.farq, st.far_parity);
  const int32_t np = st.near_parity;
  int32_t *Qn = pick(a.nearq, np ^ 1);
  int32_t *Sn = pick(a.nearS, np ^ 1);
  const int32_t len = st.far_len;
  const unsigned long long T = st.T, T_old = st.T_old;
  const int32_t iter = st.iter, epoch = st.far_epoch + 1;
  uint32_t local_min = 0xFFFFFFFFu;
  const long long per_round = (long long)gridDim.x * kSsspThreads;
  const long long rounds = (len + per_round - 1) / per_round;
  for (long long r = 0; r < rounds; ++r) {
    const long long i = (r * gridDim.x + blockIdx.x) * kSsspThreads + threadIdx.x;
    int code = 0;
    int32_t v = 0, dv = 0;
    if (i < len && GR_IN(i, a.nv + 1, 310) && GR_IN(F[i], a.nv, 311)) {
      v = F[i];
      const uint32_t d = dist[v];
      if ((unsigned long long)d < T_old) {
        code = 0;  // stale: improved below the old threshold and expanded
      } else if ((unsigned long long)d < T) {
        if (atomicExch(a.stamp + v, iter) != iter) {
          code = 1;
          const int32_t vl = v - lane_base(v, a.n);
          dv = a.R[vl + 1] - a.R[vl];
        }
      } else {
        local_min = min(local_min, d);
        code = atomicExch(a.far_stamp + v, epoch) != epoch ? 2 : 0;
      }
    }
    emit_scanned(sm.nearb, code == 1, v, dv);
    emit_plain(sm.farb, code == 2, v);
    if ((r + 1) % ITEMS == 0 || r == rounds - 1) {
      flush_scanned<kSsspThreads>(sm.nearb, st.near_ctr, Qn, Sn, a.nv + 1);
      flush_plain<kSsspThreads>(sm.farb, st.far_ctr, st.far_dest, st.far_cap);
    }
  }
  for (int o = 16; o > 0; o >>= 1) local_min = min(local_min, __shfl_xor_sync(0xffffffffu, local_min, o));
  if ((threadIdx.x & 31) == 0 && local_min != 0xFFFFFFFFu) atomicMin(st.fmin, local_min);
}

template <bool LOW>
__device__ void relax_mode(const SsspArgs &a, SsspCtl *c, SsspSmem<kSsspItems> &sm) {
  SsspStep st;
  st.near_parity = c->near_parity;
  st.far_parity = c->far_parity;
  st.q = c->near_len;
  st.q_edges = (int32_t)c->near_edges;
  st.far_len = c->far_len;
  st.T = c->T;
  st.T_old = c->T_old;
  st.iter = c->iter;
  st.far_epoch = c->far_epoch;
  st.near_ctr = &c->near_next_packed;
  st.far_ctr = &c->far_len;  // absolute positions in the current pile
  st.far_dest = pick(a.farq, c->far_parity);
  st.far_cap = (long long)a.nv + 1;
  st.fmin = &c->far_min;
  if (LOW) relax_body_thread(a, c->dist, st);
  else if (c->mode == kSsspPull) pull_body(a, c->dist);
  else if (c->mode == kSsspSweep) sweep_body(a, c->dist, sm, st);
  else relax_body(a, c->dist, sm, st);
}

__device__ void split_mode(const SsspArgs &a, SsspCtl *c, SsspSmem<kSsspItems> &sm) {
  SsspStep st;
  st.near_parity = c->near_parity;
  st.far_parity = c->far_parity;
  st.q = c->near_len;
  st.q_edges = (int32_t)c->near_edges;
  st.far_len = c->far_len;
  st.T = c->T;
  st.T_old = c->T_old;
  st.iter = c->iter;
  st.far_epoch = c->far_epoch;
  st.near_ctr = &c->near_next_packed;
  st.far_ctr = &c->far_next_len;
  st.far_dest = pick(a.farq, c->far_parity ^ 1);
  st.far_cap = (long long)a.nv + 1;
  st.fmin = &c->far_min_next;
  split_body(a, c->dist, sm, st);
}

__device__ __forceinline__ unsigned long long bucket_end(uint32_t d, unsigned long long delta) {
  return ((unsigned long long)d / delta + 1ull) * delta;
}

// Run by the last block of an iteration.
__device__ void sssp_end(const SsspArgs &a, SsspCtl *c) {
  if (c->error) {
    c->done = 1;
    return;
  }
  if (c->mode == kSsspPull) {  // its sweep is the rest of this iteration
    c->mode = kSsspSweep;
    return;
  }
  // counters the other blocks filled with atomics: read past L1
  const unsigned long long packed = *(volatile unsigned long long *)&c->near_next_packed;
  const int32_t qn = (int32_t)(packed & 0xFFFFFFFFull);
  const long long en = (long long)(packed >> 32);
  if (c->mode != kSsspSplit) {
    c->relaxations += c->mode == kSsspSweep ? a.m : c->near_edges;
    c->pulls += c->mode == kSsspSweep;
    c->far_len = *(volatile int32_t *)&c->far_len;
    c->far_min = *(volatile uint32_t *)&c->far_min;
  } else {
    c->far_len = *(volatile int32_t *)&c->far_next_len;
    c->far_parity ^= 1;
    c->far_epoch += 1;
    c->far_min = *(volatile uint32_t *)&c->far_min_next;
    c->phases += 1;
  }
  c->near_len = qn;
  c->near_edges = en;
  c->near_parity ^= 1;
  pick(a.nearS, c->near_parity)[qn] = (int32_t)en;
  c->near_next_packed = 0ull;
  c->far_next_len = 0;
  c->far_min_next = 0xFFFFFFFFu;
  c->iter += 1;
  if (c->near_len > 0) {
    c->mode = c->near_edges >= c->pull_min_edges ? kSsspPull : kSsspRelax;
  } else if (c->far_len > 0) {
    c->mode = kSsspSplit;
    c->T_old = c->T;
    const unsigned long long t = c->T + c->delta;
    const unsigned long long j = bucket_end(c->far_min, c->delta);
    c->T = t > j ? t : j;
  } else {
    c->done = 1;
    return;
  }
  if (c->iter >= c->max_iters) {
    c->error = kDevOverflow;
    c->done = 1;
  }
}

// LOW: per-thread relaxation (graphs of small maximum degree)
template <bool LOW>
__global__ void __launch_bounds__(kSsspThreads, kSsspBlocksPerSm)
    k_sssp_iter(SsspArgs a, cudaGraphConditionalHandle h, int32_t use_cond) {
  SsspCtl *c = a.ctl;
  if (*(volatile int32_t *)&c->done) {
    // an iteration kernel after the run ended (host-driven batches enqueue a
    // few extra): every block leaves; inside a graph the loop condition is
    // cleared here too, so the while loop cannot outlive the run
    if (use_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(h, 0u);
    return;
  }
  __shared__ SsspSmem<kSsspItems> sm;
  if (threadIdx.x == 0) {
    sm.nearb.cnt = 0;
    sm.farb.cnt = 0;
  }
  __syncthreads();
  if (c->mode != kSsspSplit) relax_mode<LOW>(a, c, sm);
  else split_mode(a, c, sm);
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned long long old = atomicAdd(&c->arrivals, 1ull);
    sm.last = (old + 1ull) % gridDim.x == 0ull;
  }
  __syncthreads();
  if (sm.last && threadIdx.x == 0) {
    __threadfence();
    sssp_end(a, c);
    if (use_cond) cudaGraphSetConditional(h, c->done ? 0u : 1u);
  }
}

// ------------------------------------------------------- one block per search
// On a mesh a search is a thousand iterations of a few hundred vertices, and
// each iteration of the grid kernel costs two microseconds of barrier and a
// chain of L2 round trips from queue to queue (9 us in all). Here one block
// runs a search by itself, so a batch runs its searches side by side on SMs of
// their own: iterations are separated by one __syncthreads, the frontier and
// the near and far membership bits live in shared memory, a vertex's row is
// one 32-byte sector of low_adjacency read by four threads, an edge each, and
// the L2 chain left is row and distance, then atomicMin. 511 x 511 grid,
// weights to 16, two mean weights a bucket: 8.8 us an iteration on the grid,
// 2.5 with a thread per vertex (its four bit tests one after another) and a
// pass of its own to take the frontier off the bits, 2.1 so. What is left is
// that chain (1.4 us) and, above some 300 vertices, one L2 access a clock.
//
// A vertex leaves the frontier's membership bits when its first thread takes
// it up; that thread's read of the distance waits for the cleared word, as
// the bit test of a thread that lowers the distance waits for what its
// atomicMin returns. So whoever lowers the distance and still finds the bit
// did so before that read, everybody else finds it clear and puts the vertex
// on the next frontier, and no barrier stands between the two.
//
// A lane whose frontier outgrows kSoloHandoffEdges edges (at the graph's largest
// degree) writes it and what is left of its far pile to the grid's far pile and
// stops; k_sssp_do, next on the stream, goes on with all lanes handed over, by
// a split in its own bucket width: a graph on which the frontier grows so fast
// is no mesh, and a bucket as wide as a mesh's would hold most of it (random
// graphs of degree 8 and 16, 500,000 vertices: 0.77 and 1.61 ms in six mean
// weights from the first bucket on, 0.69 and 0.94 on the grid alone in two).
// Per lane, the ids [lane * n, (lane + 1) * n) of nearq[1] hold what the
// shared-memory queue cannot, and those of nearS[0] and nearS[1] the far pile
// by parity (both are free: per-thread relaxations use no degree scan).
struct SoloState {
  int32_t near[3];   // frontier sizes, ring by iteration
  int32_t far[2];    // far pile sizes by parity
  uint32_t far_min;  // lower bound of the far pile's distances
  int32_t near_at;   // hand-over position
  unsigned long long relaxed;
};

// Appends a warp's entries (code 1: near, 2: far), one shared-memory atomic
// per queue.
__device__ __forceinline__ void solo_append(int32_t v, int code, int32_t *near_cnt,
                                            int32_t *far_cnt, int32_t *near_s, int32_t *near_g,
                                            int32_t *far) {
  const uint32_t nb = __ballot_sync(0xffffffffu, code == 1);
  const uint32_t fb = __ballot_sync(0xffffffffu, code == 2);
  if (!(nb | fb)) return;
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  int32_t at = 0;
  if (lane == 0 && nb) at = atomicAdd(near_cnt, __popc(nb));
  if (lane == 1 && fb) at = atomicAdd(far_cnt, __popc(fb));
  const int32_t kn = __shfl_sync(0xffffffffu, at, 0) + __popc(nb & lt);
  const int32_t kf = __shfl_sync(0xffffffffu, at, 1) + __popc(fb & lt);
  if (code == 1) {
    if (kn < kSoloQueue) near_s[kn] = v;
    else near_g[kn] = v;
  } else if (code == 2) {
    far[kf] = v;
  }
}

// LONG: the graph has rows of more than four entries; FAR_BITS: the far pile's
// membership bits fit shared memory (else far_stamp holds them). The code for
// the other cases costs instruction fetches on every iteration.
template <bool LONG, bool FAR_BITS>
__global__ void __launch_bounds__(kSoloThreads, 1) k_sssp_solo(SsspArgs a, SsspSources src) {
  extern __shared__ uint32_t solo_smem[];
  __shared__ SoloState st;
  SsspCtl *c = a.ctl;
  const int32_t nwords = (a.n + 31) >> 5;
  int32_t *const q0 = (int32_t *)solo_smem, *const q1 = q0 + kSoloQueue;
  uint32_t *nbits = solo_smem + 2 * kSoloQueue;  // on the frontier or the next one
  uint32_t *fbits = nbits + nwords;              // in the far pile (FAR_BITS)
  const int32_t base = (int32_t)blockIdx.x * a.n;
  uint32_t *dist = c->dist + base;
  int32_t *near_g = a.nearq[1] + base;
  int32_t *far_stamp = a.far_stamp + base;  // -1: not in the far pile (without FAR_BITS)
  int32_t *far0 = a.nearS[0] + base, *far1 = a.nearS[1] + base;
  const unsigned long long delta = c->delta, delta_thick = c->delta_thick;
  const int32_t handoff_at = LONG ? a.solo_handoff : kSoloQueue;
  const int32_t max_iters = c->max_iters;
  const int lane = threadIdx.x & 31;
  const int32_t s0 = src.s[blockIdx.x];
  for (int32_t w = threadIdx.x; w < nwords * (FAR_BITS ? 2 : 1); w += kSoloThreads)
    nbits[w] = w == (s0 >> 5) ? 1u << (s0 & 31) : 0u;
  if (threadIdx.x == 0) {
    q0[0] = s0;
    st.near[0] = 1;
    st.near[1] = 0;
    st.far[0] = st.far[1] = 0;
    st.far_min = 0xFFFFFFFFu;
    st.relaxed = 0ull;
  }
  unsigned long long T = LONG ? delta_thick : delta;
  int64_t expanded = 0;  // LONG: vertices so far
  int32_t fp = 0, iter = 0, ring = 0, phases = 0;
  uint32_t relaxed = 0u;
  __syncthreads();
  for (;;) {
    const int32_t next = ring == 2 ? 0 : ring + 1, after = next == 2 ? 0 : next + 1;
    const int32_t q = st.near[ring], len = st.far[fp];
    const bool split = q == 0;
    if ((split && len == 0) || q > handoff_at || iter >= max_iters) break;
    if (threadIdx.x == 0) st.near[after] = 0;  // last read an iteration ago
    const int32_t *Q = iter & 1 ? q1 : q0;
    int32_t *Qn = iter & 1 ? q0 : q1;
    int32_t *far = fp ? far1 : far0;
    uint32_t local_min = 0xFFFFFFFFu;
    if (LONG) expanded += q;
    if (!split) {
      // nd < T, for distances below 0xFFFFFFFF
      const uint32_t T32 = (uint32_t)min(T, 0xFFFFFFFFull);
      for (int32_t i = threadIdx.x; i - lane < 4 * q; i += kSoloThreads) {  // warp-uniform
        int2 vw = make_int2(-1, 0);
        uint32_t du = 0xFFFFFFFFu;
        if (i < 4 * q) {
          const int32_t u = Q[i >> 2];
          vw = __ldg((const int2 *)a.adjw + 4 * (int64_t)u + (lane & 3));
          if ((lane & 3) == 0) {
            // u's bit is set: the address below is u's, once the bit is clear
            const uint32_t old = atomicAnd(&nbits[u >> 5], ~(1u << (u & 31)));
            const int32_t u_then = u - 1 + (int32_t)((old >> (u & 31)) & 1u);
            if (GR_IN(u_then, a.n, 341)) du = __ldcg(dist + u_then);  // atomics lower it: not from L1
          }
        }
        du = __shfl_sync(0xffffffffu, du, lane & ~3);
        int32_t e = 0, e1 = 0;  // a row longer than four: its quad walks it
        if (LONG && __any_sync(0xffffffffu, vw.x == -2)) {
          const int32_t tag = __shfl_sync(0xffffffffu, vw.x, lane & ~3);
          const int32_t r0 = __shfl_sync(0xffffffffu, vw.y, lane & ~3);
          const int32_t r1 = __shfl_sync(0xffffffffu, vw.x, (lane & ~3) + 1);
          if (tag == -2) {
            e = r0 + (lane & 3);
            e1 = r1;
            vw = e < e1 ? make_int2(a.C[e], (int32_t)a.W[e]) : make_int2(-1, 0);
          }
        }
        for (;;) {
          const int32_t v = vw.x;
          int code = 0;
          // below 0xFFFFFFFF, or the sum wrapped round or is no distance
          const uint32_t nd = du + (uint32_t)vw.y;
          relaxed += v >= 0;
          if (v >= 0 && nd >= du && nd != 0xFFFFFFFFu && GR_IN(v, a.n, 340) &&
              nd < atomicMin(dist + v, nd)) {  // this thread lowered dist[v]
            const uint32_t bit = 1u << (v & 31);
            if (nd < T32) {
              code = atomicOr(&nbits[v >> 5], bit) & bit ? 0 : 1;
            } else {
              local_min = min(local_min, nd);
              if (FAR_BITS) code = atomicOr(&fbits[v >> 5], bit) & bit ? 0 : 2;
              else code = atomicExch(far_stamp + v, 0) == 0 ? 0 : 2;
            }
          }
          __syncwarp();
          solo_append(v, code, &st.near[next], &st.far[fp], Qn, near_g, far);
          e += 4;
          if (!LONG || !__any_sync(0xffffffffu, e < e1)) break;
          vw = e < e1 ? make_int2(a.C[e], (int32_t)a.W[e]) : make_int2(-1, 0);
        }
      }
    } else {
      // the far pile by the raised threshold; entries that fell below the
      // old one were expanded already
      const unsigned long long width =
          LONG && (int64_t)len * kSsspFarShare > expanded ? delta_thick : delta;
      const unsigned long long T_old = T, t = T + width, b = bucket_end(st.far_min, width);
      T = t > b ? t : b;
      int32_t *far_n = fp ? far0 : far1;
      __syncthreads();  // every thread has read far_min
      if (threadIdx.x == 0) {
        st.far[fp ^ 1] = 0;
        st.far_min = 0xFFFFFFFFu;
      }
      __syncthreads();
      for (int32_t i0 = 0; i0 < len; i0 += kSoloThreads) {
        const int32_t i = i0 + (int32_t)threadIdx.x;
        if (i0 + (int32_t)(threadIdx.x & ~31) >= len) break;  // warp-uniform
        int32_t v = 0;
        int code = 0;
        if (i < len) {
          v = far[i];
          const uint32_t d = __ldcg(dist + v);
          const uint32_t bit = 1u << (v & 31);
          if ((unsigned long long)d >= T) {
            code = 2;
            local_min = min(local_min, d);
          } else {
            if (FAR_BITS) atomicAnd(&fbits[v >> 5], ~bit);
            else far_stamp[v] = -1;
            if ((unsigned long long)d >= T_old) {
              code = 1;
              atomicOr(&nbits[v >> 5], bit);
            }
          }
        }
        __syncwarp();
        solo_append(v, code, &st.near[next], &st.far[fp ^ 1], Qn, near_g, far_n);
      }
      fp ^= 1;
      phases += 1;
    }
    local_min = __reduce_min_sync(0xffffffffu, local_min);
    if (lane == 0 && local_min != 0xFFFFFFFFu) atomicMin(&st.far_min, local_min);
    iter += 1;
    ring = next;
    __syncthreads();
  }
  const uint32_t wsum = __reduce_add_sync(0xffffffffu, relaxed);
  if (lane == 0) atomicAdd(&st.relaxed, (unsigned long long)wsum);
  __syncthreads();
  const int32_t q = st.near[ring], len = st.far[fp];
  const bool over = (q > 0 || len > 0) && iter >= max_iters;
  const bool handoff = !over && q > handoff_at;
  if (threadIdx.x == 0) {
    atomicMax(&c->iter, iter);
    atomicMax(&c->phases, phases);
    atomicAdd((unsigned long long *)&c->relaxations, st.relaxed);
    if (over) atomicExch(&c->error, kDevOverflow);
    if (handoff) st.near_at = atomicAdd(&c->far_len, q);
  }
  __syncthreads();
  if (!handoff) return;
  const int32_t *Q = iter & 1 ? q1 : q0;
  const int32_t *far = fp ? far1 : far0;
  uint32_t lowest = 0xFFFFFFFFu;
  for (int32_t i = threadIdx.x; i < q; i += kSoloThreads) {
    const int32_t v = i < kSoloQueue ? Q[i] : near_g[i];
    a.farq[0][st.near_at + i] = base + v;
    lowest = min(lowest, __ldcg(dist + v));
  }
  // of the far pile what has not fallen below T: the rest is on the frontier or
  // expanded already. (far_stamp says nothing of the grid's pile, whose epochs
  // begin at 0: its first step splits all of it into epoch 1.)
  for (int32_t i = threadIdx.x; i - lane < len; i += kSoloThreads) {  // warp-uniform
    const int32_t v = i < len ? far[i] : 0;
    const uint32_t d = i < len ? __ldcg(dist + v) : 0u;
    const bool keep = i < len && (unsigned long long)d >= T;
    const uint32_t kb = __ballot_sync(0xffffffffu, keep);
    int32_t at = 0;
    if (lane == 0 && kb) at = atomicAdd(&c->far_len, __popc(kb));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(kb & ((1u << lane) - 1u));
    if (keep) {
      a.farq[0][at] = base + v;
      lowest = min(lowest, d);
    }
  }
  lowest = __reduce_min_sync(0xffffffffu, lowest);
  if (lane == 0) atomicMin(&c->far_min, lowest);
}

// Persistent form: the whole SSSP in one cooperative kernel, one grid
// barrier per iteration. After the barrier every block reads the
// iteration's counters and recomputes the same next state in registers; the
// counters form rings of three (the one an iteration fills, the one just
// read, the one block 0 clears for the next iteration).
template <bool LOW, bool PULL>
__global__ void __launch_bounds__(kSsspThreads, kSsspBlocksPerSm) k_sssp_do(SsspArgs a) {
  constexpr int ITEMS = PULL ? kSsspPullItems : kSsspItems;
  constexpr int CHUNK = kSsspThreads * ITEMS;
  SsspCtl *c = a.ctl;
  __shared__ SsspSmem<ITEMS> sm;
  if (threadIdx.x == 0) {
    sm.nearb.cnt = 0;
    sm.farb.cnt = 0;
  }
  __syncthreads();
  uint32_t *dist = c->dist;
  const unsigned long long delta = c->delta;
  const int32_t max_iters = c->max_iters;
  // the sources, or the pile that k_sssp_solo handed over (nothing: it finished
  // every search)
  int32_t mode = kSsspRelax, near_parity = 0, far_parity = 0, near_len = c->near_len,
          far_len = c->far_len;
  if (near_len == 0 && far_len == 0) return;
  // Bucket width: a mesh's thin frontiers wait for the barrier whatever their
  // size, so wide buckets save iterations (4096 x 4096: 147 ms at two mean
  // weights, 104 at six); where an iteration has more than a vertex per thread,
  // relaxing vertices again costs more (random graph of degree 16, 2 M vertices:
  // 2.8 and 5.5 ms). Each split goes by the iterations since the last.
  const unsigned long long delta_thick = c->delta_thick;
  long long expanded = 0;
  long long near_edges = c->near_edges, relaxations = c->relaxations;
  const long long pull_min_edges = c->pull_min_edges;
  int32_t iter = c->iter, far_epoch = 0, phases = c->phases, gen = 0, pulls = 0;
  uint32_t far_min = c->far_min;
  unsigned long long T = c->T, T_old = 0;
  if (LOW && near_len == 0) {
    mode = kSsspSplit;
    T = bucket_end(far_min, delta_thick);
  }
  for (;;) {
    const int32_t slot = iter % 3, clear = (iter + 1) % 3;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      c->ring_near[clear] = 0ull;
      c->ring_far[clear] = 0;
      c->ring_fmin[clear] = 0xFFFFFFFFu;
    }
    SsspStep st;
    st.near_parity = near_parity;
    st.far_parity = far_parity;
    st.q = near_len;
    st.q_edges = (int32_t)near_edges;
    st.far_len = far_len;
    st.T = T;
    st.T_old = T_old;
    st.iter = iter;
    st.far_epoch = far_epoch;
    st.near_ctr = &c->ring_near[slot];
    st.far_ctr = &c->ring_far[slot];
    st.fmin = &c->ring_fmin[slot];
    if (mode != kSsspSplit) {
      st.far_dest = pick(a.farq, far_parity) + far_len;  // appended after the pile
      st.far_cap = (long long)a.nv + 1 - far_len;
      if (PULL && mode == kSsspPull) {
        pull_body(a, dist);
        if (!grid_sync(&c->bar, &c->error, gen)) break;
        sweep_body(a, dist, sm, st);
      } else if (LOW) {
        relax_body_thread(a, dist, st);
      } else {
        // a dense frontier's chunk bounds in one grid-wide pass (every block
        // then starts its chunks without a search)
        const long long nchunks = ((long long)near_len + near_edges + CHUNK - 1) / CHUNK;
        const bool bounds = a.qcb && nchunks >= (long long)kSsspBoundsChunksPerBlock * gridDim.x;
        if (bounds) {
          frontier_chunk_bounds<CHUNK>(pick(a.nearS, near_parity), near_len, (int32_t)near_edges,
                                nchunks, a.qcb);
          if (!grid_sync(&c->bar, &c->error, gen)) break;
        }
        relax_body(a, dist, sm, st, bounds ? a.qcb : nullptr);
      }
    } else {
      st.far_dest = pick(a.farq, far_parity ^ 1);
      st.far_cap = (long long)a.nv + 1;
      split_body(a, dist, sm, st);
    }
    if (!grid_sync(&c->bar, &c->error, gen)) break;  // a wait gave up: error is set
    const unsigned long long pk = *(volatile unsigned long long *)&c->ring_near[slot];
    const int32_t fcnt = *(volatile int32_t *)&c->ring_far[slot];
    const uint32_t fmin = *(volatile uint32_t *)&c->ring_fmin[slot];
    if (mode != kSsspSplit) {
      relaxations += mode == kSsspPull ? a.m : near_edges;
      pulls += mode == kSsspPull;
      far_len += fcnt;
      far_min = min(far_min, fmin);
      if (LOW) expanded += near_len;
    } else {
      far_len = fcnt;
      far_parity ^= 1;
      far_epoch += 1;
      far_min = fmin;
      phases += 1;
    }
    near_len = (int32_t)(pk & 0xFFFFFFFFull);
    near_edges = (long long)(pk >> 32);
    near_parity ^= 1;
    iter += 1;
    bool done = false, overflow = false;
    if (near_len > 0) {
      mode = PULL && near_edges >= pull_min_edges ? kSsspPull : kSsspRelax;
    } else if (far_len > 0) {
      mode = kSsspSplit;
      T_old = T;
      unsigned long long width = delta;
      if (LOW && (long long)far_len * kSsspFarShare > expanded) width = delta_thick;
      const unsigned long long t = T + width;
      const unsigned long long j = bucket_end(far_min, width);
      T = t > j ? t : j;
    } else {
      done = true;
    }
    if (!done && iter >= max_iters) overflow = true;
    if (done || overflow) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->iter = iter;
        c->phases = phases;
        c->relaxations = relaxations;
        c->pulls = pulls;
        if (overflow) c->error = kDevOverflow;
        c->done = 1;
      }
      break;
    }
  }
}

// pred[v] = smallest u with an edge (u, v) and dist[u] + w = dist[v]
__global__ void k_sssp_pred_init(int32_t *pred, int32_t n) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    pred[v] = INT32_MAX;
}

__global__ void k_sssp_pred(const int32_t *R, const int32_t *C, const uint32_t *W,
                            const uint32_t *dist, int32_t *pred, int32_t n, int32_t src) {
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int lane = threadIdx.x & 31;
  for (int64_t uu = gw; uu < n; uu += nw) {
    const int32_t u = (int32_t)uu;
    const uint32_t du = dist[u];
    if (du == 0xFFFFFFFFu) continue;
    for (int32_t e = R[u] + lane; e < R[u + 1]; e += 32) {
      const int32_t v = C[e];
      const uint32_t dv = dist[v];
      if (v != src && dv != 0xFFFFFFFFu && (unsigned long long)du + W[e] == dv)
        atomicMin(pred + v, u);
    }
  }
}

__global__ void k_sssp_pred_fin(int32_t *pred, int32_t n, int32_t src) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    pred[v] = v == src ? src : (pred[v] == INT32_MAX ? -1 : pred[v]);
}

}  // namespace

// Dynamic shared memory k_sssp_solo may take: the compiler rounds its SoloState
// up (to 48 bytes).
constexpr size_t kSoloSmemMax = kBlockSmemMax - 64;
static_assert(sizeof(SoloState) <= 64, "the state does not fit beside the bits");

// Shared memory k_sssp_solo needs on this graph with the far pile's bits in
// it or not; 0 where the graph is not a mesh or does not fit.
static size_t solo_smem(const gr_graph *g, bool far_bits) {
  if (g->max_degree > kLowDegreeMax) return 0;
  const size_t bytes = sizeof(int32_t) * (2 * (size_t)kSoloQueue +
                                          (size_t)g->nwords * (far_bits ? 2 : 1));
  return bytes <= kSoloSmemMax ? bytes : 0;
}

// Whether a single search may pull: a row holds the in-edges and their
// weights.
static bool can_pull(const gr_graph *g) {
  return g->weights_symmetric && g->max_degree > kLowDegreeMax && g->m > 0;
}

// Most merge-path chunks a near frontier of `lanes` copies can have: n vertices
// of each and their edges.
static size_t sssp_max_chunks(const gr_graph *g, int32_t lanes) {
  const int items = lanes == 1 && can_pull(g) ? kSsspPullItems : kSsspItems;
  return (size_t)lanes * ((size_t)g->n + (size_t)g->m) / (kSsspThreads * items) + 2;
}

size_t sssp_ws_bytes(const gr_graph *g, int32_t lanes) {
  return (size_t)lanes * sssp_lane_bytes(g) + sizeof(SsspCtl) +
         (solo_smem(g, false) ? 32 * (size_t)g->n : 0) +
         (lanes == 1 && can_pull(g) ? gather_plan_bytes(g->n, g->m) + 4 * (size_t)g->nwords +
                                          4 * sssp_max_chunks(g, 1)
                                    : 0);
}

size_t sssp_lane_bytes(const gr_graph *g) {
  const size_t n = (size_t)g->n;
  return 4 * sizeof(int32_t) * (n + 1) + 2 * sizeof(int32_t) * (n + 2) + 2 * sizeof(int32_t) * n +
         (g->max_degree > kLowDegreeMax
              ? sizeof(int32_t) * ((n + (size_t)g->m) / (kSsspThreads * kSsspItems) + 3)
              : 0);
}

int32_t sssp_batch_max_lanes(const gr_graph *g) {
  // lane-major ids and queue positions (up to lanes * n + 1), and a
  // frontier's edge count (up to lanes * m), are int32
  long long k = kSsspMaxLanes;
  k = std::min<long long>(k, (INT32_MAX - 2) / std::max<int32_t>(g->n, 1));
  if (g->m > 0) k = std::min<long long>(k, INT32_MAX / g->m);
  return (int32_t)std::max<long long>(k, 1);
}

gr_status sssp_ws_create(gr_graph *g, cudaStream_t s, SsspWorkspace **out, int32_t lanes) {
  if (lanes < 1 || lanes > sssp_batch_max_lanes(g))
    return fail(GR_EINVAL, "SSSP workspace: lane count out of range for this graph");
  std::unique_ptr<SsspWorkspace> ws(new SsspWorkspace());
  ws->lanes = lanes;
  const size_t n = (size_t)g->n * (size_t)lanes;
  for (int i = 0; i < 2; ++i) {
    GR_TRY(ws->nearq[i].alloc(sizeof(int32_t) * (n + 1), "SSSP near queue"));
    GR_TRY(ws->nearS[i].alloc(sizeof(int32_t) * (n + 2), "SSSP near degree scan"));
    GR_TRY(ws->farq[i].alloc(sizeof(int32_t) * (n + 1), "SSSP far pile"));
  }
  GR_TRY(ws->stamp.alloc(sizeof(int32_t) * n, "SSSP near stamps"));
  GR_TRY(ws->far_stamp.alloc(sizeof(int32_t) * n, "SSSP far stamps"));
  GR_TRY(ws->ctl.alloc(sizeof(SsspCtl), "SSSP control"));
  if (g->max_degree > kLowDegreeMax) {
    GR_TRY(ws->qcb.alloc(sizeof(int32_t) * (sssp_max_chunks(g, lanes) + 1),
                         "SSSP frontier chunk bounds"));
  }
  if (lanes == 1 && can_pull(g)) {
    GR_TRY(gather_plan_build(&ws->plan, g->row_off.as<int32_t>(), g->n, g->m, s));
    GR_TRY(ws->lowered.alloc(sizeof(uint32_t) * (size_t)g->nwords, "SSSP pull marks"));
  }
  GR_CUDA(cudaMemsetAsync(ws->ctl.p, 0, sizeof(SsspCtl), s));
  if (solo_smem(g, false)) GR_TRY(low_adjacency(g, true, s));
  GR_CUDA(cudaStreamSynchronize(s));
  *out = ws.release();
  return GR_OK;
}

static SsspArgs sssp_args(gr_graph *g, SsspWorkspace *ws, int32_t lanes = 1) {
  SsspArgs a;
  a.R = g->row_off.as<int32_t>();
  a.C = g->col.as<int32_t>();
  a.W = g->w.as<uint32_t>();
  a.n = g->n;
  a.nv = g->n * lanes;
  a.m = g->m;
  for (int i = 0; i < 2; ++i) {
    a.nearq[i] = ws->nearq[i].as<int32_t>();
    a.nearS[i] = ws->nearS[i].as<int32_t>();
    a.farq[i] = ws->farq[i].as<int32_t>();
  }
  a.stamp = ws->stamp.as<int32_t>();
  a.far_stamp = ws->far_stamp.as<int32_t>();
  a.ctl = ws->ctl.as<SsspCtl>();
  a.low_degree = g->max_degree <= kLowDegreeMax ? 1 : 0;
  a.adjw = g->adjw4.as<int4>();
  a.solo_handoff = std::min(kSoloQueue, kSoloHandoffEdges / std::max(g->max_degree, 4));
  a.plan = ws->plan.a;  // null where nothing may be pulled (sssp_pull_min_edges)
  a.lowered = ws->lowered.as<uint32_t>();
  a.qcb = ws->qcb.as<int32_t>();  // null on low-degree graphs
  return a;
}

// Smallest near-frontier edge count at which a relaxation pulls: m /
// opts->alpha, else m / the graph's tuned alpha (0: never); GR_DIR_PUSH
// never pulls, GR_DIR_PULL pulls every relaxation. Only a single search on a
// workspace with a plan pulls: one made for several lanes has none, whatever
// the number of sources it is used for, nor has that of a graph whose rows are
// not its in-edges (weights that differ by direction among them).
static long long sssp_pull_min_edges(const gr_graph *g, const SsspWorkspace *ws, const gr_opts &o,
                                     int32_t lanes) {
  if (lanes != 1 || !ws->plan.a.desc || !ws->lowered.p || o.direction == GR_DIR_PUSH)
    return LLONG_MAX;
  if (o.direction == GR_DIR_PULL) return 1;
  const double div = o.alpha > 0.f ? (double)o.alpha : (double)g->tuned_sssp_alpha;
  if (div <= 0.0) return LLONG_MAX;
  return std::max<long long>(1, (long long)((double)g->m / div));
}

static gr_status sssp_enqueue_iter(gr_graph *g, const SsspArgs &a, cudaStream_t s,
                                   cudaGraphConditionalHandle h, int use_cond) {
  if (a.low_degree)
    k_sssp_iter<true><<<g->num_sms * kSsspBlocksPerSm, kSsspThreads, 0, s>>>(a, h, use_cond);
  else
    k_sssp_iter<false><<<g->num_sms * kSsspBlocksPerSm, kSsspThreads, 0, s>>>(a, h, use_cond);
  GR_CUDA(cudaGetLastError());
  return GR_OK;
}

static gr_status build_sssp_graph(gr_graph *g, SsspWorkspace *ws) {
  if (ws->exec) return GR_OK;
  cudaGraph_t graph;
  GR_CUDA(cudaGraphCreate(&graph, 0));
  cudaGraphConditionalHandle h;
  GR_CUDA(cudaGraphConditionalHandleCreate(&h, graph, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  GR_CUDA(cudaGraphAddNode(&node, graph, nullptr, nullptr, 0, &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  cudaStream_t cs;
  GR_CUDA(cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking));
  GR_CUDA(cudaStreamBeginCaptureToGraph(cs, body, nullptr, nullptr, 0,
                                        cudaStreamCaptureModeThreadLocal));
  gr_status st = sssp_enqueue_iter(g, sssp_args(g, ws), cs, h, 1);
  cudaGraph_t captured;
  cudaError_t e = cudaStreamEndCapture(cs, &captured);
  cudaStreamDestroy(cs);
  if (st != GR_OK) return st;
  GR_CUDA(e);
  GR_CUDA(cudaGraphInstantiate(&ws->exec, graph, 0));
  ws->graph = graph;
  return GR_OK;
}

gr_status sssp_read_ctl_error(SsspWorkspace *ws, cudaStream_t s) {
  SsspCtl h;
  // pageable destination: the copy has finished when the call returns
  GR_CUDA(cudaMemcpyAsync(&h, ws->ctl.p, sizeof(SsspCtl), cudaMemcpyDeviceToHost, s));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "iteration limit reached");
  return GR_OK;
}

gr_status sssp_check(const gr_graph *g, int32_t src, const gr_opts &o) {
  if (!g->has_weights) return fail(GR_EINVAL, "SSSP needs edge weights (w was NULL at creation)");
  if (src < 0 || src >= g->n) return fail(GR_EINVAL, "source out of range");
  if (o.mode < GR_MODE_AUTO || o.mode > GR_MODE_PERSISTENT)
    return fail(GR_EINVAL, "unknown mode");
  if (o.direction < GR_DIR_AUTO || o.direction > GR_DIR_PULL)
    return fail(GR_EINVAL, "unknown direction policy");
  if (o.direction == GR_DIR_PULL && !g->symmetric)
    return fail(GR_EINVAL, "pull relaxation needs a symmetric CSR (in-neighbours = out-neighbours)");
  if (o.alpha < 0.f) return fail(GR_EINVAL, "alpha must be >= 0");
  return GR_OK;
}

// Blocks per SM of a search over m entries, measured in tune_prior (0: all).
int32_t sssp_prior_blocks(int64_t m) {
  return m < 150'000 ? 1 : m < 4'000'000 ? 3 : m < 16'000'000 ? 4 : 0;
}

// Bucket width of thin or of thick frontiers: the caller's, or the graph's own.
static unsigned long long sssp_delta_of(const gr_graph *g, const gr_opts &o, bool thick) {
  if (o.delta == UINT32_MAX) return 1ull << 40;
  return o.delta ? o.delta : thick ? g->sssp_delta_thick : g->sssp_delta;
}

static int32_t sssp_max_iters_of(const gr_graph *g, const gr_opts &o) {
  return o.max_iters > 0 ? o.max_iters
                         : (int32_t)std::min<long long>(INT32_MAX, 8ll * g->n + 1024);
}

// Initialises the searches and runs their device-side loop with the given
// driver.
static gr_status sssp_drive(gr_graph *g, SsspWorkspace *ws, SsspArgs a, const SsspSources &src,
                            uint32_t *dist, int32_t *pred, int32_t mode, const gr_opts &o,
                            cudaStream_t s) {
  const int32_t max_iters = sssp_max_iters_of(g, o);
  const long long pull_min_edges = sssp_pull_min_edges(g, ws, o, src.k);
  // meshes whose membership bits fit one block's shared memory: one block
  // per search, up to the frontier size where the grid takes over
  const size_t near_only = mode == GR_MODE_PERSISTENT ? solo_smem(g, false) : 0;
  // the other drivers know one width
  k_sssp_init<<<g->num_sms * 8, 256, 0, s>>>(
      a, src, dist, pred, sssp_delta_of(g, o, mode != GR_MODE_PERSISTENT),
      sssp_delta_of(g, o, true), max_iters, pull_min_edges, near_only > 0);
  GR_CUDA(cudaGetLastError());
  if (near_only) {
    const size_t both = solo_smem(g, true), bytes = both ? both : near_only;
    const bool longer = g->max_degree > 4;
    auto kern = both ? (longer ? k_sssp_solo<true, true> : k_sssp_solo<false, true>)
                     : (longer ? k_sssp_solo<true, false> : k_sssp_solo<false, false>);
    GR_TRY(allow_smem(kern, kSoloSmemMax));
    kern<<<src.k, kSoloThreads, bytes, s>>>(a, src);
    GR_CUDA(cudaGetLastError());
  }
  if (mode == GR_MODE_PERSISTENT) {
    void *kern = a.low_degree ? (void *)k_sssp_do<true, false>
                 : pull_min_edges < LLONG_MAX ? (void *)k_sssp_do<false, true>
                                              : (void *)k_sssp_do<false, false>;
    const int32_t want = o.block > 0 ? o.block : g->tuned_sssp_blocks_per_sm;
    // the carveout fitted to the blocks that run leaves the rest to L1
    int bps = 1;
    GR_TRY(fit_carveout(kern, kSsspThreads, want > 0 ? std::min(want, kSsspBlocksPerSm)
                                                      : kSsspBlocksPerSm,
                        g->device, &bps));
    void *args[] = {&a};
    GR_CUDA(cudaLaunchCooperativeKernel(kern, std::max(1, bps) * g->num_sms,
                                        kSsspThreads, args, 0, s));
  } else if (mode == GR_MODE_LAUNCH) {
    // the device ends the run, at its iteration limit at the latest; a pulled
    // iteration takes two launches
    SsspCtl h;
    const long long most = 2ll * max_iters + 2;
    long long enq = 0;
    int32_t batch = 8;
    for (;;) {
      for (int i = 0; i < batch; ++i) GR_TRY(sssp_enqueue_iter(g, a, s, 0, 0));
      enq += batch;
      GR_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(h), cudaMemcpyDeviceToHost, s));
      GR_CUDA(cudaStreamSynchronize(s));
      if (h.done) break;
      if (enq > most) return fail(GR_ETIMEOUT, "SSSP did not end within its iteration limit");
      batch = std::min(batch * 2, 256);
    }
  } else {
    GR_TRY(build_sssp_graph(g, ws));
    GR_CUDA(cudaGraphLaunch(ws->exec, s));
  }
  return GR_OK;
}

// SSSP into device outputs with an explicit workspace (no locking, no
// staging): the public gr_sssp and the query server both call this.
gr_status sssp_run(gr_graph *g, SsspWorkspace *ws, int32_t src, uint32_t *dist, int32_t *pred,
                   const gr_opts &o, cudaStream_t s) {
  SsspArgs a = sssp_args(g, ws);
  SsspSources one;
  one.k = 1;
  one.s[0] = src;
  const int32_t mode = o.mode != GR_MODE_AUTO ? o.mode : g->tuned_sssp_mode;
  GR_TRY(sssp_drive(g, ws, a, one, dist, pred, mode, o, s));
  if (pred) {
    const int grid = g->num_sms * 8;
    k_sssp_pred_init<<<grid, 256, 0, s>>>(pred, g->n);
    k_sssp_pred<<<grid, 256, 0, s>>>(a.R, a.C, a.W, dist, pred, g->n, src);
    k_sssp_pred_fin<<<grid, 256, 0, s>>>(pred, g->n, src);
    GR_CUDA(cudaGetLastError());
  }
  return GR_OK;
}

// k searches as one over k copies of the graph into dist[k][n] (device).
// The CUDA-graph driver holds one-lane arguments, so every driver but the
// persistent kernel becomes the host-driven loop here.
gr_status sssp_batch_run(gr_graph *g, SsspWorkspace *ws, const int32_t *h_srcs, int32_t k,
                         uint32_t *dist, const gr_opts &o, cudaStream_t s) {
  if (k < 1 || k > ws->lanes) return fail(GR_EINVAL, "batched SSSP: k exceeds the workspace");
  SsspArgs a = sssp_args(g, ws, k);
  SsspSources srcs;
  srcs.k = k;
  for (int32_t l = 0; l < kSsspMaxLanes; ++l) srcs.s[l] = l < k ? h_srcs[l] : 0;
  int32_t mode = o.mode != GR_MODE_AUTO ? o.mode : g->tuned_sssp_mode;
  if (mode != GR_MODE_PERSISTENT) mode = GR_MODE_LAUNCH;
  gr_opts ob = o;
  // k lanes carry k times the frontier of one search per iteration: where
  // one search runs on few blocks a batch takes more (16 sources on the 4096^2
  // mesh: 282 ms at 2 blocks per SM, 321 at 1, 297 at 3, 335 at 5)
  if (k > 1 && ob.block == 0 && g->tuned_sssp_blocks_per_sm > 0) {
    const int32_t more = a.low_degree ? 2 : sssp_prior_blocks((int64_t)k * g->m);
    ob.block = more == 0 ? kSsspBlocksPerSm : std::max(more, g->tuned_sssp_blocks_per_sm);
  }
  return sssp_drive(g, ws, a, srcs, dist, nullptr, mode, ob, s);
}

}  // namespace gr

using namespace gr;

extern "C" {

gr_status gr_sssp(gr_graph *g, int32_t src, uint32_t *dist, int32_t *pred,
                  const gr_opts *opts, void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!dist) return fail(GR_EINVAL, "dist must not be NULL");
  const gr_opts &o = opts ? *opts : default_opts();
  GR_TRY(sssp_check(g, src, o));
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  if (!g->sssp) GR_TRY(sssp_ws_create(g, s, &g->sssp));
  void *d_dist, *d_pred;
  bool cp_dist, cp_pred;
  GR_TRY(resolve_output(g, 0, dist, sizeof(uint32_t) * (size_t)g->n, &d_dist, &cp_dist));
  GR_TRY(resolve_output(g, 1, pred, sizeof(int32_t) * (size_t)g->n, &d_pred, &cp_pred));
  GR_TRY(sssp_run(g, g->sssp, src, (uint32_t *)d_dist, (int32_t *)d_pred, o, s));
  if (cp_dist)
    GR_CUDA(cudaMemcpyAsync(dist, d_dist, sizeof(uint32_t) * (size_t)g->n,
                            cudaMemcpyDeviceToHost, s));
  if (cp_pred)
    GR_CUDA(cudaMemcpyAsync(pred, d_pred, sizeof(int32_t) * (size_t)g->n,
                            cudaMemcpyDeviceToHost, s));
  GR_TRY(end_call(g, s));
  return GR_OK;
}

gr_status gr_sssp_batch(gr_graph *g, const int32_t *srcs, int32_t k, uint32_t *dist,
                        const gr_opts *opts, void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!srcs || !dist) return fail(GR_EINVAL, "srcs/dist must not be NULL");
  const int32_t kmax = sssp_batch_max_lanes(g);
  if (k < 1 || k > kmax)
    return fail(GR_EINVAL, "k must be in [1, " + std::to_string(kmax) +
                               "] (64, and k*n and k*m must fit in int32)");
  const gr_opts &o = opts ? *opts : default_opts();
  for (int32_t i = 0; i < k; ++i) GR_TRY(sssp_check(g, srcs[i], o));
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  if (g->sssp_batch && g->sssp_batch->lanes < k) {
    // the old buffers may still be in use by enqueued work
    GR_CUDA(cudaStreamSynchronize(s));
    free_sssp(g->sssp_batch);
    g->sssp_batch = nullptr;
  }
  if (!g->sssp_batch) GR_TRY(sssp_ws_create(g, s, &g->sssp_batch, k));
  void *d_dist;
  bool cp;
  const size_t bytes = sizeof(uint32_t) * (size_t)k * (size_t)g->n;
  GR_TRY(resolve_output(g, 0, dist, bytes, &d_dist, &cp));
  GR_TRY(sssp_batch_run(g, g->sssp_batch, srcs, k, (uint32_t *)d_dist, o, s));
  if (cp) GR_CUDA(cudaMemcpyAsync(dist, d_dist, bytes, cudaMemcpyDeviceToHost, s));
  GR_TRY(end_call(g, s));
  return GR_OK;
}

gr_status gr_sssp_batch_stats(gr_graph *g, int32_t *iterations, int32_t *phases,
                              int64_t *relaxations) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!g->sssp_batch) return fail(GR_EINVAL, "no batched SSSP has run on this graph");
  std::lock_guard<std::mutex> lock(g->mu);
  GR_CUDA(cudaSetDevice(g->device));
  if (g->has_last) GR_CUDA(cudaEventSynchronize(g->last_done));
  SsspCtl h;
  GR_CUDA(cudaMemcpy(&h, g->sssp_batch->ctl.p, sizeof(h), cudaMemcpyDeviceToHost));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "iteration limit reached");
  if (iterations) *iterations = h.iter;
  if (phases) *phases = h.phases;
  if (relaxations) *relaxations = h.relaxations;
  return GR_OK;
}

gr_status gr_sssp_pull_stats(gr_graph *g, int32_t *pulls) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!g->sssp) return fail(GR_EINVAL, "no SSSP has run on this graph");
  std::lock_guard<std::mutex> lock(g->mu);
  GR_CUDA(cudaSetDevice(g->device));
  if (g->has_last) GR_CUDA(cudaEventSynchronize(g->last_done));
  SsspCtl h;
  GR_CUDA(cudaMemcpy(&h, g->sssp->ctl.p, sizeof(h), cudaMemcpyDeviceToHost));
  if (pulls) *pulls = h.pulls;
  return GR_OK;
}

gr_status gr_sssp_stats(gr_graph *g, int32_t *iterations, int32_t *phases,
                        int64_t *relaxations) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!g->sssp) return fail(GR_EINVAL, "no SSSP has run on this graph");
  std::lock_guard<std::mutex> lock(g->mu);
  GR_CUDA(cudaSetDevice(g->device));
  if (g->has_last) GR_CUDA(cudaEventSynchronize(g->last_done));
  SsspCtl h;
  GR_CUDA(cudaMemcpy(&h, g->sssp->ctl.p, sizeof(h), cudaMemcpyDeviceToHost));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "iteration limit reached");
  if (iterations) *iterations = h.iter;
  if (phases) *phases = h.phases;
  if (relaxations) *relaxations = h.relaxations;
  return GR_OK;
}

}  // extern "C"
