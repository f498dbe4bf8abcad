// Multi-source traversals with 64 bitmask lanes: batched BFS and Brandes
// betweenness centrality (Sec. 5.3).
//
// Up to 64 sources advance together, one bit lane each (the multi-source BFS
// idea of Then et al., VLDB 2014). Per vertex v a 64-bit mask lm[L][v] holds
// the lanes whose frontier at level L contains v; visit[v] the lanes that
// reached v at an earlier level. One level is a pull over all vertices
// (batched BFS: in 256-entry register tiles over the rows that miss a lane; BC:
// in merge-path chunks, one per warp): for an edge (v, u), bits = lm[L][u] & ~visited(v) are
// the lanes in which u is a predecessor of v, and v joins lm[L+1] in those
// lanes. Every column index is read once per level; the 64 traversals share
// that read.
//
// BC (Brandes, as the paper's Sec. 5.3 describes: a forward BFS pass
// counting shortest paths sigma, then a backward pass over the BFS levels
// accumulating dependencies) keeps per vertex 64 FP64 lanes, vertex-major
// (512 bytes per vertex), so the warp that serves an edge reads the 64
// lanes of one vertex in two coalesced 256-byte loads:
//   forward   sigma[v][s] = sum of sigma[u][s] over predecessors u in lane s
//   backward  with q[w][s] = 1/sigma[w][s] + sum over children x of q[x][s]
//             (i.e. (1 + delta[w][s]) / sigma[w][s]),
//             delta[v][s] = sigma[v][s] * sum over children w of q[w][s],
//             bc[v] += delta[v][s] for every lane s that reached v at level
//             >= 1 (v is then not lane s's source).
// This is the dependency recursion delta[v] += sigma[v]/sigma[w]*(1+delta[w])
// regrouped so that each edge needs one gathered value per lane.
//
// Path counts are integers, and FP64 arithmetic is scarce on this GPU (a few
// FP64 operations per clock per SM), so the forward pass counts them exactly
// in uint64 with integer adds (exact where FP64 rounds, beyond 2^53). A batch
// whose counts pass 2^64 - 1 (an add carries out) is counted again in FP64,
// which holds counts up to about 1.8e308.
//
// The forward level loop runs in one cooperative persistent kernel
// (k_mb_do), levels separated by the bounded grid barrier, the direction of
// every level decided on the device. Each level also emits the list of the
// vertices that joined the next level (with its degree scan), so a push
// level expands exactly its frontier and nothing scans all n vertices to
// find it. A batched BFS needs no host round trip at all; BC, which keeps
// one mask array per level, stops the kernel when the next level needs an
// array not yet allocated, and the host allocates more and resumes it.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "double_single.cuh"
#include "gather.cuh"

namespace gr {

// Items per thread of a push level's chunk: two leave the pulls' gathers more of
// the L1; the batched BFS of a directed graph of kMbPushOnlyM entries or more, which
// only pushes, takes four (R-MAT 2^20, 15.7 M entries, 16 lanes: 1053 us at two,
// 867 at four; 2^18, 3.8 M, 247 and 233; 2^16, 0.9 M, 131 and 137).
constexpr int kMbThreads = 256, kMbItems = 2, kMbPushOnlyItems = 4;
constexpr int64_t kMbPushOnlyM = 3'000'000;
// Batched BFS keeps the lane masks of its first kKeepLevels levels, each in
// its own array, and writes their depths in one pass at the end (full
// coalesced rows); deeper levels rotate through three arrays and write their
// depths as they are reached. On graphs of small maximum degree (meshes:
// thousands of levels, small frontiers) no level is kept.
constexpr int32_t kKeepLevels = 16;
// A batched BFS level pushes when its frontier has fewer than m / kPushDiv
// edges, and pulls over every vertex otherwise.
constexpr long long kPushDiv = 16;
// BC's gathers take chunks of this many items per warp: with one per block
// its warps waited for the slowest at every chunk (half of the forward's
// stalls).
constexpr int kMbWarpChunk = 128;
constexpr int kMbListChunk = 1024;  // vertices per block step of k_mb_list
// What the forward pass counts: nothing (batched BFS), path counts in uint64,
// or path counts in FP64 (a batch whose uint64 counts overflowed).
enum : int { kSigNone = 0, kSigU64 = 1, kSigF64 = 2 };


struct BatchWorkspace {
  DevMem visit, sigma, q, counter, lmp, ctl;
  GatherPlan plan;  // row structure of the batched BFS's pulls (symmetric graphs)
  DevMem full;      // a bit per vertex: it holds every lane in use
  DevMem cb_fwd;    // chunk bounds of BC's all-vertex pulls (fixed per graph)
  DevMem fq, fs;    // BC backward: one level's vertex list and degree scan
  DevMem fcb;       // BC backward: that list's merge-path chunk bounds
  DevMem lq[3], ls[3];  // forward: level lists (ring by level) and degree scans
  std::vector<DevMem *> lm;  // level mask arrays ("slots")
  int32_t uploaded = 0;      // slots whose pointers are in lmp
  ~BatchWorkspace() {
    for (DevMem *p : lm) delete p;
  }
};

void free_batch(BatchWorkspace *ws) { delete ws; }

GR_GUARD_REPORTER(guard_report_batch)

namespace {

// Forward state in device memory: where the level loop stands (so a
// stopped kernel can resume), the level lists' counters and the barrier.
struct MbCtl {
  GridBarrier bar;
  unsigned long long cnt3[3];  // level L+1's vertices: [31:0] count, [63:32] edges
  unsigned long long cnt_list;  // compaction of a pulled level's list
  int32_t level;   // next level to run
  int32_t push;    // its direction
  int32_t q, qe;   // its list's size and edge count
  int32_t q_prev;  // size of the list before it
  int32_t listed;       // the list of `level` exists (a push emitted it)
  int32_t prev_listed;  // the list of `level` - 1 exists
  int32_t done;
  int32_t paused;  // stopped before `level`: it needs a slot beyond cap
  int32_t error;   // kDevTimeout / kDevOverflow
  int32_t levels;  // levels holding vertices (when done)
  int32_t sig_overflow;  // a uint64 path count overflowed
};

struct MbArgs {
  const int32_t *R;
  const int32_t *C;
  int32_t n;
  long long m;
  unsigned long long all;  // mask of the lanes in use
  unsigned long long *visit;
  unsigned long long *const *lmp;  // level mask arrays
  int32_t cap;        // arrays in lmp
  int32_t keep;       // levels < keep have their own array; later ones rotate through 3
  int32_t *lq[3];     // level lists, ring by level: lq[L % 3] lists level L
  int32_t *ls[3];     // their exclusive degree scans
  void *sigma;        // [n][64] uint64 or FP64 path counts, or null (BFS)
  int32_t *depth;     // [k][n] or null (BC)
  int32_t k;
  int32_t symmetric;
  int32_t max_levels;
  MbCtl *ctl;
  GatherPlanArgs plan;  // batched BFS: row structure of the pull levels
  uint32_t *full;       // batched BFS: vertices with every lane, by the last pull
  // BC: chunk bounds of the all-vertex merge path, kMbWarpChunk items each
  const int32_t *cb_fwd;
};

__device__ __forceinline__ int32_t mb_slot(const MbArgs &a, int32_t L) {
  return L < a.keep ? L : a.keep + (L - a.keep) % 3;
}

__device__ __forceinline__ unsigned long long shfl_u64(unsigned long long x, int src) {
  return __shfl_sync(0xffffffffu, x, src);
}

// Path-count arithmetic in the forward pass's type: uint64 adds record a
// carry out in `ovf`, FP64 adds cannot overflow short of infinity (caught
// when the counts are used).
template <int SK>
using CountT = typename std::conditional<SK == kSigU64, unsigned long long, double>::type;

__device__ __forceinline__ unsigned long long count_add(unsigned long long x,
                                                        unsigned long long y, bool &ovf) {
  const unsigned long long t = x + y;
  ovf |= t < x;
  return t;
}
__device__ __forceinline__ double count_add(double x, double y, bool &) { return x + y; }

__device__ __forceinline__ void count_atomic_add(unsigned long long *p, unsigned long long y,
                                                 bool &ovf) {
  const unsigned long long old = atomicAdd(p, y);
  ovf |= old + y < old;
}
__device__ __forceinline__ void count_atomic_add(double *p, double y, bool &) {
  atomicAdd(p, y);
}

// Zeroes what the forward reads first: visit, the arrays of levels 0 and 1,
// the path counts and dependencies (BC) and, when no level is kept, the
// depth output (-1: unreached; kept levels' depths are all written by the
// end-of-run pass).
__global__ void k_mb_init(MbArgs a, unsigned long long *sigma, double *q) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  unsigned long long *l0 = a.lmp[mb_slot(a, 0)], *l1 = a.lmp[mb_slot(a, 1)];
  for (int64_t v = tid; v < a.n; v += stride) {
    a.visit[v] = 0ull;
    l0[v] = 0ull;
    l1[v] = 0ull;
  }
  if (sigma) {
    for (int64_t i = tid; i < (int64_t)a.n * 64; i += stride) {
      sigma[i] = 0ull;  // 0 as uint64 and as FP64
      q[i] = 0.0;
    }
  }
  if (a.depth && a.keep == 0)
    for (int64_t i = tid; i < (int64_t)a.k * a.n; i += stride) a.depth[i] = -1;
}

// Level 0: the sources' lanes, their path counts (1) and the level list
// (each distinct source vertex once, with its degree scan). One block of 64
// threads, after k_mb_init.
struct MbSources {
  int32_t s[64];
};

__global__ void k_mb_sources(MbArgs a, MbSources srcs, int32_t sk) {
  __shared__ int32_t s_v[64], s_d[64];
  __shared__ int32_t s_cnt;
  const int s = threadIdx.x;
  if (s == 0) s_cnt = 0;
  __syncthreads();
  unsigned long long *l0 = a.lmp[mb_slot(a, 0)];
  if (s < a.k && GR_IN(srcs.s[s], a.n, 205)) {
    const int32_t v = srcs.s[s];
    if (atomicOr(l0 + v, 1ull << s) == 0ull) {
      const int32_t k = atomicAdd(&s_cnt, 1);
      s_v[k] = v;
      s_d[k] = a.R[v + 1] - a.R[v];
    }
    if (sk == kSigU64) ((unsigned long long *)a.sigma)[(int64_t)v * 64 + s] = 1ull;
    if (sk == kSigF64) ((double *)a.sigma)[(int64_t)v * 64 + s] = 1.0;
  }
  __syncthreads();
  if (s == 0) {
    const int32_t cnt = s_cnt;
    int32_t run = 0;
    for (int32_t i = 0; i < cnt; ++i) {
      a.lq[0][i] = s_v[i];
      a.ls[0][i] = run;
      run += s_d[i];
    }
    MbCtl *c = a.ctl;
    grid_barrier_reset(&c->bar);
    for (int i = 0; i < 3; ++i) c->cnt3[i] = 0ull;
    c->cnt_list = 0ull;
    c->listed = 1;
    c->prev_listed = 0;
    c->level = 0;
    c->push = 1;
    c->q = cnt;
    c->qe = run;
    c->q_prev = 0;
    c->done = cnt == 0;
    c->paused = 0;
    c->error = kDevOk;
    c->levels = cnt ? 0 : 1;
    c->sig_overflow = 0;
  }
}

// Block-local list of the vertices a push level adds to the next level,
// flushed per chunk with flush_scanned (one packed atomic per block and
// chunk); a chunk adds at most as many vertices as it has items.
template <int CHUNK>
__device__ __forceinline__ void mb_emit(ScannedBuf<CHUNK> &em, const MbArgs &a, int32_t v) {
  const int32_t k = atomicAdd(&em.cnt, 1);
  em.out[k] = v;
  em.deg[k] = a.R[v + 1] - a.R[v];
}

// Packed (vertices, edges) increment for a vertex that joined the next level.
__device__ __forceinline__ unsigned long long joined(const MbArgs &a, int32_t v) {
  return 1ull | ((unsigned long long)(uint32_t)(a.R[v + 1] - a.R[v]) << 32);
}

// Shared memory of the level forms (one at a time).
template <int ITEMS>
union MbSmem {
  static constexpr int kChunk = kMbThreads * ITEMS;  // items of a push level's chunk
  struct {  // per warp
    int32_t off[kMbWarpChunk + 1];
    unsigned long long U[kMbWarpChunk + 1];
  } fwd[kMbThreads / 32];
  struct {
    int32_t off[kChunk + 1];
    int32_t row[kChunk + 1];
    unsigned long long cur[kChunk + 1];
    int32_t u[kChunk + 1];
    ScannedBuf<kChunk> em;
  } push;
  ScannedBuf<kChunk> list;  // compaction of a pulled level into its list
};

// Lanes of `c` at vertex v reach their depth at level L.
__device__ __forceinline__ void mb_write_depth(const MbArgs &a, int32_t v, unsigned long long c,
                                               int32_t L) {
  for (int s = 0; s < a.k; ++s)
    if (((c >> s) & 1ull) && GR_IN((int64_t)s * a.n + v, (int64_t)a.k * a.n, 204))
      a.depth[(int64_t)s * a.n + v] = L;
}

// A batched BFS pull level (no path counts) has two parts. The fold: every
// vertex's cur goes into visit, its depths at L are written past the kept
// levels, and the vertices that hold every lane are marked in `full`. After
// a grid barrier the gather: nxt[v] = OR over the entries (v, u) of v's row
// of cur[u], less visit[v], in registers (gather_reduce_tiles), the rows of
// full vertices skipped; whole rows are stored (nxt is zero), pieces of rows
// combined with atomicOr. It counts the vertices whose mask goes from empty
// to non-empty, and their edges; it writes no list (a push level after it
// compacts one). R-MAT 2^20, 64 sources, 31.4 M entries: the four pulls took
// 192, 237, 199 and 97 us with merge-path tables in shared memory (which take
// the masks' L1) and a lane mask looked up per edge.
__device__ void mb_pull_fold(const MbArgs &a, int32_t L, const unsigned long long *cur) {
  const bool write_depth = a.depth && L >= a.keep;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t nr = ((int64_t)a.n + 31) & ~31ll;  // warp-uniform bound
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < nr; v += stride) {
    bool all = true;
    if (v < a.n) {
      const unsigned long long c = cur[v];
      unsigned long long seen = a.visit[v];
      if (c) {
        seen |= c;
        a.visit[v] = seen;
        if (write_depth) mb_write_depth(a, (int32_t)v, c, L);
      }
      all = seen == a.all;
    }
    const uint32_t b = __ballot_sync(0xffffffffu, all);
    if ((threadIdx.x & 31) == 0) a.full[v >> 5] = b;
  }
}

struct LaneMask {
  static constexpr bool kWeighted = false;
  const unsigned long long *cur;
  __device__ __forceinline__ unsigned long long operator()(int32_t u, int32_t) const {
    return cur[u];
  }
};
struct OrU64 {
  static __device__ __forceinline__ unsigned long long identity() { return 0ull; }
  static __device__ __forceinline__ unsigned long long op(unsigned long long x,
                                                          unsigned long long y) {
    return x | y;
  }
};
struct SkipFull {
  static constexpr bool kSkips = true;
  const uint32_t *full;
  __device__ __forceinline__ bool operator()(int32_t v) const { return test_bit(full, v); }
};
struct JoinLanes {
  const MbArgs &a;
  unsigned long long *nxt;
  unsigned long long &count;
  __device__ __forceinline__ void operator()(int32_t v, unsigned long long x, bool whole) const {
    if (!x) return;
    x &= ~a.visit[v];
    if (!x) return;
    if (whole) nxt[v] = x;
    else if (atomicOr(nxt + v, x)) return;
    count += joined(a, v);
  }
};

__device__ __forceinline__ void mb_pull_gather(const MbArgs &a, const unsigned long long *cur,
                                               unsigned long long *nxt,
                                               unsigned long long *counter) {
  unsigned long long count = 0;
  gather_reduce_tiles<1, unsigned long long, OrU64>(
      a.plan, a.C, nullptr, 0, (int32_t)a.m, LaneMask{cur}, JoinLanes{a, nxt, count},
      spread_warp(), grid_warps(), SkipFull{a.full});
  count = warp_sum(count);
  if ((threadIdx.x & 31) == 0 && count) atomicAdd(counter, count);
}

// ------------------------------------------------------- lane-wise gathers
// BC adds, for an edge (v, u) and every lane s set in its `bits`, one value of
// u's row of 64 to v's sum of lane s. Few lanes are set, and they are much the
// same along v's row (the lanes whose level v is on): R-MAT 2^17, 64 sources,
// busiest level: 41.8 M (edge, lane) pairs on 2.9 M edges, 7.9 of 32 lanes in
// a half row that has any. With lane s of a warp serving source s, edge after
// edge, that is 5.3 M half-row adds of which three quarters do nothing, and
// an FP64 add holds the SM's pipe for 16 cycles whatever its lanes.
//
// Here a warp takes a window of 32 edges, packs those of one vertex that have
// bits into shared memory, and deals its threads to the vertex's lanes of a
// half row: with a lanes in it, thread t serves the (t mod a)-th of them and
// every (32 / a)-th edge. The partial sums of a lane meet in the atomics that
// add them to v's row (done in L2, not in the FP64 pipe).
struct LaneBuf {
  int32_t u[32];
  uint32_t bits[2][32];
  uint8_t lane_of[2][32];
};

// What a warp is summing: vertex `owner`; per half row the thread's source,
// its first edge and edge step (step 0: none), its sum.
template <class T>
struct LaneSums {
  int32_t owner;
  int32_t src[2], first[2], step[2];
  T acc[2];
};

template <class T>
__device__ __forceinline__ void lane_deal(LaneSums<T> &s, LaneBuf &b, int32_t owner, uint32_t m0,
                                          uint32_t m1) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  s.owner = owner;
  if ((m0 >> lane) & 1u) b.lane_of[0][__popc(m0 & lt)] = (uint8_t)lane;
  if ((m1 >> lane) & 1u) b.lane_of[1][__popc(m1 & lt)] = (uint8_t)(lane + 32);
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int32_t a = __popc(h ? m1 : m0);
    // 32 / a and lane / a, exact for these sizes
    const float r = __frcp_rn((float)max(a, 1));
    const int32_t groups = (int32_t)(32.5f * r), g = (int32_t)(((float)lane + 0.5f) * r);
    s.src[h] = a ? b.lane_of[h][lane - g * a] : 0;
    s.first[h] = g < groups ? g : 32;  // a left-over thread: no edge
    s.step[h] = a ? groups : 0;
    s.acc[h] = T(0);
  }
}

// One window: lane i's edge (owner, u) with `bits` (0: no edge) of v's lanes
// `of` (the same for all of v's edges). flush(s) takes a vertex's sums.
template <class T, class FLUSH>
__device__ __forceinline__ void lane_window(LaneSums<T> &s, LaneBuf &b, int32_t owner, int32_t u,
                                            unsigned long long bits, unsigned long long of,
                                            const T *val, FLUSH flush) {
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t act = __ballot_sync(0xffffffffu, bits != 0ull);
  while (act) {  // warp-uniform
    const int j0 = __ffs(act) - 1;
    const int32_t ov = __shfl_sync(0xffffffffu, owner, j0);
    const uint32_t seg = __ballot_sync(0xffffffffu, owner == ov) & act;
    act &= ~seg;
    const bool mine = (seg >> lane) & 1u;
    __syncwarp();  // the buffer's last readers are done
    if (ov != s.owner) {
      if (s.owner >= 0) flush(s);
      lane_deal(s, b, ov, __shfl_sync(0xffffffffu, (uint32_t)of, j0),
                __shfl_sync(0xffffffffu, (uint32_t)(of >> 32), j0));
    }
    if (mine) {
      const int k = __popc(seg & lt);
      b.u[k] = u;
      b.bits[0][k] = (uint32_t)bits;
      b.bits[1][k] = (uint32_t)(bits >> 32);
    }
    __syncwarp();
    const int cnt = __popc(seg);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int step = s.step[h];
      if (!step) continue;  // warp-uniform
      const int bit = s.src[h] & 31;
      for (int base = 0; base < cnt; base += 4 * step) {
        T x[4];
        bool has[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int j = base + k * step + s.first[h];
          has[k] = j < cnt && ((b.bits[h][j & 31] >> bit) & 1u);
          x[k] = has[k] ? val[(int64_t)b.u[j & 31] * 64 + s.src[h]] : T(0);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (base + k * step < cnt && has[k]) s.acc[h] += x[k];
      }
    }
  }
}

// A BC forward pull level: nxt[v] = OR over edges (v,u) of cur[u] &
// ~seen(v), seen(v) = visit[v] | cur[v], and the path counts of the newly
// reached lanes. The vertex loader of each chunk folds cur into visit
// (idempotent, so chunks sharing a vertex may both do it). Lane l of a warp
// counts for the sources l and l + 32: uint64 adds cost little, so the edges
// with bits are served one by one by all lanes, but four at a time, the rows of
// all four loaded before any is added (dealing the threads to the lanes in
// use, as the backward does, was slower: 1.79 against 1.48 ms on R-MAT 2^18
// with 64 sources, before the chunks became the warps' own).
template <int SK, class SMEM>
__device__ void mb_forward_level(const MbArgs &a, SMEM &sm, const unsigned long long *cur,
                                 unsigned long long *nxt, unsigned long long *counter, bool &ovf) {
  using T = CountT<SK>;
  const int lane = threadIdx.x & 31;
  const long long total = (long long)a.n + a.R[a.n];
  const long long nchunks = (total + kMbWarpChunk - 1) / kMbWarpChunk;
  unsigned long long new_vertices = 0;
  T *const sigma = (T *)a.sigma;
  int32_t *off = sm.fwd[threadIdx.x >> 5].off;
  unsigned long long *U = sm.fwd[threadIdx.x >> 5].U;
  // the vertex being summed, its lanes so far, its counts
  int32_t sum_of = -1;
  uint32_t got0 = 0u, got1 = 0u;
  T a0 = T(0), a1 = T(0);
  auto flush = [&]() {
    if (sum_of < 0) return;
    T *sg = sigma + (int64_t)sum_of * 64 + lane;
    if ((got0 >> lane) & 1u) count_atomic_add(sg, a0, ovf);
    if ((got1 >> lane) & 1u) count_atomic_add(sg + 32, a1, ovf);
    if (lane == 0 && !atomicOr(nxt + sum_of, ((unsigned long long)got1 << 32) | got0))
      new_vertices += joined(a, sum_of);
  };
  const long long warps = (long long)gridDim.x * (kMbThreads / 32);
  for (long long chunk = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; chunk < nchunks;
       chunk += warps) {
    const long long d0 = chunk * kMbWarpChunk;
    const long long d1 = min(d0 + kMbWarpChunk, total);
    const int32_t i0 = a.cb_fwd[chunk], i1 = a.cb_fwd[chunk + 1];
    const long long j0 = d0 - i0, j1 = d1 - i1;
    const int32_t nv = (i0 <= a.n - 1) ? (min(i1, a.n - 1) - i0 + 1) : 0;
    bool any = false;
    for (int32_t kk = lane; kk < nv; kk += 32) {
      const int32_t v = i0 + kk;
      const unsigned long long c = cur[v];
      const unsigned long long seen = a.visit[v] | c;
      if (c) a.visit[v] = seen;
      off[kk] = a.R[v];
      U[kk] = a.all & ~seen;
      any |= (a.all & ~seen) != 0ull;
    }
    if (!__any_sync(0xffffffffu, any)) continue;  // every lane of these vertices is there
    __syncwarp();
    const int32_t ne = (int32_t)(j1 - j0);
    for (int32_t kb = 0; kb < ne; kb += 32) {
      const int32_t kk = kb + lane;
      int32_t owner = -1, u = 0;
      uint32_t lo = 0u, hi = 0u;
      if (kk < ne) {
        const int32_t e = (int32_t)(j0 + kk);
        int32_t k = 0, top = nv - 1;
        while (k < top) {
          const int32_t mid = (k + top + 1) >> 1;
          if (off[mid] <= e) k = mid;
          else top = mid - 1;
        }
        const unsigned long long miss = U[k];
        if (miss && GR_IN(i0 + k, a.n, 201) && GR_IN(e, a.m, 202)) {
          owner = i0 + k;
          u = a.C[e];
          const unsigned long long bits = GR_IN(u, a.n, 203) ? (cur[u] & miss) : 0ull;
          lo = (uint32_t)bits;
          hi = (uint32_t)(bits >> 32);
        }
      }
      uint32_t act = __ballot_sync(0xffffffffu, (lo | hi) != 0u);
      while (act) {  // warp-uniform: one owner's edges at a time
        const int32_t ov = __shfl_sync(0xffffffffu, owner, __ffs(act) - 1);
        uint32_t seg = __ballot_sync(0xffffffffu, owner == ov) & act;
        act &= ~seg;
        if (ov != sum_of) {
          flush();
          sum_of = ov;
          got0 = got1 = 0u;
          a0 = a1 = T(0);
        }
        while (seg) {
          uint32_t l[4], h[4];
          T x[4], y[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const bool has = seg != 0u;
            const int j = has ? __ffs(seg) - 1 : 0;
            seg &= seg - 1u;
            const int32_t uj = __shfl_sync(0xffffffffu, u, j);
            l[k] = __shfl_sync(0xffffffffu, lo, j);
            h[k] = __shfl_sync(0xffffffffu, hi, j);
            if (!has) l[k] = h[k] = 0u;
            const T *su = sigma + (int64_t)uj * 64 + lane;
            x[k] = (l[k] >> lane) & 1u ? su[0] : T(0);
            y[k] = (h[k] >> lane) & 1u ? su[32] : T(0);
          }
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            got0 |= l[k];
            got1 |= h[k];
            if (l[k]) a0 = count_add(a0, x[k], ovf);  // warp-uniform
            if (h[k]) a1 = count_add(a1, y[k], ovf);
          }
        }
      }
    }
    __syncwarp();  // the tables are reused
  }
  flush();
  for (int o = 16; o > 0; o >>= 1) new_vertices += __shfl_xor_sync(0xffffffffu, new_vertices, o);
  if (lane == 0 && new_vertices) atomicAdd(counter, new_vertices);
}

// A push level, for levels whose list has few edges (the sources' level,
// the last levels, every level of a mesh): the listed vertices send their
// lanes over their edges (merge-path chunks over the list's degree scan).
// For an edge (u, v): bits = cur[u] & ~seen(v), seen(v) = visit[v] | cur[v]
// (v may be on the list itself, its cur not yet folded into visit), and
// nxt[v] |= bits; with SIGMA (BC's forward pass) those lanes also add u's
// path counts to v's, the warp serving such edges one at a time. The
// loader folds each listed vertex's cur into visit and, past the kept
// levels, writes its depths.
template <int SK, class SMEM>
__device__ void mb_push_level(const MbArgs &a, SMEM &sm, int32_t *s_red8, int32_t L,
                              const unsigned long long *cur,
                              unsigned long long *nxt, const int32_t *Q, const int32_t *S,
                              int32_t q, int32_t qe, int32_t *Qn, int32_t *Sn,
                              unsigned long long *counter, bool &ovf) {
  constexpr bool SIGMA = SK != kSigNone;
  using T = CountT<SK == kSigNone ? kSigU64 : SK>;
  const bool write_depth = a.depth && L >= a.keep;
  const int lane = threadIdx.x & 31;
  const long long total = (long long)q + qe;
  constexpr int CHUNK = SMEM::kChunk;
  const long long nchunks = (total + CHUNK - 1) / CHUNK;
  // the emission buffer shares its storage with the other level forms: its
  // count starts at zero here
  if (threadIdx.x == 0) sm.push.em.cnt = 0;
  __syncthreads();
  for (long long chunk = blockIdx.x; chunk < nchunks; chunk += gridDim.x) {
    const long long d0 = chunk * CHUNK;
    const long long d1 = min(d0 + CHUNK, total);
    int32_t i0, i1;
    block_chunk_bounds<kMbThreads>(S, q, qe, d0, d1, CHUNK, s_red8, &i0, &i1);
    const long long j0 = d0 - i0, j1 = d1 - i1;
    const int32_t nv = (i0 <= q - 1) ? (min(i1, q - 1) - i0 + 1) : 0;
    for (int32_t k = threadIdx.x; k < nv; k += kMbThreads) {
      const int32_t i = i0 + k;
      const int32_t u = GR_IN(i, a.n + 1, 207) ? Q[i] : 0;
      const bool ok = GR_IN(u, a.n, 208);
      const unsigned long long c = ok ? cur[u] : 0ull;
      if (c) {
        a.visit[u] |= c;
        if (write_depth) mb_write_depth(a, u, c, L);
      }
      sm.push.off[k] = S[i];
      sm.push.row[k] = ok ? a.R[u] : 0;
      sm.push.cur[k] = c;
      if (SIGMA) sm.push.u[k] = ok ? u : 0;
    }
    __syncthreads();
    const int32_t ne = (int32_t)(j1 - j0);
    for (int32_t kb = 0; kb < ne; kb += kMbThreads) {
      const int32_t k = kb + threadIdx.x;
      unsigned long long bits = 0ull;
      int32_t v = -1, u = 0;
      if (k < ne) {
        const int32_t er = (int32_t)(j0 + k);
        int32_t lo = 0, hi = nv - 1;
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (sm.push.off[mid] <= er) lo = mid;
          else hi = mid - 1;
        }
        const long long e = (long long)sm.push.row[lo] + (er - sm.push.off[lo]);
        v = GR_IN(e, a.m, 209) ? a.C[e] : -1;
        if (v >= 0 && GR_IN(v, a.n, 210)) {
          bits = sm.push.cur[lo] & ~(a.visit[v] | cur[v]);
          if (bits && !atomicOr(nxt + v, bits)) mb_emit(sm.push.em, a, v);
          if (SIGMA) u = sm.push.u[lo];
        }
      }
      if (SIGMA) {
        T *const sigma = (T *)a.sigma;
        uint32_t act = __ballot_sync(0xffffffffu, bits != 0ull);
        while (act) {
          const int j = __ffs(act) - 1;
          act &= act - 1u;
          const int32_t vj = __shfl_sync(0xffffffffu, v, j);
          const int32_t uj = __shfl_sync(0xffffffffu, u, j);
          const unsigned long long bj = shfl_u64(bits, j);
          const T *su = sigma + (int64_t)uj * 64;
          T *sv = sigma + (int64_t)vj * 64;
          if ((bj >> lane) & 1ull) count_atomic_add(sv + lane, su[lane], ovf);
          if ((bj >> (lane + 32)) & 1ull) count_atomic_add(sv + lane + 32, su[lane + 32], ovf);
        }
      }
    }
    flush_scanned<kMbThreads>(sm.push.em, counter, Qn, Sn, (long long)a.n + 1);
  }
}

// The list of a level reached by a pull (the vertices with lanes in cur,
// with their degree scan), for the push level that expands it.
template <class SMEM>
__device__ void mb_compact_list(const MbArgs &a, SMEM &sm, const unsigned long long *cur,
                                int32_t *Q, int32_t *S, unsigned long long *counter) {
  constexpr int CHUNK = SMEM::kChunk, PER = CHUNK / kMbThreads;
  // the list buffer shares its storage with the level forms: its count
  // starts at zero here
  if (threadIdx.x == 0) sm.list.cnt = 0;
  __syncthreads();
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < a.n;
       base += (int64_t)gridDim.x * CHUNK) {  // block-uniform
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int64_t v = base + j * kMbThreads + threadIdx.x;
      const bool take = v < a.n && cur[v] != 0ull;
      emit_scanned(sm.list, take, (int32_t)v, take ? a.R[v + 1] - a.R[v] : 0);
    }
    flush_scanned<kMbThreads>(sm.list, counter, Q, S, (long long)a.n + 1);
  }
}

// Depths of the kept levels [0, levels) from their lane masks, written once
// for every (lane, vertex), in full coalesced rows: for each lane s,
// depth[s][v] = the level L whose mask holds bit s (-1 if none). The masks
// of one vertex are disjoint, so the level of every lane follows from bit
// slices: slice j is the OR of the masks of the levels whose index has bit j
// set.
template <int SLICES>
__device__ void mb_depth_slices(const MbArgs &a, int32_t levels) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < a.n; v += stride) {
    unsigned long long b[SLICES], reached = 0ull;
#pragma unroll
    for (int j = 0; j < SLICES; ++j) b[j] = 0ull;
    for (int32_t L = 0; L < levels; ++L) {
      const unsigned long long m = a.lmp[L][v];
      reached |= m;
#pragma unroll
      for (int j = 0; j < SLICES; ++j)
        if ((L >> j) & 1) b[j] |= m;
    }
    int32_t *out = a.depth + v;
    for (int32_t s = 0; s < a.k; ++s, out += a.n) {
      int32_t d = 0;
#pragma unroll
      for (int j = 0; j < SLICES; ++j) d |= (int32_t)((b[j] >> s) & 1ull) << j;
      *out = (reached >> s) & 1ull ? d : -1;
    }
  }
}

__device__ __forceinline__ void mb_depth_pass(const MbArgs &a, int32_t levels) {
  static_assert(kKeepLevels <= 16, "four slices");
  if (levels <= 8) mb_depth_slices<3>(a, levels);
  else mb_depth_slices<4>(a, levels);
}

// Most blocks per SM of k_mb_do: 48 registers a thread for the batched BFS, 64
// for BC's forward.
template <int SK>
constexpr int mb_do_blocks_per_sm() { return SK == kSigNone ? 5 : 4; }

// The forward levels in one cooperative kernel. Every block runs every
// level; levels are separated by one bounded grid barrier, after which each
// block reads the level's packed counter (published with the release on
// large grids) and takes the same decisions: stop when no vertex joined,
// push when the next level's vertices have fewer than m / kPushDiv edges
// (or the graph is directed), else pull. A push level expands the list of
// its level (emitted by the push before it, or compacted from the masks
// after a pull, which writes no list). Lane-mask arrays: the one of level
// L + 2 is cleared while level L runs (all of it for a kept level, an
// array's first use in this run or when level L - 1, its last user, has no
// list; otherwise only the entries on that list). The kernel stops before a
// level whose arrays are not allocated (BC only) and records where;
// launched again, it resumes.
// Loop state of k_mb_do, the same in every block; kept in shared memory so
// that the level bodies have the registers to themselves.
struct MbLoop {
  int32_t L, push, q, qe, q_prev, listed, prev_listed;
};

// PULL: the graph is symmetric (else every level pushes)
template <int SK, bool PULL = true>
__global__ void __launch_bounds__(kMbThreads, mb_do_blocks_per_sm<SK>()) k_mb_do(MbArgs a) {
  MbCtl *c = a.ctl;
  __shared__ MbSmem<PULL ? kMbItems : kMbPushOnlyItems> sm;
  __shared__ int32_t s_red8[kMbThreads / 32];
  __shared__ MbLoop st;
  if (threadIdx.x == 0) {
    st.L = c->level;
    st.push = c->push;
    st.q = c->q;
    st.qe = c->qe;
    st.q_prev = c->q_prev;
    st.listed = c->listed;
    st.prev_listed = c->prev_listed;
  }
  __syncthreads();
  if (c->done) return;
  int32_t gen = 0;
  bool ovf = false;
  for (;;) {
    const int32_t L = st.L;
    if (mb_slot(a, L + 1) >= a.cap || (L + 2 < a.keep && L + 2 >= a.cap)) {
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->level = L;
        c->push = st.push;
        c->q = st.q;
        c->qe = st.qe;
        c->q_prev = st.q_prev;
        c->listed = st.listed;
        c->prev_listed = st.prev_listed;
        c->paused = 1;
      }
      break;
    }
    if (a.depth && a.keep > 0 && L == a.keep) {
      // every kept level is complete: their depths first, then the later
      // levels' writes
      mb_depth_pass(a, a.keep);
      if (!grid_sync(&c->bar, &c->error, gen)) break;
    }
    const unsigned long long *cur = a.lmp[mb_slot(a, L)];
    unsigned long long *nxt = a.lmp[mb_slot(a, L + 1)];
    if (PULL && st.push && !st.listed) {
      mb_compact_list(a, sm, cur, a.lq[L % 3], a.ls[L % 3], &c->cnt_list);
      if (!grid_sync(&c->bar, &c->error, gen)) break;
      if (threadIdx.x == 0) st.listed = 1;
      if (blockIdx.x == 0 && threadIdx.x == 0) c->cnt_list = 0ull;  // next use: a barrier later
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) c->cnt3[(L + 2) % 3] = 0ull;
    {
      const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
      const int64_t stride = (int64_t)gridDim.x * blockDim.x;
      const int32_t s2 = mb_slot(a, L + 2);
      if (s2 < a.cap) {
        unsigned long long *clr = a.lmp[s2];
        if (L - 1 < a.keep || !st.prev_listed) {
          for (int64_t v = tid; v < a.n; v += stride) clr[v] = 0ull;
        } else {
          const int32_t *Qp = a.lq[(L + 2) % 3];  // level L - 1's list
          for (int64_t i = tid; i < st.q_prev; i += stride) {
            const int32_t v = Qp[i];
            if (GR_IN(v, a.n, 211)) clr[v] = 0ull;
          }
        }
      }
    }
    unsigned long long *counter = &c->cnt3[(L + 1) % 3];
    if (!PULL || st.push) {
      mb_push_level<SK>(a, sm, s_red8, L, cur, nxt, a.lq[L % 3], a.ls[L % 3], st.q, st.qe,
                        a.lq[(L + 1) % 3], a.ls[(L + 1) % 3], counter, ovf);
    } else if (SK == kSigNone) {
      mb_pull_fold(a, L, cur);
      if (!grid_sync(&c->bar, &c->error, gen)) break;
      mb_pull_gather(a, cur, nxt, counter);
    } else {
      mb_forward_level<SK == kSigNone ? kSigU64 : SK>(a, sm, cur, nxt, counter, ovf);
    }
    unsigned long long pk = 0ull;
    if (gridDim.x > kFlatBarrierBlocks) {
      if (!grid_sync(&c->bar, &c->error, gen, counter, &pk)) break;
    } else {
      if (!grid_sync(&c->bar, &c->error, gen)) break;
      pk = *(volatile unsigned long long *)counter;
    }
    // grid_sync ends with a block barrier: every thread has read st
    const int32_t qn = (int32_t)(pk & 0xFFFFFFFFull);
    const long long en = (long long)(pk >> 32);
    const int32_t levels = L + 1;  // levels 0 .. L hold vertices
    const bool done = qn == 0;
    const bool overflow = !done && levels >= a.max_levels;
    if (done || overflow) {
      if (done && a.depth && a.keep > 0 && levels <= a.keep) mb_depth_pass(a, levels);
      if (blockIdx.x == 0 && threadIdx.x == 0) {
        c->level = levels;
        c->levels = levels;
        c->q = 0;
        if (overflow) c->error = kDevOverflow;
        c->done = 1;
      }
      break;
    }
    if (threadIdx.x == 0) {
      st.prev_listed = st.listed;
      st.listed = st.push;  // a push emitted the next level's list
      st.L = levels;
      st.q_prev = st.q;
      st.q = qn;
      st.qe = (int32_t)en;
      st.push = (!a.symmetric || en * kPushDiv < a.m) ? 1 : 0;
    }
    __syncthreads();
  }
  if (SK == kSigU64 && __any_sync(0xffffffffu, ovf) && (threadIdx.x & 31) == 0)
    atomicOr(&c->sig_overflow, 1);
}

struct BcBackArgs {
  const int32_t *R;
  const int32_t *C;
  int32_t n;
  long long m;
  const unsigned long long *lv;   // lm[L]
  const unsigned long long *lw;   // lm[L+1]
  double *q;                      // [n][64]
};

// Items per warp of the backward pass over a list of `total` items: kMbWarpChunk,
// and fewer where that would leave three quarters of the warps without a chunk
// (with all of them busy the chunks' own cost shows: R-MAT of 0.1 M vertices 1275
// us, 1263 so). A warp serves the
// vertices of its chunk one after another, each with the latency of its
// children's rows: a level of 32 vertices with two edges each took 18.7 us in
// one warp (a path of 1000 vertices, 16 sources: 46.3 ms; 39.4 with 512 items to a
// block of eight warps).
__device__ __forceinline__ int32_t list_chunk(long long total, int32_t warps) {
  const long long share = (4 * total + warps - 1) / warps;
  return (int32_t)min((long long)kMbWarpChunk, (share + 7) / 8 * 8);
}

// Chunk bounds of a level list's merge path, the list's size and edge count
// read from *fpacked (its scan S[0..q) does not store S[q]): cb[c] = the
// members whose end marker S[i + 1] + i lies before c * list_chunk,
// cb[nchunks] = q. One thread per chunk; threads past the list's chunks
// return. warps: those of the backward pass.
__global__ void k_list_bounds(const int32_t *S, const unsigned long long *fpacked, int32_t warps,
                              int32_t *cb) {
  const unsigned long long fp = *fpacked;
  const int32_t q = (int32_t)(fp & 0xFFFFFFFFull);
  const int32_t qe = (int32_t)(fp >> 32);
  const int32_t chunk = list_chunk((long long)q + qe, warps);
  if (chunk == 0) return;  // an empty list
  const long long nchunks = ((long long)q + qe + chunk - 1) / chunk;
  const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (c > nchunks) return;
  if (c == nchunks) {
    cb[c] = q;
    return;
  }
  const long long d = c * chunk;
  int32_t lo = 0, hi = q;  // first member whose end marker is not before d
  while (lo < hi) {
    const int32_t mid = (int32_t)(((long long)lo + hi) >> 1);
    const int32_t sv = mid + 1 == q ? qe : S[mid + 1];
    if ((long long)sv + mid < d) lo = mid + 1;
    else hi = mid;
  }
  cb[c] = lo;
}

// resident blocks per SM of the backward pass (its carveout is fitted to
// them, the rest of the shared-memory array left to L1 for the children's rows)
constexpr int kBcBackBlocksPerSm = 4;

// Backward level L: q[v][s] += q[w][s] over edges (v, w) with v in lane s's
// level L and w in its level L+1 (w's q is final: level L+1 was finished).
// Only the vertices of level L (listed with their degrees by k_mb_list) are
// visited, so the whole backward pass reads every edge about once instead of
// once per level.

struct BcBackWarp {  // a warp's chunk: its vertices' list scan, row starts, ids, lanes
  int32_t off[kMbWarpChunk + 1];
  int32_t row[kMbWarpChunk + 1];
  int32_t v[kMbWarpChunk + 1];
  unsigned long long A[kMbWarpChunk + 1];
  LaneBuf lanes;
};

__global__ void __launch_bounds__(kMbThreads, kBcBackBlocksPerSm) k_bc_backward(
    BcBackArgs a, const int32_t *Q, const int32_t *S, const unsigned long long *fpacked,
    const int32_t *cb) {
  __shared__ BcBackWarp s_warp[kMbThreads / 32];
  BcBackWarp &sm = s_warp[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const unsigned long long fp = *fpacked;
  const int32_t q = (int32_t)(fp & 0xFFFFFFFFull);
  const int32_t qe = (int32_t)(fp >> 32);
  const long long total = (long long)q + qe;
  const int32_t size = list_chunk(total, (int32_t)gridDim.x * (kMbThreads / 32));
  const long long nchunks = size ? (total + size - 1) / size : 0;
  auto flush = [&](const LaneSums<double> &s) {
    double *qv = a.q + (int64_t)s.owner * 64;
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (s.acc[h] != 0.0) atomicAdd(qv + s.src[h], s.acc[h]);
  };
  LaneSums<double> sums = {};
  sums.owner = -1;
  const long long warps = (long long)gridDim.x * (kMbThreads / 32);
  for (long long chunk = (long long)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; chunk < nchunks;
       chunk += warps) {
    const long long d0 = chunk * size;
    const long long d1 = min(d0 + size, total);
    const int32_t i0 = cb[chunk], i1 = cb[chunk + 1];  // k_list_bounds
    const long long j0 = d0 - i0, j1 = d1 - i1;
    const int32_t nv = (i0 <= q - 1) ? (min(i1, q - 1) - i0 + 1) : 0;
    for (int32_t k = lane; k < nv; k += 32) {
      const int32_t i = i0 + k;
      const int32_t v = GR_IN(i, a.n + 1, 220) ? Q[i] : 0;
      const bool ok = GR_IN(v, a.n, 221);
      sm.off[k] = S[i];
      sm.v[k] = ok ? v : -1;
      sm.row[k] = ok ? a.R[v] : 0;
      sm.A[k] = ok ? a.lv[v] : 0ull;
    }
    __syncwarp();
    const int32_t ne = (int32_t)(j1 - j0);
    for (int32_t kb = 0; kb < ne; kb += 32) {
      const int32_t k = kb + lane;
      int32_t owner = -1, w = 0;
      unsigned long long bits = 0ull, A = 0ull;
      if (k < ne) {
        const int32_t er = (int32_t)(j0 + k);
        int32_t lo = 0, hi = nv - 1;
        while (lo < hi) {
          const int32_t mid = (lo + hi + 1) >> 1;
          if (sm.off[mid] <= er) lo = mid;
          else hi = mid - 1;
        }
        owner = sm.v[lo];
        const long long e = (long long)sm.row[lo] + (er - sm.off[lo]);
        A = sm.A[lo];
        if (owner >= 0 && A && GR_IN(e, a.m, 222)) {
          w = a.C[e];
          bits = GR_IN(w, a.n, 223) ? (A & a.lw[w]) : 0ull;
        }
      }
      __syncwarp();
      lane_window(sums, sm.lanes, owner, w, bits, A, (const double *)a.q, flush);
    }
    __syncwarp();  // the tables are reused
  }
  if (sums.owner >= 0) flush(sums);
}

// The vertices with lanes in `lv`, with their degree scan (block-wise
// compaction, one packed atomic per block). Vertices without edges are
// listed too (a directed graph reaches some): they have no children, but
// their dependencies still have to be finished. *next_packed, the counter of
// the level after this one, is cleared on the way.
__global__ void __launch_bounds__(kMbThreads) k_mb_list(const unsigned long long *lv,
                                                         const int32_t *R, int32_t n,
                                                         int32_t *Q, int32_t *S,
                                                         unsigned long long *fpacked,
                                                         unsigned long long *next_packed) {
  __shared__ ScannedBuf<kMbListChunk> buf;
  if (threadIdx.x == 0) buf.cnt = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) *next_packed = 0ull;
  __syncthreads();
  constexpr int PER = kMbListChunk / kMbThreads;
  for (int64_t base = (int64_t)blockIdx.x * kMbListChunk; base < n;
       base += (int64_t)gridDim.x * kMbListChunk) {  // block-uniform
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const int64_t v = base + j * kMbThreads + threadIdx.x;
      int32_t d = 0;
      bool take = false;
      if (v < n && lv[v]) {
        d = R[v + 1] - R[v];
        take = true;
      }
      emit_scanned(buf, take, (int32_t)v, d);
    }
    flush_scanned<kMbThreads>(buf, fpacked, Q, S, (long long)n + 1);
  }
}

// Finish level L: delta[v][s] = sigma[v][s] * q[v][s] (q holds the child
// sum), bc[v] += delta over the lanes of lm[L][v], then q[v][s] becomes
// 1/sigma + child sum for level L-1. The vertices of level L come listed by
// k_mb_list (Q[0..q), q in fpacked; a vertex of a level >= 1 has an edge).
// Lanes over s. A warp takes kFinItems vertices at a time where the level has
// them, their list entries and masks with one load each instead of two waits
// per vertex, and the rows of two in flight; the lanes' parts of four vertices
// are added up together, 9 steps instead of 20. Large levels are bound by
// instruction issue (over 100 FP32 instructions per lane and vertex), small
// ones by the waits. 64 sources on R-MAT 2^18: 253 us for the six levels, 396
// with a warp per vertex.
constexpr int kFinItems = 8;

// The four sums of part[j] over the warp: that of j = lane / 8.
template <typename T, typename ADD, typename XOR>
__device__ __forceinline__ T warp_sum4(const T (&part)[4], int lane, ADD add, XOR xshfl) {
  const bool up = lane & 16, odd = lane & 8;
  const T a0 = add(up ? part[2] : part[0], xshfl(up ? part[0] : part[2], 16));
  const T a1 = add(up ? part[3] : part[1], xshfl(up ? part[1] : part[3], 16));
  T s = add(odd ? a1 : a0, xshfl(odd ? a0 : a1, 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s = add(s, xshfl(s, o));
  return s;
}

template <int SK>
__global__ void __launch_bounds__(256) k_bc_finalize(
    const unsigned long long *lv, const int32_t *Q, const unsigned long long *fpacked,
    const void *sigma_p, double *q, double *bc, int32_t n, int32_t *overflow) {
  const int32_t gw = (int32_t)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int32_t nw = (int32_t)(((int64_t)gridDim.x * blockDim.x) >> 5);
  const int lane = threadIdx.x & 31;
  const CountT<SK> *sigma = (const CountT<SK> *)sigma_p;
  const int32_t nq = (int32_t)(*fpacked & 0xFFFFFFFFull);
  const int32_t items = min(kFinItems, (nq + nw - 1) / nw);
  for (int64_t i0 = (int64_t)gw * items; i0 < nq; i0 += (int64_t)nw * items) {  // warp-uniform
    int32_t my_v = -1;
    unsigned long long my_A = 0ull;
    if (lane < items && i0 + lane < nq) {
      my_v = Q[i0 + lane];
      if (GR_IN(my_v, n, 230)) my_A = lv[my_v];
    }
    double add = 0.0;  // lane j: what vertex j of the group gains
#pragma unroll 1
    for (int j0 = 0; j0 < items; j0 += 4) {
      using P = typename std::conditional<SK == kSigU64, DS, double>::type;
      P part[4] = {};
#pragma unroll
      for (int jj = 0; jj < 4; jj += 2) {
        unsigned long long A[2];
        int64_t at[2];
        double child[2][2];
        CountT<SK> cnt[2][2];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          A[j] = __shfl_sync(0xffffffffu, my_A, j0 + jj + j);
          at[j] = (int64_t)__shfl_sync(0xffffffffu, my_v, j0 + jj + j) * 64 + lane;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            child[j][h] = 0.0;
            cnt[j][h] = 0;
            if ((A[j] >> (lane + 32 * h)) & 1ull) {
              child[j][h] = q[at[j] + 32 * h];
              cnt[j][h] = sigma[at[j] + 32 * h];
            }
          }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if ((uint32_t)(A[j] >> (32 * h)) == 0u) continue;  // warp-uniform
            if (!((A[j] >> (lane + 32 * h)) & 1ull)) continue;
            if constexpr (SK == kSigU64) {
              // double-single: delta = sigma * (child sum), q = 1/sigma + child sum
              const unsigned long long c = (unsigned long long)cnt[j][h];
              if (c == 0ull) *overflow = 1;  // a reached lane has at least one path
              const DS ch = ds_from_double(child[j][h]);
              const DS sg = ds_from_u64(c);
              part[jj + j] = ds_add(part[jj + j], ds_mul(sg, ch));
              q[at[j] + 32 * h] = ds_to_double(ds_add(ds_rcp(sg), ch));
            } else {
              const double sg = (double)cnt[j][h];
              if (!isfinite(sg) || sg <= 0.0) *overflow = 1;
              part[jj + j] = fma(sg, child[j][h], part[jj + j]);
              q[at[j] + 32 * h] = 1.0 / sg + child[j][h];
            }
          }
        }
      }
      double gain;
      if constexpr (SK == kSigU64)
        gain = ds_to_double(warp_sum4(part, lane, [](DS x, DS y) { return ds_add(x, y); },
                                      [](DS x, int o) { return shfl_xor_ds(x, o); }));
      else
        gain = warp_sum4(part, lane, [](double x, double y) { return x + y; },
                         [](double x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); });
      gain = __shfl_sync(0xffffffffu, gain, (lane & 3) * 8);
      if ((lane & ~3) == j0) add = gain;
    }
    if (my_A) bc[my_v] += add;
  }
}

__global__ void k_fill_f64(double *x, int64_t n, double val) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    x[i] = val;
}

// Before k_mb_do runs again after it stopped for more level arrays: a fresh
// barrier (its generation restarts with every launch).
__global__ void k_mb_resume(MbCtl *c) {
  grid_barrier_reset(&c->bar);
  c->paused = 0;
}

}  // namespace

// Levels of a batched BFS kept in their own mask arrays on this graph.
static int32_t bfs_keep_levels(const gr_graph *g) {
  return g->max_degree <= kLowDegreeMax ? 0 : kKeepLevels;
}

size_t batch_ws_bytes(const gr_graph *g) {
  // visit masks, the level arrays of a batched BFS, the level lists
  const size_t n = (size_t)g->n;
  return sizeof(unsigned long long) * n * (1 + bfs_keep_levels(g) + 3) +
         3 * sizeof(int32_t) * (2 * n + 3) + sizeof(MbCtl) + 4096 +
         (g->symmetric ? gather_plan_bytes(g->n, g->m) + n / 8 + 4 * ((n + (size_t)g->m) / kMbWarpChunk)
                       : 0);
}

gr_status batch_ws_create(gr_graph *g, BatchWorkspace **out) {
  std::unique_ptr<BatchWorkspace> ws(new BatchWorkspace());
  GR_TRY(ws->visit.alloc(sizeof(unsigned long long) * (size_t)g->n, "lane visit masks"));
  GR_TRY(ws->counter.alloc(sizeof(unsigned long long) * 4, "batch counters"));
  GR_TRY(ws->ctl.alloc(sizeof(MbCtl), "batch control"));
  if (g->symmetric) {  // else no level pulls
    GR_TRY(gather_plan_build(&ws->plan, g->row_off.as<int32_t>(), g->n, g->m, 0));
    GR_TRY(ws->full.alloc(sizeof(uint32_t) * (size_t)g->nwords, "batch full vertices"));
    // BC's merge path over all vertices is the same on every level: its chunk
    // bounds are found once
    const int32_t *R = g->row_off.as<int32_t>();
    const int32_t cf = merge_chunks(g->n, g->m, kMbWarpChunk);
    GR_TRY(ws->cb_fwd.alloc(sizeof(int32_t) * ((size_t)cf + 1), "BC pull chunk bounds"));
    k_chunk_bounds<<<(cf + 256) / 256, 256>>>(R, g->n, kMbWarpChunk, cf, ws->cb_fwd.as<int32_t>());
    GR_CUDA(cudaGetLastError());
    GR_CUDA(cudaStreamSynchronize(0));
  }
  for (int i = 0; i < 3; ++i) {
    GR_TRY(ws->lq[i].alloc(sizeof(int32_t) * ((size_t)g->n + 1), "batch level list"));
    GR_TRY(ws->ls[i].alloc(sizeof(int32_t) * ((size_t)g->n + 2), "batch level list scan"));
  }
  *out = ws.release();
  return GR_OK;
}

// Most merge-path chunks a BC level list can have: those of all n vertices and
// m edges, or one for every warp of the backward pass (list_chunk).
static long long bc_list_max_chunks(const gr_graph *g) {
  return std::max<long long>(((long long)g->n + g->m) / kMbWarpChunk + 1,
                             (long long)g->num_sms * kBcBackBlocksPerSm * (kMbThreads / 32));
}

static gr_status ensure_batch_ws(gr_graph *g, BatchWorkspace **slot, bool need_bc) {
  if (!*slot) GR_TRY(batch_ws_create(g, slot));
  BatchWorkspace *ws = *slot;
  if (need_bc && !ws->sigma.p) {
    GR_TRY(ws->sigma.alloc(sizeof(double) * 64 * (size_t)g->n, "BC path counts"));
    GR_TRY(ws->q.alloc(sizeof(double) * 64 * (size_t)g->n, "BC dependencies"));
  }
  if (need_bc && !ws->fq.p) {
    GR_TRY(ws->fq.alloc(sizeof(int32_t) * ((size_t)g->n + 1), "BC level list"));
    GR_TRY(ws->fs.alloc(sizeof(int32_t) * ((size_t)g->n + 2), "BC level list scan"));
    GR_TRY(ws->fcb.alloc(sizeof(int32_t) * (size_t)(bc_list_max_chunks(g) + 1),
                         "BC level list chunk bounds"));
  }
  return GR_OK;
}

// At least `slots` level mask arrays, their device pointers in lmp. New
// arrays are zeroed on `s` (the forward clears the arrays it reuses itself).
static gr_status ensure_slots(gr_graph *g, BatchWorkspace *ws, int32_t slots, cudaStream_t s) {
  const size_t bytes = sizeof(unsigned long long) * (size_t)g->n;
  if ((int32_t)ws->lm.size() < slots) {
    // the old table may still be read by enqueued work
    GR_CUDA(cudaStreamSynchronize(s));
    while ((int32_t)ws->lm.size() < slots) {
      std::unique_ptr<DevMem> m(new DevMem());
      GR_TRY(m->alloc(bytes, "level lane masks"));
      GR_CUDA(cudaMemsetAsync(m->p, 0, bytes, s));
      ws->lm.push_back(m.release());
    }
  }
  if (ws->uploaded < slots || !ws->lmp.p) {
    const int32_t cap = (int32_t)ws->lm.size();
    std::vector<unsigned long long *> ptrs(cap);
    for (int32_t i = 0; i < cap; ++i) ptrs[i] = ws->lm[i]->as<unsigned long long>();
    if (ws->lmp.bytes < sizeof(void *) * (size_t)cap) {
      GR_CUDA(cudaStreamSynchronize(s));
      GR_TRY(ws->lmp.alloc(sizeof(void *) * (size_t)std::max<int32_t>(cap, 64), "level mask table"));
    }
    // pageable source: staged before the call returns, copied in stream order
    GR_CUDA(cudaMemcpyAsync(ws->lmp.p, ptrs.data(), sizeof(void *) * (size_t)cap,
                            cudaMemcpyHostToDevice, s));
    ws->uploaded = cap;
  }
  return GR_OK;
}

static MbArgs mb_args(gr_graph *g, BatchWorkspace *ws, int32_t k, int32_t *depth, int32_t keep,
                      int32_t max_levels, bool with_sigma) {
  MbArgs a;
  std::memset(&a, 0, sizeof(a));
  a.R = g->row_off.as<int32_t>();
  a.C = g->col.as<int32_t>();
  a.n = g->n;
  a.m = g->m;
  a.all = k == 64 ? ~0ull : ((1ull << k) - 1ull);
  a.visit = ws->visit.as<unsigned long long>();
  a.lmp = (unsigned long long *const *)ws->lmp.p;
  a.cap = (int32_t)ws->lm.size();
  a.keep = keep;
  for (int i = 0; i < 3; ++i) {
    a.lq[i] = ws->lq[i].as<int32_t>();
    a.ls[i] = ws->ls[i].as<int32_t>();
  }
  a.sigma = with_sigma ? ws->sigma.p : nullptr;
  a.depth = depth;
  a.k = k;
  a.symmetric = g->symmetric ? 1 : 0;
  a.max_levels = max_levels;
  a.ctl = ws->ctl.as<MbCtl>();
  a.plan = ws->plan.a;
  a.full = ws->full.as<uint32_t>();
  a.cb_fwd = ws->cb_fwd.as<int32_t>();
  return a;
}

static gr_status mb_launch(gr_graph *g, const MbArgs &a, int sk, cudaStream_t s) {
  void *kern = sk == kSigU64   ? (void *)k_mb_do<kSigU64>
               : sk == kSigF64 ? (void *)k_mb_do<kSigF64>
               : !g->symmetric && g->m >= kMbPushOnlyM ? (void *)k_mb_do<kSigNone, false>
                                                       : (void *)k_mb_do<kSigNone>;
  // small graphs are bound by the grid barrier, which costs more the more
  // blocks meet at it. Batched BFS at 1 to 5 blocks per SM, 20 lanes: R-MAT
  // 34,000 entries 81, 88, 92, 97, 99 us; 0.24 M 81, 93, 95, 101, 102; 0.64 M
  // 115, 112, 111, 114, 119; 1.1 M 133, 116, 115, 112, 115; 2.5 M 174, 138,
  // 131, 130, 132; 32 lanes 5.7 M 347, 250, 222, 209, 216; 64 lanes 15 M 744,
  // 474, 400, 366, 346. Directed, 64 lanes: 0.13 M 112, 111, 117, 120, 127;
  // 0.34 M 150, 129, 115, 120, 115; 1.3 M 337, 224, 187, 180, 173. BC at 1 to
  // 4: 40,000 entries 490, 505, 500, 518; 0.24 M 558, 491, 499, 499; 0.65 M
  // 619, 539, 501, 476.
  int want;
  if (sk != kSigNone) want = g->m < 100'000 ? 1 : g->m < 500'000 ? 2 : mb_do_blocks_per_sm<kSigU64>();
  else if (!g->symmetric) want = g->m < 300'000 ? 2 : mb_do_blocks_per_sm<kSigNone>();
  else want = g->m < 400'000 ? 1 : g->m < 900'000 ? 3 : g->m < 10'000'000 ? 4 : mb_do_blocks_per_sm<kSigNone>();
  int per_sm = 1;
  GR_TRY(fit_carveout(kern, kMbThreads, want, g->device, &per_sm));
  const int blocks = per_sm * g->num_sms;
  MbArgs arg = a;
  void *args[] = {&arg};
  GR_CUDA(cudaLaunchCooperativeKernel(kern, blocks, kMbThreads, args, 0, s));
  return GR_OK;
}

// Forward levels of one batch of k <= 64 sources (device-driven), counting
// paths as `sk` says. A batched BFS (depth != null) has every array it can
// need before it starts and never synchronises; BC (levels_out != null)
// keeps every level's array, so the kernel may stop for more and is
// resumed, and the call synchronises to report the level count and
// whether a uint64 path count overflowed.
static gr_status run_forward(gr_graph *g, BatchWorkspace *ws, const int32_t *h_srcs, int32_t k,
                             int32_t *depth, int sk, cudaStream_t s, int32_t max_levels,
                             int32_t *levels_out = nullptr, bool *overflowed = nullptr) {
  const bool with_sigma = sk != kSigNone;
  const int32_t keep = with_sigma ? INT32_MAX : bfs_keep_levels(g);
  GR_TRY(ensure_slots(g, ws, with_sigma ? std::max<int32_t>(16, (int32_t)ws->lm.size())
                                        : keep + 3, s));
  MbArgs a = mb_args(g, ws, k, depth, keep, max_levels, with_sigma);
  const int grid = g->num_sms * 8;
  k_mb_init<<<grid, 256, 0, s>>>(a, with_sigma ? ws->sigma.as<unsigned long long>() : nullptr,
                                 with_sigma ? ws->q.as<double>() : nullptr);
  MbSources src;  // by value: no host-to-device copy
  for (int32_t i = 0; i < 64; ++i) src.s[i] = i < k ? h_srcs[i] : 0;
  k_mb_sources<<<1, 64, 0, s>>>(a, src, sk);
  GR_CUDA(cudaGetLastError());
  GR_TRY(mb_launch(g, a, sk, s));
  if (!levels_out) return GR_OK;
  for (;;) {
    MbCtl h;
    GR_CUDA(cudaMemcpyAsync(&h, ws->ctl.p, sizeof(MbCtl), cudaMemcpyDeviceToHost, s));
    GR_CUDA(cudaStreamSynchronize(s));
    if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
    if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "level limit reached");
    if (h.done) {
      *levels_out = h.levels;
      if (overflowed) *overflowed = h.sig_overflow != 0;
      return GR_OK;
    }
    if (!h.paused) return fail(GR_ECUDA, "batched forward stopped without a reason");
    // the next levels need more arrays: double them and resume
    GR_TRY(ensure_slots(g, ws, 2 * (int32_t)ws->lm.size(), s));
    a = mb_args(g, ws, k, depth, keep, max_levels, with_sigma);
    k_mb_resume<<<1, 1, 0, s>>>(a.ctl);
    GR_CUDA(cudaGetLastError());
    GR_TRY(mb_launch(g, a, sk, s));
  }
}

gr_status batch_read_ctl_error(BatchWorkspace *ws, cudaStream_t s) {
  MbCtl h;
  // pageable destination: the copy has finished when the call returns
  GR_CUDA(cudaMemcpyAsync(&h, ws->ctl.p, sizeof(MbCtl), cudaMemcpyDeviceToHost, s));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "level limit reached");
  if (!h.done) return fail(GR_ECUDA, "batched BFS did not finish");
  return GR_OK;
}

// Batched BFS into a device depth array [k][n] with an explicit workspace.
gr_status bfs_batch_run(gr_graph *g, BatchWorkspace *ws, const int32_t *h_srcs, int32_t k,
                        int32_t *depth, int32_t max_levels, cudaStream_t s) {
  return run_forward(g, ws, h_srcs, k, depth, kSigNone, s, max_levels);
}

}  // namespace gr

using namespace gr;

extern "C" {

gr_status gr_bfs_batch(gr_graph *g, const int32_t *srcs, int32_t k, int32_t *depth,
                       const gr_opts *opts, void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (k < 1 || k > 64) return fail(GR_EINVAL, "k must be in [1, 64]");
  if (!srcs || !depth) return fail(GR_EINVAL, "srcs/depth must not be NULL");
  for (int32_t i = 0; i < k; ++i)
    if (srcs[i] < 0 || srcs[i] >= g->n) return fail(GR_EINVAL, "source out of range");
  const gr_opts &o = opts ? *opts : default_opts();
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  GR_TRY(ensure_batch_ws(g, &g->batch, false));
  void *d_depth;
  bool cp;
  const size_t bytes = sizeof(int32_t) * (size_t)k * (size_t)g->n;
  GR_TRY(resolve_output(g, 0, depth, bytes, &d_depth, &cp));
  const int32_t max_levels = o.max_iters > 0 ? o.max_iters : g->n + 1;
  GR_TRY(bfs_batch_run(g, g->batch, srcs, k, (int32_t *)d_depth, max_levels, s));
  if (cp) GR_CUDA(cudaMemcpyAsync(depth, d_depth, bytes, cudaMemcpyDeviceToHost, s));
  GR_TRY(end_call(g, s));
  return GR_OK;
}

gr_status gr_bfs_batch_stats(gr_graph *g, int32_t *levels) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (!g->batch) return fail(GR_EINVAL, "no batched traversal has run on this graph");
  std::lock_guard<std::mutex> lock(g->mu);
  GR_CUDA(cudaSetDevice(g->device));
  if (g->has_last) GR_CUDA(cudaEventSynchronize(g->last_done));
  MbCtl h;
  GR_CUDA(cudaMemcpy(&h, g->batch->ctl.p, sizeof(MbCtl), cudaMemcpyDeviceToHost));
  if (h.error == kDevTimeout) return fail(GR_ETIMEOUT, "a device-side wait timed out");
  if (h.error == kDevOverflow) return fail(GR_ETIMEOUT, "level limit reached");
  if (levels) *levels = h.levels;
  return GR_OK;
}

gr_status gr_bc(gr_graph *g, const int32_t *srcs, int32_t k, double *bc, const gr_opts *opts,
                void *stream) {
  clear_error();
  if (!g) return fail(GR_EINVAL, "graph must not be NULL");
  if (k < 0) return fail(GR_EINVAL, "k must be >= 0");
  if ((k > 0 && !srcs) || !bc) return fail(GR_EINVAL, "srcs/bc must not be NULL");
  for (int32_t i = 0; i < k; ++i)
    if (srcs[i] < 0 || srcs[i] >= g->n) return fail(GR_EINVAL, "source out of range");
  const gr_opts &o = opts ? *opts : default_opts();
  std::lock_guard<std::mutex> lock(g->mu);
  cudaStream_t s = (cudaStream_t)stream;
  GR_TRY(begin_call(g, s));
  GR_TRY(ensure_batch_ws(g, &g->batch, true));
  void *d_bc;
  bool cp;
  GR_TRY(resolve_output(g, 0, bc, sizeof(double) * (size_t)g->n, &d_bc, &cp));
  const int grid = g->num_sms * 8;
  k_fill_f64<<<grid, 256, 0, s>>>((double *)d_bc, g->n, 0.0);
  BatchWorkspace *ws = g->batch;
  int32_t *overflow = (int32_t *)(ws->counter.as<unsigned long long>() + 1);
  GR_CUDA(cudaMemsetAsync(overflow, 0, sizeof(int32_t), s));
  const int32_t max_levels = o.max_iters > 0 ? o.max_iters : g->n + 1;
  for (int32_t b = 0; b < k; b += 64) {
    const int32_t kb = std::min<int32_t>(64, k - b);
    int32_t levels = 0;
    // exact uint64 path counts; a batch whose counts overflow them is
    // counted again in FP64
    int sk = kSigU64;
    bool overflowed = false;
    GR_TRY(run_forward(g, ws, srcs + b, kb, nullptr, sk, s, max_levels, &levels, &overflowed));
    if (overflowed) {
      sk = kSigF64;
      GR_TRY(run_forward(g, ws, srcs + b, kb, nullptr, sk, s, max_levels, &levels));
    }
    // backward over levels levels-2 .. 1 (level levels-1 has no children;
    // level 0 holds the sources, which take no credit)
    BcBackArgs ba;
    ba.R = g->row_off.as<int32_t>();
    ba.C = g->col.as<int32_t>();
    ba.n = g->n;
    ba.m = g->m;
    ba.q = ws->q.as<double>();
    unsigned long long *packed = ws->counter.as<unsigned long long>() + 2;  // two, taken in turn
    GR_CUDA(cudaMemsetAsync(packed, 0, 2 * sizeof(unsigned long long), s));
    int32_t *fq = ws->fq.as<int32_t>(), *fs = ws->fs.as<int32_t>();
    const int list_bound_blocks = (int)((bc_list_max_chunks(g) + 1 + 255) / 256);
    int back_per_sm = 1;
    GR_TRY(fit_carveout(k_bc_backward, kMbThreads, kBcBackBlocksPerSm, g->device, &back_per_sm));
    for (int32_t L = levels - 1; L >= 1; --L) {
      // the vertices of level L (in any lane) with their degree scan
      ba.lv = ws->lm[L]->as<unsigned long long>();
      unsigned long long *fpacked = packed + (L & 1);
      k_mb_list<<<grid, kMbThreads, 0, s>>>(ba.lv, ba.R, g->n, fq, fs, fpacked,
                                            packed + (~L & 1));
      if (L + 1 < levels) {
        ba.lw = ws->lm[L + 1]->as<unsigned long long>();
        k_list_bounds<<<list_bound_blocks, 256, 0, s>>>(
            fs, fpacked, g->num_sms * back_per_sm * (kMbThreads / 32), ws->fcb.as<int32_t>());
        k_bc_backward<<<g->num_sms * back_per_sm, kMbThreads, 0, s>>>(ba, fq, fs, fpacked,
                                                                       ws->fcb.as<int32_t>());
      }
      if (sk == kSigU64)
        k_bc_finalize<kSigU64><<<grid, 256, 0, s>>>(ba.lv, fq, fpacked, ws->sigma.p,
                                                    ws->q.as<double>(), (double *)d_bc, g->n,
                                                    overflow);
      else
        k_bc_finalize<kSigF64><<<grid, 256, 0, s>>>(ba.lv, fq, fpacked, ws->sigma.p,
                                                    ws->q.as<double>(), (double *)d_bc, g->n,
                                                    overflow);
      GR_CUDA(cudaGetLastError());
    }
  }
  if (cp) GR_CUDA(cudaMemcpyAsync(bc, d_bc, sizeof(double) * (size_t)g->n,
                                  cudaMemcpyDeviceToHost, s));
  int32_t h_over = 0;
  GR_CUDA(cudaMemcpyAsync(&h_over, overflow, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  GR_CUDA(cudaStreamSynchronize(s));
  GR_TRY(end_call(g, s));
  if (h_over)
    return fail(GR_EINVAL, "shortest-path counts overflow FP64 on this graph (BC undefined)");
  return GR_OK;
}

}  // extern "C"
