// All-vertex neighbourhood gather-reduce in registers.
//
// For each vertex v of a range with entries: out[v] = OP over the entries
// e = (v, u) of v's row of f(u, e). The entries, not the vertices, are dealt
// out: a warp takes a tile of consecutive entries, 8 * G8 per lane, whatever
// the degree mix. What bounds it is the random load of x[u], one L1 line or
// L2 sector per entry, so everything else is kept out of its way:
//
//  * No shared memory. The whole L1 / shared-memory array is left to the L1,
//    which serves the hubs' values: a plain gather of an R-MAT 2^21 column
//    array takes 161 us with all of it as L1, 250 with half, 480 with the
//    shared-memory maximum.
//  * Columns come as one 32-byte load per lane and 8 entries, past the L1.
//  * Row boundaries come from a plan made once per graph: 16 bits for every
//    8 entries (which of them end a row, and how many rows end before them
//    in their 256-entry tile), so no search and no walk over row offsets.
//    That is m / 4 bytes beside the 4 m of the columns.
//
// A lane adds its entries up row by row. Rows that begin and end inside one
// lane are stored at once; a segmented scan over the lanes joins the pieces
// of rows that cross lanes (one per tile: FP64 adds are scarce on this GPU,
// so a lane takes 16 FP64 values to a scan), and the two pieces that reach
// over a tile's ends go out as atomics. out[v] must therefore hold OP's
// identity beforehand; vertices without entries are not touched.
//
// Which warp takes which tile is the caller's: neighbouring tiles on
// different SMs (spread_warp) suit the rankings and PageRank, whose loops also
// meet small graphs (PageRank 2^21 3.84 ms, 4.05 with a block's tiles
// together; HITS 512k x 128k 1.61, 1.69), tiles of a block together
// (block_warp) the single gather over FP64 values (1.5 M vertices, 45 M
// entries: 167 us, 172 spread).
#pragma once

#include "advance.cuh"

namespace gr {

constexpr int kGpTile = 256;  // entries per rank_base element

// Device side of the plan. desc[g], for entries [8 g, 8 g + 8): bits 0-7 the
// entries that are the last of their row, bits 8-15 the rows that end in the
// same tile before them. rank_base[t]: rows that end before tile t, bit 31
// set when tile t begins with a row's first entry. rows[k]: the k-th vertex
// with entries.
struct GatherPlanArgs {
  const uint16_t *desc;
  const uint32_t *rank_base;
  const int32_t *rows;
};

struct GatherPlan {
  DevMem mem;  // desc, rank_base, rows and the build's partial sums
  GatherPlanArgs a = {nullptr, nullptr, nullptr};
};

// Device memory of a plan.
inline size_t gather_plan_bytes(int32_t n, int64_t m) {
  return (size_t)m / 4 + (size_t)m / 64 + 4 * (size_t)n + 4096;
}

// Builds the plan of the CSR row offsets R (n vertices, m entries) on `s`
// unless it is there already; a stream that is being captured is refused.
// Nothing is synchronised: the caller does, or orders what may use the plan on
// another stream. In gather.cu.
gr_status gather_plan_build(GatherPlan *p, const int32_t *R, int32_t n, int64_t m, cudaStream_t s);

// The same inside a public call on g, after begin_call: whatever becomes of the
// call, the next one, on any stream, comes after the plan's kernels.
gr_status gather_plan_of_call(gr_graph *g, GatherPlan *p, const int32_t *R, cudaStream_t s);

#ifdef __CUDACC__

// 8 consecutive 32-bit values, 32-byte aligned, read once: past the L1
__device__ __forceinline__ void ld_stream8(const int32_t *p, int32_t (&v)[8]) {
  asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
                 "=r"(v[6]), "=r"(v[7])
               : "l"(p));
}

// Where a row's value goes: whole rows are stored, pieces of a row that
// crosses a tile combined atomically.
template <class T, class OP>
struct StoreReduced {
  T *out;
  __device__ __forceinline__ void operator()(int32_t v, T x, bool whole) const {
    if (whole) out[v] = x;
    else OP::atomic(out + v, x);
  }
};

struct SkipNone {
  static constexpr bool kSkips = false;
  __device__ __forceinline__ bool operator()(int32_t) const { return false; }
};

// One warp's share (tiles gw, gw + nw, ...) of the entries [eb, ee), which
// begin and end with whole rows. F: value_type operator()(u, weight) and
// F::kWeighted (whether it reads w[e], then non-null). E: operator()(v,
// value, whole), once per whole row and once per piece of the others. S:
// operator()(v), whether v's row needs no gathering (its value is then OP's
// identity), asked for every row of a lane before its columns are loaded.
template <int G8, class T, class OP, class F, class E, class S = SkipNone>
__device__ __forceinline__ void gather_reduce_tiles(const GatherPlanArgs &p, const int32_t *C,
                                                    const int32_t *W, int32_t eb, int32_t ee,
                                                    const F &f, const E &emit, int64_t gw,
                                                    int64_t nw, const S &skip = S()) {
  constexpr int ITEMS = 8 * G8;
  constexpr int TILE = 32 * ITEMS;
  static_assert(TILE % kGpTile == 0, "a warp's tile is whole rank_base tiles");
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  for (int64_t t = eb / TILE + gw; t * TILE < ee; t += nw) {  // warp-uniform
    const int64_t tb = t * TILE;
    const int64_t e0 = tb + lane * ITEMS;
    const bool whole = tb >= eb && tb + TILE <= ee;
    int32_t c[ITEMS], wt[F::kWeighted ? ITEMS : 1];
    uint32_t ends = 0u, before = 0u;
    int32_t rank;
    {
      const int64_t g = e0 >> 3;
      const uint32_t d0 = p.desc[g];
      ends = d0 & 0xFFu;
      rank = (int32_t)(p.rank_base[e0 / kGpTile] & 0x7FFFFFFFu) + (int32_t)(d0 >> 8);
      if (G8 == 2) ends |= (uint32_t)(p.desc[g + 1] & 0xFFu) << 8;
    }
    uint32_t valid = (1u << ITEMS) - 1u;  // entries to gather
    if (S::kSkips && whole) {
      uint32_t left = ends;
      int32_t r = rank;
      for (int from = 0; from < ITEMS; ++r) {
        const int to = left ? __ffs(left) : ITEMS;
        if (skip(p.rows[r])) valid &= ~((1u << to) - (1u << from));
        left &= left - 1u;
        from = to;
      }
    }
    if (whole) {
#pragma unroll
      for (int k = 0; k < G8; ++k) {
        int32_t x[8];
        if (!S::kSkips || valid) ld_stream8(C + e0 + 8 * k, x);
        else
#pragma unroll
          for (int i = 0; i < 8; ++i) x[i] = 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) c[8 * k + i] = x[i];
        if (F::kWeighted) {
          ld_stream8(W + e0 + 8 * k, x);
#pragma unroll
          for (int i = 0; i < 8; ++i) wt[F::kWeighted ? 8 * k + i : 0] = x[i];
        }
      }
    } else {
      valid = 0u;
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) {
        const int64_t e = e0 + i;
        c[i] = 0;
        if (F::kWeighted) wt[F::kWeighted ? i : 0] = 0;
        if (e < eb) before |= 1u << i;
        if (e >= eb && e < ee) {
          valid |= 1u << i;
          c[i] = C[e];
          if (F::kWeighted) wt[F::kWeighted ? i : 0] = W[e];
        }
      }
      rank += __popc(ends & before);  // rows of this group that end before eb
      ends &= valid;
    }
    T v[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i)
      v[i] = (valid >> i) & 1u ? f(c[i], wt[F::kWeighted ? i : 0]) : OP::identity();
    // the lane's rows: the first end closes a row that may have begun in an
    // earlier lane (head), the others are whole
    T acc = v[0], head = OP::identity();
    const int32_t rank_head = rank;
    bool any = false;
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      if (i) acc = (ends >> (i - 1)) & 1u ? v[i] : OP::op(acc, v[i]);
      if ((ends >> i) & 1u) {
        if (any) emit(p.rows[rank], acc, true);
        else head = acc;
        any = true;
        ++rank;
      }
    }
    // pieces of rows that go on past a lane, summed up to the lane before
    // the one that closes them
    const uint32_t em = __ballot_sync(0xffffffffu, any);
    const uint32_t le = em & (lt | (1u << lane));
    const int from = le ? 31 - __clz(le) : 0;  // lane the open row begins in
    T s = (ends >> (ITEMS - 1)) & 1u ? OP::identity() : acc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      if (!__any_sync(0xffffffffu, lane - from >= o)) break;
      const T y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane - o >= from) s = OP::op(y, s);
    }
    const T carry = __shfl_up_sync(0xffffffffu, s, 1);
    const bool opens = tb < eb || (p.rank_base[tb / kGpTile] >> 31);
    if (any) {
      if (lane) head = OP::op(carry, head);
      emit(p.rows[rank_head], head, (em & lt) || opens);
    }
    // the row that reaches into the next tile
    if (lane == 31 && tb + TILE < ee && !((ends >> (ITEMS - 1)) & 1u))
      emit(p.rows[rank], s, false);
  }
}

// This thread's warp and the number of warps, consecutive warps on different
// blocks, so that little work still spreads over every SM.
__device__ __forceinline__ int64_t spread_warp() {
  return (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
}
__device__ __forceinline__ int64_t grid_warps() {
  return (int64_t)gridDim.x * (blockDim.x >> 5);
}
// This thread's warp, a block's warps together.
__device__ __forceinline__ int64_t block_warp() {
  return (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
}

// Block-wide FP64 sum, added to *dst by thread 0. Block-uniform call of
// THREADS threads (a multiple of 128, at least 256). Four warps add the columns up in
// shared memory before one warp shuffles: a warp's FP64 add holds the SM's
// FP64 pipe for 16 cycles, and a shuffle reduction in all 32 warps of a
// 1024-thread block is 160 of them (1.2 us), this 41.
template <int THREADS>
__device__ __forceinline__ void block_add_f64(double v, double *smem, double *dst) {
  static_assert(THREADS % 128 == 0 && THREADS >= 256, "columns of 128");
  __syncthreads();
  smem[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 128) {
    double t = smem[threadIdx.x];
#pragma unroll
    for (int i = 128; i < THREADS; i += 128) t += smem[threadIdx.x + i];
    smem[threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    double t = (smem[threadIdx.x] + smem[threadIdx.x + 32]) +
               (smem[threadIdx.x + 64] + smem[threadIdx.x + 96]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (threadIdx.x == 0 && t != 0.0) atomicAdd(dst, t);
  }
}

#endif  // __CUDACC__

}  // namespace gr
