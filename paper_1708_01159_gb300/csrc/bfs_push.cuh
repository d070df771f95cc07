// Top-down push shared by the traversal kernels (bfs_kernels.cu) and the
// allocation-free entry point (bfs_static.cu): the visit of one edge and the
// edge-centric level.
#pragma once

#include "bfs_kernels.cuh"

namespace bfs {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---- output staging and per-edge visit --------------------------------------

// No __restrict__ on the queue or bitmaps: inside the persistent kernel they are
// rewritten every level, so they must not be read through the non-coherent
// read-only cache.
struct Level {
  const int32_t* qin;
  int32_t* qout;
  uint32_t* vis;       // current visited bitmap (push updates it in place; pull reads it)
  uint32_t* vis_next;  // the other bitmap (pull writes it)
  int32_t* depth;
  unsigned long long* tail;  // output queue tail (low 32 bits)
  int32_t next_depth;
  int32_t frontier;
  int32_t shared_scan;    // an edge-centric level scans its frontier in every block (pe_shared)
  int32_t latency_bound;  // the level's frontier has fewer than kLatencyEdges edges
  unsigned int* n_heavy;     // heavy list's length (edge-centric push)
  int32_t pull_sparse;    // fewer than 1/16 of the vertices with edges are still unvisited
};

// Below this many frontier edges a level cannot fill the GPU: its time is the
// latency of its chain of dependent memory accesses, not bandwidth. Such a
// level claims targets without reading their bitmap word first (one round trip
// less; the extra atomics cost nothing at this size) and prefetches the first
// adjacency sector of every vertex it reaches into L2, so the next level's
// list reads are L2 hits.
constexpr long long kLatencyEdges = 1ll << 17;

// Newly reached vertices go through a block-local stage (see stage_put) into
// the level's output queue.
__device__ __forceinline__ void stage_flush(const Stage& s, const Level& lv, unsigned int threshold) {
  stage_drain(s, lv.qout, lv.tail, threshold);
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Top-down visit of up to K edges u -> v[k] (Section 3.1.2 push). The bitmap
// words of all K targets are read (except on latency-bound levels), then the
// claims (atomicOr) issued, then the winners' row extents read, so the K
// edges' memory round trips overlap instead of forming one dependent chain per
// edge. The one thread whose atomicOr flips a vertex's bit writes its depth,
// counts its out-degree and stages it. Bound by these round trips; written as
// predicated accesses because an `if` per edge made the compiler wait for each
// claim and each row extent in turn (vertex push on R-MAT 14: 2.49 ms a
// traversal with the branches, 1.85 ms without; virtual warps on its level of
// 345k edges 78 -> 59 us; ER 2^21, level of 1.6M edges, 48 -> 41 us). The
// winners of all K edges of the converged lanes take one reservation in the
// stage, not one per edge (ER level 41 -> 36 us).
// valid: bit k set when v[k] is an edge to visit.
template <int K, int kCount = CM_BLOCK>
__device__ __forceinline__ void visit_km(const DevGraph& g, const Level& lv, const Stage& s, const int32_t (&v)[K],
                                         uint32_t valid, unsigned long long& edges) {
  const bool filter = !lv.latency_bound;
  // The filter reads through L1: the words of hubs, which most edges of a
  // skewed graph name, are then not read from one L2 slice by every SM. A stale
  // word lacks bits set since, which costs a claim, never a vertex. (R-MAT 20,
  // edge-centric level of 6.3M edges: 213 us with L2 reads, 145 so; ER 2^20 of
  // 17M edges 165 and 122. Both ends of a row in one 16-byte load instead of
  // two 4-byte ones below: 10 to 20 % slower, so not done.)
  uint32_t word[K];
#pragma unroll
  for (int k = 0; k < K; ++k) word[k] = ld_now_if(filter && ((valid >> k) & 1u), lv.vis + (v[k] >> 5), 0u);
  bool won[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const uint32_t bit = 1u << (v[k] & 31);
    word[k] = atom_or_if(((valid >> k) & 1u) && !(word[k] & bit), lv.vis + (v[k] >> 5), bit, bit);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) won[k] = !((word[k] >> (v[k] & 31)) & 1u);
  // the winners' rows, four at a time
  constexpr int kRows = K < 4 ? K : 4;
  static_assert(K % kRows == 0, "whole groups");
#pragma unroll
  for (int h = 0; h < K; h += kRows) {
    int32_t b0[kRows], d[kRows];
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      b0[k] = ld_if(won[h + k], g.off + v[h + k], 0);
      d[k] = ld_if(won[h + k], g.off + v[h + k] + 1, 0);
    }
#pragma unroll
    for (int k = 0; k < kRows; ++k) {
      d[k] -= b0[k];
      prefetch_l2_if(!filter && d[k] > 0, g.idx + b0[k]);
      edges += (unsigned long long)d[k];
    }
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (!won[k]) continue;
    lv.depth[v[k]] = lv.next_depth;
    if (kCount == CM_WARP) queue_append(lv.qout, lv.tail, v[k]);
    if (kCount == CM_ATOMIC) lv.qout[(unsigned int)atomicAdd(lv.tail, 1ull)] = v[k];
  }
  if (kCount == CM_BLOCK) stage_put_won(s, lv.qout, lv.tail, won, v);
}

// The first nv entries of v are edges to visit, four in flight at a time (more
// do not fit the registers a thread has at four blocks per SM).
template <int K, int kCount = CM_BLOCK>
__device__ __forceinline__ void visit_k(const DevGraph& g, const Level& lv, const Stage& s, const int32_t (&v)[K],
                                        int nv, unsigned long long& edges) {
  constexpr int kAtOnce = K < 4 ? K : 4;
  static_assert(K % kAtOnce == 0, "whole groups");
#pragma unroll
  for (int k = 0; k < K; k += kAtOnce) {
    int32_t w[kAtOnce];
#pragma unroll
    for (int j = 0; j < kAtOnce; ++j) w[j] = v[k + j];
    const int left = min(max(nv - k, 0), kAtOnce);
    visit_km<kAtOnce, kCount>(g, lv, s, w, (1u << left) - 1u, edges);
  }
}

template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T x, T* total) {
  __shared__ T wsum[32];
  const uint32_t lane = lane_id();
  const int w = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  T inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    T y = __shfl_up_sync(kFull, inc, o);
    if ((int)lane >= o) inc += y;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    T s = (int)lane < nw ? wsum[lane] : T(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      T y = __shfl_up_sync(kFull, s, o);
      if ((int)lane >= o) s += y;
    }
    if ((int)lane < nw) wsum[lane] = s;
  }
  __syncthreads();
  const T base = w > 0 ? wsum[w - 1] : T(0);
  *total = wsum[nw - 1];
  __syncthreads();
  return base + inc - x;
}

// ---------------------------------------------------------------------------
// Push, edge-centric (Section 3.1.1 edge list, restricted to the frontier's
// edges): a tile of frontier vertices is scanned by degree in shared memory and
// its edges are dealt to the block's threads one by one (a binary search of the
// scan finds an edge's vertex), so that a step visits 1,024 edges whatever their
// vertices' degrees.
//  - A frontier of few vertices with long lists (pe_shared) is one tile that
//    every block scans itself; each takes its share of the edges.
//  - Any other is cut into tiles of 32 to 256 vertices, as short as
//    spreads it over every block, one block a tile. Vertices of kHeavy edges or
//    more are set aside on a list and dealt over all blocks afterwards, as a
//    frontier of their own (body_push_heavy, after a grid barrier); graphs
//    without such vertices need no barrier. A list that is full leaves its
//    vertices to their block.
// A level of 53k edges from 3,149 vertices (ER 2^21) took 24 us with a scan of
// the whole frontier over the grid (three barriers), 11.5 us in tiles.
// The lanes of a warp take consecutive edges: coalesced, but where a hub's list
// names consecutive vertices 32 claims meet in one bitmap word (one vertex, 10^6
// edges: 29 us; 15 when a thread took several consecutive edges). Four consecutive
// edges a lane instead made R-MAT and Erdos-Renyi traversals 0.5 to 1.5 % slower.
// ---------------------------------------------------------------------------
// Whether every block scans the whole frontier (at most one tile) itself. On
// GB300: 763 vertices of 32.5 edges 9.5 us that way, 16.7 in tiles of 32; 359
// of 17 edges 8.2 and 8.6; 667 of 9 edges 8.3 and 7.2. With heavy vertices in
// the graph the tiles pay a grid barrier whatever the level (11 vertices of one
// edge: 5.8 and 8.3 us).
__device__ __forceinline__ bool pe_shared(long long f, long long e, bool graph_has_heavy) {
  return f <= kPeTile && (graph_has_heavy || e > 16 * f);
}

// Exclusive scan of the degrees of q[0 .. f), f <= kPeTile, into s_a (their
// total past the last), row starts into s_beg: kPeTile entries each, in an
// order of their own. Returns the total.
__device__ __forceinline__ int32_t pe_scan_all(const DevGraph& g, const int32_t* q, int f, int32_t* s_a,
                                               int32_t* s_beg) {
  int32_t beg[kPeItems], d[kPeItems];
#pragma unroll
  for (int k = 0; k < kPeItems; ++k) {
    const int i = k * kThreads + (int)threadIdx.x;
    const int32_t u = ld_now_if(i < f, q + (i < f ? i : 0), -1);
    beg[k] = ld_if(u >= 0, g.off + (u >= 0 ? u : 0), 0);
    d[k] = ld_if(u >= 0, g.off + (u >= 0 ? u : 0) + 1, 0);
  }
  int32_t run = 0;
#pragma unroll
  for (int k = 0; k < kPeItems; ++k) {
    const int32_t t = d[k] - beg[k];
    d[k] = run;
    run += t;
  }
  int32_t total;
  const int32_t ex = block_exclusive_scan<int32_t>(run, &total);
#pragma unroll
  for (int k = 0; k < kPeItems; ++k) {
    s_a[(int)threadIdx.x * kPeItems + k] = ex + d[k];
    s_beg[(int)threadIdx.x * kPeItems + k] = beg[k];
  }
  __syncthreads();
  return total;
}

// Visit edges j0 .. j1 - 1 of the scan s_a of N entries (N a power of two; s_a
// nondecreasing from 0). Uniform: every thread of the block calls it.
template <int N>
__device__ __forceinline__ void pe_visit(const DevGraph& g, const Level& lv, const Stage& stage, const int32_t* s_a,
                                         const int32_t* s_beg, uint32_t j0, uint32_t j1, unsigned long long& edges) {
  for (uint32_t e0 = j0; e0 < j1; e0 += 4 * kThreads) {  // j1 < 2^31: no wrap
    int32_t v[4];
    uint32_t valid = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t j = e0 + k * kThreads + threadIdx.x;
      int o = 0;  // the last entry with s_a[o] <= j owns edge j
      if (e0 + k * kThreads < j1) {
#pragma unroll
        for (int step = N / 2; step > 0; step >>= 1) o += (uint32_t)s_a[o + step] <= j ? step : 0;
      }
      valid |= (uint32_t)(j < j1) << k;
      v[k] = ld_if(j < j1, g.idx + ((uint32_t)s_beg[o] + (j - (uint32_t)s_a[o])), 0);
    }
    visit_km<4>(g, lv, stage, v, valid, edges);
    stage_flush(stage, lv, kStageCap / 2);
  }
}

// The frontier q[0 .. f), f <= kPeTile, every block taking its share of the edges.
__device__ void body_push_shared(const DevGraph& g, const Level& lv, const int32_t* q, int f, const Stage& stage,
                                 int32_t* s_a, int32_t* s_beg, unsigned long long& edges) {
  const int32_t total = pe_scan_all(g, q, f, s_a, s_beg);
  // a whole multiple of the block size a block, as few as spreads them over every block
  const int32_t each = (int32_t)((((long long)total + gridDim.x - 1) / gridDim.x + kThreads - 1) / kThreads * kThreads);
  const long long j0 = (long long)blockIdx.x * each;
  if (j0 < total) pe_visit<kPeTile>(g, lv, stage, s_a, s_beg, (uint32_t)j0, (uint32_t)min(j0 + each, (long long)total), edges);
  __syncthreads();  // the scan is not overwritten before every thread has read it
}

// The frontier in tiles; heavy: a list of heavy_cap vertices, its length (zero
// at the level's start) at lv.n_heavy.
__device__ void body_push_tiles(const DevGraph& g, const Level& lv, const Stage& stage, int32_t* s_a, int32_t* s_beg,
                                int32_t* heavy, int32_t heavy_cap, unsigned long long& edges) {
  const int f = lv.frontier;
  const int share = (int)(((long long)f + gridDim.x - 1) / gridDim.x);
  const int tile = min(kThreads, (share + 31) & ~31);
  for (long long t0 = (long long)blockIdx.x * tile; t0 < f; t0 += (long long)gridDim.x * tile) {
    const long long i = t0 + (long long)threadIdx.x;
    const bool have = (int)threadIdx.x < tile && i < f;
    int32_t beg = 0, deg = 0;
    if (have) {
      const int32_t u = lv.qin[i];
      beg = g.off[u];
      deg = g.off[u + 1] - beg;
      if (deg >= kHeavy) {
        const unsigned int at = atomicAdd(lv.n_heavy, 1u);
        if (at < (unsigned)heavy_cap) {
          heavy[at] = u;
          deg = 0;
        }
      }
    }
    int32_t total;
    s_a[threadIdx.x] = block_exclusive_scan<int32_t>(deg, &total);
    s_beg[threadIdx.x] = beg;
    __syncthreads();
    pe_visit<kThreads>(g, lv, stage, s_a, s_beg, 0u, (uint32_t)total, edges);
    __syncthreads();
  }
}

// The vertices set aside, `count` of them on the list (every block calls it).
__device__ void body_push_heavy(const DevGraph& g, const Level& lv, const Stage& stage, int32_t* s_a, int32_t* s_beg,
                                const int32_t* heavy, int32_t count, unsigned long long& edges) {
  for (int32_t base = 0; base < count; base += kPeTile)
    body_push_shared(g, lv, heavy + base, min(kPeTile, count - base), stage, s_a, s_beg, edges);
}

}  // namespace
}  // namespace bfs
