// Level kernels of the per-level switched BFS (sm_103a).
//
// Each variant's level is a device function ("body") written with
// block-uniform loops, so three drivers can share it:
//   - graph path: one thin kernel per body, launched by a CUDA graph whose
//     WHILE node runs the level loop and whose SWITCH node picks the variant
//     set on the device by k_decide;
//   - persistent path: k_bfs_persistent, one cooperative launch per traversal;
//     levels are separated by a grid barrier and every block evaluates the
//     decision tree itself from counters indexed by level % 3;
//   - host loop: the graph path's kernels launched from the host level by
//     level (for profilers and the per-level timing harness).
//
// Newly reached vertices are claimed by an atomicOr on the visited bitmap; the
// single thread that flips a bit writes depth L + 1, stages the vertex in a
// block-local shared-memory buffer that is flushed to the output queue with
// one global atomic per block (the queue tail is the next frontier size:
// Section 3.1.4's first variant, a global atomic counter, with warp and block
// aggregation in front of it), and adds the vertex's out-degree to the next
// level's frontier-edge count.
#include "bfs_push.cuh"

namespace bfs {

namespace {

// ---- mbarrier + bulk async copy (TMA bulk, non-tensor) --------------------

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}

// Wait for the phase with the given parity to complete, giving up after
// kWaitLimitNs. Returns false on timeout.
__device__ bool mbar_wait_bounded(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_ns() - t0 > kWaitLimitNs) return false;
  }
  return true;
}

__device__ __forceinline__ Level load_level(const DevGraph& g, const Buffers& b, RunState* st) {
  Level lv;
  // select with ternaries: indexing the by-value parameter arrays would copy them to local memory
  const bool qs = st->qsel != 0u;
  const bool vs = st->vsel != 0u;
  lv.qin = qs ? b.q[1] : b.q[0];
  lv.qout = qs ? b.q[0] : b.q[1];
  lv.vis = vs ? b.vis[1] : b.vis[0];
  lv.vis_next = vs ? b.vis[0] : b.vis[1];
  lv.depth = st->depth;
  lv.tail = &st->next_count;
  lv.next_depth = st->level + 1;
  lv.frontier = st->frontier;
  lv.n_heavy = &st->heavy3[0];
  lv.shared_scan = pe_shared(st->frontier, st->frontier_edges, g.gfeat[F_DEG_MAX] >= kHeavy);
  lv.latency_bound = st->frontier_edges < kLatencyEdges;
  lv.pull_sparse = (long long)g.n_active - st->discovered < (long long)(g.n_active >> 4);
  return lv;
}

// ---------------------------------------------------------------------------
// Init (Section 3.1: all depths infinity, the root 0): depth and bitmap fill
// ---------------------------------------------------------------------------
__device__ __forceinline__ void init_fill(const DevGraph& g, uint32_t* vis0, int32_t* depth, int32_t root) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int32_t n = g.n;
  if ((reinterpret_cast<uintptr_t>(depth) & 15u) == 0) {
    const int64_t n4 = n >> 2;
    int4* d4 = reinterpret_cast<int4*>(depth);
    for (int64_t i = tid; i < n4; i += stride) {
      int4 val = make_int4(-1, -1, -1, -1);
      if ((root >> 2) == i) {
        const int k = root & 3;
        if (k == 0) val.x = 0;
        if (k == 1) val.y = 0;
        if (k == 2) val.z = 0;
        if (k == 3) val.w = 0;
      }
      d4[i] = val;
    }
    for (int64_t i = (n4 << 2) + tid; i < n; i += stride) depth[i] = (i == root) ? 0 : -1;
  } else {
    for (int64_t i = tid; i < n; i += stride) depth[i] = (i == root) ? 0 : -1;
  }
  for (int64_t w = tid; w < g.words; w += stride)
    vis0[w] = g.vis_init[w] | ((w == (root >> 5)) ? (1u << (root & 31)) : 0u);
}

// ---------------------------------------------------------------------------
// Tree evaluation (Section 2.1 walk over the Section 4.1 features, with the
// Section 4.1 unknown-prediction rule). Returns the variant; fills feat[].
// ---------------------------------------------------------------------------
// Value of feature fi at this level, computed on demand: a walk reads at most
// the tree's depth of them, and each ppm share costs a 64-bit division.
__device__ __forceinline__ long long feature_value(const DevGraph& g, int32_t fi, int32_t L, long long f, long long e,
                                                   long long discovered) {
  if (is_graph_feature(fi)) return g.gfeat[fi];
  switch (fi) {
    case F_FRONTIER: return f;
    case F_FRONTIER_PPM: return (1000000ll * f) / g.n;
    case F_DISCOVERED: return discovered;
    case F_DISCOVERED_PPM: return (1000000ll * discovered) / g.n;
    case F_FRONTIER_EDGES: return e;
    default: return L;  // F_LEVEL
  }
}

// The split test x_fi <= t of a tree node, without dividing for the ppm
// shares: floor(1e6 c / n) <= t is 1e6 c < (t + 1) n for 0 <= t < 1e6, always
// true for t >= 1e6 (c <= n) and never for t < 0.
__device__ __forceinline__ bool feature_le(const DevGraph& g, int32_t fi, long long t, int32_t L, long long f,
                                          long long e, long long discovered) {
  if (fi == F_FRONTIER_PPM || fi == F_DISCOVERED_PPM) {
    const long long c = fi == F_FRONTIER_PPM ? f : discovered;
    if (t < 0) return false;
    if (t >= 1000000) return true;
    return 1000000ll * c < (t + 1) * (long long)g.n;
  }
  return feature_value(g, fi, L, f, e, discovered) <= t;
}

// Section 2.1 walk of an integer tree; -1 for an unknown leaf.
__device__ __forceinline__ int32_t walk_tree(const DevGraph& g, const TreeNode* tree, int32_t nodes, int32_t L,
                                             long long f, long long e, long long discovered) {
  int32_t i = 0;
  for (int32_t step = 0; step <= nodes; ++step) {
    const TreeNode nd = tree[i];
    if (nd.f < 0) return nd.v;
    i = feature_le(g, nd.f, nd.t, L, f, e, discovered) ? nd.l : nd.r;
  }
  return -1;
}

// The test x_fi <= t of a level feature without branches, so that the lanes
// of a warp, each on a different feature, do not diverge. The ppm shares do not
// occur here: the host rewrote each as the equivalent test on the count
// (floor(1e6 c / n) <= t is c <= ceil((t + 1) n / 1e6) - 1).
__device__ __forceinline__ bool level_feature_le(int32_t fi, long long t, int32_t L, long long f, long long e,
                                                 long long discovered) {
  long long x = L;
  x = (fi == F_FRONTIER) ? f : x;
  x = (fi == F_DISCOVERED) ? discovered : x;
  x = (fi == F_FRONTIER_EDGES) ? e : x;
  return x <= t;
}

// The leaf the tree's walk reaches, by the bit-parallel form, within one warp:
// lane k tests the level-feature nodes k, k + 32; the graph-feature tests are
// already folded into q.base. Every lane of the warp calls it and gets the
// same result (-1 if none); no block-wide synchronisation.
__device__ __forceinline__ int32_t qs_leaf_warp(const QsTree& q, int32_t L, long long f, long long e,
                                                long long discovered) {
  unsigned long long m = q.base;
  for (int k = lane_id(); k < q.n_int; k += 32) {
    const QsNode nd = q.node[k];
    if (!level_feature_le(nd.f, nd.t, L, f, e, discovered)) m &= nd.mask;
  }
  const uint32_t lo = __reduce_and_sync(kFull, (uint32_t)m);
  const uint32_t hi = __reduce_and_sync(kFull, (uint32_t)(m >> 32));
  const int leaf = __ffsll((long long)(((unsigned long long)hi << 32) | lo)) - 1;
  return (leaf >= 0 && leaf < q.n_leaf) ? leaf : -1;
}

// The tree's prediction (leaf class, -1 for unknown) by the bit-parallel form.
__device__ __forceinline__ int32_t qs_eval_warp(const QsTree& q, int32_t L, long long f, long long e,
                                                long long discovered) {
  const int32_t leaf = qs_leaf_warp(q, L, f, e, discovered);
  return leaf >= 0 ? q.leaf[leaf] : -1;
}

// True (in every lane) when this level's features lie in the box that lanes
// 0-7 of the warp hold in `bound` (lane 2k: lower bound of level feature k,
// lane 2k + 1: upper bound; k = frontier, discovered, frontier edges, level).
__device__ __forceinline__ bool in_leaf_box(int32_t bound, int32_t L, long long f, long long e, long long discovered) {
  const uint32_t lane = lane_id();
  // every level feature lies in [0, 2^31)
  const int32_t x = lane < 2 ? (int32_t)f : lane < 4 ? (int32_t)discovered : lane < 6 ? (int32_t)e : L;
  const bool ok = (lane & 1u) ? x <= bound : x >= bound;
  return __all_sync(kFull, lane >= 8u || ok);
}

// Section 4.1 unknown-prediction rule on a walk's result.
__device__ __forceinline__ int32_t known_variant(int32_t v, int32_t L, int32_t prev) {
  if (v < 0 || v >= V_NUM) v = (L == 0) ? kLevel0Default : prev;  // unknown prediction
  if (v < 0 || v >= V_NUM) v = kLevel0Default;
  return v;
}

// The virtual-warp width under the graph's policy: the rule is the power of
// two nearest above the frontier's mean degree floor(e / f), clamped to [4,
// 32] (floor(e / f) <= k is e < (k + 1) f).
__device__ __forceinline__ int32_t warp_width(long long f, long long e, int32_t policy) {
  const int32_t rule = (f <= 0 || e < 5 * f) ? 4 : e < 9 * f ? 8 : e < 17 * f ? 16 : 32;
  return policy == VW_RULE_X2     ? min(32, 2 * rule)
         : policy == VW_RULE_HALF ? max(4, rule / 2)
         : policy == VW_4         ? 4
         : policy == VW_8         ? 8
         : policy == VW_16        ? 16
         : policy == VW_32        ? 32
                                  : rule;
}

// ---------------------------------------------------------------------------
// Push, one thread per frontier vertex (Section 3.1.2 vertex push, over an
// explicit queue instead of a scan of all vertices). Each thread walks its
// vertex's adjacency four edges at a time. (Positions in a queue are unsigned
// in all push variants: a frontier may have 2^31 - 3 vertices, and the step past
// its end does not fit 31 bits then.)
// ---------------------------------------------------------------------------
// Lists from this length on are visited eight edges at a time, so that a hub's
// thread has eight claims in flight (R-MAT 14 by vertex push alone, four roots:
// 7.17 -> 6.14 ms with the shared reservation of visit_km); shorter ones four.
constexpr int32_t kLongList = 32;

template <int kCount = CM_BLOCK>
__device__ void body_push_thread(const DevGraph& g, const Level& lv, const Stage& stage, unsigned long long& edges) {
  const uint32_t stride = gridDim.x * blockDim.x, f = (uint32_t)lv.frontier;
  for (uint32_t base = blockIdx.x * blockDim.x; base < f; base += stride) {
    const uint32_t i = base + threadIdx.x;
    if (i < f) {
      const int32_t u = lv.qin[i];
      const int32_t end = g.off[u + 1];
      int32_t e = g.off[u];
      // a long list eight edges at a time, its entries two 16-byte loads
      if (end - e >= kLongList) {
        const int32_t head = min(end, (e + 3) & ~3);
        int32_t first[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) first[k] = e + k < head ? g.idx[e + k] : 0;
        visit_k<4, kCount>(g, lv, stage, first, head - e, edges);
        for (e = head; e + 8 <= end; e += 8) {
          const int4 lo = *reinterpret_cast<const int4*>(g.idx + e), hi = *reinterpret_cast<const int4*>(g.idx + e + 4);
          const int32_t v[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
          visit_km<8, kCount>(g, lv, stage, v, 0xffu, edges);
        }
      }
      for (; e < end; e += 4) {
        const int nv = min(4, end - e);
        int32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = k < nv ? g.idx[e + k] : 0;
        visit_k<4, kCount>(g, lv, stage, v, nv, edges);
      }
    }
    stage_flush(stage, lv, kStageCap / 2);
  }
}

// ---------------------------------------------------------------------------
// Push, virtual warp of W lanes per frontier vertex (Section 3.1.3, after Hong
// et al. 2011). Lanes stride the adjacency; W = 32 reads long lists with
// 16-byte vector loads. Positions in the lists that a step may carry past the
// lists' end are unsigned: the end may lie 65 below 2^31.
// ---------------------------------------------------------------------------
template <int W>
__device__ __forceinline__ void push_vwarp(const DevGraph& g, const Level& lv, const Stage& stage,
                                           unsigned long long& edges) {
  constexpr int G = kThreads / W;  // groups per block
  const int lane = threadIdx.x & (W - 1);
  const uint32_t f = (uint32_t)lv.frontier;
  if (W < 32 && f > gridDim.x * G) {
    // More frontier vertices than groups: a group takes kR consecutive
    // frontier vertices per step, and each round every lane visits one edge of
    // each of them (edge lane, lane + W, ...), so kR independent chains of
    // loads are in flight per lane and the level needs a quarter of the steps
    // (a high-diameter graph's levels on a narrow grid). A frontier that fits
    // one step keeps one vertex per group, spread over every block.
    constexpr int kR = 4;
    const uint32_t grp = threadIdx.x / W;
    for (uint32_t base = blockIdx.x * G * kR; base < f; base += gridDim.x * G * kR) {
      uint32_t e[kR], end[kR];
#pragma unroll
      for (int j = 0; j < kR; ++j) {
        const uint32_t i = base + grp * kR + j;
        e[j] = end[j] = 0;
        if (i < f) {
          const int32_t u = lv.qin[i];
          e[j] = (uint32_t)(g.off[u] + lane);
          end[j] = (uint32_t)g.off[u + 1];
        }
      }
      uint32_t valid;
      do {
        int32_t v[kR];
        valid = 0;
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          const bool ok = e[j] < end[j];
          v[j] = ok ? g.idx[e[j]] : 0;
          valid |= (uint32_t)ok << j;
          e[j] += W;
        }
        if (valid) visit_km<kR>(g, lv, stage, v, valid, edges);
      } while (valid);
      stage_flush(stage, lv, kStageCap / 2);
    }
    return;
  }
  for (uint32_t base = blockIdx.x * G; base < f; base += gridDim.x * G) {
    const uint32_t i = base + threadIdx.x / W;
    if (i < f) {
      const int32_t u = lv.qin[i];
      const int32_t beg = g.off[u], end = g.off[u + 1];
      if (W == 32 && end - beg >= 256) {
        const int32_t a0 = (beg + 3) & ~3, a1 = end & ~3;
        {
          int32_t v[1] = {beg + lane < a0 ? g.idx[beg + lane] : 0};
          visit_k<1>(g, lv, stage, v, beg + lane < a0 ? 1 : 0, edges);
        }
        for (uint32_t e = (uint32_t)(a0 + 4 * lane); e < (uint32_t)a1; e += 128) {
          const int4 q = *reinterpret_cast<const int4*>(g.idx + e);
          int32_t v[4] = {q.x, q.y, q.z, q.w};
          visit_k<4>(g, lv, stage, v, 4, edges);
        }
        {
          int32_t v[1] = {a1 + lane < end ? g.idx[a1 + lane] : 0};
          visit_k<1>(g, lv, stage, v, a1 + lane < end ? 1 : 0, edges);
        }
      } else {
        for (uint32_t e = (uint32_t)(beg + lane); e < (uint32_t)end; e += 4 * W) {
          int32_t v[4];
          int nv = 0;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t ek = e + k * W;
            v[k] = ek < (uint32_t)end ? g.idx[ek] : 0;
            nv += ek < (uint32_t)end ? 1 : 0;
          }
          visit_k<4>(g, lv, stage, v, nv, edges);
        }
      }
    }
    stage_flush(stage, lv, kStageCap / 2);
  }
}

__device__ void body_push_warp(const DevGraph& g, const Level& lv, const Stage& stage, int32_t vw,
                               unsigned long long& edges) {
  switch (vw) {
    case 4: push_vwarp<4>(g, lv, stage, edges); break;
    case 8: push_vwarp<8>(g, lv, stage, edges); break;
    case 16: push_vwarp<16>(g, lv, stage, edges); break;
    default: push_vwarp<32>(g, lv, stage, edges); break;
  }
}

// ---------------------------------------------------------------------------
// Push, one CTA per frontier vertex. Long adjacency lists are streamed into a
// double-buffered shared-memory stage by bulk async copies (cp.async.bulk with
// an mbarrier transaction count); the CTA's threads then test and claim the
// staged neighbours. Copies are 16-byte aligned: the range is widened to
// multiples of 4 entries (idx is padded) and the extra entries are skipped.
// ---------------------------------------------------------------------------
struct CtaPipe {
  int32_t* chunk;  // 2 x kCtaChunk entries of shared memory
  uint64_t* bar;   // 2 mbarriers, initialised once per block
  uint32_t parity0, parity1;
  uint32_t extra_tx;  // test hook: bytes the next copy's barrier expects beyond the copy (0 normally)
};

__device__ __forceinline__ void cta_pipe_init(uint64_t* bar) {
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  __syncthreads();
}

// Returns false if a copy never completed (status set; block stopped early).
__device__ bool body_push_cta(const DevGraph& g, const Level& lv, const Stage& stage, CtaPipe& pp, int32_t* status,
                              unsigned long long& edges) {
  const int tid = threadIdx.x;
  constexpr int kPer = kCtaChunk / kThreads;  // staged entries per thread per chunk
  int iter = 0;
  for (uint32_t i = blockIdx.x; i < (uint32_t)lv.frontier; i += gridDim.x, ++iter) {
    const int32_t u = lv.qin[i];
    const int32_t beg = g.off[u], end = g.off[u + 1];
    if (end - beg < kCtaDirect) {
      // short lists: read directly; check the stage every 4th vertex (4 x 512
      // entries fit it), not after each one, to keep barriers rare
      for (uint32_t e = (uint32_t)beg + (uint32_t)tid; e < (uint32_t)end; e += 4 * kThreads) {  // unsigned as above
        int32_t v[4];
        int nv = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t ek = e + k * kThreads;
          v[k] = ek < (uint32_t)end ? g.idx[ek] : 0;
          nv += ek < (uint32_t)end ? 1 : 0;
        }
        visit_k<4>(g, lv, stage, v, nv, edges);
      }
      if ((iter & 3) == 3) stage_flush(stage, lv, kStageCap / 2);
      continue;
    }
    stage_flush(stage, lv, 1);  // empty the stage before a long list
    const int32_t abeg = beg & ~3, aend = (end + 3) & ~3;
    const int32_t nch = (aend - abeg + kCtaChunk - 1) / kCtaChunk;
    auto issue = [&](int32_t c) {
      const int32_t cb = abeg + c * kCtaChunk;
      const uint32_t bytes = (uint32_t)min(kCtaChunk, aend - cb) * 4u;
      uint64_t* br = &pp.bar[c & 1];
      mbar_expect_tx(br, bytes + pp.extra_tx);
      pp.extra_tx = 0;
      bulk_g2s(pp.chunk + (c & 1) * kCtaChunk, g.idx + cb, bytes, br);
    };
    if (tid == 0) {
      issue(0);
      if (nch > 1) issue(1);
    }
    for (int32_t c = 0; c < nch; ++c) {
      const int s = c & 1;
      const bool ok = mbar_wait_bounded(&pp.bar[s], s ? pp.parity1 : pp.parity0);
      if (s)
        pp.parity1 ^= 1u;
      else
        pp.parity0 ^= 1u;
      if (ok) {
        const int32_t cb = abeg + c * kCtaChunk;
        const int32_t len = min(kCtaChunk, aend - cb);
        const int32_t* buf = pp.chunk + s * kCtaChunk;
        int32_t v[kPer];
        int nv = 0;
        // entries tid, tid + 256, ... of the chunk, compacted to the valid ones
#pragma unroll
        for (int k = 0; k < kPer; ++k) {
          const int32_t kk = tid + k * kThreads;
          const int32_t e = cb + kk;
          if (kk < len && e >= beg && e < end) v[nv++] = buf[kk];
        }
        visit_k<kPer>(g, lv, stage, v, nv, edges);
      }
      stage_flush(stage, lv, kStageCap / 2);
      if (!__syncthreads_and(ok)) {
        // a copy never completed: flag it, let the other in-flight copy land (bounded) and stop
        if (tid == 0) {
          *status = ST_TIMEOUT;
          if (c + 1 < nch) mbar_wait_bounded(&pp.bar[s ^ 1], s ? pp.parity0 : pp.parity1);
        }
        return false;
      }
      if (tid == 0 && c + 2 < nch) issue(c + 2);
    }
  }
  return true;
}

// ---------------------------------------------------------------------------
// Pull, bottom-up over the visited bitmap (Section 3.1.2 vertex pull). A warp
// owns 32 consecutive vertices (one bitmap word); each unvisited lane scans its
// in-neighbours, four at a time, and stops at the first visited one. At the
// start of level L a visited in-neighbour of an unvisited vertex has depth
// exactly L (a smaller depth would already have reached the vertex), so the
// current bitmap is the frontier test. New bits go to the other bitmap (read
// and write sets stay apart); the found vertices are staged and appended to
// the queue, which is also the bitmap-to-queue conversion a following push
// level needs. kReadOnlyCache: the bitmap is read through the non-coherent
// read-only cache, valid only when no earlier level ran in the same launch
// (graph and host-loop drivers); the persistent kernel passes false.
// ---------------------------------------------------------------------------
template <bool kReadOnlyCache>
__device__ __forceinline__ uint32_t vis_bit(const uint32_t* vis, int32_t u) {
  const uint32_t word = kReadOnlyCache ? ld_nc_u32(vis + (u >> 5)) : vis[u >> 5];
  return (word >> (u & 31)) & 1u;
}

// A warp takes kWords bitmap words (kWords x 32 vertices) per step and each
// lane interleaves the scans of its kWords vertices, four in-neighbours of each
// per round, so kWords times as many independent loads are in flight per
// thread as with one vertex per lane (a scan is a chain of dependent loads:
// row extent, adjacency entries, bitmap words). The bitmap words of the next
// step are loaded at the start of the current one. Found vertices go to a
// warp-private slice of the block stage, flushed by the warp alone (one queue
// atomic per slice), so warps never wait for one another inside the level.
constexpr int kPullWordsLaunch = 2;      // k_pull
constexpr int kPullWordsPersistent = 2;  // pull level of the persistent kernel
constexpr int kWarpStage = kStageCap / (kThreads / 32);
static_assert(kStageCap % (kThreads / 32) == 0, "stage slices");

__device__ __forceinline__ void warp_stage_flush(int32_t* wbuf, unsigned int cnt, const Level& lv) {
  __syncwarp();
  unsigned int base = 0;
  if (lane_id() == 0) base = (unsigned int)atomicAdd(lv.tail, (unsigned long long)cnt);
  base = __shfl_sync(kFull, base, 0);
  for (unsigned int i = lane_id(); i < cnt; i += 32) lv.qout[base + i] = wbuf[i];
  __syncwarp();
}

// A pull level runs in two phases per warp. The hint pass takes kWords bitmap
// words per step (w[j] < 0: none; cw[j] the current word): each lane takes
// vertex w[j] * 32 + lane of every word and, when it is unvisited, tests its
// hint (the in-neighbour of largest out-degree among the first entries of its
// in-list, chosen at graph create); a vertex whose hint is in the frontier is
// found there, without reading its in-list, and the next bitmap's words are
// written. The others (misses) go to the warp's miss list in shared memory;
// whenever it holds 32, the miss pass scans their in-lists, one vertex per
// lane, four in-neighbours per round, stopping at the first visited one, and
// sets the found vertices' bits in the next bitmap. So a step of the hint pass
// costs one round trip to the hint and its bitmap word, and no lane of a miss
// scan waits on vertices that need no scan. Found vertices get their depth and
// a slot of the warp's stage.
template <int kWords>
struct PullMisses {
  static constexpr int kCap = 32 * (kWords + 1);  // up to 31 left over plus one step's misses
  int32_t* v;                                     // kCap entries each, in shared memory
  int32_t* beg;
  int32_t* end;
};

// Shared-memory ints the miss lists of a block's warps take.
template <int kWords>
constexpr int pull_scratch_ints() {
  return (kThreads / 32) * 3 * PullMisses<kWords>::kCap;
}

template <bool kReadOnlyCache, int kWords>
__device__ __forceinline__ void pull_words(const DevGraph& g, const Level& lv, const int32_t (&w)[kWords],
                                           const uint32_t (&cw)[kWords], int32_t* wbuf, unsigned int& wcnt,
                                           const PullMisses<kWords>& ms, int& mcnt, unsigned long long& edges) {
  const uint32_t lane = lane_id();
  int32_t v[kWords], beg[kWords], end[kWords], h[kWords];
  bool active[kWords], found[kWords];
#pragma unroll
  for (int j = 0; j < kWords; ++j) {
    v[j] = w[j] * 32 + (int32_t)lane;
    active[j] = w[j] >= 0 && cw[j] != kFull && v[j] < g.n && !((cw[j] >> lane) & 1u);
    beg[j] = end[j] = 0;
    h[j] = -1;
    if (active[j]) {  // three coalesced loads, issued together
      beg[j] = g.in_off[v[j]];
      end[j] = g.in_off[v[j] + 1];
      h[j] = g.hint[v[j]];
    }
    active[j] = active[j] && beg[j] < end[j];
  }
#pragma unroll
  for (int j = 0; j < kWords; ++j) found[j] = active[j] && h[j] >= 0 && vis_bit<kReadOnlyCache>(lv.vis, h[j]);
#pragma unroll
  for (int j = 0; j < kWords; ++j) {
    const uint32_t fm = __ballot_sync(kFull, found[j]);
    if (found[j]) {
      const int32_t deg = g.symmetric ? end[j] - beg[j] : g.off[v[j] + 1] - g.off[v[j]];
      lv.depth[v[j]] = lv.next_depth;
      edges += (unsigned long long)deg;
      wbuf[wcnt + __popc(fm & lanemask_lt())] = v[j];
    }
    wcnt += (unsigned)__popc(fm);
    if (lane == 0 && w[j] >= 0) lv.vis_next[w[j]] = cw[j] | fm;
    const bool miss = active[j] && !found[j];
    const uint32_t mm = __ballot_sync(kFull, miss);
    if (miss) {
      const int slot = mcnt + __popc(mm & lanemask_lt());
      ms.v[slot] = v[j];
      ms.beg[slot] = beg[j];
      ms.end[slot] = end[j];
    }
    mcnt += __popc(mm);
  }
}

// The miss pass over entries base .. base + cnt - 1 (cnt <= 32) of the warp's
// miss list.
template <bool kReadOnlyCache, int kWords>
__device__ __forceinline__ void pull_misses(const DevGraph& g, const Level& lv, const PullMisses<kWords>& ms,
                                            int base, int cnt, int32_t* wbuf, unsigned int& wcnt,
                                            unsigned long long& edges) {
  // orders the list entries and this warp's next-bitmap word stores before
  // the reads and bit sets below
  __syncwarp();
  const uint32_t lane = lane_id();
  bool active = (int)lane < cnt;
  int32_t v = 0, beg = 0, pos = 0, end = 0;
  if (active) {
    v = ms.v[base + lane];
    beg = ms.beg[base + lane];
    end = ms.end[base + lane];
    pos = beg;
  }
  bool found = false;
  while (__any_sync(kFull, active)) {
    const int nv = active ? min(4, end - pos) : 0;
    int32_t u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) u[k] = nv ? g.in_idx[k < nv ? pos + k : pos] : 0;
    if (active) {
      uint32_t hit = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) hit |= vis_bit<kReadOnlyCache>(lv.vis, u[k]);
      pos += 4;
      if (hit) {
        found = true;
        active = false;
      } else if (pos >= end) {
        active = false;
      }
    }
  }
  const uint32_t fm = __ballot_sync(kFull, found);
  if (found) {
    const int32_t deg = g.symmetric ? end - beg : g.off[v + 1] - g.off[v];
    lv.depth[v] = lv.next_depth;
    edges += (unsigned long long)deg;
    wbuf[wcnt + __popc(fm & lanemask_lt())] = v;
    atomicOr(lv.vis_next + (v >> 5), 1u << (v & 31));
  }
  wcnt += (unsigned)__popc(fm);
  __syncwarp();  // the list entries are read before the hint pass overwrites them
}

// After a hint-pass step: scan the misses 32 at a time while the list holds
// that many (all of them when drain), keeping the warp's stage below capacity.
template <bool kReadOnlyCache, int kWords>
__device__ __forceinline__ void pull_settle(const DevGraph& g, const Level& lv, const PullMisses<kWords>& ms,
                                            int& mcnt, bool drain, int32_t* wbuf, unsigned int& wcnt,
                                            unsigned long long& edges) {
  if (wcnt > (unsigned)(kWarpStage - kWords * 32)) {
    warp_stage_flush(wbuf, wcnt, lv);
    wcnt = 0;
  }
  while (mcnt >= 32 || (drain && mcnt > 0)) {  // uniform
    const int take = min(32, mcnt);
    mcnt -= take;
    pull_misses<kReadOnlyCache, kWords>(g, lv, ms, mcnt, take, wbuf, wcnt, edges);
    if (wcnt > (unsigned)(kWarpStage - kWords * 32)) {
      warp_stage_flush(wbuf, wcnt, lv);
      wcnt = 0;
    }
  }
}

// Two walks over the bitmap words share the hint pass. This warp's k-th word
// is (k / kWords) * stride + base0 + (k % kWords) * kWarps (consecutive warps
// take consecutive words; increasing in k), and it takes kWords per step.
//  - dense (most reachable vertices still unvisited): each step's words are
//    loaded one step ahead, and their row extents and hints prefetched into
//    L2, so those round trips overlap the current step;
//  - sparse (few left): a batch of 32 of the warp's words is loaded at once,
//    one per lane; words with no unvisited vertex are settled right there
//    (their next-bitmap word is all ones), the row extents and hints of the
//    others are prefetched into L2, and only those are taken. A late level
//    whose words are nearly all full then costs one round trip per 32 words
//    instead of one per kWords.
// scratch: pull_scratch_ints<kWords>() ints of the block's shared memory.
template <bool kReadOnlyCache>
__device__ __forceinline__ uint32_t pull_load_word(const uint32_t* vis, int32_t w) {
  return kReadOnlyCache ? ld_nc_u32(vis + w) : vis[w];
}

template <bool kReadOnlyCache, int kWords>
__device__ void body_pull(const DevGraph& g, const Level& lv, const Stage& stage, int32_t* scratch,
                          unsigned long long& edges) {
  static_assert(kWords * 32 <= kWarpStage, "a step must fit a stage slice");
  static_assert(32 % kWords == 0, "a batch holds whole steps");
  const uint32_t lane = lane_id();
  constexpr int kWarps = kThreads / 32;
  const int wib = threadIdx.x >> 5;
  int32_t* wbuf = stage.buf + wib * kWarpStage;  // the block stage is empty on entry
  unsigned int wcnt = 0;
  constexpr int kCap = PullMisses<kWords>::kCap;
  int32_t* mine = scratch + wib * 3 * kCap;
  const PullMisses<kWords> ms{mine, mine + kCap, mine + 2 * kCap};
  int mcnt = 0;
  const int stride = gridDim.x * kWarps * kWords;
  const int base0 = blockIdx.x * kWarps * kWords + wib;
  if (!lv.pull_sparse) {
    uint32_t cw_next[kWords];
#pragma unroll
    for (int j = 0; j < kWords; ++j) {
      const int wn = base0 + j * kWarps;
      cw_next[j] = wn < g.words ? pull_load_word<kReadOnlyCache>(lv.vis, wn) : kFull;
    }
    for (int wb = base0; wb < g.words; wb += stride) {
      int32_t w[kWords];
      uint32_t cw[kWords];
#pragma unroll
      for (int j = 0; j < kWords; ++j) {
        w[j] = wb + j * kWarps;
        w[j] = w[j] < g.words ? w[j] : -1;
        cw[j] = cw_next[j];
        const int wn = wb + j * kWarps + stride;
        cw_next[j] = wn < g.words ? pull_load_word<kReadOnlyCache>(lv.vis, wn) : kFull;
        if (wn < g.words) {  // the next step's row extents and hints
          prefetch_l2(g.in_off + (size_t)wn * 32);
          prefetch_l2(g.hint + (size_t)wn * 32);
        }
      }
      pull_words<kReadOnlyCache, kWords>(g, lv, w, cw, wbuf, wcnt, ms, mcnt, edges);
      pull_settle<kReadOnlyCache, kWords>(g, lv, ms, mcnt, false, wbuf, wcnt, edges);
    }
  } else {
    for (int k0 = 0;; k0 += 32) {
      const int kk = k0 + (int)lane;
      const int wl = (kk / kWords) * stride + base0 + (kk % kWords) * kWarps;
      if (__shfl_sync(kFull, wl, 0) >= g.words) break;  // uniform: lane 0 holds the batch's smallest word
      const bool inb = wl < g.words;
      const uint32_t cwl = inb ? pull_load_word<kReadOnlyCache>(lv.vis, wl) : kFull;
      const bool open = inb && cwl != kFull;
      if (inb && !open) lv.vis_next[wl] = kFull;
      if (open) {
        prefetch_l2(g.in_off + (size_t)wl * 32);
        prefetch_l2(g.hint + (size_t)wl * 32);
      }
      uint32_t todo = __ballot_sync(kFull, open);
      while (todo) {  // uniform
        int32_t w[kWords];
        uint32_t cw[kWords];
#pragma unroll
        for (int j = 0; j < kWords; ++j) {
          const int src = todo ? __ffs(todo) - 1 : 0;
          const bool have = todo != 0u;
          todo &= todo - 1u;
          w[j] = have ? __shfl_sync(kFull, wl, src) : -1;
          cw[j] = have ? __shfl_sync(kFull, cwl, src) : kFull;
        }
        pull_words<kReadOnlyCache, kWords>(g, lv, w, cw, wbuf, wcnt, ms, mcnt, edges);
        pull_settle<kReadOnlyCache, kWords>(g, lv, ms, mcnt, false, wbuf, wcnt, edges);
      }
    }
  }
  pull_settle<kReadOnlyCache, kWords>(g, lv, ms, mcnt, true, wbuf, wcnt, edges);
  if (wcnt) warp_stage_flush(wbuf, wcnt, lv);
}

// ---------------------------------------------------------------------------
// Edge list and reverse edge list (Section 3.1.1): one thread per edge of the
// whole graph, every level, four edges per thread per step (coalesced). Edge
// list: CSR entry e is the edge origin_out[e] -> idx[e], whose target is
// reached when its source is in the frontier (depth L). Reverse edge list:
// transpose entry e is in_idx[e] -> origin_in[e]; the destination's bitmap
// bit is read first, so settled destinations cost no depth read. Targets are
// claimed through the visited bitmap like the push variants', so frontier
// counts and queues stay exact.
// ---------------------------------------------------------------------------
template <bool kReverse>
__device__ void body_edge_list(const DevGraph& g, const Level& lv, const Stage& stage, unsigned long long& edges) {
  const int32_t L = lv.next_depth - 1;
  const long long m = g.m;
  const int32_t* origin = kReverse ? g.aux->origin_in : g.aux->origin_out;
  const int32_t* other = kReverse ? g.in_idx : g.idx;
  const long long step = (long long)blockDim.x * 4;
  for (long long base = (long long)blockIdx.x * step; base < m; base += (long long)gridDim.x * step) {
    int32_t v[4] = {0, 0, 0, 0};
    int nv = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const long long e = base + k * (long long)blockDim.x + threadIdx.x;
      if (e < m) {
        if (kReverse) {
          const int32_t dst = origin[e];
          if (!vis_bit<false>(lv.vis, dst) && lv.depth[other[e]] == L) v[nv++] = dst;
        } else {
          if (lv.depth[origin[e]] == L) v[nv++] = other[e];
        }
      }
    }
    visit_k<4>(g, lv, stage, v, nv, edges);
    stage_flush(stage, lv, kStageCap / 2);
  }
}

}  // namespace

// ===========================================================================
// Graph path: init, decide, and one kernel per body
// ===========================================================================
__global__ void __launch_bounds__(kThreads) k_init(DevGraph g, Buffers b, RunState* st, int32_t* depth, int32_t root,
                                                   int32_t forced, const TreeNode* tree, int32_t tree_nodes,
                                                   const QsTree* tree_qs, int32_t use_handles,
                                                   unsigned long long h_while, unsigned long long h_switch) {
  if (blockIdx.x == 0 && threadIdx.x == 0) st->t_entry = (long long)global_ns();
  init_fill(g, b.vis[0], depth, root);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->depth = depth;
    st->tree = tree;
    st->tree_qs = tree_qs;
    st->tree_nodes = tree_nodes;
    st->root = root;
    st->forced = forced;
    st->h_while = h_while;
    st->h_switch = h_switch;
    st->use_handles = use_handles;
    st->level = -1;
    st->variant = -1;
    st->qsel = 0;
    st->vsel = 0;
    st->frontier = 0;
    st->status = ST_OK;
    st->vw = 32;
    st->vw_policy = g.vw_policy;
    st->levels = 0;
    st->frontier_edges = 0;
    st->discovered = 0;
    st->edges_reached = 0;
    st->small_tail = 0;
    // the root is the output of "level -1": the first decide turns it into the frontier of level 0
    b.q[1][0] = root;
    st->next_count = 1;
    st->next_edges = (unsigned long long)(g.off[root + 1] - g.off[root]);
  }
}

// First node of the level-loop graph: opens the WHILE loop from the device.
// (The handle has no launch-time default: a value applied by the host when a
// launch is enqueued could reach a still-running earlier launch of the same
// graph on that stream; a kernel inside the launch is ordered with it.)
__global__ void k_loop_start(DevGraph g, Buffers b, RunState* st) {
  (void)g;
  (void)b;
  if (threadIdx.x == 0 && blockIdx.x == 0) cudaGraphSetConditional((cudaGraphConditionalHandle)st->h_while, 1u);
}

// Level end + tree evaluation, between levels on the device. Launched with
// kDecideThreads threads (one warp): lane 0 closes the level and keeps the
// state; the warp evaluates a tree that has a bit-parallel form, else lane 0
// walks it.
__global__ void __launch_bounds__(kDecideThreads) k_decide(DevGraph g, Buffers b, RunState* st) {
  (void)b;
  __shared__ long long s_in[3];  // f, e, discovered
  __shared__ int32_t s_go;       // 1: evaluate the tree this level
  RunState& s = *st;
  int32_t L = 0;
  if (threadIdx.x == 0) {
    // close level L-1: its output queue becomes the frontier of level L
    const unsigned int f = (unsigned int)*reinterpret_cast<volatile unsigned long long*>(&s.next_count);
    const unsigned long long e = *reinterpret_cast<volatile unsigned long long*>(&s.next_edges);
    s.next_count = 0;
    s.next_edges = 0;
    s.heavy3[0] = 0;
    if (s.level >= 0 && s.variant == V_PULL) s.vsel ^= 1u;  // pull wrote the other bitmap
    s.qsel ^= 1u;
    L = s.level + 1;
    s.level = L;
    s.frontier = (int32_t)f;
    s.frontier_edges = (long long)e;
    s.discovered += f;
    s.edges_reached += (long long)e;
    // a traversal has at most n nonempty levels; more means corrupted state, so
    // end the loop with an error instead of iterating on
    if (L > g.n || s.discovered > g.n) s.status = ST_TIMEOUT;
    if (L < s.log_cap) s.log_time[L] = (long long)global_ns();
    s_go = 1;
    if (f == 0 || s.status != ST_OK) {
      s.levels = L;
      if (s.use_handles) {
        cudaGraphSetConditional((cudaGraphConditionalHandle)s.h_while, 0u);
        cudaGraphSetConditional((cudaGraphConditionalHandle)s.h_switch, (unsigned)V_FORCED_NUM);
      }
      s_go = 0;
    }
    s_in[0] = f;
    s_in[1] = (long long)e;
    s_in[2] = s.discovered;
  }
  __syncthreads();
  if (!s_go) return;  // uniform
  const long long f = s_in[0], e = s_in[1], discovered = s_in[2];
  L = st->level;
  int32_t v = s.forced;
  const QsTree* qs = s.tree_qs;
  if (v < 0 && qs != nullptr) v = qs_eval_warp(*qs, L, f, e, discovered);  // the whole warp
  if (threadIdx.x != 0) return;
  if (v < 0 && qs == nullptr && s.tree != nullptr && s.tree_nodes > 0)
    v = walk_tree(g, s.tree, s.tree_nodes, L, f, e, discovered);
  if (s.forced < 0) v = known_variant(v, L, s.variant);
  const int32_t vw = warp_width(f, e, s.vw_policy);
  for (int i = 0; i < F_NUM; ++i) s.feat[i] = feature_value(g, i, L, f, e, discovered);
  s.variant = v;
  s.vw = vw;
  if (L < s.log_cap) {
    s.log_variant[L] = v;
    s.log_frontier[L] = f;
    s.log_edges[L] = e;
  }
  if (s.use_handles) cudaGraphSetConditional((cudaGraphConditionalHandle)s.h_switch, (unsigned)v);
}

// Vertex push with the other frontier-count modes (Section 3.1.4 comparison).
__global__ void __launch_bounds__(kThreads) k_push_thread_warp_count(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_push_thread<CM_WARP>(g, lv, stage, edges);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_push_thread_atomic_count(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_push_thread<CM_ATOMIC>(g, lv, stage, edges);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_push_thread(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_push_thread(g, lv, stage, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_push_warp(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_push_warp(g, lv, stage, st->vw, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_push_cta(DevGraph g, Buffers b, RunState* st) {
  __shared__ alignas(128) int32_t chunk[2 * kCtaChunk];
  __shared__ alignas(8) uint64_t bar[2];
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  cta_pipe_init(bar);
  CtaPipe pp{chunk, bar, 0u, 0u, 0u};
  unsigned long long edges = 0;
  body_push_cta(g, lv, stage, pp, &st->status, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_push_edge(DevGraph g, Buffers b, RunState* st) {
  __shared__ int32_t s_a[kPeTile];
  __shared__ int32_t s_beg[kPeTile];
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  if (lv.shared_scan)
    body_push_shared(g, lv, lv.qin, lv.frontier, stage, s_a, s_beg, edges);
  else
    body_push_tiles(g, lv, stage, s_a, s_beg, b.heavy, b.heavy_cap, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

// (Returns at once when nothing was set aside.)
__global__ void __launch_bounds__(kThreads) k_push_heavy(DevGraph g, Buffers b, RunState* st) {
  __shared__ int32_t s_a[kPeTile];
  __shared__ int32_t s_beg[kPeTile];
  const unsigned int count = st->heavy3[0];
  if (count == 0u) return;
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_push_heavy(g, lv, stage, s_a, s_beg, b.heavy, (int32_t)min(count, (unsigned)b.heavy_cap), edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_edge_list(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_edge_list<false>(g, lv, stage, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

__global__ void __launch_bounds__(kThreads) k_rev_edge_list(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  body_edge_list<true>(g, lv, stage, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

// fn(e, v) for every CSR entry e and the vertex v whose row [off[v], off[v + 1])
// holds it. A block takes kPeTile consecutive entries, finds the rows that hold
// them and each entry's row by binary search (in shared memory unless empty
// rows make them many), so a hub's row is shared out like any other. (A thread
// per row spent 19.9 ms in the transpose of a directed R-MAT graph of 2^20
// vertices and 15.9M edges, walking its longest row; creation with one traversal
// takes 2.2 ms in all with this and the summaries in one pass, 24.1 before.)
template <typename Fn>
__device__ __forceinline__ void for_each_entry(const int32_t* off, int32_t n, int32_t m, Fn fn) {
  __shared__ int32_t s_off[kPeTile];
  __shared__ int32_t s_row[2];
  for (long long c0 = (long long)blockIdx.x * kPeTile; c0 < m; c0 += (long long)gridDim.x * kPeTile) {
    const int32_t c1 = (int32_t)min(c0 + kPeTile, (long long)m);
    if (threadIdx.x < 2) {  // the last row that starts at or before the chunk's first / last entry
      const int32_t e = threadIdx.x ? c1 - 1 : (int32_t)c0;
      int32_t lo = 0, hi = n - 1;
      while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (off[mid] <= e)
          lo = mid;
        else
          hi = mid - 1;
      }
      s_row[threadIdx.x] = lo;
    }
    __syncthreads();
    const int32_t r0 = s_row[0], rows = s_row[1] - r0 + 1;
    const bool shared = rows <= kPeTile;  // uniform
    if (shared)
      for (int32_t r = threadIdx.x; r < rows; r += blockDim.x) s_off[r] = off[r0 + r];
    __syncthreads();
    const int32_t* start = shared ? s_off : off + r0;
    const int32_t len = c1 - (int32_t)c0;  // stepped from 0: an entry number past the end might not fit 32 bits
    for (int32_t i = (int32_t)threadIdx.x; i < len; i += kThreads) {
      const int32_t e = (int32_t)c0 + i;
      int32_t lo = 0, hi = rows - 1;
      while (lo < hi) {
        const int32_t mid = lo + (hi - lo + 1) / 2;
        if (start[mid] <= e)
          lo = mid;
        else
          hi = mid - 1;
      }
      fn(e, r0 + lo);
    }
    __syncthreads();
  }
}

// Origin of every CSR entry: the vertex whose row holds it.
__global__ void __launch_bounds__(kThreads) k_build_origin(const int32_t* off, int32_t n, int32_t m, int32_t* origin) {
  for_each_entry(off, n, m, [=](int32_t e, int32_t v) { origin[e] = v; });
}

__global__ void __launch_bounds__(kThreads) k_pull(DevGraph g, Buffers b, RunState* st) {
  BFS_DECLARE_STAGE(stage);
  const Level lv = load_level(g, b, st);
  unsigned long long edges = 0;
  __shared__ int32_t s_scratch[pull_scratch_ints<kPullWordsLaunch>()];
  body_pull<true, kPullWordsLaunch>(g, lv, stage, s_scratch, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &st->next_edges);
}

// ===========================================================================
// Persistent path: the whole traversal in one cooperative launch
// ===========================================================================
// Timing harness: undo one level run from the graph path's state. The vertices
// the level discovered are exactly the entries it appended to the output
// queue, so resetting their depth and visited bit restores the state it
// started from, in time proportional to the level's output (pull wrote only
// the other bitmap, which is rewritten whole before it is read again).
__global__ void k_undo_level(Buffers b, RunState* st) {
  const unsigned int count = (unsigned int)st->next_count;
  const int32_t* qout = st->qsel ? b.q[0] : b.q[1];
  uint32_t* vis = st->vsel ? b.vis[1] : b.vis[0];
  int32_t* depth = st->depth;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
    const int32_t v = qout[i];
    depth[v] = -1;
    atomicAnd(&vis[v >> 5], ~(1u << (v & 31)));
  }
}

// One shared-memory buffer serves the CTA variant's copy stage or the
// edge-centric tile of the persistent kernels.
constexpr int kPeSlot = kPeTile + 32;
static_assert(2 * kCtaChunk <= 2 * kPeSlot, "union sizing");
static_assert(pull_scratch_ints<kPullWordsPersistent>() <= 2 * kPeSlot, "union sizing");

// Level L of a persistent traversal (frontier in q[L & 1], appending to
// q[(L + 1) & 1] and to the level words of the given slot; current bitmap
// vis[vsel]).
__device__ __forceinline__ Level persistent_level(const DevGraph& g, const Buffers& b, RunState* st, int32_t* depth,
                                                  int32_t L, unsigned int f, unsigned long long e,
                                                  long long discovered, uint32_t vsel, uint32_t slot) {
  Level lv;
  lv.qin = (L & 1) ? b.q[1] : b.q[0];
  lv.qout = (L & 1) ? b.q[0] : b.q[1];
  lv.vis = vsel ? b.vis[1] : b.vis[0];
  lv.vis_next = vsel ? b.vis[0] : b.vis[1];
  lv.depth = depth;
  lv.tail = &st->tail3[slot];
  lv.n_heavy = &st->heavy3[slot];
  lv.next_depth = L + 1;
  lv.frontier = (int32_t)f;
  lv.shared_scan = pe_shared(f, (long long)e, g.gfeat[F_DEG_MAX] >= kHeavy);
  lv.latency_bound = (long long)e < kLatencyEdges;
  lv.pull_sparse = (long long)g.n_active - discovered < (long long)(g.n_active >> 4);
  return lv;
}

// The level's work with variant v inside a persistent kernel (every block of
// the cooperative grid calls it); returns the block's sum of the reached
// vertices' out-degrees, after the block's appends are flushed.
__device__ __forceinline__ unsigned long long persistent_level_work(const DevGraph& g, const Buffers& b, RunState* st,
                                                                    const Level& lv, int32_t v, int32_t vw,
                                                                    const Stage& stage, CtaPipe& pp, int32_t* ubuf,
                                                                    unsigned long long& bar_target) {
  unsigned long long edges = 0;
  switch (v) {
    case V_PUSH_THREAD: body_push_thread(g, lv, stage, edges); break;
    case V_PUSH_WARP: body_push_warp(g, lv, stage, vw, edges); break;
    case V_PUSH_CTA: body_push_cta(g, lv, stage, pp, &st->status, edges); break;
    case V_PUSH_EDGE:
      if (lv.shared_scan) {
        body_push_shared(g, lv, lv.qin, lv.frontier, stage, ubuf, ubuf + kPeSlot, edges);
        break;
      }
      body_push_tiles(g, lv, stage, ubuf, ubuf + kPeSlot, b.heavy, b.heavy_cap, edges);
      if (g.gfeat[F_DEG_MAX] < kHeavy) break;  // nothing can have been set aside
      if (!grid_arrive_wait(&st->bar64, bar_target, &st->status)) break;
      body_push_heavy(g, lv, stage, ubuf, ubuf + kPeSlot, b.heavy,
                      (int32_t)min(*reinterpret_cast<volatile unsigned int*>(lv.n_heavy), (unsigned)b.heavy_cap), edges);
      break;
    case V_EDGE_LIST: body_edge_list<false>(g, lv, stage, edges); break;
    case V_REV_EDGE_LIST: body_edge_list<true>(g, lv, stage, edges); break;
    default: body_pull<false, kPullWordsPersistent>(g, lv, stage, ubuf, edges); break;
  }
  stage_flush(stage, lv, 1);
  return block_sum_u64(edges);
}

// The tree's choice of a level's variant, for every lane of the calling warp.
struct TreeChoice {
  const QsTree* qs;  // bit-parallel form (shared memory), or null
  const TreeNode* tree;
  int32_t nodes;
  // lanes 0-7 of each warp: the box of the leaf the last evaluated level
  // reached (in_leaf_box); leaf < 0 until a level has been evaluated
  mutable int32_t bound, leaf;

  // Section 4.1's rule for unknown predictions included.
  __device__ __forceinline__ int32_t choose(const DevGraph& g, int32_t L, unsigned int f, long long e,
                                            long long discovered, int32_t prev) const {
    int32_t v = -1;
    if (qs != nullptr) {
      // same leaf box as the previous level: the walk reaches the same leaf, and
      // the level repeats the previous level's choice (for an unknown leaf too)
      if (leaf >= 0 && in_leaf_box(bound, L, f, e, discovered)) {
        v = prev;
      } else {
        leaf = qs_leaf_warp(*qs, L, f, e, discovered);
        v = leaf >= 0 ? qs->leaf[leaf] : -1;
        bound = (leaf >= 0 && lane_id() < 8u) ? qs->box[leaf][lane_id()] : 0;
      }
    } else if (tree != nullptr && nodes > 0) {
      v = walk_tree(g, tree, nodes, L, f, e, discovered);
    }
    return known_variant(v, L, prev);
  }
};

// The per-level log's buffers, read once per launch.
struct RunLog {
  int32_t cap;
  int32_t* variant;
  long long* frontier;
  long long* edges;
  long long* time;
};

__device__ __forceinline__ void log_level(const RunLog& log, int32_t L, int32_t v, unsigned int f, long long e) {
  if (L < log.cap) {
    log.variant[L] = v;
    log.frontier[L] = f;
    log.edges[L] = e;
    log.time[L] = (long long)global_ns();
  }
}

}  // namespace bfs

#include "bfs_small.cuh"

namespace bfs {

// epoch: a number the host changes on every launch on this workspace. Block 0
// clears the barrier counter and the status word left by the previous run
// (which a failed run may leave set) and then publishes epoch; every other
// block waits for it before its first barrier, so no separate reset launch is
// needed.
// stall: STALL_NONE, or the test hook's choice of one bounded wait to run out.
// kRecord: 0, or the entries of the graph's vertex records (4 or 8); then small
// levels run on the leader cluster (bfs_small.cuh).
// Four blocks an SM: at their 64 registers 60 to 68 bytes a thread are spilled (120
// to 144 read back); five blocks at 48 registers spilled 216 and ran R-MAT 22 9 %
// slower.
template <int kRecord>
__global__ void __launch_bounds__(kThreads, 4) k_bfs_persistent(const __grid_constant__ DevGraph g,
                                                             const __grid_constant__ Buffers b, RunState* st,
                                                             int32_t* depth, int32_t root, int32_t forced,
                                                             const TreeNode* tree, int32_t tree_nodes,
                                                             const QsTree* qs, uint32_t epoch, int32_t stall) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->t_entry = (long long)global_ns();
    st->bar64 = 0;
    st->status = ST_OK;
    for (int k = 0; k < 3; ++k) {
      st->tail3[k] = 0;
      st->edg3[k] = 0;
      st->heavy3[k] = 0;
    }
    st->small_tail = 0;
    st->small_seq = 0;
    st->small_beat = 0;
    st_release_u32(&st->run_epoch, epoch);
  }
  __shared__ alignas(128) int32_t ubuf[2 * kPeSlot];
  static_assert(2 * kPeSlot >= 4 * kCandCap && kStageCap >= kWonCap, "the leader's queues");
  __shared__ alignas(8) uint64_t bar[2];
  __shared__ SmallShared s_small;
  __shared__ RunLog s_log;
  // the tree is evaluated by every warp every level: its bit-parallel form
  // (trees of up to 64 leaves) is kept in shared memory; larger trees are
  // walked in global memory
  __shared__ QsTree s_qs;
  const bool use_qs = qs != nullptr;
  if (use_qs) {
    static_assert(sizeof(QsTree) % 4 == 0, "QsTree copy");
    const uint32_t* src = reinterpret_cast<const uint32_t*>(qs);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&s_qs);
    for (int i = threadIdx.x; i < (int)(sizeof(QsTree) / 4); i += blockDim.x) dst[i] = src[i];
  }
  BFS_DECLARE_STAGE(stage);
  init_fill(g, b.vis[0], depth, root);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->depth = depth;
    st->root = root;
    st->forced = forced;
    b.q[0][0] = root;
  }
  if (threadIdx.x == 0) {
    s_log = RunLog{st->log_cap, st->log_variant, st->log_frontier, st->log_edges, st->log_time};
    const bool late = kRecord > 0 && stall == STALL_LEADER_MESSAGE && blockIdx.x + 1u == cluster_size();
    mbar_init(&s_small.bar[0], 1);
    mbar_init(&s_small.bar[1], late ? 2 : 1);
    s_small.failed = s_small.run_no = 0u;
    for (int i = 0; i < kMaxCluster; ++i) s_small.ended[i] = 0u;
    s_small.mute = stall == STALL_LEADER_STATE ? 1u : 0u;
  }
  cta_pipe_init(bar);
  CtaPipe pp{ubuf, bar, 0u, 0u, stall == STALL_BULK_COPY ? 16u : 0u};
  // the previous run's barrier state is cleared before any block arrives
  if (blockIdx.x != 0 && threadIdx.x == 0) {
    const unsigned long long t0 = global_ns();
    while (ld_acquire_u32(&st->run_epoch) != epoch)
      if (global_ns() - t0 > kWaitLimitNs) break;  // the first barrier then times out and reports it
  }
  // small levels go to cluster 0 when the tree drives the run (a forced
  // variant is timed as itself; a launch whose grid barriers are stalled keeps them)
  const bool small_on = kRecord > 0 && forced < 0 && (stall == STALL_NONE || stall >= STALL_LEADER_MESSAGE) &&
                        cluster_size() > 1u && cluster_size() <= (uint32_t)kMaxCluster;
  uint32_t vsel = 0;
  uint32_t slot = 0;  // level words: this level's slot (the levels run on the whole grid, modulo 3)
  const TreeChoice tc{use_qs ? &s_qs : nullptr, tree, tree_nodes, 0, -1};
  if (threadIdx.x == 0) {
    s_small.out.reached = 0;
    s_small.out.exchanges = 0;
    s_small.runs = 0;
  }
  int32_t L = 0, prev = -1;
  bool force_full = false;
  long long discovered = 0;
  // level 0's frontier is the root; later levels' f and e arrive with the barrier
  unsigned int f = 1;
  unsigned long long e = (unsigned long long)(g.off[root + 1] - g.off[root]);
  unsigned long long bar_target = 0;  // this block's copy of the grid barriers' arrival target
  bool ok = grid_arrive_wait(&st->bar64, bar_target, &st->status, stall == STALL_GRID_BARRIER ? 1u : 0u);
  while (ok && f != 0) {
    if (L > g.n || discovered + f > g.n) {  // corrupted state: stop with an error
      if (blockIdx.x == 0 && threadIdx.x == 0) st->status = ST_TIMEOUT;
      break;
    }
    const int32_t v = forced >= 0 ? forced : tc.choose(g, L, f, (long long)e, discovered + f, prev);
    if (kRecord > 0 && small_on && !force_full && v != V_PULL && small_fits(f, e, cluster_size())) {
      if (blockIdx.x < cluster_size()) {
        if (threadIdx.x == 0) {
          s_small.out.discovered = discovered;
          s_small.out.e = e;
          s_small.out.f = f;
          s_small.out.L = L;
          s_small.out.prev = prev;
        }
        __syncthreads();
        small_run<kRecord == 8 ? 8 : 4>(g, b, vsel ? b.vis[1] : b.vis[0], depth, st, tc.qs, tree, tree_nodes, s_log, s_small, ubuf, stage.buf,
                  v);
      } else {
        small_park(st, s_small);
      }
      __syncthreads();
      discovered = s_small.out.discovered;
      e = s_small.out.e;
      f = s_small.out.f;
      L = s_small.out.L;
      prev = s_small.out.prev;
      force_full = s_small.out.force_full != 0;
      ok = s_small.out.ok != 0;
      tc.leaf = -1;  // prev is not the class of this block's last leaf any more
      __syncthreads();
      continue;
    }
    force_full = false;
    discovered += f;
    if (threadIdx.x == 0) s_small.out.reached += (long long)e;
    const uint32_t next = slot == 2u ? 0u : slot + 1u;
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) {
        const uint32_t after = next == 2u ? 0u : next + 1u;
        st->tail3[after] = 0;  // the slot of a barrier every block has left
        st->edg3[after] = 0;
        st->heavy3[after] = 0;
      }
      if (threadIdx.x == kThreads - 1) log_level(s_log, L, v, f, (long long)e);
    }
    const Level lv = persistent_level(g, b, st, depth, L, f, e, discovered, vsel, next);
    const int32_t vw = warp_width(f, (long long)e, g.vw_policy);
    const unsigned long long e_block = persistent_level_work(g, b, st, lv, v, vw, stage, pp, ubuf, bar_target);
    if (v == V_PULL) vsel ^= 1u;
    prev = v;
    ok = level_arrive_wait(&st->tail3[next], &st->edg3[next], e_block, &st->status, &f, &e,
                           (stall == STALL_LEVEL_BARRIER && L == 0) ? 1u : 0u);
    slot = next;
    ++L;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->levels = L;
    if (L < s_log.cap) s_log.time[L] = (long long)global_ns();
    st->discovered = discovered;
    st->edges_reached = s_small.out.reached;
  }
  // no block of a cluster ends while another may still send to its shared memory
  if (kRecord > 0 && cluster_size() > 1u) small_end(s_small, cluster_size(), cluster_rank(), ~0u, ok);
}

// Graph driver, before each level's decision, for graphs with vertex records
// (one cluster): runs the next level and those after it while they are small,
// and leaves the state as k_decide expects it (the output queue of the level
// before is in q[qsel ^ 1]). In this driver level L's queue is q[(L + 1) & 1].
// (777 x 1021 grid, 1,338 levels, in this driver: 17 us a level with a decision
// and a level kernel each, 1.6 us in runs; 22 -> 2.2 ms a traversal.)
template <int kRecord>
__global__ void __launch_bounds__(kThreads) k_small_levels(const __grid_constant__ DevGraph g, Buffers b,
                                                           RunState* st) {
  __shared__ alignas(128) int32_t ubuf[4 * kCandCap];
  __shared__ int32_t sbuf[kWonCap];
  __shared__ SmallShared s_small;
  __shared__ RunLog s_log;
  const int32_t L = st->level + 1;
  const unsigned int f = (unsigned int)st->next_count;
  const unsigned long long e = st->next_edges;
  const long long discovered = st->discovered;
  // k_decide switches to the bitmap a pull level wrote; this kernel runs first
  const uint32_t vsel = st->vsel ^ (uint32_t)(st->level >= 0 && st->variant == V_PULL);
  if (st->forced >= 0 || st->status != ST_OK || f == 0 || !small_fits(f, e, cluster_size())) return;  // uniform
  const TreeChoice tc{st->tree_qs, st->tree, st->tree_nodes, 0, -1};
  const int32_t v = tc.choose(g, L, f, (long long)e, discovered + f, st->variant);
  if (v == V_PULL) return;  // uniform over the cluster: every block reads the same state
  if (threadIdx.x == 0) {
    s_log = RunLog{st->log_cap, st->log_variant, st->log_frontier, st->log_edges, st->log_time};
    s_small.out = TravState{discovered, st->edges_reached, e, f, L, st->variant, 0, 1, 0u};
    s_small.failed = s_small.mute = s_small.run_no = 0u;
    for (int i = 0; i < kMaxCluster; ++i) s_small.ended[i] = 0u;
    mbar_init(&s_small.bar[0], 1);
    mbar_init(&s_small.bar[1], 1);
    mbar_fence_init();
  }
  cluster_barrier();  // the state is read and every block's mbarriers are ready
  const Buffers swapped{{b.q[1], b.q[0]}, {b.vis[0], b.vis[1]}, b.heavy, b.heavy_cap, 0};
  small_run<kRecord>(g, swapped, vsel ? b.vis[1] : b.vis[0], st->depth, st, tc.qs, tc.tree, tc.nodes, s_log,
                     s_small, ubuf, sbuf, v);
  if (cluster_rank() == 0u && threadIdx.x == 0 && s_small.out.L > L) {
    const TravState& t = s_small.out;
    st->level = t.L - 1;
    st->vsel = vsel;
    st->qsel = (uint32_t)(t.L & 1);
    st->variant = t.prev;
    st->next_count = t.f;
    st->next_edges = t.e;
    st->discovered = t.discovered;
    st->edges_reached = t.reached;
  }
  cluster_barrier();  // no block ends while another may still send to its shared memory
}

void* small_levels_kernel(int32_t record) {
  return record == 8 ? reinterpret_cast<void*>(&k_small_levels<8>) : reinterpret_cast<void*>(&k_small_levels<4>);
}

void* persistent_kernel(int32_t record) {
  return record == 8   ? reinterpret_cast<void*>(&k_bfs_persistent<8>)
         : record == 4 ? reinterpret_cast<void*>(&k_bfs_persistent<4>)
                       : reinterpret_cast<void*>(&k_bfs_persistent<0>);
}

// Per-level timing harness inside the persistent driver: one cooperative
// launch expands level L of a traversal whose state (queues, bitmaps, depths)
// the host has advanced to that level, with variant v, exactly as the
// persistent traversal would (the same level code, grid and barrier), and
// records the device time from the start barrier to the end of the
// level-ending barrier, with the next frontier's size and edge count. The host
// clears the arrival count and the (L + 1) % 3 level words before each launch.
__global__ void __launch_bounds__(kThreads, 4) k_profile_level(DevGraph g, Buffers b, RunState* st, int32_t* depth,
                                                            int32_t L, int32_t v, uint32_t f, unsigned long long e,
                                                            long long discovered, uint32_t vsel) {
  __shared__ alignas(128) int32_t ubuf[2 * kPeSlot];
  __shared__ alignas(8) uint64_t bar[2];
  BFS_DECLARE_STAGE(stage);
  cta_pipe_init(bar);
  CtaPipe pp{ubuf, bar, 0u, 0u, 0u};
  const int32_t vw = warp_width(f, (long long)e, g.vw_policy);
  unsigned long long bar_target = 0;
  if (!grid_arrive_wait(&st->bar64, bar_target, &st->status)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) st->prof_t0 = (long long)global_ns();
  const Level lv = persistent_level(g, b, st, depth, L, f, e, discovered, vsel, (uint32_t)((L + 1) % 3));
  const unsigned long long e_block = persistent_level_work(g, b, st, lv, v, vw, stage, pp, ubuf, bar_target);
  unsigned int fn = 0;
  unsigned long long en = 0;
  if (!level_arrive_wait(&st->tail3[(L + 1) % 3], &st->edg3[(L + 1) % 3], e_block, &st->status, &fn, &en)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->prof_t1 = (long long)global_ns();
    st->prof_f = fn;
    st->prof_e = en;
  }
}

// Before a profiled level: clear the arrival count, the status and the level
// words the level appends to.
__global__ void k_profile_reset(RunState* st, int32_t slot) {
  st->bar64 = 0;
  st->status = ST_OK;
  st->tail3[slot] = 0;
  st->edg3[slot] = 0;
  st->heavy3[slot] = 0;
}

// Undo a profiled level in the persistent layout: the `count` vertices it
// appended to q[qout] lose their depth and their bit in vis[vsel] (pull set no
// bit there; it wrote the other bitmap, which the next pull rewrites whole).
__global__ void k_undo_level_p(Buffers b, int32_t* depth, uint32_t qout, unsigned int count, uint32_t vsel) {
  const int32_t* q = qout ? b.q[1] : b.q[0];
  uint32_t* vis = vsel ? b.vis[1] : b.vis[0];
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += stride) {
    const int32_t v = q[i];
    depth[v] = -1;
    atomicAnd(&vis[v >> 5], ~(1u << (v & 31)));
  }
}

// ---------------------------------------------------------------------------
// Graph creation: validation, out-degree statistics, transpose
// ---------------------------------------------------------------------------
__global__ void k_validate(const int32_t* off, const int32_t* idx, int32_t n, int32_t m, int32_t* bad) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int32_t my = 0;
  if (tid == 0 && (off[0] != 0 || off[n] != m)) my = 1;
  for (int64_t v = tid; v < n; v += stride)
    if (off[v + 1] < off[v]) my = 1;
  for (int64_t e = tid; e < m; e += stride)
    if (idx[e] < 0 || idx[e] >= n) my = 1;
  if (my) atomicOr(bad, 1);
}

// Degrees for the statistics: out (row length in off), in (in off_in) and
// total, three summaries in one pass over the vertices; off_in null for a
// symmetric graph, whose in-degree summary is its out-degree one and whose
// total degrees are twice the out-degrees, so that only the first is taken.
__device__ __forceinline__ void stat_degrees(const int32_t* off, const int32_t* off_in, int64_t v, unsigned int (&d)[3]) {
  d[0] = (unsigned int)(off[v + 1] - off[v]);
  d[1] = off_in ? (unsigned int)(off_in[v + 1] - off_in[v]) : 0u;
  d[2] = d[0] + d[1];
}

// Sums, sums of squares, minima and maxima of the (up to) three degrees.
__global__ void __launch_bounds__(kThreads) k_deg_reduce(const int32_t* off, const int32_t* off_in, int32_t n,
                                                         DegSums* out) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int kinds = off_in ? 3 : 1;
  unsigned long long a[3] = {0, 0, 0}, q[3] = {0, 0, 0};
  unsigned int hi[3] = {0, 0, 0};
  for (int64_t v = tid; v < n; v += stride) {
    unsigned int d[3];
    stat_degrees(off, off_in, v, d);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k] += (unsigned long long)d[k];
      q[k] += (unsigned long long)d[k] * (unsigned long long)d[k];
      hi[k] = max(hi[k], d[k]);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (k >= kinds) break;  // uniform
    block_add_u64(a[k], &out[k].s1);
    block_add_u64(q[k], &out[k].s2);
    const unsigned int h = __reduce_max_sync(kFull, hi[k]);
    if (lane_id() == 0) atomicMax(&out[k].dmax, h);
  }
}

// Histograms of the degrees, kind k's at hist + at[k]. Degrees below kDegShared
// are counted in shared memory first (most vertices share a few small degrees).
constexpr int kDegShared = 512;
__global__ void __launch_bounds__(kThreads) k_deg_hist(const int32_t* off, const int32_t* off_in, int32_t n,
                                                       long long at1, long long at2, int32_t* hist) {
  __shared__ int32_t s_hist[3 * kDegShared];
  const int kinds = off_in ? 3 : 1;
  for (int i = threadIdx.x; i < 3 * kDegShared; i += blockDim.x) s_hist[i] = 0;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    unsigned int d[3];
    stat_degrees(off, off_in, v, d);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (k < kinds) {
        if (d[k] < (unsigned)kDegShared)
          atomicAdd(&s_hist[k * kDegShared + d[k]], 1);
        else
          atomicAdd(&hist[(k == 0 ? 0 : k == 1 ? at1 : at2) + d[k]], 1);
      }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kinds * kDegShared; i += blockDim.x)
    if (s_hist[i]) {
      const int kk = i / kDegShared;
      atomicAdd(&hist[(kk == 0 ? 0 : kk == 1 ? at1 : at2) + i % kDegShared], s_hist[i]);
    }
}

namespace {
__device__ unsigned long long isqrt_u128(unsigned __int128 x) {
  unsigned long long lo = 0, hi = 0xffffffffull << 32 | 0xffffffffull;
  // largest r with r*r <= x (r < 2^64)
  while (lo < hi) {
    const unsigned long long mid = lo + ((hi - lo) >> 1) + 1;
    if ((unsigned __int128)mid * mid <= x)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}
}  // namespace

// Block b: 5-number summary by nearest rank (q_k = sorted[floor(k (n-1)/4)])
// from kind b's degree histogram, and floor(256 sigma) exactly: isqrt(65536 (n
// S2 - S1^2)) / n. symmetric: block 1 gives the total degree's summary, whose
// values are twice the out-degree's.
constexpr int kDegItems = 4;
__global__ void __launch_bounds__(kDegFinishThreads) k_deg_finish(const int32_t* hist, long long at1, long long at2,
                                                                  int32_t n, const DegSums* sums, int32_t symmetric,
                                                                  long long* out) {
  __shared__ long long carry_s;
  const int kind = symmetric ? 0 : (int)blockIdx.x;
  const long long twice = symmetric && blockIdx.x == 1 ? 2 : 1;
  const int32_t* h = hist + (kind == 0 ? 0 : kind == 1 ? at1 : at2);
  const long long maxdeg = sums[kind].dmax;
  long long* out6 = out + 6 * blockIdx.x;
  long long rank[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) rank[k] = ((long long)k * (n - 1)) / 4;
  if (threadIdx.x == 0) carry_s = 0;
  __syncthreads();
  for (long long base = 0; base <= maxdeg; base += (long long)blockDim.x * kDegItems) {
    const long long d0 = base + (long long)threadIdx.x * kDegItems;
    long long c[kDegItems], sum = 0;
#pragma unroll
    for (int i = 0; i < kDegItems; ++i) {
      c[i] = d0 + i <= maxdeg ? h[d0 + i] : 0;
      sum += c[i];
    }
    long long tot;
    long long before = carry_s + block_exclusive_scan<long long>(sum, &tot);  // vertices with degree < d0
#pragma unroll
    for (int i = 0; i < kDegItems; ++i) {
      // d is the k-th quantile when before <= rank_k < before + c
#pragma unroll
      for (int k = 0; k < 5; ++k)
        if (c[i] > 0 && before <= rank[k] && rank[k] < before + c[i]) out6[k] = twice * (d0 + i);
      before += c[i];
    }
    __syncthreads();
    if (threadIdx.x == 0) carry_s += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const unsigned __int128 S1 = sums[kind].s1, S2 = sums[kind].s2;
    const unsigned __int128 var_n2 = ((unsigned __int128)n * S2 - S1 * S1) * (unsigned)(twice * twice);
    out6[5] = (long long)(isqrt_u128(var_n2 * 65536u) / (unsigned long long)n);
  }
}

__global__ void k_tr_count(const int32_t* idx, int32_t m, int32_t* cnt) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = tid; e < m; e += stride) atomicAdd(&cnt[idx[e]], 1);
}

// Generic exclusive scan of int32 (three kernels): per-block sums, scan of the
// block sums, apply. Blocks of kThreads threads x kPeItems items.
__global__ void __launch_bounds__(kThreads) k_scan_reduce(const int32_t* in, int32_t len, long long* bsum) {
  const int nblk = (int)(((long long)len + kPeTile - 1) / kPeTile);  // len may lie 1 below 2^31 - 1
  for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    long long s = 0;
#pragma unroll
    for (int k = 0; k < kPeItems; ++k) {
      const long long i = (long long)blk * kPeTile + k * kThreads + threadIdx.x;
      if (i < len) s += in[i];
    }
    long long tot;
    block_exclusive_scan<long long>(s, &tot);
    if (threadIdx.x == 0) bsum[blk] = tot;
  }
}

__global__ void __launch_bounds__(kThreads) k_scan_top(long long* bsum, int32_t nblk) {
  long long carry = 0;
  for (int base = 0; base < nblk; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const long long x = i < nblk ? bsum[i] : 0;
    long long tot;
    const long long ex = block_exclusive_scan<long long>(x, &tot);
    if (i < nblk) bsum[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) bsum[nblk] = carry;
}

__global__ void __launch_bounds__(kThreads) k_scan_apply(const int32_t* in, int32_t len, const long long* bsum,
                                                         int32_t* out) {
  const int nblk = (int)(((long long)len + kPeTile - 1) / kPeTile);  // len may lie 1 below 2^31 - 1
  for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    const long long base = (long long)blk * kPeTile + threadIdx.x * kPeItems;
    int32_t d[kPeItems];
#pragma unroll
    for (int k = 0; k < kPeItems; ++k) d[k] = (base + k < len) ? in[base + k] : 0;
    long long run = 0;
    long long ex_k[kPeItems];
#pragma unroll
    for (int k = 0; k < kPeItems; ++k) {
      ex_k[k] = run;
      run += d[k];
    }
    long long tot;
    const long long ex = block_exclusive_scan<long long>(run, &tot);
    const long long o = bsum[blk] + ex;
#pragma unroll
    for (int k = 0; k < kPeItems; ++k)
      if (base + k < len) out[base + k] = (int32_t)(o + ex_k[k]);
    if (blk == nblk - 1 && threadIdx.x == 0) out[len] = (int32_t)bsum[nblk];
  }
}

__global__ void __launch_bounds__(kThreads) k_tr_scatter(const int32_t* off, const int32_t* idx, int32_t n, int32_t m,
                                                          int32_t* cursor, int32_t* in_idx) {
  for_each_entry(off, n, m, [=](int32_t e, int32_t v) { in_idx[atomicAdd(&cursor[idx[e]], 1)] = v; });
}

// Bit v of the starting bitmap: set iff v has neither in- nor out-edges. No
// level can reach such a vertex, and it is nobody's in-neighbour, so marking it
// visited changes no depth; pull then skips it, and skips whole words of them.
// (A vertex with out-edges only must stay clear: pull would take its set bit
// for a frontier in-neighbour.) Bits past n stay clear.
__global__ void k_vis_init(const int32_t* off, const int32_t* in_off, int32_t n, int32_t words, uint32_t* vis_init,
                           unsigned int* isolated_count) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < (int64_t)words * 32; v += stride) {
    // 32 consecutive threads share one word; every lane of a warp runs the same trips
    const bool isolated = v < n && off[v + 1] == off[v] && in_off[v + 1] == in_off[v];
    const uint32_t word = __ballot_sync(kFull, isolated);
    if ((v & 31) == 0) {
      vis_init[v >> 5] = word;
      if (word) atomicAdd(isolated_count, (unsigned)__popc(word));
    }
  }
}

// Vertex records of a graph whose out-degrees are at most w (4 or 8).
__global__ void k_records(const int32_t* off, const int32_t* idx, int32_t n, int32_t w, int32_t* rec) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    const int32_t b = off[v], d = off[v + 1] - b;
    for (int32_t j = 0; j < w; j += 4) {
      int4 r;
      r.x = j < d ? idx[b + j] : -1;
      r.y = j + 1 < d ? idx[b + j + 1] : -1;
      r.z = j + 2 < d ? idx[b + j + 2] : -1;
      r.w = j + 3 < d ? idx[b + j + 3] : -1;
      *reinterpret_cast<int4*>(rec + v * w + j) = r;
    }
  }
}

// Pull hint of every vertex: among the first kHintScan entries of its in-list,
// the in-neighbour with the largest out-degree (the first such on ties; -1
// without in-edges). Any in-neighbour is a valid first test, so the cap only
// bounds the cost on hubs' long lists.
__global__ void k_pull_hint(const int32_t* off, const int32_t* in_off, const int32_t* in_idx, int32_t n,
                            int32_t* hint) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
    const int32_t b = in_off[v];
    const int32_t e = min(in_off[v + 1], b + kHintScan);
    int32_t best = -1, best_deg = -1;
    for (int32_t k = b; k < e; ++k) {
      const int32_t u = in_idx[k];
      const int32_t d = off[u + 1] - off[u];
      if (d > best_deg) {
        best_deg = d;
        best = u;
      }
    }
    hint[v] = best;
  }
}

}  // namespace bfs
