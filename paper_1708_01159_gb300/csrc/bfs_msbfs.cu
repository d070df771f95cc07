// Multi-source BFS: up to 64 traversals of one graph in one persistent kernel.
//
// Each vertex carries three 64-bit masks: visit (bit i: reached by root i),
// frontier (bit i: at depth L for root i) and next (bits pushed to it during
// the level). Every level runs one direction for all roots at once:
//   push: the vertices of the frontier list OR their frontier mask, minus the
//         target's visited bits, into each neighbour's next mask (atomicOr);
//         a target whose next mask leaves zero joins a touched list, and a
//         commit pass over that list turns next into the new frontier;
//   pull: every vertex still unvisited in some lane ORs its in-neighbours'
//         frontier masks, stopping once every unvisited lane is found. Lanes
//         whose frontier is empty (their traversal has ended) are not waited
//         for; what is left of a long list after a lane's first 64 entries is
//         dealt to the warps of the whole grid, 128 entries at a time, and
//         committed like the targets of a push.
//
// What a wave spends its time on: the gathers of 8-byte masks by random vertex
// ids (a pull level of ER 2^22, degree 8, makes 33.5M of them, 190 us: 1.8
// cycles each on every SM), and the output. R-MAT 18, 64 roots, grid of 64
// blocks: 11.5 to 33 ms a wave with one lane scanning a hub's in-list of 30,000
// (every level of it, when one root lay outside the giant component), 0.63 to
// 0.79 ms with the lists dealt out; ER 2^22: 2.10 -> 1.59 ms with the lists'
// entries loaded a round ahead, the roots set up in parallel (45 us before),
// and the final pass's reached-edge counts by a transpose of the visit masks in
// place of 64 warp reductions (480 -> 250 us).
// Push and commit touch only the frontier and its neighbours (so thousands of
// small levels stay cheap); pull sweeps every vertex, a warp per 32
// consecutive vertices. The result equals k independent single-source
// traversals (each lane is one level-synchronous BFS from its root, Section
// 3.1).
//
// Output. A depth found at a level is not written to the k x n output then:
// each output sector holds 8 vertices of one root, which would be filled piece
// by piece over several levels (and, being far larger than L2, read back and
// merged each time). Instead the frontier masks of depths below kMsHistLevels
// are kept, one n-mask array per depth (the history: hist[d][u] holds the
// roots that reached u at depth d, disjoint over d), and a final pass builds
// every vertex's depths from its history masks and writes every output sector
// once, -1 included. Depths of kMsHistLevels and beyond (high-diameter graphs)
// are written when found; the final pass leaves an entry whose root reached
// the vertex but whose history holds no depth.
//
// The traversal's own frontier masks alternate between front[0] and front[1]
// (zeroed with visit and next when a wave starts, so they stay in L2); the
// history is written beside them, one plain store per vertex and depth it is
// reached at, and read only by the final pass, which zeroes what it read, so
// that the history arrays are zero whenever a wave starts (a wave that did
// not finish leaves the next one to zero them all).
//
// Level L uses frontier slot L % 4 (ftail, fedges), appends to (L + 1) % 4 and
// clears (L + 2) % 4, which every block finished reading two levels ago; the
// previous level's list (slot (L + 3) % 4) names the masks of front[(L+1) & 1]
// to clear before that array receives the new frontier.
#include "bfs_msbfs.cuh"

namespace bfs {

namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kMsTile = kMsThreads;      // push_mode 0: frontier vertices whose edges a block deals out together
constexpr int32_t kMsChunk = 128;        // pull, a list dealt over the grid: entries a warp takes at a time

// Predicated accesses, one instruction each (see ld_if in bfs_internal.cuh).
__device__ __forceinline__ unsigned long long ld64_if(bool p, const unsigned long long* a, unsigned long long otherwise) {
  unsigned long long x = otherwise;
  asm volatile("{\n .reg .pred q;\n setp.ne.s32 q, %2, 0;\n @q ld.global.u64 %0, [%1];\n}\n"
               : "+l"(x)
               : "l"(a), "r"((int)p));
  return x;
}

__device__ __forceinline__ unsigned long long atom_or64_if(bool p, unsigned long long* a, unsigned long long bits,
                                                           unsigned long long otherwise) {
  unsigned long long x = otherwise;
  asm volatile("{\n .reg .pred q;\n setp.ne.s32 q, %3, 0;\n @q atom.global.or.b64 %0, [%1], %2;\n}\n"
               : "+l"(x)
               : "l"(a), "l"(bits), "r"((int)p)
               : "memory");
  return x;
}

__device__ __forceinline__ unsigned long long reduce_or64(unsigned long long x) {
  return (unsigned long long)__reduce_or_sync(kFullMask, (unsigned)x) |
         (unsigned long long)__reduce_or_sync(kFullMask, (unsigned)(x >> 32)) << 32;
}

// Transpose of the warp's 32 x 32 bits: bit c of lane r's word becomes bit r of lane c's.
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const uint32_t m = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu : j == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(kFullMask, x, j);
    x = (threadIdx.x & j) ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y & m) << j);
  }
  return x;
}

// Bit k of x (k < 16) moved to bit 4k, through a table of the 256 byte
// spreads (lut[x]: bit k of x at bit 4k of a 32-bit word).
__device__ __forceinline__ unsigned long long nibble_spread16(const uint32_t* lut, unsigned long long x) {
  return (unsigned long long)lut[x & 255ull] | ((unsigned long long)lut[(x >> 8) & 255ull] << 32);
}

// Exclusive scan over the block (kMsThreads threads); *total: the sum.
__device__ __forceinline__ int32_t ms_block_scan(int32_t x, int32_t* total) {
  __shared__ int32_t part[kMsThreads / 32];
  int32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(kFullMask, inc, o);
    if ((int)lane_id() >= o) inc += y;
  }
  if (lane_id() == 31) part[threadIdx.x >> 5] = inc;
  __syncthreads();
  int32_t before = 0, sum = 0;
#pragma unroll
  for (int w = 0; w < kMsThreads / 32; ++w) {
    before += w < (int)(threadIdx.x >> 5) ? part[w] : 0;
    sum += part[w];
  }
  *total = sum;
  __syncthreads();
  return before + inc - x;
}

// Vertex u was reached at depth d by the roots in nb: the history keeps the
// depths below kMsHistLevels; deeper ones are written to their rows now.
__device__ __forceinline__ void ms_record(const MsBuffers& mb, const MsRows& rows, int64_t n, int64_t u,
                                          unsigned long long nb, int32_t d) {
  if (d < kMsHistLevels) {
    mb.hist[(size_t)d * (size_t)n + (size_t)u] = nb;
  } else {
    for (unsigned long long m = nb; m; m &= m - 1) rows.row[__ffsll((long long)m) - 1][u] = d;
  }
}

}  // namespace

// Five blocks an SM: 48 registers, 60 bytes a thread spilled (88 read back).
__global__ void __launch_bounds__(kMsThreads, 5) k_msbfs(DevGraph g, MsBuffers mb, MsState* st, int32_t k,
                                                       MsRows rows, MsConfig cfg, int32_t stall) {
  __shared__ unsigned long long s_edges[64];
  __shared__ uint32_t s_spread[256];
  __shared__ int32_t s_scan[kMsTile], s_beg[kMsTile];        // push: a tile's degrees scanned, row starts
  __shared__ unsigned long long s_mask[kMsTile];             // and frontier masks
  int32_t* const s_long = reinterpret_cast<int32_t*>(s_mask);  // pull: vertices with long lists and their ends
  int32_t* const s_end = s_long + kMsTile;
  __shared__ unsigned int s_fc;
  __shared__ unsigned long long s_fe;
  BFS_DECLARE_STAGE(stage);
  const int64_t n = g.n;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const unsigned long long act = k >= 64 ? ~0ull : ((1ull << k) - 1ull);
  const uint32_t lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  constexpr int kWarps = kMsThreads / 32;
  for (int i = threadIdx.x; i < 64; i += blockDim.x) s_edges[i] = 0;
  for (int x = threadIdx.x; x < 256; x += blockDim.x) {
    uint32_t y = 0;
    for (int b = 0; b < 8; ++b) y |= ((uint32_t)(x >> b) & 1u) << (4 * b);
    s_spread[x] = y;
  }
  // init: visit, frontier and next masks cleared; the history is zero unless
  // the last wave on this set did not finish (then it is zeroed here); the
  // output rows are written once, at the end. Every block reads the counts
  // before the first barrier, block 0 resets them after it.
  const bool hist_dirty = *reinterpret_cast<volatile unsigned int*>(&st->clean_blocks) !=
                          *reinterpret_cast<volatile unsigned int*>(&st->clean_grid);
  for (int64_t v = tid; v < n; v += stride) {
    mb.visit[v] = 0;
    mb.front[0][v] = 0;
    mb.front[1][v] = 0;
    mb.next[v] = 0;
    if (hist_dirty)
      for (int d = 0; d < kMsHistLevels; ++d) mb.hist[(size_t)d * (size_t)n + (size_t)v] = 0;
  }
  unsigned long long bar_target = 0;  // this block's copy of the barriers' arrival target
  if (!grid_arrive_wait(&st->bar64, bar_target, &st->status, stall == STALL_GRID_BARRIER ? 1u : 0u)) return;
  if (blockIdx.x == 0) {
    // roots, a thread each: the level 0 frontier; a vertex repeated as several roots carries several bits
    if (threadIdx.x == 0) {
      st->clean_blocks = 0;
      st->clean_grid = gridDim.x;
      s_fc = 0;
      s_fe = 0;
    }
    if (threadIdx.x < 64) st->edges[threadIdx.x] = 0;
    __syncthreads();
    if ((int)threadIdx.x < k) {
      const int32_t r = rows.root[threadIdx.x];
      const unsigned long long bit = 1ull << threadIdx.x;
      const bool first = atomicOr(&mb.visit[r], bit) == 0ull;
      atomicOr(&mb.front[0][r], bit);
      atomicOr(&mb.hist[r], bit);  // depth 0
      if (first) {
        mb.flist[0][atomicAdd(&s_fc, 1u)] = r;
        atomicAdd(&s_fe, (unsigned long long)(g.off[r + 1] - g.off[r]));
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int s = 0; s < 4; ++s) {
        st->ftail[s] = 0;
        st->fedges[s] = 0;
        st->alive[s] = 0;
      }
      st->ftail[0] = s_fc;
      st->fedges[0] = s_fe;
      st->alive[0] = act;
      st->ttail[0] = st->ttail[1] = 0;
    }
  }
  bool ok = grid_arrive_wait(&st->bar64, bar_target, &st->status);
  const int64_t words = (n + 31) / 32;
  const bool has_long = g.gfeat[F_IN_DEG_MAX] >= kMsLongList;  // some pull may set a vertex aside
  int32_t L = 0;
  for (; ok; ++L) {
    const unsigned int f = *reinterpret_cast<volatile unsigned int*>(&st->ftail[L % 4]);
    const unsigned int pf = *reinterpret_cast<volatile unsigned int*>(&st->ftail[(L + 3) % 4]);
    const unsigned long long fe = *reinterpret_cast<volatile unsigned long long*>(&st->fedges[L % 4]);
    // roots whose frontier is not empty: the others reach nothing any more, and
    // no vertex need look for them
    const unsigned long long alive = *reinterpret_cast<volatile unsigned long long*>(&st->alive[L % 4]);
    if (f == 0) break;
    if (L > g.n) {
      if (blockIdx.x == 0 && threadIdx.x == 0) st->status = ST_TIMEOUT;
      break;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      st->ftail[(L + 2) % 4] = 0;
      st->fedges[(L + 2) % 4] = 0;
      st->alive[(L + 2) % 4] = 0;
      st->ttail[(L + 1) % 2] = 0;
    }
    const unsigned long long* cur = (L & 1) ? mb.front[1] : mb.front[0];
    unsigned long long* nxt = (L & 1) ? mb.front[0] : mb.front[1];
    const int32_t* list = (L & 1) ? mb.flist[1] : mb.flist[0];
    int32_t* out_list = (L & 1) ? mb.flist[0] : mb.flist[1];  // holds level L-1's list until the commit
    unsigned int* out_tail = &st->ftail[(L + 1) % 4];
    unsigned long long my_fe = 0, my_alive = 0;
    // direction: pull once the frontier's edges exceed m / alpha (Beamer's rule, alpha tuned)
    const bool pull = fe * (unsigned long long)cfg.alpha > (unsigned long long)g.m;
    unsigned int* ttail = &st->ttail[L % 2];
    if (!pull) {
      // nxt still holds level L-1's frontier: clear exactly those masks
      for (int64_t i = tid; i < (int64_t)pf; i += stride) nxt[out_list[i]] = 0;
      if (cfg.push_mode == 0) {
        // a tile of frontier vertices a block (32 to 256 of them, as few as
        // spreads them over every block), their edges dealt to its threads one by
        // one through a scan of the degrees, so a hub never serialises on one
        // thread; four edges a thread and step, their adjacency entries, then
        // their targets' visit masks, then the pushes issued together
        const int share = (int)(((int64_t)f + gridDim.x - 1) / gridDim.x);
        const int tile = min(kMsTile, (share + 31) & ~31);
        for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < f; t0 += (int64_t)gridDim.x * tile) {
          const int64_t i = t0 + threadIdx.x;
          int32_t beg = 0, deg = 0;
          unsigned long long fv = 0;
          if ((int)threadIdx.x < tile && i < f) {
            const int32_t v = list[i];
            beg = g.off[v];
            deg = g.off[v + 1] - beg;
            fv = cur[v];
          }
          int32_t total;
          s_scan[threadIdx.x] = ms_block_scan(deg, &total);
          s_beg[threadIdx.x] = beg;
          s_mask[threadIdx.x] = fv;
          __syncthreads();
          for (uint32_t e0 = 0; e0 < (uint32_t)total; e0 += 4 * kMsThreads) {
            int32_t u[4];
            unsigned long long nb[4], old[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t e = e0 + q * kMsThreads + threadIdx.x;
              int o = 0;  // the last entry with s_scan[o] <= e owns edge e
#pragma unroll
              for (int step = kMsTile / 2; step > 0; step >>= 1) o += (uint32_t)s_scan[o + step] <= e ? step : 0;
              const bool have = e < (uint32_t)total;
              u[q] = ld_now_if(have, g.idx + ((uint32_t)s_beg[o] + (e - (uint32_t)s_scan[o])), 0);
              nb[q] = have ? s_mask[o] : 0ull;
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) old[q] = ld64_if(nb[q] != 0ull, mb.visit + u[q], 0ull);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              nb[q] &= ~old[q];
              // a hub that many edges name: its bits are seen in L1 (stale at
              // worst, within the level) before they are set again in one place
              old[q] = ld64_if(nb[q] != 0ull, mb.next + u[q], 0ull);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
              old[q] = atom_or64_if((nb[q] & ~old[q]) != 0ull, mb.next + u[q], nb[q], ~0ull);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (old[q] == 0ull) stage_put(stage, mb.tlist, ttail, u[q]);
            stage_drain(stage, mb.tlist, ttail, kStageCap / 2);
          }
          __syncthreads();
        }
      } else {
        for (int64_t base = (int64_t)blockIdx.x * kWarps; base < f; base += (int64_t)gridDim.x * kWarps) {
          const int64_t i = base + wib;
          if (i < f) {
            const int32_t v = list[i];
            const unsigned long long fv = cur[v];
            for (int32_t e = g.off[v] + (int32_t)lane; e < g.off[v + 1]; e += 32) {
              const int32_t u = g.idx[e];
              const unsigned long long nb = fv & ~mb.visit[u];
              if (nb && atomicOr(&mb.next[u], nb) == 0ull) stage_put(stage, mb.tlist, ttail, u);
            }
          }
          stage_drain(stage, mb.tlist, ttail, kStageCap / 2);
        }
      }
      stage_drain(stage, mb.tlist, ttail, 1);
    } else {
      // pull: OR the in-neighbours' frontier masks until every unvisited lane is
      // found. A lane looks at the first kMsRounds * 4 of its own vertex's (the
      // next four entries loaded while the last four's masks arrive), the warp
      // at what is left of a longer list together; vertices with kMsLong or more
      // left are set aside for all blocks.
      // Neighbouring words go to different blocks: the low ids of a skewed graph
      // are its hubs.
      for (int64_t w0 = 0; w0 < words; w0 += (int64_t)gridDim.x * kWarps) {
        const int64_t w = w0 + (int64_t)wib * gridDim.x + blockIdx.x;
        const int64_t u = w * 32 + lane;
        const bool valid = w < words && u < n;
        const unsigned long long vis = valid ? mb.visit[u] : 0ull;
        const unsigned long long unv = valid ? ~vis & alive : 0ull;
        int32_t e = 0, end = 0;
        if (unv) {
          e = g.in_off[u];
          end = g.in_off[u + 1];
        }
        unsigned long long acc = 0;
        bool open = e < end;
        int32_t x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = ld_now_if(e + q < end, g.in_idx + e + q, 0);
        for (int round = 0; round < kMsRounds && __any_sync(kFullMask, open); ++round) {
          unsigned long long m[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) m[q] = ld64_if(open && e + q < end, cur + x[q], 0ull);
          if (open) e = min(e + 4, end);
#pragma unroll
          for (int q = 0; q < 4; ++q) x[q] = ld_now_if(open && e + q < end, g.in_idx + e + q, 0);
          acc |= (m[0] | m[1]) | (m[2] | m[3]);
          open = open && e < end && (acc & unv) != unv;
        }
        bool later = false;
        if (__any_sync(kFullMask, open)) {
          if (open && end - e >= kMsLong) {
            // set aside for all blocks, with what has been found so far
            mb.next[u] = acc;
            mb.tlist[atomicAdd(ttail, 1u)] = (int32_t)u;
            later = true;
            open = false;
          }
          uint32_t left = __ballot_sync(kFullMask, open);
          while (left) {
            const int src = __ffs(left) - 1;
            left &= left - 1u;
            const int32_t to = __shfl_sync(kFullMask, end, src);
            const unsigned long long want = __shfl_sync(kFullMask, unv, src);
            unsigned long long got = __shfl_sync(kFullMask, acc, src), part = 0;
            for (int32_t p = __shfl_sync(kFullMask, e, src); p < to && (got & want) != want; p += min(128, to - p)) {
              int32_t y[4];
              unsigned long long m[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) y[q] = ld_now_if(to - p > 32 * q + (int)lane, g.in_idx + p + 32 * q + lane, 0);
#pragma unroll
              for (int q = 0; q < 4; ++q) m[q] = ld64_if(to - p > 32 * q + (int)lane, cur + y[q], 0ull);
              part |= (m[0] | m[1]) | (m[2] | m[3]);
              got |= reduce_or64(part);
            }
            if ((int)lane == src) acc = got;
          }
        }
        if (valid && !later) {
          const unsigned long long nb = acc & unv;
          if (nb) {
            my_alive |= nb;
            mb.visit[u] = vis | nb;
            my_fe += (unsigned long long)(g.off[u + 1] - g.off[u]);
            stage_put(stage, out_list, out_tail, (int32_t)u);
            ms_record(mb, rows, n, u, nb, L + 1);
          }
          nxt[u] = nb;
        }
        stage_drain(stage, out_list, out_tail, kStageCap - kMsThreads);
      }
      stage_drain(stage, out_list, out_tail, 1);
    }
    // the touched vertices of a push level, the long lists a pull level set aside
    unsigned int t = 0;
    if (!pull || has_long) {
      ok = grid_arrive_wait(&st->bar64, bar_target, &st->status);
      if (!ok) break;
      t = *reinterpret_cast<volatile unsigned int*>(ttail);
    }
    if (pull && t > 0u) {
      // chunks of the lists' entries past those their lanes looked at, dealt over
      // all blocks: the vertices a tile at a time, their chunks counted by a scan
      int64_t dealt = 0;  // chunks of the tiles before
      for (unsigned int base = 0; base < t; base += kMsTile) {
        const unsigned int i = base + threadIdx.x;
        int32_t u = 0, from = 0, to = 0;
        if (i < t) {
          u = mb.tlist[i];
          from = g.in_off[u] + 4 * kMsRounds;
          to = g.in_off[u + 1];
        }
        int32_t total;
        s_scan[threadIdx.x] = ms_block_scan((to - from + kMsChunk - 1) / kMsChunk, &total);
        s_beg[threadIdx.x] = from;
        s_long[threadIdx.x] = u;
        s_end[threadIdx.x] = to;
        __syncthreads();
        const int64_t warps = (int64_t)gridDim.x * kWarps, me = (int64_t)wib * gridDim.x + blockIdx.x;
        for (int64_t c = (me + warps - dealt % warps) % warps; c < total; c += warps) {  // uniform over the warp
          int o = 0;  // the last entry with s_scan[o] <= c owns chunk c
#pragma unroll
          for (int step = kMsTile / 2; step > 0; step >>= 1) o += s_scan[o + step] <= (int32_t)c ? step : 0;
          const int32_t v = s_long[o];
          const int32_t p = s_beg[o] + ((int32_t)c - s_scan[o]) * kMsChunk, left = s_end[o] - p;
          const unsigned long long want = ~mb.visit[v] & alive;
          const unsigned long long got = *reinterpret_cast<volatile unsigned long long*>(&mb.next[v]);
          if (__all_sync(kFullMask, (got & want) == want)) continue;  // other chunks have found the rest
          int32_t y[4];
          unsigned long long m[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) y[q] = ld_now_if(left > 32 * q + (int)lane, g.in_idx + p + 32 * q + lane, 0);
#pragma unroll
          for (int q = 0; q < 4; ++q) m[q] = ld64_if(left > 32 * q + (int)lane, cur + y[q], 0ull);
          const unsigned long long part = reduce_or64((m[0] | m[1]) | (m[2] | m[3])) & want & ~got;
          if (lane == 0 && part) atomicOr(&mb.next[v], part);
        }
        dealt += total;
        __syncthreads();
      }
      ok = grid_arrive_wait(&st->bar64, bar_target, &st->status);
      if (!ok) break;
    }
    // commit them: next -> new frontier, depths, next frontier list
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < t; base += stride) {
      const int64_t i = base + threadIdx.x;
      if (i < t) {
        const int32_t u = mb.tlist[i];
        const unsigned long long vis = mb.visit[u];
        const unsigned long long nb = mb.next[u] & ~vis;
        mb.next[u] = 0;
        nxt[u] = nb;
        if (nb) {
          mb.visit[u] = vis | nb;
          my_alive |= nb;
          my_fe += (unsigned long long)(g.off[u + 1] - g.off[u]);
          stage_put(stage, out_list, out_tail, u);
          ms_record(mb, rows, n, u, nb, L + 1);
        }
      }
      stage_drain(stage, out_list, out_tail, kStageCap / 2);
    }
    stage_drain(stage, out_list, out_tail, 1);
    block_add_u64(my_fe, &st->fedges[(L + 1) % 4]);
    my_alive = reduce_or64(my_alive);
    if (lane == 0 && my_alive) atomicOr(&st->alive[(L + 1) % 4], my_alive);
    ok = grid_arrive_wait(&st->bar64, bar_target, &st->status);
  }
  // Final pass, a warp per 32 consecutive vertices: every output sector written
  // once from the history (coalesced 128-byte row segments, one per root),
  // the per-root reached-edge counts (for each root, the sum of out-degrees of
  // the vertices whose visit mask carries its bit), and the history cleared
  // for the next wave. (The loop ended right after a grid barrier, so
  // every block's masks are visible.) Depths 0 .. L - 1 occurred; those below
  // kMsHistLevels are in the history.
  const int32_t dmax = min(L - 1, kMsHistLevels - 1);
  const bool deep = L > kMsHistLevels;  // depths of kMsHistLevels and beyond occurred
  unsigned long long edges_lo = 0, edges_hi = 0;  // reached edges of roots lane and lane + 32, this warp's vertices
  for (int64_t wbase = (int64_t)blockIdx.x * kWarps; wbase < words; wbase += (int64_t)gridDim.x * kWarps) {
    const int64_t w = wbase + wib;
    if (w >= words) continue;  // whole warp
    const int64_t u = w * 32 + lane;
    const bool valid = u < n;
    const unsigned long long vis = valid ? mb.visit[u] : 0ull;
    if (ok && valid) {
      // bit b of the code (d + 1 for depth d) of root i is bit i of plane b
      // (the history masks of u are disjoint); loads five depths at a time
      unsigned long long p0 = 0ull, p1 = 0ull, p2 = 0ull, p3 = 0ull;
      constexpr int kChunk = 5;
      static_assert(kMsHistLevels % kChunk == 0, "whole chunks");
      static_assert(kMsHistLevels <= 15, "codes d + 1 fit four bits");
#pragma unroll 1
      for (int32_t d0 = 0; d0 <= dmax; d0 += kChunk) {
        unsigned long long m[kChunk];
#pragma unroll
        for (int j = 0; j < kChunk; ++j)  // an unreached vertex has no history
          m[j] = vis && d0 + j <= dmax ? mb.hist[(size_t)(d0 + j) * (size_t)n + (size_t)u] : 0ull;
#pragma unroll
        for (int j = 0; j < kChunk; ++j) {
          if (m[j]) {
            mb.hist[(size_t)(d0 + j) * (size_t)n + (size_t)u] = 0ull;
            const int c = d0 + j + 1;
            if (c & 1) p0 |= m[j];
            if (c & 2) p1 |= m[j];
            if (c & 4) p2 |= m[j];
            if (c & 8) p3 |= m[j];
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (16 * q >= k) break;  // uniform
        // nibble r: the code of root 16 q + r
        const unsigned long long word = nibble_spread16(s_spread, p0 >> (16 * q)) |
                                        (nibble_spread16(s_spread, p1 >> (16 * q)) << 1) |
                                        (nibble_spread16(s_spread, p2 >> (16 * q)) << 2) |
                                        (nibble_spread16(s_spread, p3 >> (16 * q)) << 3);
        // reached, but not in the history: a deeper depth, written when found
        const unsigned later = deep ? (unsigned)(vis >> (16 * q)) & 0xffffu : 0u;
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          if (16 * q + r >= k) break;  // uniform
          const int32_t code = (int32_t)((unsigned)(word >> (4 * r)) & 15u);
          if (code != 0 || !((later >> r) & 1u)) __stcs(rows.row[16 * q + r] + u, code - 1);
        }
      }
    }
    const unsigned deg = valid ? (unsigned)(g.off[u + 1] - g.off[u]) : 0u;
    // lane c: the vertices (bits) roots c and c + 32 reached, their degrees summed
    const uint32_t lo = transpose32((uint32_t)vis), hi = transpose32((uint32_t)(vis >> 32));
    unsigned sum_lo = 0, sum_hi = 0;
#pragma unroll 8
    for (int v = 0; v < 32; ++v) {
      const unsigned d = __shfl_sync(kFullMask, deg, v);
      sum_lo += ((lo >> v) & 1u) ? d : 0u;
      sum_hi += ((hi >> v) & 1u) ? d : 0u;
    }
    edges_lo += sum_lo;
    edges_hi += sum_hi;
  }
  if (edges_lo) atomicAdd(&s_edges[lane], edges_lo);
  if (edges_hi) atomicAdd(&s_edges[lane + 32], edges_hi);
  __syncthreads();
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    if (s_edges[i]) atomicAdd(&st->edges[i], s_edges[i]);
  if (blockIdx.x == 0 && threadIdx.x == 0) st->levels = L;
  // this block's share of the history is zero again (a block that stopped
  // early or saw an error does not count, and the next wave zeroes it all)
  if (threadIdx.x == 0 && ok && *reinterpret_cast<volatile int32_t*>(&st->status) == ST_OK)
    atomicAdd(&st->clean_blocks, 1u);
}

__global__ void k_ms_reset(MsState* st) {
  st->status = ST_OK;
  st->bar64 = 0;
}

}  // namespace bfs
