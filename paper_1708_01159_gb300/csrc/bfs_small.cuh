// Small levels of the persistent driver (included by bfs_kernels.cu), for
// graphs whose vertices all have few out-edges (roads, grids, chains): their
// traversals are thousands of levels of a few thousand edges each.
//
// A small level on the whole grid spends its time on the way through it: the
// queue in global memory, row extent and list in turn, the queue tail, the two
// release reductions and the polls of the level barrier, each a trip to L2. So
// one cluster (the leader: cluster 0) expands such levels alone while the
// other blocks wait until the frontier outgrows it. The leader keeps the
// frontier in its blocks' shared memory as candidates, the neighbours its
// vertices name (each with the vertex that names it, so that nobody tries his
// own parent again), and every vertex's whole list is one record of 4 or 8
// entries read by one vector load. A level is then: candidate (shared memory),
// claim (one atomicOr in L2), record of the vertices won, their neighbours to
// the next candidates. It ends with one message per pair of blocks: each block
// sends its counts into every block's shared memory with st.async, which
// completes on the receiver's mbarrier: no fence and no global memory on the
// way. The claims' results need no order, and depths are written once and not
// read again in the launch.
//
// What bounds such a level: the claim's trip to L2, the record's, the message,
// and some hundreds of instructions between them; from about 4,000 edges also
// the rate at which 16 SMs issue scattered requests. 4096^2 grid with a tenth
// of the edges dropped (6,194 levels, 2,708 vertices and 9,750 edges on
// average): 6.66 us a level on the whole grid, 2.76 us here (1.9 below 1,024
// vertices, 3.6 above 4,096), the traversal 41.3 -> 17.1 ms (17.1 to 20.2 over
// boxes and roots). Other forms measured on the same graph and box: row extents
// and lists read from the CSR by four edges of a thread 28.4 ms; records without
// the prefetch 23.8; 8 blocks instead of 16 32.0; two candidates a thread at most
// instead of four 20.9. At the 64 registers of the persistent kernel small_run<4>
// spills 108 bytes on the way, in the graph driver's kernel (80 registers) none.
#pragma once

namespace bfs {
namespace {

constexpr int kCandCap = 1040;    // candidates per block
constexpr int kWonCap = 1040;     // vertices won per block and level
// A level is left to a leader of c blocks when it has at most c * kSmallEdges
// edges; about three quarters of them name a candidate, and the blocks' shares drift
// apart between two dealings.
constexpr unsigned kSmallEdges = 1088;

// A neighbour `v` named by `from`.
struct Candidate {
  int32_t v, from;
};

struct SmallShared {
  unsigned long long msg[2][kMaxCluster];  // counts of every block of the cluster, by exchange parity
  uint64_t bar[2];
  // candidates (high half) and vertices won (low half) of a level: level k of a
  // run reads its candidates' count from cnt[k % 3], level k - 1 wrote it
  unsigned int cnt[3];
  unsigned int valid;  // candidates below this index are complete (an append that did not fit ends the run)
  unsigned int valid_won;
  unsigned int leave;
  unsigned int part_f[kThreads / 32], part_e[kThreads / 32];
  unsigned int runs;  // small runs so far (the blocks that wait count them)
  TravState out;
  unsigned int run_no;              // leader: small runs so far
  unsigned int ended[kMaxCluster];  // each block of the cluster: the last run it has ended, ~0 after its last level
                                    // (written by that block)
  unsigned int failed;              // a block of the cluster gave a wait up (written by that block)
  unsigned int mute;                // test hook: the state is not published
};

__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t x;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(x));
  return x;
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t x;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(x));
  return x;
}
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank) {
  uint32_t x;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(x) : "r"(addr), "r"(rank));
  return x;
}
__device__ __forceinline__ Candidate ld_cluster(uint32_t addr) {
  Candidate x;
  asm volatile("ld.shared::cluster.v2.s32 {%0, %1}, [%2];" : "=r"(x.v), "=r"(x.from) : "r"(addr) : "memory");
  return x;
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, unsigned int x) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(x) : "memory");
}
__device__ __forceinline__ void st_async_u64(uint32_t addr, unsigned long long x, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(addr), "l"(x),
               "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.aligned;\nbarrier.cluster.wait.aligned;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
      "p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0u;
}

// Whether a level of f vertices and e frontier edges is left to a leader of c
// blocks. The vertices count too: they are dealt out evenly when a run starts,
// and a frontier of a directed graph may be a million vertices without an edge.
__device__ __forceinline__ bool small_fits(unsigned int f, unsigned long long e, uint32_t c) {
  return f <= c * (unsigned)kWonCap && e <= c * kSmallEdges;
}

// Vertex v's record: its W out-neighbours, -1 past its degree.
template <int W>
__device__ __forceinline__ void ld_record_if(bool p, const int32_t* rec, int32_t v, int32_t (&r)[W]) {
#pragma unroll
  for (int j = 0; j < W; j += 4) {
    r[j] = r[j + 1] = r[j + 2] = r[j + 3] = -1;
    asm volatile("{\n .reg .pred q;\n setp.ne.s32 q, %5, 0;\n @q ld.global.v4.s32 {%0, %1, %2, %3}, [%4];\n}\n"
                 : "+r"(r[j]), "+r"(r[j + 1]), "+r"(r[j + 2]), "+r"(r[j + 3])
                 : "l"(rec + (size_t)v * W + j), "r"((int)p));
  }
}

// The vertices won by a warp (lane: v[k] named by from[k], record r[k]) go to
// the block's list of won vertices, the neighbours they name to the next
// candidates. When either list is full, the vertices go to the global queue
// qout (unless null) and the run ends after the level. Adds to the warp's
// vertices f_warp and the lane's out-degrees e_lane.
template <int K, int W>
__device__ __forceinline__ void small_append(const int32_t* rec, Candidate* cand, int32_t* wonq, unsigned int* cnt, SmallShared& ss,
                                             const bool (&won)[K], const int32_t (&v)[K], const int32_t (&from)[K],
                                             const int32_t (&r)[K][W], int32_t* qout, unsigned long long* tail,
                                             unsigned int& f_warp, unsigned int& e_lane) {
  uint32_t m[K];
  unsigned int wins = 0, names = 0;  // names: neighbours this lane adds, at most K * W < 32
#pragma unroll
  for (int k = 0; k < K; ++k) {
    m[k] = __ballot_sync(kFull, won[k]);
    wins += __popc(m[k]);
#pragma unroll
    for (int j = 0; j < W; ++j) {
      e_lane += (unsigned)(r[k][j] >= 0);  // records not won are all -1
      names += (unsigned)(r[k][j] >= 0 && r[k][j] != from[k]);
    }
  }
  if (wins == 0) return;  // uniform
  f_warp += wins;
  // prefix sums over the lanes, a bit plane of the count at a time
  constexpr int kPlanes = K * W < 8 ? 3 : K * W < 16 ? 4 : 5;
  unsigned int before = 0, total = 0;
#pragma unroll
  for (int p = 0; p < kPlanes; ++p) {
    const uint32_t plane = __ballot_sync(kFull, (names >> p) & 1u);
    before += (unsigned)__popc(plane & lanemask_lt()) << p;
    total += (unsigned)__popc(plane) << p;
  }
  unsigned int base = 0;
  if (lane_id() == 0) base = atomicAdd(cnt, total << 16 | wins);
  base = __shfl_sync(kFull, base, 0);
  unsigned int at = base >> 16, wat = base & 0xffffu;
  if (at + total > (unsigned)kCandCap || wat + wins > (unsigned)kWonCap) {
    if (qout) {
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (won[k]) queue_append(qout, tail, v[k]);
    }
    if (lane_id() == 0) {
      atomicMin(&ss.valid, at);
      atomicMin(&ss.valid_won, wat);
      ss.leave = 1u;
    }
    __syncwarp();
    return;
  }
  at += before;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (won[k]) wonq[wat + __popc(m[k] & lanemask_lt())] = v[k];
    wat += __popc(m[k]);
#pragma unroll
    for (int j = 0; j < W; ++j)
      if (r[k][j] >= 0 && r[k][j] != from[k]) {
        prefetch_l2(rec + (size_t)r[k][j] * W);  // its record, should it be won
        cand[at++] = Candidate{r[k][j], v[k]};
      }
  }
}

// Candidates base + tid, base + tid + kThreads, ... (K of them) of the level.
template <int K, int W>
__device__ __forceinline__ void small_step(const int32_t* rec, uint32_t* vis, int32_t* depth, int32_t next_depth,
                                           const Candidate* cur, unsigned int base, unsigned int n, Candidate* nxt,
                                           int32_t* wonq, unsigned int* cnt, SmallShared& ss, int32_t* qout,
                                           unsigned long long* tail, unsigned int& f_warp, unsigned int& e_lane) {
  int32_t v[K], from[K], r[K][W];
  uint32_t seen[K];
  bool won[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const unsigned int i = base + (unsigned)threadIdx.x + (unsigned)(k * kThreads);
    v[k] = from[k] = 0;
    if (i < n) {
      v[k] = cur[i].v;
      from[k] = cur[i].from;
    }
    const uint32_t bit = 1u << (v[k] & 31);
    seen[k] = atom_or_if(i < n, vis + (v[k] >> 5), bit, bit);
  }
#pragma unroll
  for (int k = 0; k < K; ++k) {
    won[k] = !((seen[k] >> (v[k] & 31)) & 1u);
    ld_record_if<W>(won[k], rec, v[k], r[k]);
  }
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (won[k]) depth[v[k]] = next_depth;
  small_append<K, W>(rec, nxt, wonq, cnt, ss, won, v, from, r, qout, tail, f_warp, e_lane);
}

// Level end within the leader: the block's counts (vertices of the warp,
// out-degrees of the lane, candidates of the block) go to every block; returns
// the totals, the largest block's candidates and whether some block has to
// leave. False when a message never came.
__device__ __forceinline__ bool small_exchange(SmallShared& ss, uint32_t c, uint32_t rank, unsigned int xc,
                                               const unsigned int* cnt, unsigned int f_warp, unsigned int e_lane,
                                               unsigned int* f, unsigned int* e, unsigned int* most,
                                               unsigned int* cands, bool* leave) {
  const uint32_t par = xc & 1u;
  e_lane = __reduce_add_sync(kFull, e_lane);
  if (lane_id() == 0) {
    ss.part_f[threadIdx.x >> 5] = f_warp;
    ss.part_e[threadIdx.x >> 5] = e_lane;
  }
  __syncthreads();
  if (threadIdx.x < c) {
    unsigned int fs = 0, es = 0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) {
      fs += ss.part_f[w];
      es += ss.part_e[w];
    }
    // a block tries at most kCandCap candidates in a level, and wins 8 entries with each at most
    const unsigned long long m = (unsigned long long)es | (unsigned long long)fs << 16 |
                                 (unsigned long long)min(*cnt >> 16, ss.valid) << 32 |
                                 (unsigned long long)(ss.leave != 0u) << 48;
    if (threadIdx.x == 0) mbar_expect_tx(&ss.bar[par], 8u * c);
    st_async_u64(map_rank(smem_u32(&ss.msg[par][rank]), threadIdx.x), m,
                 map_rank(smem_u32(&ss.bar[par]), threadIdx.x));
  }
  bool ok = mbar_try_wait_cluster(&ss.bar[par], (xc >> 1) & 1u);
  if (!ok) {
    const unsigned long long t0 = global_ns();
    while (!(ok = mbar_try_wait_cluster(&ss.bar[par], (xc >> 1) & 1u)))
      if (global_ns() - t0 > kWaitLimitNs) break;
  }
  const unsigned long long m = lane_id() < c ? ss.msg[par][lane_id()] : 0ull;
  const unsigned int cand = (unsigned)(m >> 32) & 0xffffu;
  *e = __reduce_add_sync(kFull, (unsigned)m & 0xffffu);
  // vertices (15 bits), candidates
  const unsigned int both = __reduce_add_sync(kFull, ((unsigned)(m >> 16) & 0xffffu) | cand << 15);
  *most = __reduce_max_sync(kFull, cand);
  *f = both & 0x7fffu;
  *cands = both >> 15;
  *leave = __any_sync(kFull, (unsigned)(m >> 48) & 1u) != 0;
  return __syncthreads_and(ok) != 0;
}
// (a run's first exchange: kWonCap vertices a block at most, small_fits)
static_assert(kCandCap * 8 < (1 << 16) && kMaxCluster * kCandCap < (1 << 15) && kWonCap * 8 < (1 << 16) &&
                  kMaxCluster * kWonCap < (1 << 15),
              "message fields and their sums");

// Deal the candidates out again, candidate i of the whole cluster to block i %
// c: a wavefront that started in one block spreads over the others. xc - 1 is
// the exchange whose messages hold every block's count.
__device__ __forceinline__ void small_deal(SmallShared& ss, uint32_t c, uint32_t rank, unsigned int xc,
                                           const Candidate* from, Candidate* to, unsigned int total,
                                           unsigned int* to_cnt) {
  const uint32_t par = (xc - 1u) & 1u;
  cluster_barrier();  // every block's candidates are written
  for (unsigned int i = rank + c * threadIdx.x; i < total; i += c * kThreads) {
    unsigned int at = i;
    uint32_t src = 0;
    for (; src + 1u < c; ++src) {
      const unsigned int n = (unsigned)(ss.msg[par][src] >> 32) & 0xffffu;
      if (at < n) break;
      at -= n;
    }
    to[i / c] = ld_cluster(map_rank(smem_u32(from + at), src));
  }
  if (threadIdx.x == 0) *to_cnt = (total > rank ? (total - rank + c - 1u) / c : 0u) << 16 | (*to_cnt & 0xffffu);
  cluster_barrier();  // every block has read what it takes
}

// The end of small run `no`, for every block of the leader, and (~0) of the levels,
// for every block of a cluster: true when none has given a wait up. A block that
// did is here before the others, who may be dealing, or at the end of a run it did
// not start: their barriers are answered until they have given up waiting for its
// messages and have come here too. So no block leaves, let alone ends, while
// another may still send to its shared memory. (Telling the others of the failure
// in the dealing's barrier instead cost every level 0.5 to 1 %.)
__device__ __forceinline__ bool small_end(SmallShared& ss, uint32_t c, uint32_t rank, unsigned int no, bool ok) {
  if (threadIdx.x < c) {
    if (!ok) st_cluster_u32(map_rank(smem_u32(&ss.failed), threadIdx.x), 1u);
    st_cluster_u32(map_rank(smem_u32(&ss.ended[rank]), threadIdx.x), no);
  }
  __syncwarp();
  bool here;  // the block of this lane is
  do {
    cluster_barrier();
    here = lane_id() >= c || *reinterpret_cast<volatile unsigned int*>(&ss.ended[lane_id()]) >= no;
  } while (!__syncthreads_and(here));
  return *reinterpret_cast<volatile unsigned int*>(&ss.failed) == 0u;
}

// The leader's part of a run of small levels, from level t.L (variant v, which
// the log records) until the frontier outgrows the leader, the tree asks for a
// pull, or nothing is left. ss.out holds the state before the run's first
// level, and on return the state before the next level, whose frontier is in
// the global queue (q[L & 1]) for the whole grid. A run that a block's wait
// failed in fails in every block. (Not inlined: the kernel's
// other levels keep their registers. ubuf, sbuf, log and ss are in shared
// memory.)
template <int W>
__device__ __noinline__ void small_run(const DevGraph& g, const Buffers& b, uint32_t* vis, int32_t* depth,
                                       RunState* st, const QsTree* qs, const TreeNode* tree, int32_t nodes,
                                       const RunLog& log, SmallShared& ss, int32_t* ubuf, int32_t* sbuf, int32_t v) {
  __builtin_assume(__isShared(&ss));
  __builtin_assume(__isShared(&log));
  __builtin_assume(__isShared(ubuf));
  __builtin_assume(__isShared(sbuf));
  constexpr int kMost = W == 4 ? 4 : 2;  // candidates a thread tries at once (registers)
  const uint32_t c = cluster_size(), rank = cluster_rank();
  const int tid = (int)threadIdx.x;
  const TreeChoice tc{qs, tree, nodes, 0, -1};
  // what every level reads, out of the parameter block (a load each time otherwise)
  const int32_t* const rec = g.rec;
  int32_t* const q0 = b.q[0];
  int32_t* const q1 = b.q[1];
  const int32_t n = g.n;
  TravState t = ss.out;
  Candidate* cur = reinterpret_cast<Candidate*>(ubuf);
  Candidate* nxt = cur + kCandCap;
  int32_t* const wonq = sbuf;
  if (tid == 0) {
    ss.cnt[0] = ss.cnt[1] = ss.cnt[2] = 0u;
    ss.valid = ss.valid_won = ~0u;
    ss.leave = 0u;
    ++ss.run_no;
  }
  __syncthreads();
  // the frontier from the global queue, vertex i to block i % c
  const int32_t* qin = (t.L & 1) ? q1 : q0;
  unsigned int my_f = 0, my_e = 0;
  for (unsigned int base = 0; base < t.f; base += c * kThreads) {
    const unsigned int i = base + rank + c * (unsigned)tid;
    const bool have[1] = {i < t.f};
    const int32_t u[1] = {ld_now_if(have[0], qin + i, 0)};
    const int32_t none[1] = {-2};
    int32_t r[1][W];
    ld_record_if<W>(have[0], rec, u[0], r[0]);
    small_append<1, W>(rec, cur, wonq, &ss.cnt[0], ss, have, u, none, r, nullptr, nullptr, my_f, my_e);
  }
  unsigned int f, e, most, cands;
  bool leave;
  bool ok = small_exchange(ss, c, rank, t.exchanges++, &ss.cnt[0], my_f, my_e, &f, &e, &most, &cands, &leave);
  unsigned int k = 0;  // levels of this run
  unsigned int k3 = 0;
  t.force_full = leave ? 1 : 0;  // a frontier that does not fit: nothing has changed yet
  const bool loaded = ok && !leave;
  if (loaded) {
    t.discovered += t.f;
    t.reached += (long long)t.e;
  }
  while (loaded && ok) {
    const unsigned int k3n = k3 == 2u ? 0u : k3 + 1u;
    const unsigned int count = ss.cnt[k3] >> 16;
    if (tid == 0) ss.cnt[k3n == 2u ? 0u : k3n + 1u] = 0u;  // the counter of level k - 1, appended to at level k + 1
    if (rank == 0u && tid == kThreads - 1) {
      log_level(log, t.L, v, t.f, (long long)t.e);
      *reinterpret_cast<volatile int32_t*>(&st->small_beat) = t.L;
    }
    int32_t* qout = (t.L & 1) ? q0 : q1;
    my_f = my_e = 0;
    for (unsigned int base = 0; base < count; base += kMost * kThreads) {
      if (kMost > 2 && count - base > 2u * kThreads)
        small_step<kMost, W>(rec, vis, depth, t.L + 1, cur, base, count, nxt, wonq, &ss.cnt[k3n], ss, qout,
                             &st->small_tail, my_f, my_e);
      else if (count - base > (unsigned)kThreads)
        small_step<2, W>(rec, vis, depth, t.L + 1, cur, base, count, nxt, wonq, &ss.cnt[k3n], ss, qout, &st->small_tail,
                         my_f, my_e);
      else
        small_step<1, W>(rec, vis, depth, t.L + 1, cur, base, count, nxt, wonq, &ss.cnt[k3n], ss, qout, &st->small_tail,
                         my_f, my_e);
    }
    ok = small_exchange(ss, c, rank, t.exchanges++, &ss.cnt[k3n], my_f, my_e, &f, &e, &most, &cands, &leave);
    t.prev = v;
    t.L += 1;
    t.f = f;
    t.e = e;
    t.force_full = leave ? 1 : 0;
    ++k;
    k3 = k3n;
    Candidate* x = cur;
    cur = nxt;
    nxt = x;
    if (!ok || leave || f == 0u) break;
    if (t.L > n || t.discovered > n) break;  // corrupted state: the caller reports it
    v = tc.choose(g, t.L, f, (long long)e, t.discovered + f, t.prev);
    if (v == V_PULL || !small_fits(f, e, c)) break;
    t.discovered += f;
    t.reached += (long long)e;
    // dealt out when one block has twice its share, or needs a step more than they do
    constexpr unsigned int kStep = 2u * kThreads;
    if ((most > 128u && most * c > 2u * cands) || (most + kStep - 1u) / kStep > (cands / c + 64u + kStep - 1u) / kStep) {
      small_deal(ss, c, rank, t.exchanges, cur, nxt, cands, &ss.cnt[k3]);
      x = cur;
      cur = nxt;
      nxt = x;
    }
  }
  if (k > 0u && t.f > 0u) {
    // the frontier's vertices (those that did not fit are there already) to the global queue
    int32_t* qout = (t.L & 1) ? q1 : q0;
    const unsigned int count = min(ss.cnt[k3] & 0xffffu, ss.valid_won);
    for (unsigned int i = (unsigned)tid; i < count; i += kThreads) queue_append(qout, &st->small_tail, wonq[i]);
  }
  ok = small_end(ss, c, rank, ss.run_no, ok);
  t.ok = ok ? 1 : 0;
  if (tid == 0) ss.out = t;
  if (rank == 0u && tid == 0) {
    if (!ok) st->status = ST_TIMEOUT;
    st->small_tail = 0;
    if (gridDim.x > c && ss.mute == 0u) {
      st->small_out = t;
      __threadfence();
      st_release_u32(&st->small_seq, st->small_seq + 1u);
    }
  }
}

// The other blocks' part: wait until the leader has published the state before
// the next level of the whole grid, giving up when its level counter stands
// still for kWaitLimitNs.
__device__ __noinline__ void small_park(RunState* st, SmallShared& ss) {
  if (threadIdx.x == 0) {
    const unsigned int run = ss.runs;
    ss.runs = run + 1u;
    bool ok = true;
    unsigned long long t0 = global_ns();
    int32_t beat = -1;
    while (ld_acquire_u32(&st->small_seq) == run) {
      __nanosleep(400);
      if (global_ns() - t0 <= kWaitLimitNs) continue;
      const int32_t now = *reinterpret_cast<volatile int32_t*>(&st->small_beat);
      if (now == beat) {
        ok = false;
        break;
      }
      beat = now;
      t0 = global_ns();
    }
    if (ok) {
      ss.out = *const_cast<const TravState*>(&st->small_out);
    } else {
      st->status = ST_TIMEOUT;
      ss.out.ok = 0;
    }
  }
  __syncthreads();
}

}  // namespace
}  // namespace bfs
