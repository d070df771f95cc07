// Kernel declarations and launch shapes shared by the kernel and host sources.
#pragma once

#include "bfs_internal.cuh"

namespace bfs {

constexpr int kThreads = 256;     // block size of the level kernels
constexpr int kMaxCluster = 16;   // blocks of a cluster that runs small levels (bfs_small.cuh)
constexpr int kDecideThreads = 32;  // block size of k_decide: one warp evaluates the bit-parallel tree
constexpr int kCtaChunk = 2048;   // int32 per shared-memory stage of the CTA variant (8 KB)
constexpr int kCtaDirect = 512;   // adjacency shorter than this is read directly, not staged
constexpr int kPeItems = 8;       // entries per thread in a scan
constexpr int kPeTile = kThreads * kPeItems;  // entries per block of a scan
constexpr int kHeavy = 1024;        // degree from which an edge-centric level deals a vertex over all blocks
constexpr int kHeavyCap = 1 << 16;  // most vertices an edge-centric level sets aside

__global__ void k_init(DevGraph g, Buffers b, RunState* st, int32_t* depth, int32_t root, int32_t forced,
                       const TreeNode* tree, int32_t tree_nodes, const QsTree* tree_qs, int32_t use_handles,
                       unsigned long long h_while, unsigned long long h_switch);
__global__ void k_decide(DevGraph g, Buffers b, RunState* st);
__global__ void k_loop_start(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_thread(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_warp(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_cta(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_edge(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_heavy(DevGraph g, Buffers b, RunState* st);
__global__ void k_pull(DevGraph g, Buffers b, RunState* st);
// Vertex push appending by CM_WARP or CM_ATOMIC (count-mode comparison)
__global__ void k_push_thread_warp_count(DevGraph g, Buffers b, RunState* st);
__global__ void k_push_thread_atomic_count(DevGraph g, Buffers b, RunState* st);
__global__ void k_edge_list(DevGraph g, Buffers b, RunState* st);
__global__ void k_rev_edge_list(DevGraph g, Buffers b, RunState* st);
__global__ void k_build_origin(const int32_t* off, int32_t n, int32_t m, int32_t* origin);
__global__ void k_undo_level(Buffers b, RunState* st);
// The persistent traversal kernel for graphs with vertex records of the given
// width (0: none); parameters DevGraph, Buffers, RunState*, depth, root, forced,
// tree, tree nodes, bit-parallel tree, epoch, stall.
void* persistent_kernel(int32_t record);
// The graph driver's kernel for runs of small levels (record 4 or 8; one cluster
// of kThreads-thread blocks); parameters DevGraph, Buffers, RunState*.
void* small_levels_kernel(int32_t record);
__global__ void k_profile_level(DevGraph g, Buffers b, RunState* st, int32_t* depth, int32_t L, int32_t v, uint32_t f,
                                unsigned long long e, long long discovered, uint32_t vsel);
__global__ void k_profile_reset(RunState* st, int32_t slot);
__global__ void k_undo_level_p(Buffers b, int32_t* depth, uint32_t qout, unsigned int count, uint32_t vsel);

// graph creation
__global__ void k_validate(const int32_t* off, const int32_t* idx, int32_t n, int32_t m, int32_t* bad);
// degree statistics: out-, in- and total degree (in null: a symmetric graph, out-degree only)
struct DegSums {
  unsigned long long s1, s2;
  unsigned int dmax, pad;
};
constexpr int kDegFinishThreads = 1024;
__global__ void k_deg_reduce(const int32_t* off, const int32_t* off_in, int32_t n, DegSums* out);
__global__ void k_deg_hist(const int32_t* off, const int32_t* off_in, int32_t n, long long at1, long long at2,
                           int32_t* hist);
__global__ void k_deg_finish(const int32_t* hist, long long at1, long long at2, int32_t n, const DegSums* sums,
                             int32_t symmetric, long long* out);
__global__ void k_tr_count(const int32_t* idx, int32_t m, int32_t* cnt);
__global__ void k_scan_reduce(const int32_t* in, int32_t len, long long* bsum);
__global__ void k_scan_top(long long* bsum, int32_t nblocks);
__global__ void k_scan_apply(const int32_t* in, int32_t len, const long long* bsum, int32_t* out);
__global__ void k_tr_scatter(const int32_t* off, const int32_t* idx, int32_t n, int32_t m, int32_t* cursor,
                             int32_t* in_idx);
__global__ void k_records(const int32_t* off, const int32_t* idx, int32_t n, int32_t w, int32_t* rec);
__global__ void k_pull_hint(const int32_t* off, const int32_t* in_off, const int32_t* in_idx, int32_t n,
                            int32_t* hint);
__global__ void k_vis_init(const int32_t* off, const int32_t* in_off, int32_t n, int32_t words, uint32_t* vis_init,
                           unsigned int* isolated_count);

}  // namespace bfs
