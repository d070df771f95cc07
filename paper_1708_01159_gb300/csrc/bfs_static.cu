// bfs_run_static: a single-source BFS that allocates no memory.
//
// Some callers cannot allocate device memory while they run: code inside a
// memory-pool arena they do not own, a plugin handed fixed buffers by its host
// application, or a real-time loop where a cudaMalloc (which may synchronise
// the device or fail under fragmentation) is not allowed. For them this file
// keeps the traversal's scratch (two frontier queues, the visited bitmap and
// the level counters) in one file-scope device array of fixed size, and the
// entry point calls no allocating routine at all; the caller passes the graph
// and the output in device memory it already owns.
//
// One cooperative launch checks the CSR and runs the whole traversal: every
// level is the main library's edge-centric push (bfs_push.cuh), levels separated
// by its grid barriers; the host reads one status block back at the end.
#include <algorithm>
#include <cstdio>

#include "bfs.h"
#include "bfs_push.cuh"

namespace bfs {
namespace {

constexpr int64_t kStaticMaxVertices = 1 << 20;  // 1,048,576 vertices
constexpr int64_t kStaticWords = kStaticMaxVertices / 32;

constexpr int32_t kStaticHeavyCap = 1 << 14;

// What a call starts from zero, and reads back.
struct StaticControl {
  unsigned long long tail3[3], edg3[3];  // level words, as the persistent traversal's (bfs_internal.cuh)
  unsigned long long bar64;
  unsigned int heavy3[3];
  int32_t bad;        // the CSR is malformed
  int32_t has_heavy;  // some vertex has kHeavy edges or more
  int32_t status;
};

// Layout: queue 0 | queue 1 | visited bitmap | heavy list | control
struct StaticScratch {
  int32_t q[2][kStaticMaxVertices];
  uint32_t vis[kStaticWords];
  int32_t heavy[kStaticHeavyCap];
  StaticControl c;
};

// Held by every GPU that loads the library, until the process exits (about 8.2 MB).
static __device__ __align__(256) StaticScratch g_static_scratch;

// The control block is zero when the kernel starts. A malformed CSR ends it
// before anything reads through it, with depth untouched. R-MAT 18 (262,144
// vertices, 7.7M edges): 0.25 to 0.30 ms a call; one thread per frontier vertex and a
// read of the next frontier size on the host for every level took 16.3 ms, a
// hub's list being walked one edge at a time.
__global__ void __launch_bounds__(kThreads, 4)
    k_static_bfs(StaticScratch* s, const int32_t* off, const int32_t* idx, int32_t n, int32_t m, int32_t root,
                 int32_t* depth) {
  __shared__ int32_t s_a[kPeTile];
  __shared__ int32_t s_beg[kPeTile];
  BFS_DECLARE_STAGE(stage);
  StaticControl& c = s->c;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int32_t bad = tid == 0 && (off[0] != 0 || off[n] != m);
  int32_t heavy = 0;
  for (int64_t v = tid; v < n; v += stride) {
    const int32_t d = off[v + 1] - off[v];
    bad |= off[v + 1] < off[v];
    heavy |= d >= kHeavy;
  }
  // 16 bytes a load where the caller's array allows it
  const int64_t head = min((int64_t)((16u - (reinterpret_cast<uintptr_t>(idx) & 15u)) & 15u) / 4, (int64_t)m);
  const int64_t quads = (m - head) / 4;
  const int4* idx4 = reinterpret_cast<const int4*>(idx + head);
  for (int64_t i = tid; i < quads; i += stride) {
    const int4 x = idx4[i];
    bad |= (uint32_t)x.x >= (uint32_t)n || (uint32_t)x.y >= (uint32_t)n || (uint32_t)x.z >= (uint32_t)n ||
           (uint32_t)x.w >= (uint32_t)n;
  }
  for (int64_t e = tid; e < head; e += stride) bad |= (uint32_t)idx[e] >= (uint32_t)n;
  for (int64_t e = head + quads * 4 + tid; e < m; e += stride) bad |= (uint32_t)idx[e] >= (uint32_t)n;
  const int64_t words = (n + 31) / 32;
  for (int64_t w = tid; w < words; w += stride) s->vis[w] = (w == (root >> 5)) ? (1u << (root & 31)) : 0u;
  if (bad) atomicOr(&c.bad, 1);
  if (heavy) atomicOr(&c.has_heavy, 1);
  if (tid == 0) s->q[0][0] = root;
  unsigned long long target = 0;
  if (!grid_arrive_wait(&c.bar64, target, &c.status)) return;
  if (*reinterpret_cast<volatile int32_t*>(&c.bad)) return;  // uniform over the grid
  const bool has_heavy = *reinterpret_cast<volatile int32_t*>(&c.has_heavy) != 0;
  for (int64_t i = tid; i < n; i += stride) depth[i] = (i == root) ? 0 : -1;
  bool ok = grid_arrive_wait(&c.bar64, target, &c.status);
  DevGraph g;
  g.off = off;
  g.idx = idx;
  unsigned int f = 1;
  unsigned long long e = (unsigned long long)(off[root + 1] - off[root]);
  uint32_t slot = 0;
  for (int32_t L = 0; ok && f != 0u; ++L) {
    if (L > n) {
      if (tid == 0) c.status = ST_TIMEOUT;
      break;
    }
    const uint32_t next = slot == 2u ? 0u : slot + 1u;
    if (tid == 0) {  // the slot of a barrier every block has left
      const uint32_t after = next == 2u ? 0u : next + 1u;
      c.tail3[after] = 0;
      c.edg3[after] = 0;
      c.heavy3[after] = 0;
    }
    Level lv{};
    lv.qin = (L & 1) ? s->q[1] : s->q[0];
    lv.qout = (L & 1) ? s->q[0] : s->q[1];
    lv.vis = s->vis;
    lv.depth = depth;
    lv.tail = &c.tail3[next];
    lv.n_heavy = &c.heavy3[next];
    lv.next_depth = L + 1;
    lv.frontier = (int32_t)f;
    lv.latency_bound = (long long)e < kLatencyEdges;
    unsigned long long edges = 0;
    if (pe_shared(f, (long long)e, has_heavy)) {
      body_push_shared(g, lv, lv.qin, lv.frontier, stage, s_a, s_beg, edges);
    } else {
      body_push_tiles(g, lv, stage, s_a, s_beg, s->heavy, kStaticHeavyCap, edges);
      if (has_heavy) {
        if (!grid_arrive_wait(&c.bar64, target, &c.status)) break;
        const unsigned int count = *reinterpret_cast<volatile unsigned int*>(lv.n_heavy);
        body_push_heavy(g, lv, stage, s_a, s_beg, s->heavy, (int32_t)min(count, (unsigned)kStaticHeavyCap), edges);
      }
    }
    stage_flush(stage, lv, 1);
    ok = level_arrive_wait(lv.tail, &c.edg3[next], block_sum_u64(edges), &c.status, &f, &e);
    slot = next;
  }
}

int static_fail(int code, const char* msg) { return bfs::set_error_detail(code, msg); }

// A launch that could not start (a stream of another device, say) reports its
// CUDA error string instead of surfacing later as a failed copy.
int launch_status(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return BFS_OK;
  char buf[256];
  snprintf(buf, sizeof buf, "%s launch: %s", what, cudaGetErrorString(e));
  return static_fail(BFS_ERR_CUDA, buf);
}

}  // namespace
}  // namespace bfs

using namespace bfs;

#define TRY_LAUNCH(what)                     \
  do {                                       \
    const int r_ = launch_status(what);      \
    if (r_ != BFS_OK) return r_;             \
  } while (0)

extern "C" {

int bfs_run_static(const int32_t* row_offsets, const int32_t* col_indices, int64_t n, int64_t m, int32_t root,
                   int32_t* depth_out, bfs_stream_t stream_) {
  if (!row_offsets || !depth_out || (m > 0 && !col_indices))
    return static_fail(BFS_ERR_INVALID_ARG, "null pointer argument");
  if (n < 1 || n > kStaticMaxVertices)
    return static_fail(BFS_ERR_INVALID_ARG, "n must be in [1, 1048576] for bfs_run_static (fixed scratch size)");
  if (m < 0 || m >= INT32_MAX) return static_fail(BFS_ERR_INVALID_ARG, "m out of range");
  if (root < 0 || root >= n) return static_fail(BFS_ERR_INVALID_ARG, "root not in [0, n)");
  cudaStream_t stream = reinterpret_cast<cudaStream_t>(stream_);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return static_fail(BFS_ERR_CUDA, "cudaGetDevice failed");
  if (stream) {
    int sdev = -1;
    if (cudaStreamGetDevice(stream, &sdev) != cudaSuccess) {
      cudaGetLastError();
      return static_fail(BFS_ERR_INVALID_ARG, "stream is not a valid CUDA stream");
    }
    if (sdev != dev) return static_fail(BFS_ERR_INVALID_ARG, "stream belongs to another device than the current one");
  }
  // The array's device address in the current device's context, looked up on
  // every call (the lookup allocates nothing), so a device reset between calls
  // never leaves a stale address behind; in host code the array's name is only
  // a host-side stand-in and must not be passed to a kernel.
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_static_scratch) != cudaSuccess || !p) {
    cudaGetLastError();
    return static_fail(BFS_ERR_CUDA, "cudaGetSymbolAddress failed");
  }
  StaticScratch* s = static_cast<StaticScratch*>(p);
  const int32_t nn = (int32_t)n, mm = (int32_t)m;
  int sms = 0, per_sm = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_static_bfs, kThreads, 0) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  cudaGetLastError();
  if (cudaMemsetAsync(&s->c, 0, sizeof s->c, stream) != cudaSuccess) return static_fail(BFS_ERR_CUDA, "control reset failed");
  const int32_t* off = row_offsets;
  const int32_t* idx = col_indices;
  void* args[] = {&s, &off, &idx, const_cast<int32_t*>(&nn), const_cast<int32_t*>(&mm), &root, &depth_out};
  // every block of the grid resident (the levels are separated by grid barriers)
  cudaLaunchCooperativeKernel(reinterpret_cast<const void*>(&k_static_bfs), dim3(sms * std::min(per_sm, 4)),
                              dim3(kThreads), args, 0, stream);
  TRY_LAUNCH("traversal");
  StaticControl c{};
  if (cudaMemcpyAsync(&c, &s->c, sizeof c, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
      cudaStreamSynchronize(stream) != cudaSuccess)
    return static_fail(BFS_ERR_CUDA, "traversal failed to run");
  if (c.bad) return static_fail(BFS_ERR_BAD_GRAPH, "CSR failed validation");
  if (c.status != ST_OK) return static_fail(BFS_ERR_TIMEOUT, "a bounded device-side wait gave up");
  return BFS_OK;
}

}  // extern "C"
