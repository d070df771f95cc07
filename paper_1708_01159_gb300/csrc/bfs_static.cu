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
// Every level is the main library's edge-centric push (bfs_push.cuh) in ordinary
// launches, so that a traversal takes whatever part of the GPU is free: a caller
// of this kind may well have a kernel of its own resident, which a cooperative
// launch (every block resident at once) would have to wait for. The launches of
// several levels are enqueued together, each let in while the one before it ends
// (programmatic dependent launch), and the control block is read back after them;
// a level past the last finds an empty frontier and returns. Bound by the chain of
// launches and dependent loads: R-MAT 18 (262,144 vertices, 7.7M edges) 184 to 246 us a
// call, Erdos-Renyi of 2^17 vertices and degree 8 101 to 104; as one cooperative
// launch 214 to 265 and 115, without the early launches 231 to 284 and 166, with
// one thread per frontier vertex and a read for every level 16,300 on R-MAT 18.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "bfs.h"
#include "bfs_push.cuh"

namespace bfs {
namespace {

constexpr int64_t kStaticMaxVertices = 1 << 20;  // 1,048,576 vertices
constexpr int64_t kStaticWords = kStaticMaxVertices / 32;

constexpr int32_t kStaticHeavyCap = 1 << 14;

// What a call starts from zero, and reads back. Level L reads its frontier's size
// and edge count from slot L % 3, appends to slot (L + 1) % 3 and clears slot
// (L + 2) % 3, which level L - 1 was the last to read.
struct StaticControl {
  unsigned long long frontier[3], edges[3];
  unsigned int heavy[3];  // vertices level L sets aside, slot (L + 1) % 3
  int32_t bad;            // the CSR is malformed
  int32_t has_heavy;      // some vertex has kHeavy edges or more
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

// CSR well-formedness, so a malformed graph is refused instead of read out of
// bounds; the visited bitmap's start. The control block is zero before.
__global__ void __launch_bounds__(kThreads)
    k_static_check(StaticScratch* s, const int32_t* off, const int32_t* idx, int32_t n, int32_t m, int32_t root) {
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
}

// Start of a kernel that is launched while the one before it may still run
// (programmatic dependent launch): waits for that one's end and its writes.
__device__ __forceinline__ void after_launch() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Depths and the first frontier, unless the CSR is malformed: then depth stays
// as it is, and every level finds an empty frontier.
__global__ void __launch_bounds__(kThreads)
    k_static_init(StaticScratch* s, const int32_t* off, int32_t n, int32_t root, int32_t* depth) {
  after_launch();
  if (s->c.bad) return;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = tid; i < n; i += stride) depth[i] = (i == root) ? 0 : -1;
  if (tid == 0) {
    s->q[0][0] = root;
    s->c.frontier[0] = 1;
    s->c.edges[0] = (unsigned long long)(off[root + 1] - off[root]);
  }
}

// Level L. kHeavyPart: the vertices its first launch set aside.
template <bool kHeavyPart>
__global__ void __launch_bounds__(kThreads, 4)
    k_static_level(StaticScratch* s, const int32_t* off, const int32_t* idx, int32_t* depth, int32_t L) {
  __shared__ int32_t s_a[kPeTile];
  __shared__ int32_t s_beg[kPeTile];
  after_launch();
  StaticControl& c = s->c;
  const int here = L % 3, next = (L + 1) % 3, after = (L + 2) % 3;
  const unsigned int f = (unsigned int)c.frontier[here], count = kHeavyPart ? c.heavy[next] : 0u;
  const unsigned long long e = c.edges[here];
  if (!kHeavyPart && blockIdx.x == 0 && threadIdx.x == 0) {  // in every launch: a level past the last reads it
    c.frontier[after] = 0;
    c.edges[after] = 0;
    c.heavy[after] = 0;
  }
  if (kHeavyPart ? count == 0u : f == 0u) return;
  BFS_DECLARE_STAGE(stage);
  DevGraph g;
  g.off = off;
  g.idx = idx;
  Level lv{};
  lv.qin = (L & 1) ? s->q[1] : s->q[0];
  lv.qout = (L & 1) ? s->q[0] : s->q[1];
  lv.vis = s->vis;
  lv.depth = depth;
  lv.tail = &c.frontier[next];
  lv.n_heavy = &c.heavy[next];
  lv.next_depth = L + 1;
  lv.frontier = (int32_t)f;
  lv.latency_bound = (long long)e < kLatencyEdges;
  unsigned long long edges = 0;
  if (kHeavyPart)
    body_push_heavy(g, lv, stage, s_a, s_beg, s->heavy, (int32_t)min(count, (unsigned)kStaticHeavyCap), edges);
  else if (pe_shared(f, (long long)e, c.has_heavy != 0))
    body_push_shared(g, lv, lv.qin, lv.frontier, stage, s_a, s_beg, edges);
  else
    body_push_tiles(g, lv, stage, s_a, s_beg, s->heavy, kStaticHeavyCap, edges);
  stage_flush(stage, lv, 1);
  block_add_u64(edges, &c.edges[next]);
}

// Levels enqueued before the control block is read: a read costs about 25 us, a
// level past the last 1.7 us (3.3 with the vertices set aside). First what a
// random graph of this mean degree needs, 1.75 ln n / ln(m / n) (6 levels for
// R-MAT 14 and 18, 10 for Erdos-Renyi of 2^17 vertices and degree 8, 17 for 2^20
// and 4), from then on as many as have run.
constexpr int32_t kFewestLevels = 8, kMostAtFirst = 20, kMostLevels = 64;
int32_t levels_at_first(int64_t n, int64_t m) {
  const double degree = (double)m / (double)n;
  const double levels = degree > 1.0 ? 1.75 * std::log((double)n) / std::log(degree) : 0.0;
  const double enough = std::min<double>(std::max<double>(std::ceil(levels), kFewestLevels), kMostAtFirst);
  return (int32_t)std::min<double>(enough, (double)n);
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
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  const int grid = sms * 4;
  if (cudaMemsetAsync(&s->c, 0, sizeof s->c, stream) != cudaSuccess) return static_fail(BFS_ERR_CUDA, "control reset failed");
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  k_static_check<<<grid, kThreads, 0, stream>>>(s, row_offsets, col_indices, nn, mm, root);
  TRY_LAUNCH("validate");
  cudaLaunchKernelEx(&cfg, k_static_init, s, row_offsets, nn, root, depth_out);
  TRY_LAUNCH("init");
  bool has_heavy = m >= kHeavy;  // as far as is known before the first read
  int32_t L = 0;
  for (int32_t levels = levels_at_first(n, m); L <= nn; levels = std::min(std::max(L, kFewestLevels), kMostLevels)) {
    for (const int32_t end = L + levels; L < end; ++L) {
      cudaLaunchKernelEx(&cfg, k_static_level<false>, s, row_offsets, col_indices, depth_out, L);
      TRY_LAUNCH("level");
      if (!has_heavy) continue;
      cudaLaunchKernelEx(&cfg, k_static_level<true>, s, row_offsets, col_indices, depth_out, L);
      TRY_LAUNCH("level");
    }
    StaticControl c{};
    if (cudaMemcpyAsync(&c, &s->c, sizeof c, cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
      return static_fail(BFS_ERR_CUDA, "traversal failed to run");
    if (c.bad) return static_fail(BFS_ERR_BAD_GRAPH, "CSR failed validation");
    if (c.frontier[L % 3] == 0) return BFS_OK;
    has_heavy = c.has_heavy != 0;
  }
  return static_fail(BFS_ERR_TIMEOUT, "more levels than vertices");
}

}  // extern "C"
