"""Index arithmetic at the largest sizes the library accepts (n below 2^31 - 1,
m up to 2^31 - 65): the device functions' own sources, run on the host over
arrays that end the program when an access leaves them. Only the accesses at
the far end are made, so a case takes a moment and no memory."""
import pytest

from tests import device_source as ds

M_MAX = 2 ** 31 - 1 - 64  # bfs_graph_create's limit

CONSTANTS = "".join(ds.constant("bfs_kernels.cuh", k) for k in ("kThreads", "kPeItems", "kPeTile"))

ENTRIES = r"""
int main(int, char** argv) {
  const int32_t m = atoi(argv[1]);
  const int32_t off[3] = {0, m / 3, m};
  const int64_t first = (int64_t)(m - 1) / kPeTile * kPeTile;  // the last chunk
  gridDim.x = 1u << 20;
  blockIdx.x = (unsigned)((m - 1) / kPeTile);
  std::vector<int> seen((size_t)(m - first));
  run_block(kThreads, [&] {
    for_each_entry(off, 2, m, [&](int32_t e, int32_t v) {
      if (e < first || e >= m || v != (e >= m / 3)) {
        printf("entry %d of row %d\n", e, v);
        fflush(stdout);
        _exit(1);
      }
      atomicAdd(&seen[(size_t)(e - first)], 1);
    });
  });
  for (int s : seen)
    if (s != 1) return 2;
  return 0;
}
"""


@pytest.mark.parametrize("m", [2048, 2 ** 31 - 256, 2 ** 31 - 255, 2 ** 31 - 129, M_MAX - 1, M_MAX])
def test_every_entry_of_the_last_chunk_once(tmp_path, m):
    rc, out = ds.run(str(tmp_path), CONSTANTS + ds.function("bfs_kernels.cu", "for_each_entry") + ENTRIES, m)
    assert rc == 0, (rc, out)


# The push levels' own loops; the visits only count the edges they are given.
PUSH_STUBS = r"""
enum { CM_BLOCK, ST_TIMEOUT = 5 };
struct Stage {};
struct DevGraph { const int32_t *off, *idx; };
struct Level { const int32_t* qin; int32_t frontier; };
struct CtaPipe { int32_t* chunk; uint64_t* bar; uint32_t parity0, parity1, extra_tx; };
inline void stage_flush(const Stage&, const Level&, unsigned int) {}
inline void mbar_expect_tx(uint64_t*, uint32_t) {}
inline void bulk_g2s(void*, const void*, uint32_t, uint64_t*) {}
inline bool mbar_wait_bounded(uint64_t*, uint32_t) { return true; }
volatile int32_t named;  // keeps the loads of the neighbours
template <int K, int kCount = CM_BLOCK>
void visit_km(const DevGraph&, const Level&, const Stage&, const int32_t (&v)[K], uint32_t valid, unsigned long long& e) {
  for (int k = 0; k < K; ++k) named = v[k];
  e += (unsigned)__builtin_popcount(valid);
}
template <int K, int kCount = CM_BLOCK>
void visit_k(const DevGraph&, const Level&, const Stage&, const int32_t (&v)[K], int nv, unsigned long long& e) {
  for (int k = 0; k < K; ++k) named = v[k];
  e += (unsigned)max(nv, 0);
}
"""

PUSH_BODIES = r"""
// Edges the block visits, its threads one after another (no list long enough to be staged).
static unsigned long long visited(int body, const DevGraph& g, const Level& lv) {
  const Stage s{};
  unsigned long long edges = 0;
  blockDim.x = kThreads;
  for (threadIdx.x = 0; threadIdx.x < kThreads; ++threadIdx.x) {
    int32_t status = 0;
    CtaPipe pp{};
    switch (body) {
      case 0: body_push_thread(g, lv, s, edges); break;
      case 4: push_vwarp<4>(g, lv, s, edges); break;
      case 8: push_vwarp<8>(g, lv, s, edges); break;
      case 16: push_vwarp<16>(g, lv, s, edges); break;
      case 32: push_vwarp<32>(g, lv, s, edges); break;
      default: body_push_cta(g, lv, s, pp, &status, edges); break;
    }
  }
  return edges;
}
"""

LAST_ROW = r"""
int main(int, char** argv) {
  const int body = atoi(argv[1]);
  const int32_t m = atoi(argv[2]), d = atoi(argv[3]);
  const int32_t off[4] = {0, 400, m - d, m};  // vertex 0: 400 edges, vertex 2: the last d
  const DevGraph g{off, guarded_zeros((int64_t)m + 8)};
  const int32_t one[1] = {2};
  if (visited(body, g, Level{one, 1}) != (unsigned)d) return 1;
  // more vertices than the block has groups, long and short lists side by side
  int32_t q[100];
  for (int i = 0; i < 100; ++i) q[i] = i % 2 * 2;
  return visited(body, g, Level{q, 100}) != 50ull * (400u + (unsigned)d);
}
"""

PUSHES = [0, 4, 8, 16, 32, 99]  # thread, virtual warps, CTA


def push_source():
    names = ["body_push_thread", "push_vwarp", "body_push_cta"]
    consts = [ds.constant("bfs_kernels.cu", "kLongList"), ds.constant("bfs_internal.cuh", "kStageCap")] + \
        [ds.constant("bfs_kernels.cuh", k) for k in ("kCtaChunk", "kCtaDirect")]
    return CONSTANTS + "".join(consts) + PUSH_STUBS + "".join(ds.function("bfs_kernels.cu", n) for n in names) + \
        PUSH_BODIES


@pytest.mark.parametrize("body", PUSHES)
def test_pushes_visit_every_edge_of_the_last_row_once(tmp_path, body):
    exe = ds.build(str(tmp_path), push_source() + LAST_ROW)
    for m, d in [(5000, 7), (M_MAX, 1), (M_MAX, 5), (M_MAX - 3, 33), (M_MAX, 100), (M_MAX, 255), (M_MAX - 1, 300),
                 (M_MAX, 511)]:
        rc, out = ds.execute(exe, body, m, d)
        assert rc == 0, (m, d, rc, out)


FULL_QUEUE = r"""
int main(int, char** argv) {  // a frontier of f vertices without edges, the grid's last block
  const int body = atoi(argv[1]);
  const int32_t f = atoi(argv[2]);
  const int32_t off[2] = {0, 0};
  gridDim.x = 608;
  blockIdx.x = 607;
  return visited(body, DevGraph{off, nullptr}, Level{guarded_zeros(f), f}) != 0;
}
"""

N_MAX = 2 ** 31 - 2  # bfs_graph_create's limit; a frontier has at most n - 1 vertices


@pytest.mark.parametrize("body", PUSHES)
def test_pushes_end_at_the_end_of_the_largest_queue(tmp_path, body):
    exe = ds.build(str(tmp_path), push_source() + FULL_QUEUE)
    for f in (1, 1000003, N_MAX - 1):
        rc, out = ds.execute(exe, body, f)
        assert rc == 0, (f, rc, out)


UNDO = r"""
struct Buffers { const int32_t* q[2]; uint32_t* vis[2]; };
struct RunState { unsigned long long next_count; uint32_t qsel, vsel; int32_t* depth; };
inline uint32_t atomicAnd(uint32_t* p, uint32_t x) { return __atomic_fetch_and(p, x, __ATOMIC_SEQ_CST); }
"""

UNDO_MAIN = r"""
int main(int, char** argv) {
  const unsigned int f = (unsigned)atoi(argv[1]);
  const int32_t* q = guarded_zeros(f);
  int32_t depth = 7;
  uint32_t vis = ~0u;
  RunState st{f, 0, 0, &depth};
  const Buffers b{{q, q}, {&vis, &vis}};
  gridDim.x = 1216;
  blockIdx.x = 1215;
  blockDim.x = kThreads;
  for (threadIdx.x = 0; threadIdx.x < kThreads; ++threadIdx.x) {
    k_undo_level(b, &st);
    k_undo_level_p(b, &depth, 0, f, 0);
  }
  return 0;
}
"""


def test_undo_ends_at_the_end_of_the_largest_queue(tmp_path):
    src = CONSTANTS + UNDO + ds.function("bfs_kernels.cu", "k_undo_level") + \
        ds.function("bfs_kernels.cu", "k_undo_level_p") + UNDO_MAIN
    rc, out = ds.run(str(tmp_path), src, N_MAX - 1)
    assert rc == 0, (rc, out)


SCAN = r"""
template <typename T>
T block_exclusive_scan(T x, T* total) {
  *total = x;
  return 0;
}
"""

SCAN_MAIN = r"""
int main(int, char** argv) {  // the block of the last entries alone
  const int32_t len = atoi(argv[1]);
  const int64_t nblk = ((int64_t)len + kPeTile - 1) / kPeTile;
  std::vector<long long> bsum((size_t)nblk + 1, -1);
  gridDim.x = 608;
  blockIdx.x = (unsigned)((nblk - 1) % 608);
  blockDim.x = kThreads;
  const int32_t* in = guarded_zeros(len);
  int32_t* out = (int32_t*)mmap(nullptr, ((size_t)len + 1) * 4, PROT_READ | PROT_WRITE,
                                MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (out == MAP_FAILED) return 4;
  threadIdx.x = 0;
  k_scan_reduce(in, len, bsum.data());
  if (bsum[(size_t)nblk - 1] != 0) return 1;  // its sum was written
  bsum[(size_t)nblk] = 12345;
  k_scan_apply(in, len, bsum.data(), out);
  return out[len] != 12345;  // and the total
}
"""


@pytest.mark.parametrize("n", [1, 2048, 2049, 2 ** 31 - 2047, N_MAX])
def test_scan_reaches_its_last_block(tmp_path, n):
    src = CONSTANTS + SCAN + ds.function("bfs_kernels.cu", "k_scan_reduce") + \
        ds.function("bfs_kernels.cu", "k_scan_apply") + SCAN_MAIN
    rc, out = ds.run(str(tmp_path), src, n)
    assert rc == 0, (rc, out)
