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
