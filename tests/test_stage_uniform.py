"""The block stage's drain is decided once for the whole block, whatever a
thread adds to the stage as soon as it has left the drain: stage_drain's own
source, run by two host threads of which one is held back at the barrier until
the other has put its next entries."""
import pytest

from tests import device_source as ds

BODY = r"""
static int32_t buf[kStageCap], out[2 * kStageCap];
static unsigned int cnt = 0, base = 0;
static unsigned long long tail = 0;
static int barriers[2][3];  // of each thread, drain by drain
static thread_local int passed = 0;
static void hold_back() {  // thread 1 leaves its first barrier late
  if (++passed == 1 && threadIdx.x == 1) std::this_thread::sleep_for(std::chrono::milliseconds(200));
}
int main(int, char** argv) {
  const unsigned int threshold = (unsigned)atoi(argv[1]);
  after_barrier = hold_back;
  run_block(2, [=] {
    const Stage s{buf, &cnt, &base};
    auto put = [&](int32_t v) { buf[atomicAdd(&cnt, 1u)] = v; };
    auto drain = [&](int i, unsigned int at) {
      const int before = passed;
      stage_drain(s, out, &tail, at);
      barriers[threadIdx.x][i] = passed - before;
    };
    if (threadIdx.x == 0)
      for (unsigned int i = 0; i + 1 < threshold; ++i) put((int32_t)i);
    drain(0, threshold);  // one entry short: nothing moves
    if (threadIdx.x == 0) put((int32_t)threshold - 1);
    drain(1, threshold);  // full: all of it moves
    drain(2, 1u);         // empty
  });
  for (int i = 0; i < 3; ++i) printf("drain %d: %d and %d barriers\n", i, barriers[0][i], barriers[1][i]);
  for (int i = 0; i < 3; ++i)
    if (barriers[0][i] != barriers[1][i]) return 5;
  if (tail != threshold || cnt != 0) return 1;
  for (unsigned int i = 0; i < threshold; ++i)
    if (out[i] != (int32_t)i) return 2;
  return 0;
}
"""


@pytest.mark.parametrize("threshold", [1, 2, 1024, 2048])
def test_drain_is_uniform(tmp_path, threshold):
    src = ds.constant("bfs_internal.cuh", "kStageCap") + ds.function("bfs_internal.cuh", "Stage") + \
        ds.function("bfs_internal.cuh", "stage_drain")
    rc, out = ds.run(str(tmp_path), src + BODY, threshold)
    assert rc == 0, (rc, out)
