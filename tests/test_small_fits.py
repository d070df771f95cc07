"""What a small level may be: every level that the rule leaves to the leader
cluster fits the lists its vertices are dealt into, and the fields its counts
are packed into (16 bits each in a block's counter and message)."""
from tests import device_source as ds

SOURCE = r"""
int main() {
  for (uint32_t c = 2; c <= kMaxCluster; c *= 2)
    for (unsigned long long f = 1; f <= 1ull << 31; f = f < 70000 ? f + 1 : f * 3 / 2)
      for (unsigned long long e : {0ull, 1ull, 1000ull, c * (unsigned long long)kSmallEdges})
        if (small_fits((unsigned)f, e, c)) {
          const unsigned long long most = (f + c - 1) / c;  // vertices of the first block
          if (most > kWonCap || most * 8 > 0xffff) {
            printf("%llu vertices, %llu edges, %u blocks\n", f, e, c);
            return 1;
          }
        }
  // what the rule is for: a grid's small levels
  return !small_fits(4500, 16 * kSmallEdges, 16) || small_fits(4500, 16 * kSmallEdges + 1, 16);
}
"""


def test_every_small_level_fits_the_leader(tmp_path):
    src = ds.constant("bfs_kernels.cuh", "kMaxCluster") + \
        "".join(ds.constant("bfs_small.cuh", k) for k in ("kCandCap", "kWonCap", "kSmallEdges")) + \
        ds.function("bfs_small.cuh", "small_fits")
    rc, out = ds.run(str(tmp_path), src + SOURCE)
    assert rc == 0, out
