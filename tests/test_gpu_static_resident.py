"""bfs_run_static beside a kernel that stays on the GPU: the call finishes while
the other kernel is still running (its launches need no particular part of the
GPU to be free), and its depths are right on graphs that end just before, at and
just after the levels it enqueues together (8, then 4, 6, 9, ...)."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def static(off, idx, g, root, stream):
    out = torch.full((g.n,), 7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = bfs.lib().bfs_run_static(off.data_ptr(), idx.data_ptr(), g.n, g.m, int(root), out.data_ptr(),
                                  stream.cuda_stream)
    assert rc == bfs.BFS_OK, bfs.lib().bfs_last_error_detail().decode()
    return out


def test_runs_beside_a_resident_kernel():
    bfs.build()
    g = gg.rmat(14, 16, seed=1001)
    root = int(gg.sample_roots(g, 1, seed=2001, giant=True)[0])
    off, idx = torch.from_numpy(g.off).cuda(), torch.from_numpy(g.idx).cuda()
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    torch.cuda._sleep(1000)
    static(off, idx, g, root, mine)  # kernels loaded
    out = torch.full((g.n,), 7, dtype=torch.int32, device="cuda")
    done = torch.cuda.Event()
    torch.cuda.synchronize()
    with torch.cuda.stream(other):
        torch.cuda._sleep(2_000_000_000)  # one block, about a second
        done.record(other)
    rc = bfs.lib().bfs_run_static(off.data_ptr(), idx.data_ptr(), g.n, g.m, root, out.data_ptr(), mine.cuda_stream)
    still_there = not done.query()
    torch.cuda.synchronize()
    assert rc == bfs.BFS_OK and still_there
    assert np.array_equal(out.cpu().numpy(), oracle.bfs(g.off, g.idx, root).depth)


@pytest.mark.parametrize("levels", [1, 2, 7, 8, 9, 11, 12, 13, 18, 19, 300])
def test_paths_around_the_levels_enqueued_together(levels):
    bfs.build()
    g = gg.from_edges(levels + 1, np.arange(levels - 1), np.arange(1, levels))  # and one vertex apart
    off = torch.from_numpy(g.off).cuda()
    idx = torch.from_numpy(g.idx if g.m else np.zeros(1, np.int32)).cuda()
    got = static(off, idx, g, 0, torch.cuda.current_stream()).cpu().numpy()
    assert np.array_equal(got, np.r_[np.arange(levels), -1].astype(np.int32))
