"""The bounded waits of the small levels' cluster, run out through the test hook:
one block's count exchange that never completes, and a state that is never
published to the blocks that wait for it. The run reports BFS_ERR_TIMEOUT after
a few seconds and the next one on the same graph is exact. Such a run can only
time out if the cluster ran its small levels, so the same calls show that it
does, and that a graph of out-degree 9 and a frontier too large for the cluster
do without."""
import time

import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

MESSAGE, STATE = 5, 6


@pytest.fixture(scope="module", autouse=True)
def built():
    bfs.build()
    yield
    bfs.bfs_debug_stall_next_launch(0)
    bfs.bfs_load_tree(None)


@pytest.fixture
def pushes(tmp_path):
    """Trees that pull the first `pulls` levels and push (virtual warps) after them:
    whether small levels run must not depend on the default tree."""
    def load(pulls=0):
        p = tmp_path / "tree"
        level = bfs.FEATURES.index("level")
        p.write_text(f"bfs-tree 1 3\n{level} {pulls - 1} 1 2 -1\n-1 0 -1 -1 {bfs.VARIANTS.index('pull')}\n"
                     f"-1 0 -1 -1 {bfs.VARIANTS.index('push_warp')}\n")
        bfs.bfs_load_tree(str(p))
    load()
    return load


def out_degree(d, n):
    rng = np.random.default_rng(d)
    return gg.Graph((d * np.arange(n + 1)).astype(np.int32), rng.integers(0, n, d * n).astype(np.int32), f"out{d}")


def run(G, g, root, blocks=0):
    d = torch.empty(g.n, dtype=torch.int32, device="cuda")
    st = bfs.bfs_run_ex(G.handle, root, d, stats=True, mode=bfs.MODE_PERSISTENT, grid_blocks=blocks)
    ref = oracle.bfs(g.off, g.idx, root)
    assert np.array_equal(d.cpu().numpy(), ref.depth) and st["edges_reached"] == ref.edges_reached


@pytest.mark.parametrize("stall,blocks", [(MESSAGE, 0), (MESSAGE, 16), (MESSAGE, 2), (STATE, 0), (STATE, 32)])
@pytest.mark.parametrize("name", ["grid", "one", "out8"])
def test_waits_run_out_then_the_next_run_is_exact(pushes, name, stall, blocks):
    g, flags = {"grid": lambda: (gg.grid(60, 50, 0.1, seed=920), bfs.BFS_SYMMETRIC),
                "one": lambda: (gg.Graph(np.zeros(2, np.int32), np.zeros(0, np.int32), "one"), bfs.BFS_SYMMETRIC),
                "out8": lambda: (out_degree(8, 30000), 0)}[name]()
    root = int(np.argmax(np.diff(g.off)))
    with bfs.Graph(g.off, g.idx, flags) as G:
        run(G, g, root, blocks)
        bfs.bfs_debug_stall_next_launch(stall)
        t0 = time.perf_counter()
        with pytest.raises(bfs.BFSError) as e:
            run(G, g, root, blocks)
        assert e.value.code == bfs.BFS_ERR_TIMEOUT and 1.0 < time.perf_counter() - t0 < 30.0
        run(G, g, root, blocks)


def uneven():
    """A tree of arity 8, its 4,096 vertices of level 4 numbered 0 to 4,095; every
    16th of the first 2,048 has 8 children, each with one child, the others have
    none. Dealt out in that order, one block of 16 names all of the next level."""
    level, first = np.array([4096]), 4097
    src, dst = [], []
    for k in range(4):
        children = np.arange(8 ** (k + 1)) if k == 3 else np.arange(first, first + 8 ** (k + 1))
        first += 0 if k == 3 else len(children)
        src.append(np.repeat(level, 8)), dst.append(children)
        level = children
    some = np.repeat(np.arange(0, 2048, 16), 8)
    a = np.arange(first, first + len(some))
    src += [some, a]
    dst += [a, a + len(a)]
    return gg.from_edges(first + 2 * len(a), np.concatenate(src), np.concatenate(dst), symmetrize=False, name="uneven")


def test_wait_runs_out_while_the_others_deal(pushes):
    """The other blocks are in the barrier in front of a dealing when the last
    one's wait runs out."""
    pushes(4)
    g = uneven()
    with bfs.Graph(g.off, g.idx, 0) as G:
        run(G, g, 4096)
        bfs.bfs_debug_stall_next_launch(MESSAGE)
        with pytest.raises(bfs.BFSError) as e:
            run(G, g, 4096)
        assert e.value.code == bfs.BFS_ERR_TIMEOUT
        run(G, g, 4096)


@pytest.mark.parametrize("stall", [MESSAGE, STATE])
def test_graphs_without_small_levels_end_normally(pushes, stall):
    g = out_degree(9, 3000)
    with bfs.Graph(g.off, g.idx, 0) as G:
        bfs.bfs_debug_stall_next_launch(stall)
        run(G, g, 5)
    # one block alone is no cluster
    g = gg.grid(60, 50, 0.1, seed=920)
    with bfs.Graph(g.off, g.idx) as G:
        bfs.bfs_debug_stall_next_launch(stall)
        run(G, g, int(np.argmax(np.diff(g.off))), 1)
