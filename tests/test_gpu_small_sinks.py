"""Directed graphs of small out-degree whose frontiers are far larger than
their edges: a level of up to two million vertices without an out-edge, and one
with a few edges left, in both drivers, equal to the oracle."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def tree(arity, levels, tail):
    """Complete tree, parent to child; `tail` of its leaves start a path of two more edges."""
    n = sum(arity ** k for k in range(levels))
    child = np.arange(1, n, dtype=np.int64)
    src, dst = [(child - 1) // arity], [child]
    ends = np.arange(n - tail, n, dtype=np.int64)
    for _ in range(2):
        new = np.arange(n, n + tail, dtype=np.int64)
        src.append(ends), dst.append(new)
        ends, n = new, n + tail
    return gg.from_edges(n, np.concatenate(src), np.concatenate(dst), symmetrize=False, name=f"tree{arity}")


@pytest.mark.parametrize("arity,levels,tail", [(8, 8, 0), (8, 8, 3), (4, 9, 17000), (4, 8, 0), (2, 16, 1), (2, 15, 0)])
def test_frontiers_of_sinks(arity, levels, tail):
    bfs.build()
    bfs.bfs_load_tree(None)
    g = tree(arity, levels, tail)
    with bfs.Graph(g.off, g.idx, 0) as G:
        d = torch.empty(g.n, dtype=torch.int32, device="cuda")
        ref = oracle.bfs(g.off, g.idx, 0)
        for mode, blocks in ((bfs.MODE_PERSISTENT, 0), (bfs.MODE_PERSISTENT, 8), (bfs.MODE_GRAPH, 0)):
            d.fill_(-7)
            st = bfs.bfs_run_ex(G.handle, 0, d, mode=mode, grid_blocks=blocks, stats=True, log_capacity=ref.num_levels)
            assert np.array_equal(d.cpu().numpy(), ref.depth), (mode, blocks)
            assert st["levels"] == ref.num_levels and st["edges_reached"] == ref.edges_reached
            assert np.array_equal(st["frontier"], ref.level_count), (mode, blocks)
            assert np.array_equal(st["frontier_edges"], ref.level_edges), (mode, blocks)
