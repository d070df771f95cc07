"""Graphs of out-degree 8 or less: runs driven by the tree and forced variants
take turns on one workspace (in the persistent driver with and without clusters,
in the graph driver on two level-loop graphs), each equal to the oracle, and no
run leaves anything behind for the next."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def out8(n=5000):
    rng = np.random.default_rng(8)
    off = (8 * np.arange(n + 1)).astype(np.int32)
    return gg.Graph(off, rng.integers(0, n, 8 * n).astype(np.int32), "out8"), 0


GRAPHS = {"grid": lambda: (gg.grid(120, 211, 0.1, seed=911), bfs.BFS_SYMMETRIC), "out8": out8}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("mode,blocks", [(bfs.MODE_PERSISTENT, 0), (bfs.MODE_PERSISTENT, 16), (bfs.MODE_PERSISTENT, 608),
                                         (bfs.MODE_GRAPH, 0)])
def test_tree_and_forced_runs_in_turn(name, mode, blocks):
    bfs.build()
    bfs.bfs_load_tree(None)
    g, flags = GRAPHS[name]()
    turns = [-1, 1, 3, -1, -1, 4, 0, 2, -1, bfs.VARIANT_EDGE_LIST, bfs.VARIANT_REVERSE_EDGE_LIST, -1]
    roots = [int(r) for r in gg.sample_roots(g, len(turns), seed=912)]
    with bfs.Graph(g.off, g.idx, flags) as G:
        refs = [oracle.bfs(g.off, g.idx, r) for r in roots]
        outs = [torch.full((g.n,), -7, dtype=torch.int32, device="cuda") for _ in turns]
        for v, r, d in zip(turns, roots, outs):  # queued behind one another
            bfs.bfs_run_ex(G.handle, r, d, mode=mode, grid_blocks=blocks, forced_variant=v)
        torch.cuda.synchronize()
        for v, ref, d in zip(turns, refs, outs):
            assert np.array_equal(d.cpu().numpy(), ref.depth), v
        for v, r, ref, d in zip(turns, roots, refs, outs):
            st = bfs.bfs_run_ex(G.handle, r, d, mode=mode, grid_blocks=blocks, forced_variant=v, stats=True,
                                log_capacity=ref.num_levels)
            assert st["levels"] == ref.num_levels and st["edges_reached"] == ref.edges_reached, v
            assert np.array_equal(st["frontier"], ref.level_count), v
            assert v < 0 or (st["variant"] == v).all()
