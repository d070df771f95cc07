"""The default grid of a multi-source wave at the edges of its rule (32 roots, long
in-lists, out-degrees of 8 and 9, vertex counts around two blocks an SM): every row
equals the oracle's, and one on a grid the caller names."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def out_degree(d, n, hub=0):
    """Out-degree d; the first `hub` entries all name vertex 0."""
    rng = np.random.default_rng(d)
    idx = rng.integers(0, n, d * n).astype(np.int32)
    idx[:hub] = 0
    return gg.Graph((d * np.arange(n + 1)).astype(np.int32), idx, f"out{d}")


GRAPHS = {
    "out8": lambda: out_degree(8, 4000),
    "out9": lambda: out_degree(9, 4000),
    "out8, long in-list": lambda: out_degree(8, 4000, 400),
    "grid, 311,296 vertices": lambda: gg.grid(512, 608, 0.1, seed=930),
    "er, 312,000 vertices": lambda: gg.erdos_renyi(312000, 6.0, seed=931),
    "one": lambda: gg.Graph(np.zeros(2, np.int32), np.zeros(0, np.int32), "one"),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
def test_waves_on_default_grids(name):
    bfs.build()
    g = GRAPHS[name]()
    symmetric = not name.startswith("out")
    with bfs.Graph(g.off, g.idx, bfs.BFS_SYMMETRIC if symmetric else 0) as G:
        for k in (1, 31, 32):
            roots = np.random.default_rng(k).integers(0, g.n, k).astype(np.int32)
            D, E = oracle.bfs_batch(g.off, g.idx, roots)
            for blocks in (0, 7):
                bfs.bfs_batch_set_config(G.handle, 0, 16, blocks)
                out = torch.full((k * g.n,), -7, dtype=torch.int32, device="cuda")
                edges = bfs.bfs_run_batch(G.handle, roots, out, edges=True)
                assert np.array_equal(out.cpu().numpy().reshape(k, g.n), D), (k, blocks)
                assert np.array_equal(edges, E), (k, blocks)
