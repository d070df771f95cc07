"""The edge-centric push at the edges of its tiles and lists: degrees around the
heavy threshold (1024), frontiers around one scan tile (2048) and one block's
tile (32 to 256), a heavy list that overflows (the allocation-free entry point's
16,384 vertices) and a CSR at an unaligned address. Depths equal the oracle's."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
EDGE = bfs.VARIANTS.index("push_edge")


@pytest.fixture(scope="module", autouse=True)
def built():
    bfs.build()
    bfs.bfs_load_tree(None)
    yield


def fan(front, degrees, n):
    """Root 0 -> vertices 1 .. front, the k-th with degrees[k % len] random out-edges; directed, n vertices."""
    rng = np.random.default_rng(front + n)
    deg = np.zeros(n, np.int64)
    deg[0] = front
    deg[1:front + 1] = np.resize(degrees, front)
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    idx = rng.integers(0, n, int(off[-1])).astype(np.int32)
    idx[:front] = np.arange(1, front + 1)
    return gg.Graph(off, idx, f"fan{front}")


CASES = {
    "heavy edges": lambda: fan(40, [1023, 1024, 1025, 0, 4097, 1], 20000),
    "tile - 1": lambda: fan(2047, [3, 0, 17], 30000),
    "tile": lambda: fan(2048, [3, 0, 17], 30000),
    "tile + 1": lambda: fan(2049, [3, 0, 17], 30000),
    "tile + 1, heavy": lambda: fan(2049, [3, 0, 17, 1, 2, 1024, 5], 60000),
    "many heavy": lambda: fan(5000, [1024], 40000),
    "no edges": lambda: fan(3000, [0], 4000),
    "wide": lambda: fan(200001, [1, 2], 300000),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_edge_centric_push_matches_the_oracle(name):
    g = CASES[name]()
    ref = oracle.bfs(g.off, g.idx, 0)
    with bfs.Graph(g.off, g.idx, 0) as G:
        for mode, blocks in ((bfs.MODE_PERSISTENT, 0), (bfs.MODE_PERSISTENT, 3), (bfs.MODE_GRAPH, 0),
                             (bfs.MODE_HOST_LOOP, 0)):
            d = torch.full((g.n,), -7, dtype=torch.int32, device="cuda")
            st = bfs.bfs_run_ex(G.handle, 0, d, mode=mode, grid_blocks=blocks, forced_variant=EDGE, stats=True,
                                log_capacity=ref.num_levels + 1)
            assert np.array_equal(d.cpu().numpy(), ref.depth), (mode, blocks)
            assert st["edges_reached"] == ref.edges_reached
            assert np.array_equal(st["frontier"], ref.level_count)


@pytest.mark.parametrize("name", sorted(CASES) + ["list overflows"])
def test_allocation_free_entry_matches_the_oracle(name):
    g = fan(17000, [1024], 40000) if name == "list overflows" else CASES[name]()
    ref = oracle.bfs(g.off, g.idx, 0)
    for shift in (0, 1, 3):  # entries the arrays are off a 16-byte boundary
        off = torch.zeros(g.n + 1 + shift, dtype=torch.int32, device="cuda")[shift:]
        idx = torch.zeros(max(g.m, 1) + shift, dtype=torch.int32, device="cuda")[shift:]
        out = torch.full((g.n + shift,), 7, dtype=torch.int32, device="cuda")[shift:]
        off.copy_(torch.from_numpy(g.off))
        idx[:g.m].copy_(torch.from_numpy(g.idx))
        bfs.bfs_run_static(off, idx[:g.m], 0, out)
        assert np.array_equal(out.cpu().numpy(), ref.depth), shift
