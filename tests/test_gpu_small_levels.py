"""Runs of small levels on the leader cluster (graphs whose out-degrees are at
most 8): depths and per-level counts equal the oracle's where the frontier
outgrows the leader and comes back, where a block's lists overflow, at both
record widths and the edges of both, and on every cluster size a grid allows."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1708_01159_gb300 as bfs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def built():
    bfs.build()
    bfs.bfs_load_tree(None)
    yield


def tree_edges(arity, levels, first=0):
    """Parent -> child pairs of a complete tree whose root is vertex `first`."""
    n = sum(arity ** k for k in range(levels))
    child = np.arange(1, n, dtype=np.int64)
    return first + (child - 1) // arity, first + child, n


def dumbbell():
    """Chain, binary tree, chain from one of its leaves, second tree, chain:
    small and large levels in turn."""
    src, dst, n = [], [], 0
    for _ in range(2):
        s = np.arange(n, n + 40)
        src.append(s), dst.append(s + 1)
        a, b, k = tree_edges(2, 16, n + 40)
        src.append(a), dst.append(b)
        n += 40 + k
        src.append(np.array([n - 1])), dst.append(np.array([n]))
    s = np.arange(n, n + 30)
    src.append(s), dst.append(s + 1)
    return gg.from_edges(n + 31, np.concatenate(src), np.concatenate(dst), symmetrize=True, name="dumbbell"), True


def regular_directed(degree, n=6000):
    """Out-degree exactly `degree` for most vertices, self-loops and duplicates kept."""
    rng = np.random.default_rng(degree)
    deg = np.where(rng.random(n) < 0.9, degree, rng.integers(0, degree + 1, n))
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    return gg.Graph(off, rng.integers(0, n, int(off[-1])).astype(np.int32), f"regular{degree}"), False


def arity8():
    a, b, n = tree_edges(8, 6)
    return gg.from_edges(n, a, b, symmetrize=False, name="arity8"), False


CASES = {
    "single": lambda: (gg.Graph(np.array([0, 0], np.int32), np.zeros(0, np.int32), "single"), True),
    "loop": lambda: (gg.Graph(np.array([0, 1], np.int32), np.zeros(1, np.int32), "loop"), True),
    "path": lambda: (gg.from_edges(3000, np.arange(2999), np.arange(1, 3000)), True),
    "grid": lambda: (gg.grid(300, 211, 0.1, seed=901), True),
    "wide": lambda: (gg.grid(1500, 1500, 0.02, seed=902), True),
    "dumbbell": dumbbell,
    "arity8": arity8,
    "out4": lambda: regular_directed(4),
    "out5": lambda: regular_directed(5),
    "out8": lambda: regular_directed(8),
    "out9": lambda: regular_directed(9),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_small_levels_match_the_oracle(name):
    g, symmetric = CASES[name]()
    roots = sorted({0, g.n // 2, g.n - 1})
    with bfs.Graph(g.off, g.idx, bfs.BFS_SYMMETRIC if symmetric else 0) as G:
        d = torch.empty(g.n, dtype=torch.int32, device="cuda")
        for root in roots:
            ref = oracle.bfs(g.off, g.idx, root)
            for mode, blocks in ((bfs.MODE_PERSISTENT, 0), (bfs.MODE_PERSISTENT, 1), (bfs.MODE_PERSISTENT, 8),
                                 (bfs.MODE_PERSISTENT, 12), (bfs.MODE_PERSISTENT, 16), (bfs.MODE_GRAPH, 0)):
                d.fill_(-7)
                st = bfs.bfs_run_ex(G.handle, root, d, mode=mode, grid_blocks=blocks, stats=True,
                                    log_capacity=ref.num_levels + 1)
                assert np.array_equal(d.cpu().numpy(), ref.depth), (root, mode, blocks)
                assert st["levels"] == ref.num_levels and st["edges_reached"] == ref.edges_reached
                assert st["vertices_reached"] == int((ref.depth >= 0).sum())
                assert np.array_equal(st["frontier"], ref.level_count), (root, mode, blocks)
                assert np.array_equal(st["frontier_edges"], ref.level_edges), (root, mode, blocks)
