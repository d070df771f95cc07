"""Multi-source waves where a level's work is uneven: in-lists around the
lengths at which a lane, a warp and the whole grid look at them (64 entries, 128
more), hubs, roots whose traversals end early (small components), repeated
roots, and every number of roots around a wave. Each row equals the oracle's."""
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


def stars(sizes, chain=0):
    """Disjoint stars with the given numbers of leaves, and a chain of `chain` vertices."""
    src, dst, n = [], [], 0
    for k in sizes:
        src.append(np.full(k, n)), dst.append(np.arange(n + 1, n + 1 + k))
        n += k + 1
    if chain:
        src.append(np.arange(n, n + chain - 1)), dst.append(np.arange(n + 1, n + chain))
        n += chain
    return gg.from_edges(n, np.concatenate(src), np.concatenate(dst), symmetrize=True, name="stars")


def hubs(n=9000, k=40, extra=20000):
    """Directed: the first k vertices are named by most others; every in-degree a little different."""
    rng = np.random.default_rng(n)
    src, dst = [rng.integers(0, n, extra)], [rng.integers(0, n, extra)]
    for h in range(k):
        m = int(n * (0.9 - 0.02 * h))
        src.append(rng.permutation(n)[:m]), dst.append(np.full(m, h))
        src.append(np.full(5, h)), dst.append(rng.integers(0, n, 5))
    return gg.from_edges(n, np.concatenate(src), np.concatenate(dst), symmetrize=False, name="hubs")


CASES = {
    "list lengths": (lambda: stars([1, 63, 64, 65, 191, 192, 193, 320, 321, 1000], chain=5), True),
    "hubs": (hubs, False),
    "hubs and small components": (lambda: stars([5000, 3, 7000, 2, 128], chain=70), True),
    "rmat": (lambda: gg.rmat(13, 16, seed=911), True),
    "deep": (lambda: stars([4000], chain=400), True),
}


@pytest.mark.parametrize("name", sorted(CASES))
@pytest.mark.parametrize("push_mode,alpha,grid", [(0, 16, 0), (1, 16, 0), (0, 1, 3), (0, 1 << 20, 0), (0, 1 << 20, 5)])
def test_batch_rows_match_the_oracle(name, push_mode, alpha, grid):
    make, symmetric = CASES[name]
    g = make()
    with bfs.Graph(g.off, g.idx, bfs.BFS_SYMMETRIC if symmetric else 0) as G:
        bfs.bfs_batch_set_config(G.handle, push_mode, alpha, grid)
        for k in (1, 33, 64, 65):
            # spread over the ids (hubs first, small components and the chain last), one root twice
            roots = np.linspace(0, g.n - 1, k).astype(np.int32)
            if k > 2:
                roots[k // 2] = roots[0]
            out = torch.full((k, g.n), -7, dtype=torch.int32, device="cuda")
            edges = bfs.bfs_run_batch(G.handle, roots, out, edges=True)
            D, E = oracle.bfs_batch(g.off, g.idx, roots)
            assert np.array_equal(out.cpu().numpy(), D), k
            assert np.array_equal(edges, E), k
