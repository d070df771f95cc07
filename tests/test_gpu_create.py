"""Graph creation at the edges of its kernels: rows longer than a block's chunk
of entries (2048), runs of empty rows longer than one, degrees around the
histograms' shared part (512), one vertex. The transpose is checked through
pull levels and the reverse edge list, the summaries against the oracle."""
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


def rows(degrees, seed):
    """Directed graph whose vertex v has degrees[v] random out-edges."""
    deg = np.asarray(degrees, np.int64)
    off = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    idx = np.random.default_rng(seed).integers(0, len(deg), int(off[-1])).astype(np.int32)
    return gg.Graph(off, idx, f"rows{seed}")


CASES = {
    "one vertex": lambda: rows([0], 1),
    "one loop": lambda: rows([3], 2),
    "long rows": lambda: rows([5, 2047, 2048, 2049, 0, 9000, 1], 3),
    "empty runs": lambda: rows([0] * 2100 + [7] + [0] * 5000 + [2048] + [0] * 2047 + [1], 4),
    "degrees 511-513": lambda: rows([511, 512, 513, 0, 1] * 40, 5),
    "ends empty": lambda: rows([0, 0, 3, 0], 6),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_create_matches_the_oracle(name):
    g = CASES[name]()
    with bfs.Graph(g.off, g.idx, 0) as G:
        info = G.info()
        for key, got in (("out", info["deg_summary"] + [info["deg_sd256"]]),
                         ("in", info["in_deg_summary"] + [info["in_deg_sd256"]]),
                         ("total", info["tot_deg_summary"] + [info["tot_deg_sd256"]])):
            out = np.diff(g.off.astype(np.int64))
            into = np.bincount(g.idx, minlength=g.n).astype(np.int64)
            d = np.sort({"out": out, "in": into, "total": out + into}[key])
            want = [int(d[k * (g.n - 1) // 4]) for k in range(5)]
            s1, s2 = int(d.sum()), int((d * d).sum())
            var = 65536 * (g.n * s2 - s1 * s1)
            r = int(np.sqrt(float(var)))
            while r * r > var:
                r -= 1
            while (r + 1) * (r + 1) <= var:
                r += 1
            assert got == want + [r // g.n], key
        d = torch.empty(g.n, dtype=torch.int32, device="cuda")
        for root in sorted({0, g.n // 2, g.n - 1}):
            ref = oracle.bfs(g.off, g.idx, root)
            for variant in (bfs.VARIANT_TREE, bfs.VARIANTS.index("pull"), bfs.VARIANT_EDGE_LIST,
                            bfs.VARIANT_REVERSE_EDGE_LIST):
                bfs.bfs_run_ex(G.handle, root, d, forced_variant=variant)
                assert np.array_equal(d.cpu().numpy(), ref.depth), (root, variant)


def test_symmetric_total_degree_summary_is_twice_the_out_degree():
    g = gg.rmat(12, 16, seed=91)
    with bfs.Graph(g.off, g.idx) as G:
        info = G.info()
        assert info["in_deg_summary"] == info["deg_summary"] and info["in_deg_sd256"] == info["deg_sd256"]
        assert info["tot_deg_summary"] == [2 * x for x in info["deg_summary"]]
        d = 2 * np.diff(g.off.astype(np.int64))
        assert info["tot_deg_sd256"] == int(256 * np.std(d.astype(np.float64)))
