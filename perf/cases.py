"""Performance cases: the calls a user of this library makes, over the sizes it is used at.

Every case builds seeded graphs on the GPU (R-MAT with a/b/c/d = .57/.19/.19/.05, permuted 2D grids with
dropped edges, Erdos-Renyi graphs; the families and sizes of the benchmark and the tests), hands the CSR to
the library and times public entry points. `listed()` holds the fixed cases, `draw()` more of the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1708_01159_gb300 as bfs

DEVICE = "cuda"
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19
GRID_DROP = 0.1


def listed():
    return [
        # one query on a small graph: launch and level latency are all of its time
        {"name": "rmat14 one root", "kind": "run", "family": "rmat", "n": 1 << 14, "degree": 16, "directed": False,
         "roots": 1, "variant": -1, "mode": 0, "host": False},
        # the plain method: every level by one fixed top-down push kernel, from several roots
        {"name": "rmat14 fixed push", "kind": "run", "family": "rmat", "n": 1 << 14, "degree": 16, "directed": False,
         "roots": 4, "variant": 0, "mode": 0, "host": False},
        # the headline: a large skewed graph, the tree choosing every level, several roots in turn
        {"name": "rmat22 switched", "kind": "run", "family": "rmat", "n": 1 << 22, "degree": 16, "directed": False,
         "roots": 4, "variant": -1, "mode": 0, "host": False},
        # directed graph with an odd vertex count: pull reads a transpose of its own
        {"name": "directed rmat odd", "kind": "run", "family": "rmat", "n": 1000003, "degree": 16, "directed": True,
         "roots": 2, "variant": -1, "mode": 0, "host": False},
        # high diameter: thousands of small levels, ids in random order
        {"name": "grid4096", "kind": "run", "family": "grid", "n": 4096, "degree": 4096, "directed": False,
         "roots": 1, "variant": -1, "mode": 0, "host": False},
        # the same family through the captured CUDA graph driver, odd side lengths
        {"name": "grid cuda graph", "kind": "run", "family": "grid", "n": 777, "degree": 1021, "directed": False,
         "roots": 1, "variant": -1, "mode": 2, "host": False},
        # end to end: the depths land in the caller's pinned host memory
        {"name": "er21 to host", "kind": "run", "family": "er", "n": 1 << 21, "degree": 16, "directed": False,
         "roots": 2, "variant": -1, "mode": 0, "host": True},
        # 64 roots of one large uniform graph in one launch
        {"name": "er22 batch 64", "kind": "batch", "family": "er", "n": 1 << 22, "degree": 8, "graphs": 1, "roots": 64,
         "streams": 1},
        # many uneven graphs, a batch of roots each, spread over streams
        {"name": "uneven rmat batches", "kind": "batch", "family": "rmat", "n": 1 << 18, "degree": 16, "graphs": 10,
         "roots": 64, "streams": 5},
        # a burst of mixed queries to a server that holds four graphs of different shapes
        {"name": "serve burst", "kind": "serve", "n": 1 << 18, "degree": 16, "queries": 128},
        # a graph that is analysed once: create (transpose, statistics), one traversal, destroy
        {"name": "create directed", "kind": "create", "family": "rmat", "n": 1 << 20, "degree": 16, "directed": True},
        # the entry point for callers that cannot allocate: CSR and output are theirs
        {"name": "allocation-free", "kind": "static", "family": "rmat", "n": 1 << 18, "degree": 16, "directed": False},
    ]


def _log_int(rng, lo, hi):
    """An integer spread evenly over the logarithm of [lo, hi]; a power of two now and then, any other value else."""
    x = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    if rng.random() < 0.25:
        x = 2.0 ** round(math.log2(x))
    return int(min(hi, max(lo, round(x))))


def _draw_graph(rng, lo, hi, families=("rmat", "er", "grid"), grid_hi=2048):
    family = rng.choice(families)
    if family == "grid":
        return {"family": "grid", "n": _log_int(rng, 32, grid_hi), "degree": _log_int(rng, 32, grid_hi),
                "directed": False}
    n = _log_int(rng, lo, hi)
    degree = rng.choice((4, 8, 16, 24, 32)) if n <= hi // 2 else rng.choice((4, 8, 16))
    return {"family": family, "n": n, "degree": degree, "directed": family == "rmat" and rng.random() < 0.4}


def draw(rng):
    kind = rng.choice(("run", "run", "run", "fixed", "graph", "host", "batch", "batch", "serve", "create", "static"))
    if kind == "run":
        return dict(_draw_graph(rng, 1 << 12, 1 << 22, grid_hi=4096), kind="run", roots=rng.randint(1, 4), variant=-1,
                    mode=0, host=False)
    if kind == "fixed":
        return dict(_draw_graph(rng, 1 << 12, 1 << 16, ("rmat", "er")), kind="run", roots=rng.randint(1, 4),
                    variant=rng.randrange(bfs.NUM_VARIANTS - 1), mode=0, host=False)
    if kind == "graph":
        return dict(_draw_graph(rng, 1 << 12, 1 << 20, grid_hi=1021), kind="run", roots=1, variant=-1, mode=2,
                    host=False)
    if kind == "host":
        return dict(_draw_graph(rng, 1 << 12, 1 << 22, ("rmat", "er")), kind="run", roots=rng.randint(1, 3),
                    variant=-1, mode=0, host=True)
    if kind == "batch":
        if rng.random() < 0.5:
            return {"kind": "batch", "family": rng.choice(("rmat", "er")), "n": _log_int(rng, 1 << 12, 1 << 22),
                    "degree": 8, "graphs": 1, "roots": rng.randint(1, 64), "streams": 1}
        return {"kind": "batch", "family": rng.choice(("rmat", "er")), "n": _log_int(rng, 1 << 14, 1 << 18),
                "degree": rng.choice((8, 16)), "graphs": rng.randint(2, 12), "roots": rng.choice((16, 33, 64, 100)),
                "streams": rng.randint(1, 8)}
    if kind == "serve":
        return {"kind": "serve", "n": _log_int(rng, 1 << 13, 1 << 18), "degree": rng.choice((8, 16)),
                "queries": _log_int(rng, 8, 128)}
    if kind == "create":
        return dict(_draw_graph(rng, 1 << 12, 1 << 20, ("rmat", "er", "grid"), 512), kind="create")
    return dict(_draw_graph(rng, 1 << 12, 1 << 20, ("rmat", "er", "grid"), 400), kind="static")


# ------------------------------------------------------------------------------------------------- the inputs

def _csr(n, u, v, symmetrise):
    """CSR (int32 offsets and indices) of the pairs u -> v: self-loops and duplicates removed, rows ascending."""
    keep = u != v
    u, v = u[keep], v[keep]
    keys = u * n + v
    if symmetrise:
        keys = torch.cat((keys, v * n + u))
    del u, v, keep
    keys = torch.unique(keys)
    off = torch.searchsorted(keys, torch.arange(n + 1, device=DEVICE, dtype=torch.int64) * n).to(torch.int32)
    return off, (keys % n).to(torch.int32)


def _rmat(n, degree, directed, gen):
    """R-MAT over the next power of two, restricted to the first n ids; degree * n generated edges in all."""
    scale = max(1, (n - 1).bit_length())
    edges = degree * n
    u = torch.zeros(edges, dtype=torch.int64, device=DEVICE)
    v = torch.zeros(edges, dtype=torch.int64, device=DEVICE)
    for _ in range(scale):
        r = torch.rand(edges, generator=gen, device=DEVICE)
        low = r >= RMAT_A + RMAT_B
        u.mul_(2).add_(low)
        v.mul_(2).add_(((r >= RMAT_A) & ~low) | (r >= RMAT_A + RMAT_B + RMAT_C))
    if n != 1 << scale:
        keep = (u < n) & (v < n)
        u, v = u[keep], v[keep]
    return _csr(n, u, v, not directed)


def _er(n, degree, gen):
    """Uniform random graph with n * degree / 2 undirected edges."""
    pairs = torch.randint(0, n, (2, n * degree // 2), generator=gen, device=DEVICE)
    return _csr(n, pairs[0], pairs[1], True)


def _grid(rows, cols, gen):
    """rows x cols lattice, a tenth of the undirected edges dropped, ids permuted."""
    n = rows * cols
    ids = torch.randperm(n, generator=gen, device=DEVICE).view(rows, cols)
    u = torch.cat((ids[:, :-1].reshape(-1), ids[:-1].reshape(-1)))
    v = torch.cat((ids[:, 1:].reshape(-1), ids[1:].reshape(-1)))
    keep = torch.rand(u.numel(), generator=gen, device=DEVICE) >= GRID_DROP
    return _csr(n, u[keep], v[keep], True)


def _graph(c, gen):
    if c["family"] == "grid":
        return _grid(c["n"], c["degree"], gen)
    if c["family"] == "er":
        return _er(c["n"], c["degree"], gen)
    return _rmat(c["n"], c["degree"], c.get("directed", False), gen)


def _roots(off, count, gen):
    """Uniform over the vertices with out-edges."""
    live = torch.nonzero(off[1:] > off[:-1]).view(-1)
    pick = torch.randint(0, live.numel(), (count,), generator=gen, device=DEVICE)
    return [int(x) for x in live[pick].tolist()]


def _flags(c):
    return 0 if c.get("directed") else bfs.BFS_SYMMETRIC


def _members(c):
    """The graphs of a batch or a server, as single-graph cases: sizes fall geometrically from n."""
    if c["kind"] == "serve":
        side = max(24, int(math.sqrt(c["n"]) * 0.75))
        return [{"family": "rmat", "n": c["n"], "degree": c["degree"]},
                {"family": "rmat", "n": max(64, c["n"] // 5), "degree": c["degree"]},
                {"family": "er", "n": max(64, c["n"] // 2 + 1), "degree": c["degree"]},
                {"family": "grid", "n": side, "degree": side + 3}]
    if c["graphs"] == 1:
        return [{"family": c["family"], "n": c["n"], "degree": c["degree"]}]
    got = []
    for i in range(c["graphs"]):
        n = int(c["n"] / 64.0 ** (i / (c["graphs"] - 1)))
        got.append({"family": c["family"], "n": max(64, n - i), "degree": c["degree"] * (1, 2)[i % 2]})
    return got


def _inputs(c, seed):
    """Every graph's CSR and the roots, from the seed alone."""
    gen = torch.Generator(device=DEVICE)
    gen.manual_seed(seed)
    if c["kind"] in ("batch", "serve"):
        graphs = [_graph(m, gen) for m in _members(c)]
        if c["kind"] == "batch":
            return graphs, [_roots(off, c["roots"], gen) for off, _ in graphs]
        which = [i % len(graphs) for i in torch.randperm(c["queries"], generator=gen, device=DEVICE).tolist()]
        pools = [_roots(off, c["queries"], gen) for off, _ in graphs]
        return graphs, [(g, pools[g][i]) for i, g in enumerate(which)]
    off, idx = _graph(c, gen)
    return [(off, idx)], [_roots(off, c.get("roots", 1), gen)]


# ------------------------------------------------------------------------------------------------ the programs

class State:
    """What a program keeps between calls; gives its library objects back when it goes."""

    def __init__(self, c):
        self.case = c
        self.graphs = []
        self.server = None

    def __del__(self):
        try:
            if self.server is not None:
                bfs.bfs_serve_destroy(self.server)
                self.server = None
            for g in self.graphs:
                g.close()
        except Exception:  # interpreter shutdown
            pass


def prepare(case, seed):
    s = State(case)
    csr, roots = _inputs(case, seed)
    kind = case["kind"]
    if kind in ("create", "static"):
        s.off, s.idx = csr[0]
        s.root = roots[0][0]
        s.out = torch.empty(s.off.numel() - 1, dtype=torch.int32, device=DEVICE)
        return s
    torch.cuda.synchronize()
    s.graphs = [bfs.Graph(off, idx, _flags(case)) for off, idx in csr]
    if kind == "run":
        n = s.graphs[0].n
        s.roots = roots[0]
        s.out = torch.empty((case["roots"], n), dtype=torch.int32, device="cpu" if case["host"] else DEVICE,
                            pin_memory=case["host"])
        s.rows = list(s.out)
    elif kind == "batch":
        s.roots = [np.array(r, dtype=np.int32) for r in roots]
        s.out = [torch.empty((case["roots"], g.n), dtype=torch.int32, device=DEVICE) for g in s.graphs]
        s.streams = [torch.cuda.Stream() for _ in range(case["streams"])] if case["streams"] > 1 else []
    else:
        s.server = bfs.bfs_serve_create(max_inflight=64, num_streams=64, merge_batch=64)
        s.ids = [bfs.bfs_serve_add_graph(s.server, g.handle) for g in s.graphs]
        count = [max(1, sum(1 for g, _ in roots if g == i)) for i in range(len(s.graphs))]
        s.out = [torch.full((k, g.n), -1, dtype=torch.int32, device=DEVICE) for k, g in zip(count, s.graphs)]
        rows = [0] * len(s.graphs)
        s.queries = []
        for g, r in roots:
            s.queries.append((s.ids[g], r, s.out[g][rows[g]]))
            rows[g] += 1
        torch.cuda.synchronize()  # the server writes the rows on streams of its own
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "run":
        g = s.graphs[0].handle
        variant, mode = s.case["variant"], s.case["mode"]
        for root, row in zip(s.roots, s.rows):
            if variant < 0 and mode == 0 and not s.case["host"]:
                bfs.bfs_run(g, root, row)
            else:
                bfs.bfs_run_ex(g, root, row, forced_variant=variant, mode=mode)
        return s.out
    if kind == "batch":
        if not s.streams:
            for g, roots, out in zip(s.graphs, s.roots, s.out):
                bfs.bfs_run_batch(g.handle, roots, out)
            return s.out
        main = torch.cuda.current_stream()
        for st in s.streams:
            st.wait_stream(main)
        for i, (g, roots, out) in enumerate(zip(s.graphs, s.roots, s.out)):
            bfs.bfs_run_batch(g.handle, roots, out, stream=s.streams[i % len(s.streams)])
        for st in s.streams:
            main.wait_stream(st)
        return s.out
    if kind == "serve":
        tickets = [bfs.bfs_serve_submit(s.server, gid, root, row) for gid, root, row in s.queries]
        status = [bfs.bfs_serve_wait(s.server, t) for t in tickets]
        return {"depth": s.out, "status": np.array(status, dtype=np.int32)}
    if kind == "create":
        with bfs.Graph(s.off, s.idx, _flags(s.case)) as g:
            info = g.info()
            bfs.bfs_run(g.handle, s.root, s.out)
        return {"depth": s.out, "degrees": np.array(info["deg_summary"] + info["in_deg_summary"] +
                                                    info["tot_deg_summary"], dtype=np.int64)}
    bfs.bfs_run_static(s.off, s.idx, s.root, s.out)
    return s.out


# ------------------------------------------------------------------------------------- work and exact results

def _sizes(m, directed):
    """(vertices, directed edges) a graph case has, to within a few per cent."""
    if m["family"] == "grid":
        n = m["n"] * m["degree"]
        return n, int(2 * (1 - GRID_DROP) * (2 * n - m["n"] - m["degree"]))
    if m["family"] == "er":
        return m["n"], m["n"] * m["degree"]
    kept = min(0.98, 0.81 + 0.018 * (math.log2(m["n"]) - 14))  # duplicates thin out with size
    return m["n"], int(m["n"] * m["degree"] * kept * (1 if directed else 2))


def work(case):
    """Every CSR read once per call and every depth written once; a comparison per edge."""
    if case["kind"] == "batch":
        parts = [(_sizes(m, False), case["roots"], 1) for m in _members(case)]
    elif case["kind"] == "serve":
        k = case["queries"] / 4.0
        parts = [(_sizes(m, False), k, k) for m in _members(case)]
    else:
        k = case.get("roots", 1)
        parts = [(_sizes(case, case.get("directed", False)), k, k)]
    total = sum(4.0 * n * rows + reads * 4.0 * (n + 1 + m) for (n, m), rows, reads in parts)
    edges = sum(rows * float(m) for (n, m), rows, _ in parts)
    return {"bytes": total, "flops": edges}


def _depths(off, idx, root):
    """Level by level with whole-frontier tensor operations, int64."""
    n = off.numel() - 1
    off = off.to(torch.int64)
    depth = torch.full((n,), -1, dtype=torch.int64, device=DEVICE)
    front = torch.tensor([root], device=DEVICE)
    depth[front] = 0
    level = 0
    while front.numel():
        beg = off[front]
        deg = off[front + 1] - beg
        ends = torch.cumsum(deg, 0)
        total = int(ends[-1])
        first = torch.repeat_interleave(beg - (ends - deg), deg, output_size=total)
        near = idx[first + torch.arange(total, device=DEVICE)].to(torch.int64)
        near = near[depth[near] < 0]
        level += 1
        depth[near] = level
        front = torch.unique(near)
    return depth


def _degrees(off, idx):
    """The five-number summaries of out-, in- and total degree: sorted[floor(k (n - 1) / 4)]."""
    n = off.numel() - 1
    out = (off[1:] - off[:-1]).to(torch.int64)
    into = torch.bincount(idx.to(torch.int64), minlength=n)
    at = torch.tensor([k * (n - 1) // 4 for k in range(5)], device=DEVICE)
    return torch.cat([torch.sort(d).values[at] for d in (out, into, out + into)])


def exact(case, seed):
    csr, roots = _inputs(case, seed)
    if case["kind"] == "serve":
        rows = [[] for _ in csr]
        for g, r in roots:
            rows[g].append(_depths(*csr[g], r))
        full = [torch.stack(r) if r else torch.full((1, csr[g][0].numel() - 1), -1, dtype=torch.int64, device=DEVICE)
                for g, r in enumerate(rows)]
        return {"depth": full, "status": np.zeros(case["queries"], dtype=np.int64)}
    if case["kind"] == "batch":
        return [torch.stack([_depths(off, idx, r) for r in rs]) for (off, idx), rs in zip(csr, roots)]
    off, idx = csr[0]
    depth = torch.stack([_depths(off, idx, r) for r in roots[0]])
    if case["kind"] == "create":
        return {"depth": depth[0], "degrees": _degrees(off, idx)}
    return depth[0] if case["kind"] == "static" else depth
