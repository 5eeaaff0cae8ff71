"""Timed cases of the library: one pass of each public entry point that a Graph500 program
or a serving program calls, on seeded synthetic graphs.

A case is a dict of plain values.  Its "kind" names the call:

  search     bfs() from each of `roots` start vertices, one after another (kernel 2)
  validated  the benchmark's loop over one root: bfs(), then bfs_validate() of the tree
             against the graph and the input tuples
  mesh       bfs() on a caller's own CSR: a rectangular grid with some edges missing, many
             levels of few vertices
  batch      bfs_batch(): `roots` searches of one graph in one launch
  graphs     bfs_multi_graph(): `roots` searches on each of several graphs in one launch
  build      graph_build_csr(): kernel 1 from int64 tuples
  wbuild     graph_build_csr_weighted(): kernel 1 with the weight row
  sssp       sssp() from `roots` start vertices (kernel 3)
  serve      a burst of queries to a Server over resident graphs, each result fetched

Graphs are Kronecker graphs (initiator 0.57, 0.19, 0.19, 0.05, vertices renumbered at
random) of 2^scale vertices and `tuples` tuples, or, with skew false, uniform random ones.

Outputs.  Levels, CSR arrays, weights, distances and canonical parents are unique, so they
have to stay what they are.  Outside canonical mode any valid tree is a right answer and the
claiming order decides which one comes out, so the parents of those searches are not
compared value by value: "validated" returns the verdict on the tree instead, and the
canonical searches return the parents themselves.
"""
import math

import numpy as np
import torch

import paper_2012_13548_gb300 as gb


def listed():
    return [
        # One query on a small graph in canonical mode: launch and barrier latency.
        dict(name="search_s10_canonical", kind="search", scale=10, tuples=16 << 10, skew=True, roots=1,
             canonical=True),
        # Plain searches of the mid-size benchmark graph: about 0.1 ms each.
        dict(name="search_s20", kind="search", scale=20, tuples=16 << 20, skew=True, roots=8, canonical=False),
        # The headline: single-source searches of the SCALE 26 graph.
        dict(name="search_s26", kind="search", scale=26, tuples=16 << 26, skew=True, roots=4, canonical=False),
        # A caller's own graph, nothing about it a power of two: a mesh with about 1,500 levels.
        dict(name="mesh_997x601", kind="mesh", width=997, height=601, canonical=False),
        # One root of the benchmark as it is reported: the search and the validation of its tree.
        dict(name="validated_s22", kind="validated", scale=22, tuples=16 << 22, skew=True, canonical=False),
        # 64 roots in one launch on the SCALE 22 graph.
        dict(name="batch_s22_k64", kind="batch", scale=22, tuples=16 << 22, skew=True, roots=64, canonical=False),
        # 32 graphs of SCALE 12 to 18, 8 roots each, in one launch.
        dict(name="graphs32_s12_18", kind="graphs", graphs=32, lo=12, hi=18, roots=8, canonical=False),
        # Kernel 1 at full size: 1.07 billion tuples.
        dict(name="build_s26", kind="build", scale=26, tuples=16 << 26, skew=True),
        # Kernel 1 of a small graph with an odd number of tuples: launches, allocations and waits count.
        dict(name="build_s16_odd", kind="build", scale=16, tuples=(16 << 16) - 12345, skew=True),
        # Kernel 1 with the weight row, for kernel 3.
        dict(name="wbuild_s22", kind="wbuild", scale=22, tuples=16 << 22, skew=True),
        # Shortest paths on the SCALE 22 weighted graph, bucket width as the tuning table has it.
        dict(name="sssp_s22", kind="sssp", scale=22, tuples=16 << 22, skew=True, roots=1, delta=0.05,
             canonical=False),
        # Six resident graphs, SCALE 14 to 24; 48 queries arrive at once, the graph chosen uniformly.
        dict(name="serve_burst48", kind="serve", queries=48, lo=14, hi=24, step=2),
    ]


def draw(rng):
    kind = rng.choice(["search", "search", "mesh", "validated", "batch", "graphs", "build", "build", "wbuild",
                       "sssp", "serve"])

    def kron(lo, hi):
        # sizes uniform in their logarithm; any number of tuples, not only multiples of 2^scale
        scale = rng.randint(lo, hi)
        return dict(scale=scale, tuples=int(math.exp2(scale + rng.uniform(2.5, 4.5))) | 1,
                    skew=rng.random() < 0.8)

    if kind == "search":
        return dict(kind=kind, **kron(10, 25), roots=rng.randint(1, 8), canonical=rng.random() < 0.3)
    if kind == "mesh":
        return dict(kind=kind, width=rng.randint(17, 1000), height=rng.randint(17, 700),
                    canonical=rng.random() < 0.3)
    if kind == "validated":
        return dict(kind=kind, **kron(12, 23), canonical=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, **kron(12, 22), roots=rng.randint(2, 64), canonical=rng.random() < 0.3)
    if kind == "graphs":
        lo = rng.randint(8, 15)
        return dict(kind=kind, graphs=rng.randint(2, 32), lo=lo, hi=rng.randint(lo, 18), roots=rng.randint(1, 8),
                    canonical=rng.random() < 0.3)
    if kind in ("build", "wbuild"):
        return dict(kind=kind, **(kron(10, 24) if kind == "build" else kron(10, 21)))
    if kind == "sssp":
        return dict(kind=kind, **kron(10, 21), roots=rng.randint(1, 3), delta=round(rng.uniform(0.03, 0.2), 3),
                    canonical=rng.random() < 0.3)
    lo = rng.randint(12, 16)
    return dict(kind="serve", queries=rng.randint(4, 64), lo=lo, hi=rng.randint(lo, 21), step=rng.randint(1, 3))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _tuples(scale, tuples, skew, gen):
    """int64 [2, tuples]: each tuple draws a quadrant per bit, then the vertices are renumbered
    at random.  The draws depend on the case alone, so that every seed's graph has the same
    number of edges (outputs keep their shapes); the numbering comes from the seed."""
    a, b, c = (0.57, 0.19, 0.19) if skew else (0.25, 0.25, 0.25)
    e = torch.zeros((2, tuples), dtype=torch.int64, device="cuda")
    draws = _generator(scale)
    for _ in range(scale):
        r = torch.rand(tuples, generator=draws, device="cuda")
        row = r >= a + b
        e[0].mul_(2).add_(row)
        col = (r >= a).logical_and_(~row).logical_or_(r >= a + b + c)
        e[1].mul_(2).add_(col)
        del r, row, col
    perm = torch.randperm(1 << scale, generator=gen, device="cuda")
    for i in (0, 1):
        torch.index_select(perm, 0, e[i].clone(), out=e[i])
    return e


def _weights(tuples, gen):
    """float32 [tuples], uniform on the multiples of 2^-24 in (0, 1]."""
    return (torch.randint(0, 1 << 24, (tuples,), generator=gen, device="cuda") + 1).to(torch.float32) * 2.0 ** -24


def _roots(graph, k, gen):
    """k start vertices drawn uniformly among those with an edge."""
    off, _ = graph.csr()
    cand = torch.nonzero(off[1:] > off[:-1]).flatten()
    pick = torch.randint(0, cand.numel(), (k,), generator=gen, device="cuda")
    return [int(r) for r in cand[pick].tolist()]


def _mesh(width, height, gen):
    """CSR (off int64 [n+1], col int32 [nnz]) of a width x height grid, one edge in 50 missing."""
    n = width * height
    v = torch.arange(n, device="cuda")
    right = v[(v % width) != width - 1]
    down = v[v < n - width]
    u = torch.cat([right, down])
    w = torch.cat([right + 1, down + width])
    keep = torch.rand(u.numel(), generator=gen, device="cuda") >= 0.02
    u, w = u[keep], w[keep]
    key = torch.sort(torch.cat([u * n + w, w * n + u])).values
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.bincount(key // n, minlength=n), 0)
    return off, (key % n).to(torch.int32)


def _uniform(lo, hi, count):
    """`count` whole numbers from lo..hi, the same for every seed of a case."""
    return torch.randint(lo, hi + 1, (count,), generator=_generator(count), device="cuda").tolist()


def prepare(case, seed):
    gen = _generator(seed)
    kind = case["kind"]
    gb.bfs_set_options(canonical_parents=1 if case.get("canonical") else 0)
    st = dict(kind=kind, canonical=bool(case.get("canonical")))
    if kind == "mesh":
        off, col = _mesh(case["width"], case["height"], gen)
        st["graph"] = gb.graph_from_csr(off, col)
        st["roots"] = _roots(st["graph"], 1, gen)
    elif kind == "graphs":
        scales = _uniform(case["lo"], case["hi"], case["graphs"])
        scales[0], scales[-1] = case["hi"], case["lo"]  # both ends of the range are there
        st["graphs"] = [gb.graph_build_csr(_tuples(s, 16 << s, True, gen), s) for s in scales]
        st["roots"] = [_roots(g, case["roots"], gen) for g in st["graphs"]]
    elif kind == "serve":
        scales = range(case["lo"], case["hi"] + 1, case["step"])
        graphs = [gb.graph_build_csr(_tuples(s, 16 << s, True, gen), s) for s in scales]
        which = _uniform(0, len(graphs) - 1, case["queries"])
        st["queries"] = [(w, _roots(graphs[w], 1, gen)[0]) for w in which]
        st["server"] = gb.Server(graphs, 64 << 30)
    else:
        e = _tuples(case["scale"], case["tuples"], case["skew"], gen)
        st["scale"] = case["scale"]
        if kind in ("build", "wbuild"):
            st["edges"] = e
            if kind == "wbuild":
                st["weights"] = _weights(case["tuples"], gen)
        elif kind == "sssp":
            st["graph"] = gb.graph_build_csr_weighted(e, _weights(case["tuples"], gen), case["scale"])
            st["roots"] = _roots(st["graph"], case["roots"], gen)
            st["delta"] = case["delta"]
        else:
            st["graph"] = gb.graph_build_csr(e, case["scale"])
            st["roots"] = _roots(st["graph"], case.get("roots", 1), gen)
            if kind == "validated":
                st["edges"] = e
    return st


def run(state):
    kind = state["kind"]
    if kind in ("search", "mesh"):
        got = [gb.bfs(state["graph"], r) for r in state["roots"]]
        if state["canonical"]:
            return [list(x) for x in got]
        return [level for _, level in got]
    if kind == "validated":
        root = state["roots"][0]
        parent, level = gb.bfs(state["graph"], root)
        verdict = gb.bfs_validate(state["graph"], root, parent, level, state["edges"])
        return dict(level=level, **verdict)
    if kind == "batch":
        parents, levels = gb.bfs_batch(state["graph"], state["roots"])
        return [parents, levels] if state["canonical"] else [levels]
    if kind == "graphs":
        parents, levels = gb.bfs_multi_graph(state["graphs"], state["roots"])
        return parents + levels if state["canonical"] else levels
    if kind == "build":
        return list(gb.graph_build_csr(state["edges"], state["scale"]).csr())
    if kind == "wbuild":
        g = gb.graph_build_csr_weighted(state["edges"], state["weights"], state["scale"])
        return [*g.csr(), g.weights()]
    if kind == "sssp":
        return [list(gb.sssp(state["graph"], r, state["delta"])) for r in state["roots"]]
    srv = state["server"]
    tickets = [(srv.submit(g, r), g) for g, r in state["queries"]]
    levels = [srv.result(t, g)[1] for t, g in tickets]
    torch.cuda.current_stream().synchronize()  # the copies are made before the server reuses its buffers
    for t, _ in tickets:
        srv.release(t)
    return levels


def work(case):
    """Bytes that a pass cannot do without: its inputs once, its outputs once.  A search
    needs the offsets and one column of every vertex; a shortest-path search and a
    validation need every entry.  nnz is taken as two entries per tuple."""
    kind = case["kind"]
    if kind == "mesh":
        n = case["width"] * case["height"]
        return dict(bytes=n * (8 + 4 * 4 + 8), flops=0)
    if kind == "graphs":
        # SCALE uniform in lo..hi: every size as often as the others
        sizes = [1 << s for s in range(case["lo"], case["hi"] + 1)]
        n = case["graphs"] * sum(sizes) / len(sizes)
        return dict(bytes=n * (8 + 32 * 4 + 8 * case["roots"]), flops=0)
    if kind == "serve":
        sizes = [1 << s for s in range(case["lo"], case["hi"] + 1, case["step"])]
        return dict(bytes=case["queries"] * sum(sizes) / len(sizes) * (8 + 4 + 8), flops=0)
    n, m = 1 << case["scale"], case["tuples"]
    nnz = 2 * m
    b = {
        "search": lambda: case["roots"] * n * (8 + 4 + 8),
        "validated": lambda: n * (8 + 4 + 8) + 8 * n + 4 * nnz + 8 * n + 8 * m,
        "batch": lambda: 8 * n + 4 * nnz + 8 * n * case["roots"],
        "build": lambda: 16 * m + 8 * n + 4 * nnz,
        "wbuild": lambda: 20 * m + 8 * n + 16 * nnz,
        "sssp": lambda: case["roots"] * (8 * n + 8 * nnz + 12 * n),
    }[kind]()
    return dict(bytes=b, flops=0)


def tolerance(case):
    if case["kind"] == "sssp":
        # Distances are exact sums of multiples of 2^-24: the same to the last bit.  Two tight
        # parents of one vertex are rare; outside canonical mode either may be recorded.
        return dict(rel=0.0, max=0.0, differ=0.0 if case["canonical"] else 2e-5)
    return "exact"


def exact(case, seed):
    """Distances by repeated relaxation of every tuple in 64 bits (kernel 3 only: all other
    outputs are whole numbers)."""
    if case["kind"] != "sssp":
        return None
    gen = _generator(seed)
    n = 1 << case["scale"]
    e = _tuples(case["scale"], case["tuples"], case["skew"], gen)
    w = _weights(case["tuples"], gen).to(torch.float64)
    loop = e[0] == e[1]
    deg = torch.bincount(e[0][~loop], minlength=n) + torch.bincount(e[1][~loop], minlength=n)
    cand = torch.nonzero(deg > 0).flatten()
    pick = torch.randint(0, cand.numel(), (case["roots"],), generator=gen, device="cuda")
    out = []
    for r in cand[pick].tolist():
        dist = torch.full((n,), np.inf, dtype=torch.float64, device="cuda")
        dist[int(r)] = 0.0
        while True:
            before = dist.clone()
            dist.scatter_reduce_(0, e[1], before[e[0]] + w, "amin")
            dist.scatter_reduce_(0, e[0], before[e[1]] + w, "amin")
            if torch.equal(before, dist):
                break
        out.append([dist, None])
    return out
