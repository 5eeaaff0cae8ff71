"""Settle steps of the shortest-path search from either end, against the oracle.

A bucket's heavy edges are read from the settled rows or from the rows of what is
still unsettled, whichever is less; rows below and above 64 and 1024 entries, buckets
from one unit of the weights to the whole search, equal weights (ties at every
bound), unreachable parts.  How often the second end is taken follows from the final
distances; the searches have to take it as often, and the cases hold both.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2012_13548_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


def graph(kind, rng):
    if kind == "hubs":        # a few rows of thousands, the rest short
        scale = 13
        n, m = 1 << scale, 60000
        u = np.where(rng.random(m) < 0.5, rng.integers(0, 5, m) * 1000, rng.integers(0, n, m))
        v = rng.integers(0, n, m)
    elif kind == "middle":    # rows of 40 to 100 entries
        scale = 10
        n, m = 1 << scale, 35000
        u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    elif kind == "path":      # one long path beside a star that it does not touch
        scale = 11
        n = 1 << scale
        u = np.concatenate([np.arange(500), np.full(1400, 600)])
        v = np.concatenate([np.arange(1, 501), rng.integers(601, n, 1400)])
    else:                     # two dense parts joined by one edge
        scale = 12
        n, m = 1 << scale, 40000
        u, v = rng.integers(0, n // 2, m), rng.integers(0, n // 2, m)
        u = np.concatenate([u, u + n // 2, [0]])
        v = np.concatenate([v, v + n // 2, [n // 2]])
    return scale, np.stack([u, v]).astype(np.int64)


def expected_pulls(off, dist, delta):
    """The settle steps from the unsettled end: those where the degrees of the vertices
    that the bucket settles exceed a quarter of what is left (the unsettled degrees and
    the length of the list of vertices to look at: all at first, then those that
    the last such step left)."""
    units = dist * 2.0 ** 24                       # whole numbers
    width = max(1.0, np.floor(delta * 2.0 ** 24 + 0.5))
    deg = np.diff(off)
    n, nnz, settled, listed, pulls, before = len(deg), int(off[-1]), 0.0, float(len(deg)), 0, 0
    top = width
    while True:
        below = units < top
        settled = int(deg[below].sum())
        if settled - before > 0.25 * (nnz - settled + listed):
            pulls += 1
            listed = float(np.count_nonzero(~below & (deg > 0)))
        before = settled
        left = units[~below]
        least = left.min() if left.size else np.inf
        if not np.isfinite(least):
            return pulls
        top = (least // width + 1) * width


@pytest.mark.parametrize("weights", ["any", "one", "tiny"])
@pytest.mark.parametrize("kind", ["hubs", "middle", "path", "parts"])
def test_distances_equal_the_oracle(kind, weights):
    rng = np.random.default_rng(len(kind))
    scale, e = graph(kind, rng)
    m = e.shape[1]
    w = {"any": lambda: (rng.integers(0, 1 << 24, m) + 1) * 2.0 ** -24, "one": lambda: np.ones(m),
         "tiny": lambda: (rng.integers(0, 4, m) + 1) * 2.0 ** -24}[weights]().astype(np.float32)
    off, col, wr = oracle.csr_build_weighted(e, w, scale)
    G = gb.graph_build_csr_weighted(torch.as_tensor(e).cuda(), torch.as_tensor(w).cuda(), scale)
    edges = torch.as_tensor(e).cuda()
    deg = np.diff(off)
    roots = [int(deg.argmax()), int(np.nonzero(deg > 0)[0][0]), int(rng.choice(np.nonzero(deg > 0)[0]))]
    saved, ends = gb.bfs_get_options(), set()
    try:
        for r in roots:
            d_ref, _ = oracle.sssp(off, col, wr, r)
            for delta in (2.0 ** -22 if weights == "tiny" else 0.004, 0.07, 0.6, 5.0):
                for canonical in (0, 1):
                    gb.bfs_set_options(canonical_parents=canonical)
                    dist, parent = gb.sssp(G, r, delta)
                    pulls = gb.debug_sssp_pulls()
                    assert pulls == expected_pulls(off, d_ref, delta)
                    ends.add(pulls > 0)
                    assert np.array_equal(dist.cpu().numpy(), d_ref), (r, delta, canonical)
                    if canonical:
                        assert np.array_equal(parent.cpu().numpy(), oracle.sssp_tree(off, col, wr, r, d_ref))
                    assert gb.sssp_validate(G, r, parent, dist, edges)["code"] == 0
    finally:
        gb.bfs_set_options(**saved)
    if weights == "any" and kind != "middle":   # rows of every length: some searches never pull
        assert ends == {True, False}
    gb.gb_device_status()
