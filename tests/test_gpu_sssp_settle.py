"""Settle steps of the shortest-path search from either end, against the oracle.

A bucket's heavy edges are read from the settled rows or from the rows of what is
still unsettled, whichever is less; rows below and above 64 and 1024 entries, buckets
from one unit of the weights to the whole search, equal weights (ties at every
bound), unreachable parts.
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
    saved = gb.bfs_get_options()
    try:
        for r in roots:
            d_ref, _ = oracle.sssp(off, col, wr, r)
            for delta in (2.0 ** -22 if weights == "tiny" else 0.004, 0.07, 0.6, 5.0):
                for canonical in (0, 1):
                    gb.bfs_set_options(canonical_parents=canonical)
                    dist, parent = gb.sssp(G, r, delta)
                    assert np.array_equal(dist.cpu().numpy(), d_ref), (r, delta, canonical)
                    if canonical:
                        assert np.array_equal(parent.cpu().numpy(), oracle.sssp_tree(off, col, wr, r, d_ref))
                    assert gb.sssp_validate(G, r, parent, dist, edges)["code"] == 0
    finally:
        gb.bfs_set_options(**saved)
    gb.gb_device_status()
