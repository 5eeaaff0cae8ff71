"""Searches whose levels are narrow: one block runs them alone (bfs.cu,
solo_levels).  Graphs with levels on both sides of its limits (1024 frontier
vertices, 1024 edges, 4096 edges of short rows), numbered at random, against
the oracle: levels always, parents in canonical mode, the Graph500 rules
otherwise.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2012_13548_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _reset_options():
    gb.bfs_set_options(canonical_parents=0, big_degree=256, blocks_per_sm=2, timeout_ms=5000.0)
    yield
    gb.bfs_set_options(canonical_parents=0, big_degree=256, blocks_per_sm=2, timeout_ms=5000.0)
    gb.gb_device_status()


def _csr(n, pairs, rng):
    """CSR of the undirected pairs under a random numbering, and the number of vertex 0."""
    perm = rng.permutation(n)
    p = perm[np.asarray(pairs, dtype=np.int64)]
    key = np.unique(np.concatenate([p[:, 0] * n + p[:, 1], p[:, 1] * n + p[:, 0]]))
    off = np.zeros(n + 1, dtype=np.int64)
    off[1:] = np.cumsum(np.bincount(key // n, minlength=n))
    return off, (key % n).astype(np.int32), int(perm[0])


def _layers(widths, rng, extra):
    """Consecutive layers, every vertex joined to at least one of the layer before."""
    pairs, first, n = [], 0, widths[0]
    for w in widths[1:]:
        prev = n - first
        for i in range(w):
            for j in {i % prev, *rng.integers(0, prev, extra)}:
                pairs.append((first + int(j), n + i))
        first, n = n, n + w
    return n, pairs


def _mesh(w, h):
    v = np.arange(w * h).reshape(h, w)
    return w * h, np.concatenate([np.stack([v[:, :-1].ravel(), v[:, 1:].ravel()], 1),
                                  np.stack([v[:-1].ravel(), v[1:].ravel()], 1)])


GRAPHS = {
    "path": lambda r: (4001, [(i, i + 1) for i in range(4000)]),
    "mesh": lambda r: _mesh(61, 83),
    "wide_mesh": lambda r: _mesh(1500, 1100),                        # frontiers above 1024 and back
    "frontier_limits": lambda r: _layers([1, 1023, 1, 1024, 1, 1025, 2, 5000, 3], r, 0),
    "edge_limits": lambda r: _layers([1, 8, 128, 128, 511, 513, 2, 2, 40], r, 7),
    "short_rows": lambda r: _layers([1, 4, 16, 64, 256, 1000, 1024, 1024, 1000, 256, 1300, 7], r, 1),
    "hubs": lambda r: _layers([1, 3, 3000, 4, 700, 1, 1], r, 2),
}


@pytest.mark.parametrize("name", sorted(GRAPHS))
@pytest.mark.parametrize("big_degree", [4, 256])
@pytest.mark.parametrize("canonical", [0, 1])
def test_narrow_levels(name, big_degree, canonical):
    rng = np.random.default_rng(len(name))
    n, pairs = GRAPHS[name](rng)
    off, col, root = _csr(n, pairs, rng)
    p_ref, l_ref = oracle.bfs(off, col, root)
    g = gb.graph_from_csr(torch.as_tensor(off).cuda(), torch.as_tensor(col).cuda())
    gb.bfs_set_options(canonical_parents=canonical, big_degree=big_degree)
    for blocks in (1, 2, 3):
        gb.bfs_set_options(blocks_per_sm=blocks)
        parent, level = gb.bfs(g, root)
        assert np.array_equal(level.cpu().numpy(), l_ref)
        if canonical:
            assert np.array_equal(parent.cpu().numpy(), p_ref)
        assert gb.bfs_validate(g, root, parent, level)["code"] == 0
        st = gb.bfs_last_stats()
        assert st["nlevels"] == l_ref.max() + 1 == st["td_levels"] + st["bu_levels"]
        assert st["reached"] == n
    g.free()


@pytest.mark.parametrize("name", ["path", "mesh", "wide_mesh"])
@pytest.mark.parametrize("canonical", [0, 1])
def test_stretches_that_the_wait_limit_cuts_short(name, canonical):
    # a quarter of the limit ends a stretch, so each of these searches is many stretches
    rng = np.random.default_rng(len(name))
    n, pairs = GRAPHS[name](rng)
    off, col, root = _csr(n, pairs, rng)
    p_ref, l_ref = oracle.bfs(off, col, root)
    g = gb.graph_from_csr(torch.as_tensor(off).cuda(), torch.as_tensor(col).cuda())
    gb.bfs_set_options(canonical_parents=canonical, timeout_ms=1.0)
    for _ in range(10):
        parent, level = gb.bfs(g, root)
        gb.gb_device_status()
        assert np.array_equal(level.cpu().numpy(), l_ref)
        if canonical:
            assert np.array_equal(parent.cpu().numpy(), p_ref)
    assert gb.bfs_validate(g, root, parent, level)["code"] == 0
    g.free()


@pytest.mark.parametrize("limit_ms", [0.2, 0.09])
@pytest.mark.parametrize("canonical", [0, 1])
def test_a_short_wait_limit_holds_for_levels_run_by_one_block(canonical, limit_ms):
    # the other blocks wait for a whole stretch of levels of up to 25 us: it has to end
    # well within their limit, as a level of the whole grid does
    n, pairs = GRAPHS["wide_mesh"](None)
    off, col, root = _csr(n, pairs, np.random.default_rng(8))
    p_ref, l_ref = oracle.bfs(off, col, root)
    g = gb.graph_from_csr(torch.as_tensor(off).cuda(), torch.as_tensor(col).cuda())
    gb.bfs_set_options(canonical_parents=canonical)
    gb.bfs(g, root)
    gb.bfs_set_options(timeout_ms=limit_ms)
    for _ in range(3):
        parent, level = gb.bfs(g, root)
        gb.gb_device_status()
        assert np.array_equal(level.cpu().numpy(), l_ref)
        if canonical:
            assert np.array_equal(parent.cpu().numpy(), p_ref)
    g.free()
