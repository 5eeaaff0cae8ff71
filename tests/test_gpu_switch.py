"""Where a search turns bottom-up, on graphs whose second level lies between two rules.

level_dir of the statistics tells how a level was run.
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
def _options():
    saved = gb.bfs_get_options()
    yield
    gb.bfs_set_options(**saved)


def hubs(scale, count, leaves, rest, rng):
    """Vertex 0 joined to `count` hubs of `leaves` neighbours each, and about `rest` edges
    among the leaves: the second frontier is the hubs."""
    n = 1 << scale
    first = 1 + count
    leaf = np.arange(first, first + count * leaves) % (n - first) + first
    u = [np.zeros(count, np.int64), np.repeat(np.arange(1, first), leaves), rng.integers(first, n, rest)]
    v = [np.arange(1, first), leaf, rng.integers(first, n, rest)]
    e = np.stack([np.concatenate(u), np.concatenate(v)]).astype(np.int64)
    off, col = oracle.csr_build(e, scale)
    hub_edges = int((off[first] - off[1]))
    return gb.graph_build_csr(torch.as_tensor(e).cuda(), scale), off, col, hub_edges


@pytest.mark.parametrize("ms_alpha,step", [(None, "td"), (16.0, "td"), (4.0, "td"), (8.0, "td"),
                                           (12.0, "bu"), (16.5, "bu"), (64.0, "bu")])
def test_ms_alpha_acts_as_it_is_set(ms_alpha, step):
    g, off, col, mf = hubs(13, 20, 200, 16000, np.random.default_rng(1))
    assert 1 / 12 < mf / off[-1] < 1 / 8.5   # between the ratios 12 and 8, and the default's 4
    if ms_alpha is not None:
        gb.bfs_set_options(ms_alpha=ms_alpha)
    for canonical in (0, 1):
        gb.bfs_set_options(canonical_parents=canonical)
        _, levels = gb.bfs_batch(g, [0, 0])
        assert gb.bfs_last_stats()["level_dir"][:2] == ["td", step]
        assert np.array_equal(levels[1].cpu().numpy(), oracle.bfs(off, col, 0)[1])


@pytest.mark.parametrize("canonical", [0, 1])
def test_edges_examined_counts_the_frontiers_edges_once(canonical):
    # top-down only: every reached vertex's row, however the smallest parents are found
    rng = np.random.default_rng(2)
    graphs = [hubs(12, 7, 300, 3000, rng)[:3], hubs(13, 300, 20, 9000, rng)[:3]]
    gb.bfs_set_options(canonical_parents=canonical, alpha=1e-9, beta=1e-9, ms_alpha=1e-9, ms_beta=1e-9)
    for g, off, col in graphs:
        _, level = oracle.bfs(off, col, 0)
        rows = int(np.diff(off)[level >= 0].sum())
        gb.bfs(g, 0)
        assert gb.bfs_last_stats()["edges_examined"] == rows
        gb.bfs_batch(g, [0, 0])
        assert gb.bfs_last_stats()["edges_examined"] == rows
