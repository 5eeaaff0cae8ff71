"""Smallest-id parents after wide top-down levels, against the oracle.

The parents come from the frontier's edges where they are fewer than the claimed
vertices' and from the claimed vertices' rows otherwise, so the graphs here grow
through hubs (rows above and below the sizes that are cut into chunks), shrink
after a wide level, and let many frontier vertices reach the same ones.
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
def _canonical():
    saved = gb.bfs_get_options()
    yield
    gb.bfs_set_options(**saved)


def hub_graph(hubs, degree, scale, rng):
    """A root joined to every hub, every hub to `degree` random vertices, some of those
    to a few more; high ids first, so that the first claim is seldom the smallest."""
    n = 1 << scale
    ids = rng.permutation(n)
    root, hub, rest = ids[0], ids[1: 1 + hubs], ids[1 + hubs:]
    u = [np.full(hubs, root), np.repeat(hub, degree)]
    v = [hub, rng.choice(rest, hubs * degree)]
    leaf = rng.choice(rest, n // 8)
    u.append(leaf)
    v.append(rng.choice(rest, n // 8))
    return int(root), np.stack([np.concatenate(u), np.concatenate(v)]).astype(np.int64)


@pytest.mark.parametrize("alpha", [14.0, 1e-3])   # 1e-3: every level stays top-down
@pytest.mark.parametrize("hubs,degree,scale", [(1, 5000, 13), (3, 257, 12), (40, 200, 13), (300, 300, 15),
                                               (7, 20000, 16), (1500, 30, 14)])
def test_parents_equal_the_oracle(hubs, degree, scale, alpha):
    rng = np.random.default_rng(hubs + degree)
    root, e = hub_graph(hubs, degree, scale, rng)
    off, col = oracle.csr_build(e, scale)
    G = gb.graph_build_csr(torch.as_tensor(e).cuda(), scale)
    gb.bfs_set_options(canonical_parents=1, alpha=alpha, ms_alpha=alpha)
    roots = [root] + [int(x) for x in rng.choice(np.nonzero(np.diff(off) > 0)[0], 7)]
    ref = [oracle.bfs(off, col, r) for r in roots]
    for r, (p_ref, l_ref) in zip(roots, ref):
        parent, level = gb.bfs(G, r)
        assert np.array_equal(level.cpu().numpy(), l_ref)
        assert np.array_equal(parent.cpu().numpy(), p_ref)
    P, L = gb.bfs_batch(G, roots)
    Pm, Lm = gb.bfs_multi_graph([G, G], [roots, roots[::-1]])
    for i, (p_ref, l_ref) in enumerate(ref):
        assert np.array_equal(L[i].cpu().numpy(), l_ref)
        assert np.array_equal(P[i].cpu().numpy(), p_ref)
        for g, row in ((0, i), (1, len(roots) - 1 - i)):
            assert np.array_equal(Lm[g][row].cpu().numpy(), l_ref)
            assert np.array_equal(Pm[g][row].cpu().numpy(), p_ref)
    gb.gb_device_status()
