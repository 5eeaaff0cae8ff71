"""The validator's pass over the CSR entries: which entry it names.

A graph built from tuples is symmetric and only the entries (u, v) with u < v
are looked up; a caller's CSR need not be, and all are.  Rows of every length:
isolated vertices in long runs, rows of one entry, a row longer than a warp's run.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2012_13548_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


def graph(kind, scale, rng):
    n = 1 << scale
    if kind == "sparse":      # long runs of isolated vertices
        u = rng.integers(0, n, n // 64)
        v = rng.integers(0, n, n // 64)
    elif kind == "star":
        u = np.full(4 * n, n // 2)
        v = rng.integers(0, n, 4 * n)
    else:
        u, v = rng.integers(0, n, 8 * n), rng.integers(0, n, 8 * n)
    return np.stack([u, v]).astype(np.int64)


def first_entry(off, col, level):
    row = np.repeat(np.arange(len(off) - 1), np.diff(off))
    lu, lw = level[row], level[col]
    five = (lu < 0) != (lw < 0)
    six = ~five & (lu >= 0) & (np.abs(lu - lw) > 1)
    bad = np.nonzero(five | six)[0]
    return (0, -1) if bad.size == 0 else (5 if five[bad[0]] else 6, int(bad[0]))


@pytest.mark.parametrize("built", [True, False])
@pytest.mark.parametrize("kind,scale", [("sparse", 13), ("star", 12), ("any", 9), ("any", 13)])
def test_the_first_failing_entry(kind, scale, built):
    rng = np.random.default_rng(scale)
    e = graph(kind, scale, rng)
    off, col = oracle.csr_build(e, scale)
    off, col = np.asarray(off), np.asarray(col)
    if built:
        G = gb.graph_build_csr(torch.as_tensor(e).cuda(), scale)
    else:
        G = gb.graph_from_csr(torch.as_tensor(off).cuda(), torch.as_tensor(col).cuda())
    root = int(np.diff(off).argmax())
    parent, level = oracle.bfs(off, col, root)
    leaves = np.nonzero((level > 0) & ~np.isin(np.arange(len(level)), parent))[0]
    for t in range(12):
        # another level for some vertices, or none: only vertices that no parent rule
        # looks at first are touched where possible, and the entry pass is compared alone
        p, lv = parent.copy(), level.copy()
        x = rng.choice(leaves if leaves.size else np.nonzero(level > 0)[0])
        if t % 3 == 0:
            p[x] = lv[x] = -1
        else:
            lv[x] += 1 + t % 4
        code, where = first_entry(off, col, lv)
        res = gb.bfs_validate(G, root, torch.as_tensor(p).cuda(), torch.as_tensor(lv).cuda())
        ref = oracle.validate(off, col, root, p, lv)
        assert res["code"] == ref
        if res["code"] in (5, 6):
            assert (res["code"], res["where"]) == (code, where)


def test_an_asymmetric_csr_is_checked_in_full():
    # 0 - 1 - 2, and an entry 3 -> 0 without its twin: vertex 3 is not reached
    off = np.array([0, 1, 3, 4, 5], dtype=np.int64)
    col = np.array([1, 0, 2, 1, 0], dtype=np.int32)
    G = gb.graph_from_csr(torch.as_tensor(off).cuda(), torch.as_tensor(col).cuda())
    p = torch.tensor([0, 0, 1, -1], dtype=torch.int32, device="cuda")
    lv = torch.tensor([0, 1, 2, -1], dtype=torch.int32, device="cuda")
    res = gb.bfs_validate(G, 0, p, lv)
    assert (res["code"], res["where"]) == (5, 4)
