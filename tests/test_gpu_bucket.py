"""Kernel 1's sort by buckets at the sizes where it can go wrong, against the oracle.

One digit up to 2^21 keys and two above; buckets longer than 4096 keys split
once, or again from the bits that their keys differ in (columns crowded at one end, all
weights equal); key ranges with no row start, rows with no entry; self-loops only; one
endpoint pair repeated.  Every output is compared bit for bit, and the way that each
build took is asserted.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2012_13548_gb300 as gb  # noqa: E402

pytestmark = pytest.mark.gpu


def tuples(kind, scale, m, rng):
    n = 1 << scale
    u, v = rng.integers(0, n, m), rng.integers(0, n, m)
    if kind == "star":      # one row of every vertex: split by row bits, then by column bits
        u[:] = n // 3
    elif kind == "loops":
        v = u.copy()
    elif kind == "pair":    # one pair m times: no split tells its copies apart
        u[:], v[:] = n - 1, n // 2
    elif kind == "pairs":   # as many copies of two pairs beside ordinary tuples
        u[: m // 2], v[: m // 2] = 1 % n, 0
        u[m // 2: 3 * m // 4], v[m // 2: 3 * m // 4] = n - 2, n - 1
    elif kind == "skew":    # endpoints crowded at both ends of the range
        u = np.minimum(n - 1, (n * rng.random(m) ** 6).astype(np.int64))
        v = n - 1 - np.minimum(n - 1, (n * rng.random(m) ** 6).astype(np.int64))
    elif kind == "band":    # neighbours close to their row
        v = np.clip(u + rng.integers(-3, 4, m), 0, n - 1)
    elif kind == "crowd":   # one row, its columns ever denser towards the last
        u[:] = n // 3
        v = n - 1 - np.minimum(n - 1, (n * rng.random(m) ** 12).astype(np.int64))
    elif kind == "geo":     # three rows, as many columns in every range [2^k, 2^(k+1))
        u = rng.integers(0, 3, m)
        v = np.minimum(n - 1, (2.0 ** (scale * rng.random(m))).astype(np.int64))
    elif kind == "rmat":    # the quadrants' own order: vertices not renumbered
        u, v = np.zeros(m, np.int64), np.zeros(m, np.int64)
        for _ in range(scale):
            r = rng.random(m)
            u, v = 2 * u + (r >= 0.76), 2 * v + (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    elif kind == "hub":     # one row of every vertex beside short ones
        u[: n - 1], v[: n - 1] = 0, np.arange(1, n)
    return np.stack([u, v]).astype(np.int64)


# kinds whose long buckets one split by length leaves too long
CROWDED = {("pairs", 14), ("crowd", 14), ("crowd", 20), ("geo", 16), ("geo", 21), ("rmat", 18)}
CASES = [("any", 1, 1), ("any", 1, 5000), ("any", 2, 4097), ("any", 5, 100003), ("any", 10, 1023),
         ("any", 11, (1 << 20) - 1), ("any", 11, (1 << 20) + 1), ("any", 16, (1 << 20) + 12345), ("any", 21, 70001),
         ("any", 22, 70001), ("any", 24, 3), ("loops", 9, 10000), ("pair", 9, 300001), ("pair", 18, 9001),
         ("pairs", 1, 100000), ("pairs", 14, 100000), ("star", 13, 4096), ("star", 18, 1 << 18), ("star", 20, 1 << 21),
         ("skew", 12, 1 << 19), ("skew", 19, (1 << 21) + 77), ("band", 17, 1 << 20), ("crowd", 14, 200000),
         ("crowd", 20, (1 << 20) + 5), ("geo", 16, 300000), ("geo", 21, (1 << 21) + 1), ("rmat", 18, 16 << 18)]


def digits(scale, m, weighted):
    """Digits of the bucket sort: one while a bucket holds 2048 keys on average, at most
    512 rows, and what is left of a key fits its type."""
    bits = max(2 * scale + 25 - 64 if weighted else 2 * scale - 32, scale - 9, int(-(-2 * m // 2048) - 1).bit_length(), 1)
    return 1 if bits <= 10 else 2


@pytest.mark.parametrize("kind,scale,m", CASES)
def test_buckets_equal_the_oracle(kind, scale, m):
    e = tuples(kind, scale, m, np.random.default_rng(scale * 1000003 + m))
    g = gb.graph_build_csr(torch.as_tensor(e).cuda(), scale)
    took, splits = gb.debug_build_route()
    assert took == digits(scale, m, False)
    if (kind, scale) in CROWDED:
        assert splits > 0
    elif kind in ("any", "loops", "band"):
        assert splits == 0
    off_ref, col_ref = oracle.csr_build(e, scale)
    off, col = g.csr()
    assert np.array_equal(off.cpu().numpy(), off_ref)
    assert np.array_equal(col.cpu().numpy(), col_ref)
    gb.gb_device_status()


@pytest.mark.parametrize("weights", ["any", "one", "few"])
@pytest.mark.parametrize("kind,scale,m", [("any", 1, 3000), ("any", 10, 1023), ("any", 16, (1 << 20) + 12345),
                                          ("any", 20, 40001), ("pair", 9, 100001), ("pairs", 14, 60000),
                                          ("star", 18, 1 << 18), ("skew", 15, 1 << 19), ("crowd", 14, 200000),
                                          ("geo", 16, 300000), ("hub", 17, 1 << 18)])
def test_weighted_buckets_equal_the_oracle(kind, scale, m, weights):
    rng = np.random.default_rng(scale * 1000003 + m)
    e = tuples(kind, scale, m, rng)
    w = {"any": lambda: (rng.integers(0, 1 << 24, m) + 1) * 2.0 ** -24, "one": lambda: np.ones(m),
         "few": lambda: 2.0 ** -rng.integers(0, 3, m).astype(np.float64)}[weights]().astype(np.float32)
    g = gb.graph_build_csr_weighted(torch.as_tensor(e).cuda(), torch.as_tensor(w).cuda(), scale)
    took, splits = gb.debug_build_route()
    assert took == digits(scale, m, True)
    if (kind, scale) in CROWDED or (kind == "hub" and weights == "one"):
        assert splits > 0
    elif kind == "any":
        assert splits == 0
    off_ref, col_ref, w_ref = oracle.csr_build_weighted(e, w, scale)
    off, col = g.csr()
    assert np.array_equal(off.cpu().numpy(), off_ref)
    assert np.array_equal(col.cpu().numpy(), col_ref)
    assert np.array_equal(g.weights().cpu().numpy() * 2.0 ** -24, w_ref)  # whole units: exact
    # the weight-ordered rows serve the searches
    deg = np.diff(off_ref)
    if deg.max() == 0:
        return
    root = int(deg.argmax())
    gb.bfs_set_options(canonical_parents=1)
    try:
        dist, _ = gb.sssp(g, root, delta=0.1)
    finally:
        gb.bfs_set_options(canonical_parents=0)
    d_ref, _ = oracle.sssp(off_ref, col_ref, w_ref, root)
    assert np.array_equal(dist.cpu().numpy(), d_ref)
    gb.gb_device_status()


def test_bad_endpoints_and_weights_are_refused():
    e = torch.randint(0, 1 << 12, (2, 50000), device="cuda")
    w = torch.ones(50000, device="cuda")
    for bad in (-1, 1 << 12):
        f = e.clone()
        f[1, 49999] = bad
        with pytest.raises(gb.GbError, match="endpoint"):
            gb.graph_build_csr(f, 12)
        w2 = w.clone()
        w2[3] = 2.0
        with pytest.raises(gb.GbError, match="endpoint"):
            gb.graph_build_csr_weighted(f, w2, 12)
    for x in (0.0, 1.5, float("nan")):
        w2 = w.clone()
        w2[49999] = x
        with pytest.raises(gb.GbError, match="weight"):
            gb.graph_build_csr_weighted(e, w2, 12)
    gb.gb_device_status()


def test_a_portion_of_the_callers_own_takes_the_radix_sort():
    e = tuples("any", 12, 50001, np.random.default_rng(3))
    off_ref, col_ref = oracle.csr_build(e, 12)
    saved = gb.sort_portion()
    try:
        gb.sort_portion(20000)
        g = gb.graph_build_csr(torch.as_tensor(e).cuda(), 12)
        assert gb.debug_build_route() == (0, 0)
        gb.graph_build_csr_weighted(torch.as_tensor(e).cuda(), torch.ones(50001, device="cuda"), 12)
        assert gb.debug_build_route() == (0, 0)
    finally:
        gb.sort_portion(saved)
    off, col = g.csr()
    assert np.array_equal(off.cpu().numpy(), off_ref) and np.array_equal(col.cpu().numpy(), col_ref)
