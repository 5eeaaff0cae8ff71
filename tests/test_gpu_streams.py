"""A graph built on one stream and searched at once on another.

Every call that builds a graph, or adds to one, returns when its arrays are complete: a
search on a stream that is not ordered after the building one reads finished arrays.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
import paper_2012_13548_gb300 as gb  # noqa: E402
from paper_2012_13548_gb300 import workloads as W  # noqa: E402

pytestmark = pytest.mark.gpu

BUILDS = {
    "buckets": lambda e, off, col, spec, s: gb.graph_build_csr(e, spec.scale, stream=s),
    "counting": lambda e, off, col, spec, s: gb.graph_build_csr_counting(e, spec.scale, stream=s),
    "fused": lambda e, off, col, spec, s: gb.graph_generate_csr(**spec.kron_args(), stream=s),
    "csr": lambda e, off, col, spec, s: gb.graph_from_csr(off, col, stream=s),
}


@pytest.mark.parametrize("scale", [10, 18])
@pytest.mark.parametrize("how", sorted(BUILDS))
def test_search_on_another_stream(how, scale):
    spec = W.GraphSpec(scale=scale)
    e_ref = oracle.kron_generate(**spec.kron_args())
    off_ref, col_ref = oracle.csr_build(e_ref, scale)
    roots = [int(r) for r in W.select_roots(off_ref, 2, spec.seeds()[3])]
    ref = [oracle.bfs(off_ref, col_ref, r)[1] for r in roots]
    e = torch.as_tensor(e_ref).cuda()
    off, col = torch.as_tensor(off_ref).cuda(), torch.as_tensor(col_ref).cuda()
    parent = torch.empty(1 << scale, dtype=torch.int32, device="cuda")
    level = torch.empty_like(parent)
    P = torch.empty((2, 1 << scale), dtype=torch.int32, device="cuda")
    L = torch.empty_like(P)
    build, search = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(5):
        torch.cuda.synchronize()
        g = BUILDS[how](e, off, col, spec, build)
        gb.bfs(g, roots[0], parent, level, stream=search)
        search.synchronize()
        assert np.array_equal(level.cpu().numpy(), ref[0])
        torch.cuda.synchronize()
        g.prepare_batched(stream=build)
        gb.bfs_batch(g, roots, P, L, stream=search)
        search.synchronize()
        assert np.array_equal(L.cpu().numpy(), np.stack(ref))
        g.free()
    gb.gb_device_status()


def test_shortest_paths_on_another_stream():
    spec = W.GraphSpec(scale=14)
    e_ref = oracle.kron_generate(**spec.kron_args())
    w_ref = oracle.kron_weights(e_ref.shape[1], spec.seed_weight())
    off, col, wgt = oracle.csr_build_weighted(e_ref, w_ref, spec.scale)
    root = int(np.diff(off).argmax())
    d_ref, _ = oracle.sssp(off, col, wgt, root)
    e, w = torch.as_tensor(e_ref).cuda(), torch.as_tensor(w_ref, dtype=torch.float32).cuda()
    dist = torch.empty(1 << spec.scale, dtype=torch.float64, device="cuda")
    parent = torch.empty(1 << spec.scale, dtype=torch.int32, device="cuda")
    build, search = torch.cuda.Stream(), torch.cuda.Stream()
    for _ in range(5):
        torch.cuda.synchronize()
        g = gb.graph_build_csr_weighted(e, w, spec.scale, stream=build)
        gb.sssp(g, root, 0.1, dist, parent, stream=search)
        search.synchronize()
        assert np.array_equal(dist.cpu().numpy(), d_ref)
        g.free()
    gb.gb_device_status()
