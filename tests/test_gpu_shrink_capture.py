"""A shrinking captured into a graph by a context that has the boundary triangles
but has not shrunk yet: the search index it needs belongs to the context, not to
the graph, so shrinking outside the graph works before the first replay, and
every replay gives the same spheres."""
import pytest
import torch

from paper_2403_18761_gb300 import build_workload
from paper_2403_18761_gb300.rpd import _ptr, load
from rpd_inputs import genus_slab

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("warm", [False, True])
def test_first_shrinking_under_capture(warm):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = genus_slab(2, h=0.15, ns=64)
    want = build_workload(w)
    pts, normals, faces = want.rpd_surface_samples()
    centres, radii, iters = want.rpd_shrink(pts, normals, faces)
    start = 1.5 * radii
    stream = torch.cuda.Stream()
    ctx = build_workload(w, stream=stream)
    ctx.rpd_surface_samples()
    n = len(pts)
    c, r = torch.zeros_like(centres), torch.zeros_like(radii)
    it, re = torch.zeros_like(iters), torch.zeros_like(iters)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        if warm:
            st = load().rpd_shrink_warm(ctx.handle, _ptr(pts), _ptr(normals), _ptr(faces), n, _ptr(start), _ptr(c), _ptr(r),
                                        _ptr(it), _ptr(re))
        else:
            st = load().rpd_shrink(ctx.handle, _ptr(pts), _ptr(normals), _ptr(faces), n, _ptr(c), _ptr(r), _ptr(it))
        assert st == 0
    now = ctx.rpd_shrink(pts, normals, faces)   # outside the graph, before any replay
    assert torch.equal(now[0], centres) and torch.equal(now[1], radii)
    for _ in range(2):
        r.zero_()
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        if warm:
            assert torch.allclose(r, radii, rtol=1e-9, atol=0)
        else:
            assert torch.equal(c, centres) and torch.equal(r, radii) and torch.equal(it, iters)
