"""Envelope distances of samples with no finite position, or far from the shape,
among ordinary ones: they change no distance of the others, and they do not make
the others' packets test every primitive.  (Which of several primitives at the same
distance is named follows from the samples' order, so strays may change that.)

A sample with a coordinate that is not a number, infinite, or whose square FP32
cannot hold has no nearest primitive: (infinity, -1).  The time bound is three
times that of the ordinary samples alone; with shared margins and bounds one such
sample made it six times.
"""
import numpy as np
import pytest
import torch

from paper_2403_18761_gb300 import build_workload
from rpd_inputs import blob_c3

pytestmark = pytest.mark.gpu

NAN, INF = float("nan"), float("inf")


@pytest.fixture(scope="module")
def shape():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    ctx = build_workload(blob_c3(target_tets=300_000, ns=3000, n_ellipsoids=60))
    pts = ctx.rpd_surface_samples()[0]
    return ctx, pts, ctx.rpd_envelope_distance(pts)[0]


def _ms(ctx, pts):
    best = INF
    for _ in range(5):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        ctx.rpd_envelope_distance(pts)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("rows", ["one", "every_37th", "last_quarter"])
@pytest.mark.parametrize("value", [NAN, INF, -INF, 1e30, 1e10, -1e4])
def test_strays(shape, rows, value):
    ctx, pts, dist = shape
    n = len(pts)
    at = torch.zeros(n, dtype=torch.bool, device=pts.device)
    at[{"one": slice(5, 6), "every_37th": slice(0, n, 37), "last_quarter": slice(n - n // 4, n)}[rows]] = True
    q = pts.clone()
    q[at, 1] = value
    d, a = ctx.rpd_envelope_distance(q)
    assert torch.equal(d[~at], dist[~at]) and bool((a[~at] >= 0).all())
    if np.isfinite(value) and abs(value) < 1e19:
        assert bool((a[at] >= 0).all())
        # every primitive lies within the shape, whose size is below 20
        assert bool(((d[at] - abs(value)).abs() <= 20 + 1e-5 * abs(value)).all())
    else:
        assert bool((a[at] == -1).all()) and bool(torch.isinf(d[at]).all())
    if rows == "one":
        assert _ms(ctx, q) < 3 * _ms(ctx, pts)


def test_nothing_but_strays(shape):
    ctx, pts, _ = shape
    d, a = ctx.rpd_envelope_distance(torch.full_like(pts, NAN))
    assert bool((a == -1).all()) and bool(torch.isinf(d).all())
