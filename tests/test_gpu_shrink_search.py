"""The sphere shrinking's search over groups of 32 boundary triangles against
the CPU restatement (oracle/shrink.py): fewer triangles than a group, a ragged
last group, many groups; plain and proposed first radii; pins off the
triangles' centroids.

Tolerance: both sides run in FP64; a radius |p - q|^2 / (2 n.(q - p)) carries
the rounding of n.(q - p) amplified by r / |q - p|, below 1e-9 of the radius
for the shapes here (the same bound as the repair tests').
"""
import numpy as np
import pytest
import torch

from oracle.shrink import boundary_triangles, shrink as cpu_shrink
from paper_2403_18761_gb300 import build_workload
from rpd_inputs import genus_slab, tiny, torus_c1
from rpd_inputs.configs import Workload

pytestmark = pytest.mark.gpu


def _one_tet():
    v = np.array([[0, 0, 0], [1.0, 0, 0], [0, 0.75, 0], [0, 0, 1.25]])
    c, r = np.array([[0.25, 0.25, 0.25]]), np.array([0.25])
    return Workload("one_tet", v, np.array([[0, 1, 2, 3]], dtype=np.int32), c, r, 18, 4, "fp32", {})


CASES = {"one_tet": _one_tet, "box": lambda: tiny("box", 1, 5), "ring": lambda: tiny("ring", 3, 0),
         "torus": torus_c1, "slab": lambda: genus_slab(2, h=0.15, ns=64)}


@pytest.mark.parametrize("which", sorted(CASES))
def test_search_matches_a_scan_of_all_triangles(which):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = CASES[which]()
    ctx = build_workload(w)
    tris, ids = boundary_triangles(w)
    q, _, _ = w.ints()
    sc = 1.0 / float(1 << w.grid_bits)
    rng = np.random.default_rng(7)
    pick = np.sort(rng.choice(len(ids), size=min(16, len(ids)), replace=False))
    pick = np.concatenate([pick, [0, len(ids) - 1]])   # the first and the last triangle of the groups' input order
    pins, nrm = [], []
    for j, k in enumerate(pick):
        T = tris[k]
        n = np.cross(T[1] - T[0], T[2] - T[0])
        n /= np.linalg.norm(n)
        lam = np.ones(3) / 3 if j % 2 == 0 else rng.dirichlet((2.0, 2.0, 2.0))
        p = lam @ T
        t, f = int(ids[k]) >> 2, int(ids[k]) & 3
        if n @ (q[w.tets[t, f]] * sc - p) < 0:
            n = -n
        pins.append(p)
        nrm.append(n)
    pins, nrm, faces = np.array(pins + [pins[0]]), np.array(nrm + [nrm[0]]), ids[pick].astype(np.int32)
    faces = np.append(faces, np.int32(-1))   # a row without a face
    r0 = 2.0 ** (23 - w.grid_bits)
    want = [cpu_shrink(tris, int(k), pins[j], nrm[j], r0) for j, k in enumerate(pick)]
    c, r, it = (x.cpu().numpy() for x in ctx.rpd_shrink(pins, nrm, faces))
    # proposals above, at and below the fixed point
    start = np.array([rr * (1.5, 1.0 + 1e-7, 0.4)[j % 3] for j, (_, rr, _) in enumerate(want)] + [1.0])
    cw, rw, iw, re = (x.cpu().numpy() for x in ctx.rpd_shrink_warm(pins, nrm, faces, start))
    for j, (cc, rr, _) in enumerate(want):
        for got_c, got_r in ((c[j], r[j]), (cw[j], rw[j])):
            assert abs(got_r - rr) <= 1e-9 * rr, (j, got_r, rr)
            assert np.linalg.norm(got_c - cc) <= 1e-9 * rr
        if j % 3 == 2:
            assert re[j] == 1   # an empty proposed ball starts over
    assert np.isnan(r[-1]) and np.isnan(rw[-1]) and it[-1] == 0 and iw[-1] == 0
