"""The packet search for the tets' candidate spheres (csrc/cand.cu) against the
per-vertex neighbour lists (debug bit 4, csrc/knn.cu): the candidate sets are
exact in both, so every table, piece and volume must be the same bit for bit,
whatever the order of the mesh, the number of spheres (one leaf, a ragged leaf,
several nodes) and the list length k (which sends tets to the fallback)."""
import numpy as np
import pytest
import torch

from paper_2403_18761_gb300 import rpd_build, rpd_build_batch
from paper_2403_18761_gb300.rpd import collect
from rpd_inputs import blob_c3, block_c2, genus_slab, torus_c1

pytestmark = pytest.mark.gpu


def _same(a, b):
    for kind in (1, 2, 3, 4):
        for f in ("keys", "chi", "beta0", "flag"):
            assert np.array_equal(a["kinds"][kind][f], b["kinds"][kind][f]), (kind, f)
    for f in ("tet", "sphere", "vol", "moment"):
        assert np.array_equal(a[f], b[f]), f


def _both(v, t, c, r, bits, k=16, precision="fp32"):
    a, b = (collect(rpd_build(v, t, c, r, precision=precision, k=k, grid_bits=bits, debug=d)) for d in (0, 4))
    _same(a, b)
    return a


def _shuffled(w, seed):
    """The same shape with its vertices, tets and spheres in random order."""
    rng = np.random.default_rng(seed)
    pv, pt, ps = rng.permutation(len(w.verts)), rng.permutation(len(w.tets)), rng.permutation(len(w.centers))
    at = np.empty(len(pv), dtype=np.int32)
    at[pv] = np.arange(len(pv), dtype=np.int32)
    return w.verts[pv], at[w.tets[pt]], w.centers[ps], w.radii[ps]


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


@pytest.mark.parametrize("ns", [1, 2, 31, 32, 33, 64, 65, 300])
def test_sphere_counts(ns):
    w = block_c2(h=0.15, ns=300)
    _both(w.verts, w.tets, w.centers[:ns], w.radii[:ns], w.grid_bits)


@pytest.mark.parametrize("make", [lambda: torus_c1(), lambda: block_c2(h=0.1, ns=1500),
                                  lambda: blob_c3(target_tets=60_000, ns=3000, n_ellipsoids=40)])
def test_orders(make):
    w = make()
    _both(w.verts, w.tets, w.centers, w.radii, w.grid_bits, k=32)
    _both(*_shuffled(w, 3), w.grid_bits, k=32)


@pytest.mark.parametrize("k", [1, 2, 7])
def test_short_lists_take_the_fallback(k):
    w = block_c2(h=0.15, ns=300)
    a = _both(w.verts, w.tets, w.centers, w.radii, w.grid_bits, k=k)
    assert k > 1 or a["stats"]["cand_fallback"] > 0   # up to 4 k spheres are gathered per tet


def test_batch_of_uneven_shapes():
    ws = [torus_c1(), block_c2(h=0.15, ns=300), genus_slab(1, h=0.2, ns=1), genus_slab(3, h=0.15, ns=70)]
    shapes = [(w.verts, w.tets, w.centers, w.radii) for w in ws]
    a = collect(rpd_build_batch(shapes, k=16, grid_bits=18))
    at = 0
    for s in shapes:
        one = collect(rpd_build(*s, k=16, grid_bits=18, debug=4))
        n = len(one["tet"])
        assert np.array_equal(a["vol"][at:at + n], one["vol"])
        at += n
    assert at == len(a["tet"])
