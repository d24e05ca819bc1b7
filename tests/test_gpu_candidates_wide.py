"""The packet search for candidate spheres (csrc/cand.cu) where one of its fixed
sizes is exceeded, against the per-vertex neighbour lists (debug bit 4): the
candidate sets are exact in both, so every table, piece and volume must be the
same bit for bit.

More than 32,768 spheres: more than 32 nodes of the sphere tree, so that a warp's
walk over them takes two rounds, and (above that number) the library's scan in
the finalisation.  A packet of tets that is far apart: more than 16 distinct
owners, of which only 16 serve to reject spheres, and with a crowd of spheres
between the tets more than the 256 that a packet holds, which sends all its
tets to the fallback."""
import numpy as np
import pytest
import torch

from paper_2403_18761_gb300 import rpd_build
from paper_2403_18761_gb300.rpd import collect
from rpd_inputs import block_c2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


def _both(v, t, c, r, bits):
    a, b = (collect(rpd_build(v, t, c, r, k=32, grid_bits=bits, debug=d)) for d in (0, 4))
    for kind in (1, 2, 3, 4):
        for f in ("keys", "chi", "beta0", "flag"):
            assert np.array_equal(a["kinds"][kind][f], b["kinds"][kind][f]), (kind, f)
    for f in ("tet", "sphere", "vol", "moment"):
        assert np.array_equal(a[f], b[f]), f
    return a


@pytest.mark.parametrize("ns", [32768, 32769, 36000])
def test_many_spheres(ns):
    w = block_c2(h=0.06, ns=10)
    rng = np.random.default_rng(9)
    c = rng.uniform(w.verts.min(axis=0), w.verts.max(axis=0), (ns, 3))
    a = _both(w.verts, w.tets, c, rng.uniform(0.05, 0.06, ns), w.grid_bits)
    assert len(np.unique(a["sphere"])) > 25000


@pytest.mark.parametrize("crowd", [100, 600])
def test_scattered_packet(crowd):
    """Eight small tets at the corners of a box, one packet, eight spheres about
    each, and a crowd in the middle that owns nothing."""
    rng = np.random.default_rng(31)
    one = np.array([[0, 0, 0], [0.25, 0, 0], [0, 0.2, 0], [0, 0, 0.3]])
    at = np.array([[x, y, z] for x in (-1.5, 1.5) for y in (-1.4, 1.4) for z in (-1.3, 1.3)])
    v = (at[:, None, :] + one + rng.uniform(-0.01, 0.01, (8, 4, 3))).reshape(-1, 3)
    t = np.arange(32, dtype=np.int32).reshape(8, 4)
    near = (at[:, None, :] + rng.uniform(-0.05, 0.3, (8, 8, 3))).reshape(-1, 3)
    mid = rng.normal(0, 0.05, (crowd, 3))
    c = np.concatenate([near, mid])
    r = np.concatenate([rng.uniform(0.05, 0.06, 64), rng.uniform(0.01, 0.02, crowd)])
    a = _both(v, t, c, r, 18)
    assert a["sphere"].max() < 64
    owners = {tuple(np.argmin(((v[k] - c[:64]) ** 2).sum(axis=1) - r[:64] ** 2, keepdims=True)) for k in range(32)}
    assert len(owners) > 16
    # the packet holds 256 spheres
    assert (a["stats"]["cand_fallback"] > 0) == (crowd > 256)
