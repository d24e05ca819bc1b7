"""The clip's first stage (csrc/clip.cu) in the bins that keep the planes' rows in
shared memory and in those that compute them again, against the exact stage for
every predicate (debug value 2): the combinatorial tables and the set of pieces
must be the same.  Both precisions, few and many candidates per tet.

Volumes come from the same vertices in either form: equal up to the rounding of
the volume pass (double-float or FP64, 1e-9 of the largest piece at most).
"""
import numpy as np
import pytest
import torch

from paper_2403_18761_gb300 import rpd_build
from paper_2403_18761_gb300.rpd import collect
from rpd_inputs import block_c2

pytestmark = pytest.mark.gpu


# most pairs with 3 to 8, 9 to 16, and 9 to 32 candidates
@pytest.mark.parametrize("ns", [150, 1500, 4000])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_rows(ns, precision):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w = block_c2(h=0.15, ns=10)
    rng = np.random.default_rng(ns)
    c = rng.uniform(w.verts.min(axis=0), w.verts.max(axis=0), (ns, 3))
    r = rng.uniform(0.05, 0.06, ns)
    a, b = (collect(rpd_build(w.verts, w.tets, c, r, precision=precision, k=32, grid_bits=w.grid_bits, debug=d))
            for d in (0, 2))
    for kind in (1, 2, 3, 4):
        for f in ("keys", "chi", "beta0", "flag"):
            assert np.array_equal(a["kinds"][kind][f], b["kinds"][kind][f]), (kind, f)
    assert np.array_equal(a["tet"], b["tet"]) and np.array_equal(a["sphere"], b["sphere"])
    assert np.abs(a["vol"] - b["vol"]).max() <= 1e-9 * b["vol"].max()
    bins = a["stats"]["bin_pairs"]
    assert max(bins[2:6]) > 1000 if ns == 150 else bins[6] > 5000
    assert bins[7] > 0 or ns < 4000
