"""A batch takes up to 5600 spheres per shape, and refuses one more."""
import numpy as np
import pytest
import torch

from paper_2403_18761_gb300 import RpdError, rpd_build, rpd_build_batch
from paper_2403_18761_gb300.rpd import collect
from rpd_inputs import block_c2, torus_c1

pytestmark = pytest.mark.gpu


def test_spheres_per_shape():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    w, u = block_c2(h=0.06, ns=5601), torus_c1()   # small tets: at most 32 candidates each
    big = (w.verts, w.tets, w.centers[:5600], w.radii[:5600])
    small = (u.verts, u.tets, u.centers, u.radii)
    a = collect(rpd_build_batch([small, big], k=32, grid_bits=18))
    one = collect(rpd_build(*big, k=32, grid_bits=18))
    assert np.array_equal(a["vol"][-len(one["vol"]):], one["vol"])
    with pytest.raises(RpdError):
        rpd_build_batch([small, (w.verts, w.tets, w.centers, w.radii)], k=32, grid_bits=18)
