"""The batch rows of a training run: launches that overlap hand the cursor (the
next batch's first row) from one step to the next, wrapping around the data.

Against the same steps one call at a time on the batch's rows gathered
beforehand: every reduction has a fixed order, so the two are equal bit for bit,
and a step that read the cursor, the weights or the Adam moments of an earlier
step would differ.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


# batches that do not divide the rows: small and large, nearly all rows, more tiles than SMs
@pytest.mark.parametrize("n,batch", [(7, 3), (129, 128), (3001, 1024), (20011, 8192), (40000, 152 * 128 + 1)])
def test_overlapped_batches_equal_gathered_batches(n, batch):
    from paper_2403_18761_gb300 import Mlp
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.normal(0, 1, (n, 30)).astype(np.float32)).cuda()
    t = torch.sin(2 * x[:, 0]) + 0.5 * x[:, 1] ** 2
    a, b = Mlp(n_in=30, seed=7), Mlp(n_in=30, seed=7)
    steps = 40
    last = a.train(x, t, steps, batch=batch)
    for i in range(steps):
        rows = (i * batch + torch.arange(batch, device="cuda")) % n
        one = b.train(x[rows].contiguous(), t[rows].contiguous(), 1, batch=batch)
    assert last == one
    assert torch.equal(a.params(), b.params())
