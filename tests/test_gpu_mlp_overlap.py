"""Training steps whose launches overlap against the same steps one call at a
time, where every launch follows the last call's synchronisation.

Every reduction has a fixed order, so the two are equal bit for bit; a launch
that read weights, partial gradients or the cursor too early would differ.
The batch is all rows: a call starts at row 0.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


# one row, a ragged second tile, fewer tiles than SMs, two tiles and a ragged third for some CTAs
@pytest.mark.parametrize("n", [1, 130, 8192, 2 * 152 * 128 + 5])
@pytest.mark.parametrize("own_stream", [False, True])
def test_overlapped_steps_equal_single_steps(n, own_stream):
    from paper_2403_18761_gb300 import Mlp
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.normal(0, 1, (n, 30)).astype(np.float32)).cuda()
    t = torch.sin(2 * x[:, 0]) + 0.5 * x[:, 1] ** 2
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if own_stream else None
    a, b = Mlp(n_in=30, seed=7, stream=stream), Mlp(n_in=30, seed=7, stream=stream)
    steps = 40
    last = a.train(x, t, steps, batch=n)
    for _ in range(steps):
        one = b.train(x, t, 1, batch=n)
    assert last == one
    assert torch.equal(a.params(), b.params())
