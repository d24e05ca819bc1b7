"""The network's sums in the order and with the precision that its results are
defined by, bit for bit or within derived bounds.

The weights are chosen so that everything before a sum is exact: small whole
inputs, a W0 of zeros and ones, W1 and W2 the identity, so that all three
hidden layers hold the same small whole numbers (exact in bfloat16 whatever the
tensor cores' order), and w3 of ten significant bits, whose products with them
are exact in FP32.
"""
import numpy as np
import pytest
import torch

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


def _exact_net(n, seed):
    """A network with exact hidden layers, its inputs, and their activations (float32)."""
    from paper_2403_18761_gb300 import Mlp
    rng = np.random.default_rng(seed)
    x = rng.integers(0, 4, (n, 30)).astype(np.float32)
    p = np.zeros(ref.NPARAM, dtype=np.float32)
    w0 = np.zeros((ref.HID, ref.NIN), dtype=np.float32)
    w0[:, :30] = rng.random((ref.HID, 30)) < 0.3
    p[ref.OW0:ref.OB0] = w0.ravel()
    p[ref.OW1:ref.OB1] = p[ref.OW2:ref.OB2] = np.eye(ref.HID, dtype=np.float32).ravel()
    p[ref.OW3:ref.OB3] = np.ldexp(rng.integers(512, 1024, ref.HID), rng.integers(-20, 4, ref.HID)) * rng.choice((-1, 1), ref.HID)
    p[ref.OB3] = 0.5
    net = Mlp(n_in=30, seed=1)
    net.set_params(torch.from_numpy(p).cuda())
    h = x @ w0[:, :30].T
    assert h.max() <= 256   # whole numbers that bfloat16 holds
    return net, p, x, h


def _head(h, w3, b3):
    """y in the head's order: groups of four columns in turn, then the groups
    16, 8, 4, 2 and 1 apart (every product is exact in FP32)."""
    prod = (h * w3).reshape(len(h), 32, 4)
    s = prod[:, :, 0]
    for q in (1, 2, 3):
        s = s + prod[:, :, q]
    for off in (16, 8, 4, 2, 1):
        s = s[:, :off] + s[:, off:2 * off]
    assert s.dtype == np.float32
    return s[:, 0] + b3


@pytest.mark.parametrize("n", [1, 127, 128, 1000])
def test_head_order(n):
    net, p, x, h = _exact_net(n, 21)
    y = net.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    assert np.array_equal(y, _head(h, p[ref.OW3:ref.OB3], p[ref.OB3]))
