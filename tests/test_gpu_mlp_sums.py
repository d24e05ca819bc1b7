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


U = 2.0 ** -24   # half a unit in the last place of FP32


# one row; ragged tiles; a tile per CTA; a CTA with two tiles; a hundred tiles and more per CTA
@pytest.mark.parametrize("n", [1, 130, 8192, 152 * 128 + 5, 2_000_000])
def test_gradient_sums(n):
    """Every gradient against its terms' sum in 64 bits.  All residuals are
    positive, so a sum's terms have one sign and its relative error is at most
    that of its chain of additions: within a tile eight MMAs, each rounding
    its running sum towards zero (2 U) and aligning its products to it (2 U
    more), or, for the biases and w3, 64 rows (w3's products are rounded too) and the other half; then the
    CTA's tiles, the 19 partials of a group and the 8 groups (U each)."""
    net, p, x, h = _exact_net(n, 22)
    f, dev = torch.float64, "cuda"
    X = torch.from_numpy(x).cuda()
    H = torch.from_numpy(h).cuda()
    y = net.forward(X)
    t = y - (1 + torch.rand(n, device=dev, generator=torch.Generator(device=dev).manual_seed(n)))
    g, loss = net.grad(X, t)
    w3 = torch.from_numpy(p[ref.OW3:ref.OB3]).cuda()
    dy = 2 * (y - t) / torch.full_like(y, n)   # (a division, as the kernel has; by a scalar torch multiplies)
    assert float(dy.min()) > 0
    want = torch.zeros(ref.NPARAM, dtype=f, device=dev)
    ww = torch.zeros((3, ref.HID, ref.HID), dtype=f, device=dev)
    bb = torch.zeros((3, ref.HID), dtype=f, device=dev)
    for a in range(0, n, 100_000):
        d, hh, xx = dy[a:a + 100_000], H[a:a + 100_000].to(f), X[a:a + 100_000].to(f)
        want[ref.OW3:ref.OB3] += d.to(f) @ hh
        want[ref.OB3] += d.to(f).sum()
        # W1 and W2 are the identity: dZ2 = dZ1 = dZ0
        z = ((d[:, None] * w3) * (hh > 0)).bfloat16().to(f)
        ww[:2] += z.T @ hh
        ww[2][:, :30] += z.T @ xx
        bb += z.sum(0)
    want[ref.OW2:ref.OB2], want[ref.OW1:ref.OB1] = ww[0].flatten(), ww[1].flatten()
    want[ref.OW0:ref.OB0] = ww[2][:, :32].flatten()
    want[ref.OB2:ref.OW3], want[ref.OB1:ref.OW2], want[ref.OB0:ref.OW1] = bb[0], bb[1], bb[2]
    tiles = -(-n // 128)
    across = -(-tiles // 152) + 19 + 8
    off = (g.to(f) - want).abs()
    for lo, hi, chain in ((ref.OW0, ref.OB0, 32), (ref.OW1, ref.OB1, 32), (ref.OW2, ref.OB2, 32), (ref.OB0, ref.OW1, 65),
                          (ref.OB1, ref.OW2, 65), (ref.OB2, ref.OW3, 65), (ref.OW3, ref.NPARAM, 66)):
        assert bool((off[lo:hi] <= (chain + across) * U * want[lo:hi].abs()).all()), (lo, float((off[lo:hi] / want[lo:hi].abs()).nan_to_num().max()))
