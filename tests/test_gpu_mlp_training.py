"""A hundred training steps against a replay with the same bfloat16 roundings, sums
in FP64 and Adam in FP32 (torch).

Both round the same values to bfloat16; their gradients differ by the rounding of
FP32 sums (1e-7 in norm), and training amplifies that one flipped bfloat16
rounding at a time.  Two runs whose FP32 sums only differ in their order are
1.3e-4 apart in the parameters after 100 steps of 8192 rows (2-norm of the
difference over the 2-norm; up to 1.6e-4 over the seeds measured), and their last losses
scatter by 7.2e-5 (one standard deviation, relative).  The bounds are three times the
former's largest and seven of the latter.
"""
import pytest
import torch

from oracle import mlp as ref

pytestmark = pytest.mark.gpu

BLOCKS = {"W0": (ref.OW0, ref.OB0), "b0": (ref.OB0, ref.OW1), "W1": (ref.OW1, ref.OB1), "b1": (ref.OB1, ref.OW2),
          "W2": (ref.OW2, ref.OB2), "b2": (ref.OB2, ref.OW3), "w3": (ref.OW3, ref.OB3), "b3": (ref.OB3, ref.NPARAM)}


def _grad(p, x, t):
    """Gradient and loss in FP64 from FP32 parameters, bfloat16 where the library rounds."""
    def bf(a):
        return a.float().bfloat16().double()
    W = {k: p[a:b].double() for k, (a, b) in BLOCKS.items()}
    W0, W1, W2 = bf(W["W0"]).view(128, 32)[:, :30], bf(W["W1"]).view(128, 128), bf(W["W2"]).view(128, 128)
    X = bf(x)
    H0 = bf((X @ W0.T + W["b0"]).clamp(min=0))
    H1 = bf((H0 @ W1.T + W["b1"]).clamp(min=0))
    H2 = bf((H1 @ W2.T + W["b2"]).clamp(min=0))
    e = H2 @ W["w3"] + W["b3"] - t.double()
    dy = 2 * e / len(x)
    Z2 = bf(torch.outer(dy, W["w3"]) * (H2 > 0))
    Z1 = bf((Z2 @ W2) * (H1 > 0))
    Z0 = bf((Z1 @ W1) * (H0 > 0))
    g0 = torch.zeros(128, 32, dtype=torch.float64, device=p.device)
    g0[:, :30] = Z0.T @ X
    parts = [g0, Z0.sum(0), Z1.T @ H0, Z1.sum(0), Z2.T @ H1, Z2.sum(0), dy @ H2, dy.sum()]
    return torch.cat([a.reshape(-1) for a in parts]).float(), float((e * e).mean())


@pytest.mark.parametrize("seed", [1, 2, 3])
def test_hundred_steps(seed):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2403_18761_gb300 import Mlp
    n, batch, steps, lr = 20000, 8192, 100, 1e-3
    gen = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand(n, 30, device="cuda", generator=gen) * 2 - 1
    t = torch.sin(2 * x[:, 0]) + 0.5 * x[:, 1] * x[:, 2] - 2
    net = Mlp(n_in=30, seed=seed)
    p = net.params().clone()
    loss = net.train(x, t, steps, batch=batch, lr=lr)
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    for i in range(steps):
        rows = (i * batch + torch.arange(batch, device="cuda")) % n
        g, want = _grad(p, x[rows], t[rows])
        m = 0.9 * m + (1 - 0.9) * g
        v = 0.999 * v + (1 - 0.999) * g * g
        p = p - lr * (m / (1 - 0.9 ** (i + 1))) / (torch.sqrt(v / (1 - 0.999 ** (i + 1))) + 1e-8)
    got = net.params()
    assert float((got - p).norm() / p.norm()) <= 3 * 1.6e-4
    assert abs(loss - want) <= 7 * 7.2e-5 * want
