"""A training batch with more tiles than the loss has partial sums (4096 of 64
rows): its loss comes from a kernel of its own.  Against the same rows in two
halves, whose loss is an epilogue: the mean of the two losses, FP64 sums of the
same errors (1e-12), and the mean of the gradients, FP32 sums of 2^18 products
of one sign here (targets zero, inputs and weights positive: 2^18 2^-24 relative
in the worst order)."""
import numpy as np
import pytest
import torch

from paper_2009_10917_gb300 import bs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split", [False, True])
def test_loss_of_more_tiles_than_partials(split):
    D, H, B = 8, 32, 2 * 64 * 2052
    rng = np.random.default_rng(3)
    net = bs.MLP(rng.uniform(0.1, 1, (H, D)).astype(np.float32),
                 rng.uniform(0.1, 1, (D, H)).astype(np.float32), split=split)
    X = torch.from_numpy(rng.uniform(0.1, 1, (B, D)).astype(np.float32)).cuda()
    T = torch.zeros_like(X)
    loss, g1, g2 = net.loss_grad(X, T)
    halves = [net.loss_grad(X[i:i + B // 2], T[i:i + B // 2]) for i in (0, B // 2)]
    want = 0.5 * (float(halves[0][0]) + float(halves[1][0]))
    assert abs(float(loss) - want) <= 1e-12 * want
    for got, a, b in ((g1, halves[0][1], halves[1][1]), (g2, halves[0][2], halves[1][2])):
        mean = 0.5 * (a.double() + b.double())
        assert torch.all((got.double() - mean).abs() <= 2.0 ** -5 * mean.abs())
