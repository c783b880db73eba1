"""The small-tile GEMMs of a training step at the edges of their tiles.

Gradients: the entrywise bounds of test_gradients_element_by_element (their
derivation holds for any D, H and batch).  Adam: the step's arithmetic is
plain FP32 (no contraction), so the weights after a step from zero moments
are bitwise numpy's float32 evaluation on the gradients that loss_grad
returns (the same products in the same order), and the refreshed operands
give bitwise the forward pass of a new network made from those weights.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2009_10917_gb300 import bs, synth

pytestmark = pytest.mark.gpu

SHAPES = [(8, 32, 32), (27, 96, 32), (125, 64, 160), (216, 256, 96), (343, 32, 64),
          (100, 160, 10240)]  # the last one: 64 x 64 tiles


def data(D, H, B):
    W1 = (synth.uniform(H * D, 42, 0).reshape(H, D) * np.sqrt(3.0 / D)).astype(np.float32)
    W2 = (synth.uniform(D * H, 42, 1).reshape(D, H) * np.sqrt(3.0 / H)).astype(np.float32)
    X = synth.uniform(B * D, 43).reshape(B, D).astype(np.float32)
    T = synth.uniform(B * D, 44).reshape(B, D).astype(np.float32)
    return W1, W2, X, T


@pytest.mark.parametrize("D,H,B", SHAPES)
def test_gradients_at_tile_edges(D, H, B):
    W1, W2, X, T = data(D, H, B)
    net = bs.MLP(W1, W2)
    loss, g1, g2 = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    g1, g2 = g1.cpu().numpy().astype(np.float64), g2.cpu().numpy().astype(np.float64)
    lo, g1o, g2o = oracle.mlp_loss_grad(W1, W2, X, T, prec=oracle.PREC_BF16)
    Yo, _ = oracle.mlp_forward(W1, W2, X, prec=oracle.PREC_BF16)
    xb, w1b, w2b = (oracle.bf16_round(a).astype(np.float64) for a in (X, W1, W2))
    h = np.maximum(xb @ w1b.T, 0.0)
    scale = 2.0 / (B * D)
    dy = scale * (Yo - T.astype(np.float64))
    Sy = h @ np.abs(w2b.T)
    bound2 = 2.0 ** -6 * (np.abs(dy).T @ h) + scale * 2.0 ** -7 * (Sy.T @ h)
    assert np.all(np.abs(g2 - g2o) <= bound2 + 1e-30)
    mask = (xb @ w1b.T) > 0.0
    S1 = (mask * (np.abs(dy) @ np.abs(w2b))).T @ np.abs(xb)
    E1 = (mask * (scale * 2.0 ** -7 * Sy @ np.abs(w2b))).T @ np.abs(xb)
    assert np.mean(np.abs(g1 - g1o) <= 2.0 ** -6 * S1 + E1 + 1e-30) >= 0.99
    assert abs(loss.item() - lo) <= 2.0 ** -6 * (np.mean(Sy * np.abs(Yo - T)) + lo)


@pytest.mark.parametrize("D,H,B", SHAPES)
@pytest.mark.parametrize("split", [False, True])
def test_adam_and_operands_are_bitwise(D, H, B, split):
    W1, W2, X, T = data(D, H, B)
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    net, lr = bs.MLP(W1, W2, split=split), 1e-3
    loss, g1, g2 = net.loss_grad(Xd, Td)
    assert torch.equal(net.train_step(Xd, Td, lr), loss)
    f = np.float32
    b1, b2, eps, one = f(0.9), f(0.999), f(1e-8), f(1.0)
    for w, g, got in zip((W1, W2), (g1, g2), net.weights()):
        g = g.cpu().numpy()
        m = b1 * f(0.0) + (one - b1) * g
        v = b2 * f(0.0) + (one - b2) * g * g
        want = w - f(lr) * (m / (one - b1)) / (np.sqrt(v / (one - b2)) + eps)
        assert np.array_equal(got, want)
    again = bs.MLP(*net.weights(), split=split)
    assert torch.equal(net.forward(Xd), again.forward(Xd))
