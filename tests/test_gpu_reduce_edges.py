"""Reductions on both sides of the sizes where one block gives way to several:
16, 13 and 6 vectors (two FP64 or four FP32 values) for each of 256 threads.

FP64 sums of n <= 2^15 products: within n 2^-53 of the sum of their sizes in any
order, plus the products' own rounding.  The FP32 forms carry float pairs: 2^-40
of it.  A repeated call gives the same bits."""
import math

import pytest
import torch

from paper_2009_10917_gb300 import bs, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("most", [6, 13, 16])
@pytest.mark.parametrize("off", [-1, 0, 1, 2, 5])
@pytest.mark.parametrize("shift", [0, 1])  # operands of different alignment: value by value
def test_around_the_line(dtype, most, off, shift):
    w = 2 if dtype == torch.float64 else 4
    n = (most * 256 if shift else most * 256 * w) + off
    x, y, p, q = [torch.from_numpy(synth.uniform(n + 1, 5 + i)).to(dtype).cuda()[o:n + o]
                  for i, o in enumerate((shift, 0, shift, 0))]
    eps = n * 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -40

    def exact(a, b):
        t = [u * v for u, v in zip(a.double().tolist(), b.double().tolist())]
        return math.fsum(t), math.fsum(map(abs, t))
    s, size = exact(x, y)
    d = bs.dot(x, y)
    assert abs(d.item() - s) <= eps * size
    assert torch.equal(d, bs.dot(x, y))
    s, size = exact(x, x)
    v = bs.norm(x)
    assert abs(v[0].item() - s) <= eps * size and abs(v[1].item() - s ** 0.5) <= eps * s ** 0.5
    xx, r = p.clone(), q.clone()
    rr = bs.cg_update(0.25, x, y, xx, r)
    s, size = exact(r, r)
    assert abs(rr.item() - s) <= eps * size
