"""bs_apply_A_ff entry by entry on values that differ widely inside an element, at
the degrees where the fixed-point kernel runs in place of the float-float one:
within 2^-42 of the sum of the sizes of an entry's own terms, as the float-float
tests ask (the kernel lets the digits be off by 16 (2 Nq + 4) 2^-53 at most, below
2^-43 for all degrees)."""
import numpy as np
import pytest

from paper_2009_10917_gb300 import bs, synth
from tests.test_gpu_fixedpoint_entries import KINDS, LD, cuda, operator, values

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [6, 7, 11, 13, 15])
@pytest.mark.parametrize("dirichlet", [False, True])
def test_float_float_entries(N, dirichlet):
    m = synth.Mesh(2, N, seed=N, dirichlet=dirichlet)
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, 0.4)
    live = m.ids >= 0
    for kind in KINDS:
        for axis in range(3):
            p = np.zeros(m.NG)
            p[m.ids[live]] = values(kind, axis, m)[live]
            u = np.where(live, p[np.maximum(m.ids, 0)], 0.0)
            y, T = operator(N, m.h, 0.4, np.ones(m.E), u)
            want, bound = np.zeros(m.NG, LD), np.zeros(m.NG, LD)
            np.add.at(want, m.ids[live], y[live])
            np.add.at(bound, m.ids[live], T[live])
            got = P.apply_A_ff(cuda(p)).cpu().numpy()
            assert np.all(np.abs(got - want) <= LD(2) ** -42 * bound), (kind, axis)
