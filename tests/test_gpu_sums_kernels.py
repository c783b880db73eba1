"""The even-odd FP64 and float-float element kernels, and the float-float one on
general hexahedra, at the degrees where the fixed-point kernels run by default.

The even-odd kernels serve flexible PCG with a network at those degrees.  A
network of zeros adds nothing to the Jacobi correction, so three iterations
are the oracle's Jacobi-preconditioned ones: the operators' errors, 2^-46
(float-float 2^-42) of |A| |u|, grow by the condition of the three coefficients,
below 1e3 on these meshes, so x agrees within 1e-10 (1e-9) of its norm.  That the
fixed-point kernels did not run shows in the last bits.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2009_10917_gb300 import bs, synth

pytestmark = pytest.mark.gpu


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.fixture
def mode():
    prev = bs.operator_mode(-1)
    yield bs.operator_mode
    bs.operator_mode(prev)


@pytest.mark.parametrize("K,N,ff", [(5, 3, False), (4, 5, False), (3, 7, False), (2, 9, False),
                                    (3, 6, True), (3, 7, True)])
@pytest.mark.parametrize("with_coef", [False, True])
def test_learned_pcg_operators(K, N, ff, with_coef):
    m = synth.Mesh(K, N, seed=3)
    lam = 0.3
    coef = synth.lognormal(m.E, 5) if with_coef else None
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam, coef)
    D = (N + 1) ** 3
    zeros = bs.MLP(np.zeros((32, D), np.float32), np.zeros((D, 32), np.float32))
    b = synth.uniform(m.NG, 8)
    flags = bs.BS_CG_FF_OPERATOR if ff else 0
    x, _ = bs.fpcg_learned(P, zeros, cuda(b), tol=0.0, maxit=3, flags=flags, check=False)
    want = oracle.fpcg(m.E, N, m.h, lam, m.ids, m.NG, b, tol=0.0, maxit=3, coef=coef)[0]
    err = np.linalg.norm(x.cpu().numpy() - want)
    assert err <= (1e-9 if ff else 1e-10) * np.linalg.norm(want)
    y, _ = bs.fpcg_learned(P, None, cuda(b), tol=0.0, maxit=3, flags=flags, check=False)
    assert not torch.equal(x, y)


@pytest.mark.parametrize("K,N", [(2, 5), (2, 6), (2, 7)])
@pytest.mark.parametrize("with_coef", [False, True])
def test_geo_float_float_apply_direct(mode, K, N, with_coef):
    """As the general-hexahedron tests: within 1e-11 max|A p| of the oracle."""
    m = synth.Mesh(K, N, seed=3, perturb=0.2)
    c = synth.lognormal(m.E, 4) if with_coef else None
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, 0.5, c, verts=m.verts())
    p = synth.uniform(m.NG, 5)
    mode(bs.BS_OP_DIRECT)
    got = P.apply_A_ff(cuda(p))
    want = oracle.apply_A_geo(m.E, N, 0.5, m.verts(), m.ids, m.NG, p, c)
    assert np.abs(got.cpu().numpy() - want).max() <= 1e-11 * np.abs(want).max()
    assert not torch.equal(P.apply_A(cuda(p)), got)
