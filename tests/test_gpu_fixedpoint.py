"""The FP64 element operator's fixed-point contractions (degrees 2..15).

Bound, entry by entry: B = (c |K| terms + lambda M) |u| of the node's three
lines.  The direct FP64 kernel rounds every term once, so it stays within
(2 Nq + 4) 2^-53 B of the exact value; the digits are held to the same bound
wherever a column of the element does not fall more than 2^-8 below its
largest value (otherwise the element takes the FP64 sums), and the two may
differ by twice it, with the factor two of margin that the entrywise operator
tests use.
"""
import numpy as np
import pytest
import torch

from paper_2009_10917_gb300 import bs, synth
from tests import fem_ref

pytestmark = pytest.mark.gpu


@pytest.fixture
def mode():
    prev = bs.operator_mode(-1)
    yield bs.operator_mode
    bs.operator_mode(prev)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def lines(N, h, lam, coef, u):
    """B per local node."""
    _, w, D = fem_ref.gll_np(N)
    n, g = N + 1, 0.5 * h
    Ka = np.abs(D.T) @ np.diag(w) @ np.abs(D)
    a = np.abs(u).reshape(-1, n, n, n)
    b = (np.einsum("im,ekjm->ekji", Ka, a) * np.outer(w, w)[None, :, :, None]
         + np.einsum("jm,ekmi->ekji", Ka, a) * np.outer(w, w)[None, :, None, :]
         + np.einsum("km,emji->ekji", Ka, a) * np.outer(w, w)[None, None, :, :])
    w3 = w[:, None, None] * w[None, :, None] * w[None, None, :]
    return (coef[:, None, None, None] * g * b + lam * g ** 3 * w3 * a).reshape(-1)


def values(kind, m):
    u = synth.uniform(m.NL, 21)
    e = np.repeat(np.arange(m.E), m.Np)
    if kind == "column edge":  # columns 2^-7 (digits) or 2^-9 (FP64 sums) below the rest
        q = np.arange(m.NL) % (m.Nq ** 2)
        return u * np.where(q % 3 == 1, np.where(e % 2, 2.0 ** -9, 2.0 ** -7), 1.0)
    if kind == "graded":
        return u * np.exp(4.0 * synth.normal(m.NL, 5))
    if kind == "extremes":  # element by element: zero, subnormal, tiny, huge, one value alone
        scale = np.array([0.0, 2.0 ** -1060, 2.0 ** -905, 2.0 ** 905, 1.0, -3.0])[e % 6]
        u = u * scale
        u[(e % 6 == 4) & (np.arange(m.NL) % m.Np != m.Np // 2)] = 0.0
        return u
    if kind == "ones":
        return np.ones(m.NL)
    return u


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 11, 12, 15])
@pytest.mark.parametrize("kind", ["uniform", "ones", "column edge", "graded", "extremes"])
@pytest.mark.parametrize("with_coef", [False, True])
def test_local_operator_entrywise(mode, N, kind, with_coef):
    m = synth.Mesh(2 if N > 3 else 3, N, seed=N)  # 27 elements: not full warps of four
    lam = 0.4
    coef = synth.lognormal(m.E, 2) if with_coef else np.ones(m.E)
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam, coef if with_coef else None)
    u = values(kind, m)
    bound = 4 * (2 * (N + 1) + 4) * 2.0 ** -53 * lines(N, m.h, lam, coef, u)
    got = P.apply_local(cuda(u)).cpu().numpy()
    odd = torch.zeros(m.NL + 1, dtype=torch.float64, device="cuda")  # 8-byte aligned only
    odd[1:] = cuda(u)
    assert np.array_equal(P.apply_local(odd[1:]).cpu().numpy(), got)
    mode(bs.BS_OP_DIRECT)
    want = P.apply_local(cuda(u)).cpu().numpy()
    assert np.all(np.abs(got - want) <= bound + 2.0 ** -1070)


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 11, 12, 15])
def test_not_finite_values_stay_in_their_lines(mode, N):
    m = synth.Mesh(2, N, seed=1)
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, 1.0)
    u = synth.uniform(m.NL, 3)
    u[m.Np // 2] = np.inf
    u[3 * m.Np + 1] = np.nan
    got = P.apply_local(cuda(u)).cpu().numpy()
    mode(bs.BS_OP_DIRECT)
    want = P.apply_local(cuda(u)).cpu().numpy()
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
    assert np.array_equal(np.isnan(got), np.isnan(want))
    assert np.array_equal(got[np.isinf(got)], want[np.isinf(want)])


@pytest.mark.parametrize("N", [5, 6, 7])
@pytest.mark.parametrize("kind", ["uniform", "ones", "graded", "extremes"])
@pytest.mark.parametrize("with_coef", [False, True])
def test_general_hexahedra_entrywise(mode, N, kind, with_coef):
    """The same against the direct FP64 kernel on perturbed hexahedra.  Each
    gradient and flux component is a line sum within (Nq + 2) 2^-53 of the sum
    of its terms' sizes and is carried on through at most Nq + 3 more terms, so
    an entry is off by at most (2 Nq + 8) 2^-53 of B, the sum of |D|^T |G| |D|
    |u| and the mass term over the element -- here with the lines' terms
    replaced by the element's largest gradient and flux, as the digits are
    relative to those -- for either kernel; a factor two of margin."""
    m = synth.Mesh(2, N, seed=N, perturb=0.2)
    lam = 0.4
    coef = synth.lognormal(m.E, 2) if with_coef else np.ones(m.E)
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam, coef if with_coef else None,
                   verts=m.verts())
    u = values(kind, m)
    _, w, D = fem_ref.gll_np(N)
    rows, cols = np.abs(D).sum(1).max(), np.abs(D).sum(0).max()
    # |G| <= w_max (edge)^2 / det-scale: bounded through the affine size, the
    # perturbation (0.2) at most quadruples it
    big = np.abs(u).reshape(m.E, -1).max(1)
    B = coef * 3 * cols * 4 * 3 * m.h * w.max() ** 3 * rows * big + lam * m.h ** 3 * big
    got = P.apply_local(cuda(u)).cpu().numpy().reshape(m.E, -1)
    odd = torch.zeros(m.NL + 1, dtype=torch.float64, device="cuda")
    odd[1:] = cuda(u)
    assert np.array_equal(P.apply_local(odd[1:]).cpu().numpy(), got.reshape(-1))
    mode(bs.BS_OP_DIRECT)
    want = P.apply_local(cuda(u)).cpu().numpy().reshape(m.E, -1)
    bound = 4 * (2 * (N + 1) + 8) * 2.0 ** -53 * B
    assert np.all(np.abs(got - want) <= bound[:, None] + 2.0 ** -1070)


def test_general_hexahedra_not_finite(mode):
    m = synth.Mesh(2, 7, seed=1, perturb=0.2)
    P = bs.Problem(bs.Map(m.E, 7, m.NG, m.ids), m.h, 1.0, verts=m.verts())
    u = synth.uniform(m.NL, 3)
    u[m.Np // 2] = np.inf
    u[3 * m.Np + 1] = np.nan
    got = P.apply_local(cuda(u)).cpu().numpy()
    mode(bs.BS_OP_DIRECT)
    want = P.apply_local(cuda(u)).cpu().numpy()
    assert np.array_equal(np.isfinite(got), np.isfinite(want))
