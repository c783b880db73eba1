"""A p entry by entry on values that differ widely inside an element.

The fixed-point contractions (degrees 2..15) round relative to an element's
largest value; nodes whose own terms are too small for that take FP64 sums.
Either way an entry is within (2 Nq + 4) 2^-53 of the sum T of the sizes of
its own terms: three sums of Nq products and a few more roundings in FP64, and
the digits wherever the kernel finds T large enough.  The reference is the
same sum in extended precision (at least 64 bits), from quadrature tables made
in it (the oracle's, in double, are themselves off by up to 50 times this).
On general hexahedra an entry is within (2 Nq + 8) 2^-53 of B(|D|), the sum over
its lines of |D|^T |G| |D| |u| and the mass term, and so is the direct FP64 kernel
with the same G but for its table: its D, made in double, is off by up to 8 2^-53
of an entry, on the diagonal of its row's sum of sizes (the differences of nodes
alone by 7 2^-53).  With |D| + that diagonal as E the two kernels are within
2 (2 Nq + 8) 2^-53 B(|D|) + 16 2^-53 B(E).
"""
import numpy as np
import pytest
import torch

from paper_2009_10917_gb300 import bs, synth
from tests import fem_ref

pytestmark = pytest.mark.gpu
LD = np.longdouble


@pytest.fixture
def mode():
    prev = bs.operator_mode(-1)
    yield bs.operator_mode
    bs.operator_mode(prev)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def tables(N):
    """Nodes, weights and D in extended precision."""
    x0, _, _ = fem_ref.gll_np(N)
    x = x0.astype(LD)

    def legendre(z):
        p, q = np.ones_like(z), z
        for k in range(2, N + 1):
            p, q = q, ((2 * k - 1) * z * q - (k - 1) * p) / LD(k)
        return q, p
    for _ in range(4):
        pn, pm = legendre(x)
        x = x - (x * pn - pm) / ((N + 1) * pn)
    w = LD(2) / (N * (N + 1) * legendre(x)[0] ** 2)
    d = x[:, None] - x[None, :] + np.eye(N + 1, dtype=LD)
    b = LD(1) / d.prod(1)
    D = b[None, :] / b[:, None] / d
    np.fill_diagonal(D, 0)
    np.fill_diagonal(D, -D.sum(1))
    return x, w, D


def operator(N, h, lam, coef, u):
    """A_L u and T, node by node, in extended precision."""
    _, w, D = tables(N)
    Kh = (D.T @ (w[:, None] * D)) / w[:, None]
    n, g = N + 1, LD(0.5) * LD(h)
    w3 = w[:, None, None] * w[None, :, None] * w[None, None, :]
    c = coef.astype(LD)[:, None, None, None] * g

    def apply(M, v):
        s = (np.einsum("im,ekjm->ekji", M, v) + np.einsum("jm,ekmi->ekji", M, v)
             + np.einsum("km,emji->ekji", M, v))
        return (w3 * (c * s + LD(lam) * g ** 3 * v)).reshape(-1)
    v = u.astype(LD).reshape(-1, n, n, n)
    return apply(Kh, v), apply(np.abs(Kh), np.abs(v))


KINDS = ["one column", "two columns", "graded", "layer", "mild layer", "columns below",
         "layers and a zero column", "bump", "random grading"]


def values(kind, axis, m):
    """Element values [E, k, j, i], the structure along `axis` (0: r)."""
    n, E = m.Nq, m.E
    r, _, _ = fem_ref.gll_np(m.N)
    u = synth.uniform(m.NL, 7).reshape(E, n, n, n)
    t = np.arange(n)[None, :, None, None]  # the structure's direction, first of three
    a, b = np.arange(n)[None, None, :, None], np.arange(n)[None, None, None, :]
    s = r[None, :, None, None]
    if kind == "one column":  # 2^-6 a node along one line, zeros elsewhere
        v = np.where((a == n // 2) & (b == 1), 2.0 ** (-6.0 * t), 0.0) * u
    elif kind == "two columns":  # one of ones, one graded
        v = (np.where((a == n // 2) & (b == 1), 2.0 ** (-6.0 * t), 0.0)
             + np.where((a == 0) & (b == n - 1), 1.0, 0.0)) * u
    elif kind == "graded":
        v = 2.0 ** (-5.0 * t) * u
    elif kind == "layer":
        v = np.exp(-12.0 * s) * (1 + 0.1 * u)
    elif kind == "mild layer":
        v = np.exp(-2.7 * s) * (1 + 0.1 * u)
    elif kind == "columns below":
        v = u * np.where((a + b) % 3 == 1, 2.0 ** -7, 1.0)
    elif kind == "layers and a zero column":
        v = u * np.where(t == 0, 1.0, 2.0 ** -(52.0 + t)) * np.where((a == 1) & (b == 1), 0.0, 1.0)
    elif kind == "bump":
        v = np.exp(-20.0 * (s ** 2 + (r[None, None, :, None] - 0.4) ** 2
                            + r[None, None, None, :] ** 2)) * np.ones((E, 1, 1, 1))
    else:
        v = u * np.exp(3.0 * synth.normal(m.NL, 9).reshape(E, n, n, n))
    v = np.broadcast_to(v, (E, n, n, n)) * 2.0 ** np.arange(-E // 2, E - E // 2)[:, None, None, None]
    order = {0: (0, 2, 3, 1), 1: (0, 2, 1, 3), 2: (0, 1, 2, 3)}[axis]
    return np.ascontiguousarray(v.transpose(order)).reshape(-1)


@pytest.mark.parametrize("N", range(1, 16))
@pytest.mark.parametrize("with_coef", [False, True])
def test_local_entries(N, with_coef):
    m = synth.Mesh(2, N, seed=N)
    lam = 0.4
    coef = synth.lognormal(m.E, 2) if with_coef else np.ones(m.E)
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam, coef if with_coef else None)
    for kind in KINDS:
        for axis in range(3):
            u = values(kind, axis, m)
            got = P.apply_local(cuda(u)).cpu().numpy()
            want, T = operator(N, m.h, lam, coef, u)
            bound = (2 * (N + 1) + 4) * LD(2) ** -53 * T
            assert np.all(np.abs(got - want) <= bound), (kind, axis)


@pytest.mark.parametrize("N", [2, 3, 4, 5, 6, 7, 8, 11, 15])
@pytest.mark.parametrize("dirichlet", [False, True])
def test_assembled_entries(mode, N, dirichlet):
    """Through the map, also fused: a global entry adds up to eight local ones,
    seven more roundings."""
    m = synth.Mesh(2, N, seed=N, dirichlet=dirichlet)
    lam = 0.4
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam)
    live = m.ids >= 0
    for kind in KINDS:
        for axis in range(3):
            p = np.zeros(m.NG)
            p[m.ids[live]] = values(kind, axis, m)[live]
            u = np.where(live, p[np.maximum(m.ids, 0)], 0.0)
            y, T = operator(N, m.h, lam, np.ones(m.E), u)
            want, bound = np.zeros(m.NG, LD), np.zeros(m.NG, LD)
            np.add.at(want, m.ids[live], y[live])
            np.add.at(bound, m.ids[live], T[live])
            bound *= (2 * (N + 1) + 4 + 7) * LD(2) ** -53
            mode(0)
            got = P.apply_A(cuda(p)).cpu().numpy()
            assert np.all(np.abs(got - want) <= bound), (kind, axis)
            mode(bs.BS_OP_FUSED)
            assert np.array_equal(P.apply_A(cuda(p)).cpu().numpy(), got)


@pytest.mark.parametrize("N", [5, 6, 7])
@pytest.mark.parametrize("with_coef", [False, True])
def test_general_hexahedra_entries(mode, N, with_coef):
    m = synth.Mesh(2, N, seed=N, perturb=0.2)
    n, lam = N + 1, 0.4
    coef = synth.lognormal(m.E, 2) if with_coef else np.ones(m.E)
    V = m.verts()
    P = bs.Problem(bs.Map(m.E, N, m.NG, m.ids), m.h, lam, coef if with_coef else None, verts=V)
    x, w, D = tables(N)
    # J = dx/dr at every node, G = w / det J C C^T
    q = np.arange(n ** 3)
    r = np.stack([x[q % n], x[q // n % n], x[q // n ** 2]])
    sg = np.array([[1 if v >> d & 1 else -1 for d in range(3)] for v in range(8)])
    f = 1 + sg[:, :, None] * r[None]                              # [8, 3, Np]
    dN = np.stack([sg[:, d, None] * f[:, (d + 1) % 3] * f[:, (d + 2) % 3] / 8 for d in range(3)])
    J = np.einsum("evx,dvp->epxd", V.astype(LD), dN)
    Ja = np.einsum("evx,dvp->epxd", np.abs(V).astype(LD), np.abs(dN))

    def cofactors(J, sign):  # [reference direction, x]
        C = np.zeros_like(J)
        for d in range(3):
            for c in range(3):
                a, b, e, g = (c + 1) % 3, (c + 2) % 3, (d + 1) % 3, (d + 2) % 3
                C[..., d, c] = J[..., a, e] * J[..., b, g] + sign * J[..., a, g] * J[..., b, e]
        return C
    C, Ca = cofactors(J, -1), cofactors(Ja, 1)
    det = np.einsum("epx,epx->ep", J[..., 0], C[..., 0, :])
    wq = w[q % n] * w[q // n % n] * w[q // n ** 2]
    M = (wq * det).reshape(m.E, n, n, n)
    # |G| as the kernels hold it: rounded from the corners (where the exact one is
    # zero, what is left of the sums of its terms' sizes)
    G = (np.abs(np.einsum("epdx,epfx->epdf", C, C))
         + LD(2) ** -49 * np.einsum("epdx,epfx->epdf", Ca, Ca)) * (wq / det)[:, :, None, None]
    G = G.reshape(m.E, n, n, n, 3, 3)

    def B(D, v):
        grad = np.stack([np.einsum("im,ekjm->ekji", D, v), np.einsum("jm,ekmi->ekji", D, v),
                         np.einsum("km,emji->ekji", D, v)], -1)
        fl = np.einsum("ekjidf,ekjif->dekji", G, grad)
        s = (np.einsum("mi,ekjm->ekji", D, fl[0]) + np.einsum("mj,ekmi->ekji", D, fl[1])
             + np.einsum("mk,emji->ekji", D, fl[2]))
        return (coef.astype(LD)[:, None, None, None] * s + LD(lam) * M * v).reshape(-1)
    Da = np.abs(D)
    Ed = Da + np.diag(Da.sum(1))
    for kind in KINDS:
        for axis in range(3):
            u = values(kind, axis, m)
            v = np.abs(u.astype(LD)).reshape(m.E, n, n, n)
            mode(0)
            got = P.apply_local(cuda(u)).cpu().numpy()
            mode(bs.BS_OP_DIRECT)
            want = P.apply_local(cuda(u)).cpu().numpy()
            bound = (2 * (2 * n + 8) * B(Da, v) + 16 * B(Ed, v)) * LD(2) ** -53
            assert np.all(np.abs(got - want) <= bound), (kind, axis)
