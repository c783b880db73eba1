"""Performance cases of the library: the work its users have it do.

A solver built on this package spends its time in the Benchmark Streaming
vector operations (BS1-BS5), the gather and scatter over a local-to-global map
(BS6, BS7), the matrix-free Helmholtz operator on affine and on general
hexahedra, and whole conjugate-gradient solves: FP64, float-float with Jacobi,
FP32 inside FP64 refinement, many small solves at once, and flexible PCG with
the element network, which is trained on the same GPU.  Each case is one such
call, at sizes taken from the package's benchmark, tests and smoke check.

listed() and draw(rng) give cases, prepare() builds what a program holds
before the call, run() is one pass through the public entry points, work()
the bytes and operations of the pass, and exact() the same results in plain
64-bit torch, from this file's own mesh, quadrature and solver code.
"""
import functools
import math

import numpy as np
import torch

from paper_2009_10917_gb300 import bs

DEV = "cuda"


def listed():
    return [
        # the vector operations of a small solve (a few thousand unknowns):
        # launches and latency are all of it
        {"name": "stream_f64_small", "kind": "stream", "dtype": "f64", "n": 4099, "offset": 0},
        # the FP32 vectors of a refined solve, at an odd length
        {"name": "stream_f32_odd", "kind": "stream", "dtype": "f32", "n": 20000003, "offset": 0},
        # the benchmark's streaming step: vectors far larger than the caches
        {"name": "stream_f64_large", "kind": "stream", "dtype": "f64", "n": 1 << 27,
         "offset": 0},
        # scatter and gather on the benchmark's degree, FP64 and FP32
        {"name": "map_n7", "kind": "map", "N": 7, "K": 36, "masked": False},
        # one application of the FP64 operator, the inner step of every solver
        {"name": "op_n7", "kind": "op", "N": 7, "K": 36, "coef": False, "masked": False,
         "geo": False, "ff": False},
        # the same on general (perturbed) hexahedra, an even degree, odd mesh
        {"name": "op_geo_n4", "kind": "op", "N": 4, "K": 27, "coef": True, "masked": False,
         "geo": True, "ff": False},
        # FP64 CG, replayed as a graph: the headline solve
        {"name": "cg_n7", "kind": "cg", "N": 7, "K": 32, "coef": False, "masked": False,
         "jacobi": False, "ff": False, "iters": 64},
        # float-float Jacobi-PCG with strongly varying coefficients and
        # Dirichlet boundaries, at the learned workload's degree
        {"name": "cg_ff_jacobi_n5", "kind": "cg", "N": 5, "K": 33, "coef": True, "masked": True,
         "jacobi": True, "ff": True, "iters": 64},
        # an implicit time step solved with FP32 CG inside FP64 refinement
        {"name": "refined_n7", "kind": "refined", "N": 7, "K": 24, "lam": 4000.0},
        # many small solves of mixed degree advanced together to convergence
        {"name": "batched_small", "kind": "batched", "solves": 96, "nmin": 2, "nmax": 6,
         "kmin": 1, "kmax": 7},
        # flexible PCG preconditioned with the element network
        {"name": "fpcg_n5", "kind": "fpcg", "N": 5, "K": 32, "iters": 12},
        # training steps of the element network (forward, backward, Adam)
        {"name": "train_n5", "kind": "train", "N": 5, "H": 256, "batch": 256, "steps": 32},
    ]


def _spread(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh_k(rng, N, most, least=1.0):
    """Elements per direction, at least 2, spread over meshes of `least` to
    `most` local nodes."""
    lo, hi = (int((v / (N + 1) ** 3) ** (1.0 / 3.0)) for v in (least, most))
    return _spread(rng, max(2, lo + 1), max(3, lo + 2, hi))


def draw(rng):
    kind = rng.choice(["stream", "stream", "map", "map", "op", "op", "op", "cg", "cg",
                       "refined", "batched", "fpcg", "train"])
    if kind == "stream":
        return {"kind": kind, "dtype": rng.choice(["f64", "f32"]),
                "n": _spread(rng, 1000, 1 << 26), "offset": rng.choice([0, 0, 0, 1])}
    N = rng.choice([1, 2, 3, 4, 5, 6, 7, 7, 8, 9, 11, 15])
    coef, masked = rng.random() < 0.5, rng.random() < 0.3
    if kind == "map":
        return {"kind": kind, "N": N, "K": _mesh_k(rng, N, 2.0e7), "masked": masked}
    if kind == "op":
        geo = N <= 11 and rng.random() < 0.4
        return {"kind": kind, "N": N, "K": _mesh_k(rng, N, 5e6 if geo else 2.0e7),
                "coef": coef, "masked": masked, "geo": geo, "ff": rng.random() < 0.3}
    if kind == "cg":
        return {"kind": kind, "N": N, "K": _mesh_k(rng, N, 6e6, 2e4), "coef": coef,
                "masked": masked, "jacobi": rng.random() < 0.5, "ff": rng.random() < 0.5,
                "iters": rng.randrange(9, 48)}
    if kind == "refined":
        N = rng.choice([2, 3, 4, 5, 6, 7, 8])
        return {"kind": kind, "N": N, "K": _mesh_k(rng, N, 6e6, 2e3),
                "lam": float(_spread(rng, 2000, 20000))}
    if kind == "batched":
        nmin, kmin = rng.randrange(1, 5), rng.randrange(1, 4)
        return {"kind": kind, "solves": _spread(rng, 5, 80), "nmin": nmin,
                "nmax": rng.randrange(nmin, 7), "kmin": kmin, "kmax": rng.randrange(kmin, 7)}
    N = rng.choice([3, 4, 5, 6])
    if kind == "fpcg":
        return {"kind": kind, "N": N, "K": _mesh_k(rng, N, 5e6, 2e4),
                "iters": rng.randrange(4, 12)}
    return {"kind": "train", "N": N, "H": rng.choice([128, 192, 256]),
            "batch": 32 * _spread(rng, 2, 16), "steps": rng.randrange(4, 32)}


# ---------------------------------------------------------------- meshes, quadrature

@functools.lru_cache(maxsize=3)
def _mesh(N, K, masked):
    """(l2g int32 [E Np], N_G, order): a K^3 mesh of the unit cube, degree N,
    elements stored in a shuffled order; masked: boundary nodes carry -1 and
    the interior ones are numbered alone."""
    G, a = K * N + 1, np.arange(N + 1)
    order = np.random.RandomState(1000 * N + K).permutation(K ** 3)
    ex, ey, ez = order % K, order // K % K, order // (K * K)
    off = a[None, None, :] + G * (a[None, :, None] + G * a[:, None, None])
    ids = (N * (ex + G * (ey + G * ez)))[:, None] + off.reshape(1, -1)
    ids, ng = ids.reshape(-1), G ** 3
    if masked:
        inner = np.zeros((G, G, G), bool)
        inner[1:-1, 1:-1, 1:-1] = True
        new = np.full(ng, -1)
        ng = max(0, G - 2) ** 3
        new[inner.reshape(-1)] = np.arange(ng)
        ids = new[ids]
    return ids.astype(np.int32), ng, order


def _corners(N, K):
    """Corner coordinates [E, 8, 3] of the shuffled elements, interior
    vertices moved by up to a fifth of the element size."""
    _, _, order = _mesh(N, K, False)
    n1 = K + 1
    pos = np.stack(np.meshgrid(*[np.arange(n1) / K] * 3, indexing="ij")[::-1], -1)
    move = np.random.RandomState(77).uniform(-0.2 / K, 0.2 / K, pos.shape)
    move[[0, -1]] = 0
    move[:, [0, -1]] = 0
    move[:, :, [0, -1]] = 0
    pos = pos + move
    ex, ey, ez = order % K, order // K % K, order // (K * K)
    return np.stack([pos[ez + (v >> 2), ey + (v >> 1 & 1), ex + (v & 1)] for v in range(8)], 1)


def _quadrature(N):
    """GLL nodes, weights and derivative matrix D[a, i] = l_i'(x_a)."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # polish the roots of P'
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    x = (x - x[::-1]) / 2
    w = 2.0 / (N * (N + 1) * P(x) ** 2)
    d = x[:, None] - x[None, :] + np.eye(N + 1)
    b = 1.0 / d.prod(1)
    D = b[None, :] / b[:, None] / d
    np.fill_diagonal(D, 0.0)
    np.fill_diagonal(D, -D.sum(1))
    return x, w, D


def _coef(E):
    """Lognormal element coefficients (sigma 1)."""
    return np.exp(np.random.RandomState(E).standard_normal(E))


def _vector(n, seed, stream, dtype=torch.float64):
    """n values uniform in [-1, 1), on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + stream)
    return torch.rand(n, generator=g, device=DEV, dtype=dtype) * 2 - 1


def _problem(c):
    """(Map, Problem) of an affine or general mesh."""
    N, K = c["N"], c["K"]
    ids, ng, _ = _mesh(N, K, c.get("masked", False))
    m = bs.Map(K ** 3, N, ng, ids)
    return m, bs.Problem(m, 1.0 / K, c.get("lam", 1.0),
                         coef=_coef(K ** 3) if c.get("coef") else None,
                         verts=_corners(N, K) if c.get("geo") else None)


def _batch(c):
    """(N, K) of every solve."""
    r = np.random.RandomState(c["solves"])
    return [(int(r.randint(c["nmin"], c["nmax"] + 1)), int(r.randint(c["kmin"], c["kmax"] + 1)))
            for _ in range(c["solves"])]


def _slices(sizes):
    """Start of each solve's vector in one buffer (16-byte aligned), and its length."""
    starts = np.concatenate([[0], np.cumsum([n + n % 2 for n in sizes])])
    return [int(s) for s in starts]


def _element_matrix(N, K, lam):
    """One affine element's dense matrix (coefficient 1)."""
    _, w, D = _quadrature(N)
    S, W, g = D.T @ (w[:, None] * D), np.diag(w), 0.5 / K
    kron = lambda a, b, c: np.kron(a, np.kron(b, c))  # noqa: E731
    return (g * (kron(S, W, W) + kron(W, S, W) + kron(W, W, S))
            + lam * g ** 3 * kron(W, W, W))


def _network(N, K, lam, H=256):
    """Network weights whose odd part W2 W1 / 2 is the map the network is
    trained to: the element-interior error of the Jacobi-scaled residual."""
    A, n = _element_matrix(N, K, lam), N + 1
    q = np.arange(n ** 3)
    ijk = np.stack([q % n, q // n % n, q // n ** 2])
    inner = q[np.all((ijk > 0) & (ijk < N), axis=0)]
    L = np.zeros((n ** 3, n ** 3))
    d = np.diag(A)[inner]
    L[np.ix_(inner, inner)] = np.linalg.solve(A[np.ix_(inner, inner)], np.diag(d)) - np.eye(
        len(inner))
    U, s, Vt = np.linalg.svd(L)
    r = min(H, len(inner))
    W1, W2 = np.zeros((H, n ** 3), np.float32), np.zeros((n ** 3, H), np.float32)
    W1[:r], W2[:, :r] = np.sqrt(s[:r])[:, None] * Vt[:r], 2 * U[:, :r] * np.sqrt(s[:r])
    return W1, W2, inner


def _pairs(c, seed):
    """Training rows X of unit rms and targets T = G X on the interior nodes,
    and the initial weights (W2 = 0 as in training from scratch)."""
    D, H = (c["N"] + 1) ** 3, c["H"]
    rows = c["batch"] * min(c["steps"], 8)
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    X = torch.randn(rows, D, generator=g, device=DEV)
    G = torch.randn(D, D, generator=g, device=DEV) / math.sqrt(D)
    X = X / X.square().mean(1, keepdim=True).sqrt()
    T = X @ G.T
    q = torch.arange(D, device=DEV)
    n = c["N"] + 1
    edge = sum(((v == 0) | (v == c["N"])).int() for v in (q % n, q // n % n, q // n ** 2)) > 0
    T[:, edge] = 0
    W1 = np.random.RandomState(seed % (1 << 31)).uniform(-1, 1, (H, D)) * math.sqrt(3.0 / D)
    return X.contiguous(), T.contiguous(), W1.astype(np.float32), np.zeros((D, H), np.float32)


def _rate(c, t):
    """Cosine learning rate."""
    return 1e-3 * (1 + math.cos(math.pi * t / c["steps"]))


# ---------------------------------------------------------------- prepare and run

def _stream_inputs(c, seed):
    dt = torch.float64 if c["dtype"] == "f64" else torch.float32
    n, o = c["n"], c["offset"]
    return {k: _vector(n + o, seed, i, dt)[o:] for i, k in enumerate(("x", "p", "Ap", "xx", "r"))}


def prepare(case, seed):
    c, kind = case, case["kind"]
    s = {"c": c}
    if kind == "stream":
        s.update(_stream_inputs(c, seed))
    elif kind == "map":
        ids, ng, _ = _mesh(c["N"], c["K"], c["masked"])
        s["map"] = m = bs.Map(c["K"] ** 3, c["N"], ng, ids)
        for sfx, dt in (("64", torch.float64), ("32", torch.float32)):
            s["g" + sfx], s["l" + sfx] = _vector(m.NG, seed, 0, dt), _vector(m.NL, seed, 1, dt)
            s["o" + sfx] = torch.zeros(m.NL, dtype=dt, device=DEV)  # masked entries stay 0
    elif kind in ("op", "cg", "refined", "fpcg"):
        s["map"], s["prob"] = _problem(_fpcg_case(c) if kind == "fpcg" else c)
        s["b"] = _vector(s["map"].NG, seed, 0)
        s["x"] = torch.zeros_like(s["b"])
        if kind == "fpcg":
            W1, W2, _ = _network(c["N"], c["K"], _fpcg_case(c)["lam"])
            s["net"] = bs.MLP(W1, W2, split=True)
    elif kind == "batched":
        s["probs"], starts = [], None
        for N, K in _batch(c):
            s["probs"].append(_problem({"N": N, "K": K})[1])
        sizes = [p.map.NG for p in s["probs"]]
        starts = _slices(sizes)
        s["b"], s["x"] = _vector(starts[-1], seed, 0), torch.zeros(starts[-1],
                                                                    dtype=torch.float64, device=DEV)
        s["bs"] = [s["b"][o:o + n] for o, n in zip(starts, sizes)]
        s["xs"] = [s["x"][o:o + n] for o, n in zip(starts, sizes)]
    else:
        s["X"], s["T"], W1, W2 = _pairs(c, seed)
        s["net"] = bs.MLP(W1, W2, split=True)
        s["loss"] = torch.zeros(1, dtype=torch.float64, device=DEV)
    return s


def _fpcg_case(c):
    return {"N": c["N"], "K": c["K"], "lam": 0.01, "coef": True}


def run(s):
    c, kind = s["c"], s["c"]["kind"]
    if kind == "stream":  # BS1-BS5 as one CG iteration strings them together
        y = bs.copy(s["x"])
        bs.axpy(1.0, s["r"], 0.5, s["p"])
        return {"copy": y, "p": s["p"], "norm": bs.norm(s["x"]), "dot": bs.dot(s["p"], s["Ap"]),
                "rr": bs.cg_update(0.25, s["p"], s["Ap"], s["xx"], s["r"]), "x": s["xx"],
                "r": s["r"]}
    if kind == "map":
        m = s["map"]
        return [f for k in ("64", "32")
                for f in (m.scatter(s["g" + k], s["o" + k]), m.gather(s["l" + k]))]
    if kind == "op":
        return s["prob"].apply_A_ff(s["b"]) if c["ff"] else s["prob"].apply_A(s["b"])
    if kind == "cg":
        flags = (bs.BS_CG_FIXED_ITERS | bs.BS_CG_GRAPH | (bs.BS_CG_JACOBI if c["jacobi"] else 0)
                 | (bs.BS_CG_FF_OPERATOR if c["ff"] else 0))
        x, info = s["prob"].cg(s["b"], s["x"], tol=0.0, maxit=c["iters"], flags=flags)
        return x, info["rel_residual"]
    if kind == "refined":
        return s["prob"].cg_refined_f32(s["b"], s["x"], tol=1e-12, flags=bs.BS_CG_GRAPH)[0]
    if kind == "batched":
        bs.solve_batched(s["probs"], s["bs"], s["xs"], tol=1e-12, flags=bs.BS_CG_GRAPH)
        return s["x"]
    if kind == "fpcg":
        return bs.fpcg_learned(s["prob"], s["net"], s["b"], s["x"], tol=0.0, maxit=c["iters"],
                               flags=bs.BS_FPCG_ODD | bs.BS_CG_GRAPH, check=False)[0]
    B, rows = c["batch"], s["X"].shape[0]
    for t in range(c["steps"]):
        o = t * B % rows
        s["net"].train_step(s["X"][o:o + B], s["T"][o:o + B], _rate(c, t), s["loss"])
    return s["loss"], s["net"].weights()


# ---------------------------------------------------------------- work

def _sizes(c):
    N, K = c["N"], c["K"]
    NL = K ** 3 * (N + 1) ** 3
    NG = (K * N - 1) ** 3 if c.get("masked") else (K * N + 1) ** 3
    return NL, NG


def _op_work(c, w=8):
    """One A p: the map and p read, A p written; three contractions a node."""
    NL, NG = _sizes(c)
    flops = NL * ((12 if c.get("geo") else 6) * (c["N"] + 1) + (30 if c.get("geo") else 10))
    return 4 * NL + 2 * w * NG + (56 * NL if c.get("geo") else 0), flops


def work(case):
    c, kind = case, case["kind"]
    if kind == "stream":
        return {"bytes": 14 * (8 if c["dtype"] == "f64" else 4) * c["n"], "flops": 12 * c["n"]}
    if kind == "train":
        D, H, B = (c["N"] + 1) ** 3, c["H"], c["batch"]
        # forward: two products of three bf16 terms; backward: three products
        return {"bytes": c["steps"] * (24 * D * H + 8 * B * D),
                "flops": c["steps"] * 2 * B * D * H * 9}
    if kind == "batched":
        per = [(_op_work({"N": N, "K": K}), (K * N + 1) ** 3) for N, K in _batch(c)]
        its = [8 * N * K for N, K in _batch(c)]  # iterations grow with the nodes per direction
        return {"bytes": sum(i * (b + 80 * n) for i, ((b, _), n) in zip(its, per)),
                "flops": sum(i * (f + 12 * n) for i, ((_, f), n) in zip(its, per))}
    NL, NG = _sizes(c)
    if kind == "map":  # map, q_G and q_L once in each direction
        return {"bytes": 2 * (4 + 4) * NL + 2 * (8 + 4) * (NL + NG), "flops": 2 * NL}
    b, f = _op_work(c, 4 if kind == "refined" else 8)
    if kind == "op":
        return {"bytes": b, "flops": f}
    if kind == "refined":  # about 60 inner iterations
        return {"bytes": 60 * (b + 40 * NG), "flops": 60 * (f + 12 * NG)}
    extra = 0
    if kind == "fpcg":
        extra = (c["N"] + 1) ** 3 * (c["N"] - 1) ** 3 * c["K"] ** 3 * 6
    # CG: update (48 bytes a node), direction (24), p for p.Ap; Jacobi: dinv, z
    jac = 24 if c.get("jacobi") or kind == "fpcg" else 0
    return {"bytes": c["iters"] * (b + (72 + jac) * NG),
            "flops": c["iters"] * (f + 12 * NG + extra)}


# ---------------------------------------------------------------- the same in 64 bits

class _Operator:
    """A = Z^T (c S + lambda M) Z in plain 64-bit torch."""

    def __init__(self, c):
        N, K = c["N"], c["K"]
        ids, self.ng, _ = _mesh(N, K, c.get("masked", False))
        n = N + 1
        x, w, D = _quadrature(N)
        self.t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)
        self.ids = self.t(ids).long()
        self.on = self.ids >= 0
        self.ids = self.ids.clamp(min=0) if self.ng else self.ids
        self.shape, self.h2, self.lam = (K ** 3, n, n, n), 0.5 / K, c.get("lam", 1.0)
        self.D, self.S, self.w = self.t(D), self.t(D.T @ (w[:, None] * D)), self.t(w)
        self.c = (self.t(_coef(K ** 3)) if c.get("coef") else
                  torch.ones(K ** 3, dtype=torch.float64, device=DEV)).view(-1, 1, 1, 1)
        self.geo = self._factors(N, K, x) if c.get("geo") else None

    def _factors(self, N, K, x):
        X, n, t = self.t(_corners(N, K)), N + 1, self.t(x)
        r, s, q = t.view(1, 1, n), t.view(1, n, 1), t.view(n, 1, 1)
        J = torch.zeros(X.shape[0], n, n, n, 3, 3, dtype=torch.float64, device=DEV)
        for v in range(8):
            a, b, c = (2 * (v >> d & 1) - 1 for d in range(3))
            dv = torch.stack([(a * (1 + b * s) * (1 + c * q)).expand(n, n, n),
                              (b * (1 + a * r) * (1 + c * q)).expand(n, n, n),
                              (c * (1 + a * r) * (1 + b * s)).expand(n, n, n)], -1) / 8
            J += X[:, v].view(-1, 1, 1, 1, 3, 1) * dv[None, ..., None, :]
        a, b, c = J[..., 0], J[..., 1], J[..., 2]  # columns dx/dr, dx/ds, dx/dt
        C = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a),
                         torch.linalg.cross(a, b)], -2)
        det = (a * C[..., 0, :]).sum(-1)
        w3 = self._w3()
        return (w3 / det)[..., None, None] * (C @ C.transpose(-1, -2)), w3 * det

    def _w3(self):
        w = self.w
        return w.view(1, -1, 1, 1) * w.view(1, 1, -1, 1) * w.view(1, 1, 1, -1)

    def scatter(self, p):
        return torch.where(self.on, p[self.ids], torch.zeros((), dtype=p.dtype, device=DEV))

    def gather(self, q):
        q = torch.where(self.on, q.reshape(-1), torch.zeros((), dtype=q.dtype, device=DEV))
        return torch.zeros(self.ng, dtype=q.dtype, device=DEV).index_add_(0, self.ids, q)

    def _along(self, M, u):
        return (u @ M.T, torch.matmul(M, u),
                (M @ u.reshape(u.shape[0], u.shape[1], -1)).view(u.shape))

    def local(self, u):
        u = u.view(self.shape)
        w = self.w
        if self.geo is None:
            ar, as_, at = self._along(self.S, u)
            wj, wk, wi = w.view(1, 1, -1, 1), w.view(1, -1, 1, 1), w.view(1, 1, 1, -1)
            return (self.c * self.h2 * (ar * wj * wk + as_ * wi * wk + at * wi * wj)
                    + self.lam * self.h2 ** 3 * self._w3() * u)
        G, M = self.geo
        g = torch.stack(self._along(self.D, u), -1)
        f = (G @ g[..., None])[..., 0]
        del g
        return (self.c * (self._along(self.D.T, f[..., 0].contiguous())[0]
                          + self._along(self.D.T, f[..., 1].contiguous())[1]
                          + self._along(self.D.T, f[..., 2].contiguous())[2])
                + self.lam * M * u)

    def __call__(self, p):
        return self.gather(self.local(self.scatter(p)))

    def diag(self):
        d, w = torch.diagonal(self.S), self.w
        i, j, k = (1, 1, 1, -1), (1, 1, -1, 1), (1, -1, 1, 1)
        s = (d.view(i) * w.view(j) * w.view(k) + w.view(i) * d.view(j) * w.view(k)
             + w.view(i) * w.view(j) * d.view(k))
        return self.gather(self.c * self.h2 * s + self.lam * self.h2 ** 3 * self._w3())


def _cg(A, b, iters, tol=0.0, precond=None, flexible=False):
    """(x, ||r|| / ||b||) of (preconditioned) CG from x = 0."""
    M = precond or (lambda r: r)
    x, r = torch.zeros_like(b), b.clone()
    z = M(r)
    p, rz, bb = z.clone(), r @ z, b @ b
    for _ in range(iters):
        Ap = A(p)
        alpha = rz / (p @ Ap)
        x += alpha * p
        r = r - alpha * Ap
        if tol and float(r @ r) <= tol * tol * float(bb):
            break
        zo, z = z, M(r)
        rz, beta = r @ z, (r @ (z - zo if flexible else z)) / rz
        p = z + beta * p
    return x, float(torch.sqrt((r @ r) / bb))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "stream":
        v = {k: t.double() for k, t in _stream_inputs(c, seed).items()}
        xx = v["x"] @ v["x"]
        p = v["r"] + 0.5 * v["p"]
        r = v["r"] - 0.25 * v["Ap"]
        return {"copy": v["x"], "p": p, "norm": torch.stack([xx, xx.sqrt()]),
                "dot": (p @ v["Ap"]).view(1), "rr": (r @ r).view(1),
                "x": v["xx"] + 0.25 * p, "r": r}
    if kind == "map":
        A, out = _Operator(dict(c, coef=False)), []
        for dt in (torch.float64, torch.float32):
            out += [A.scatter(_vector(A.ng, seed, 0, dt)).double(),
                    A.gather(_vector(A.ids.numel(), seed, 1, dt).double())]
        return out
    if kind == "op":
        A = _Operator(c)
        return A(_vector(A.ng, seed, 0))
    if kind == "cg":
        A = _Operator(c)
        d = A.diag() if c["jacobi"] else None
        return _cg(A, _vector(A.ng, seed, 0), c["iters"],
                   precond=(lambda r: r / d) if c["jacobi"] else None)
    if kind == "refined":
        A = _Operator(c)
        return _cg(A, _vector(A.ng, seed, 0), 2000, tol=1e-14)[0]
    if kind == "batched":
        ops = [_Operator({"N": N, "K": K}) for N, K in _batch(c)]
        starts = _slices([A.ng for A in ops])
        b = _vector(starts[-1], seed, 0)
        x = torch.zeros_like(b)
        for A, o in zip(ops, starts):
            x[o:o + A.ng] = _cg(A, b[o:o + A.ng], 2000, tol=1e-14)[0]
        return x
    if kind == "fpcg":
        fc = _fpcg_case(c)
        A, n = _Operator(fc), c["N"] + 1
        W1, W2, inner = _network(c["N"], c["K"], fc["lam"])
        L = 0.5 * A.t(W2.astype(np.float64)) @ A.t(W1.astype(np.float64))
        mask = torch.zeros(n ** 3, dtype=torch.float64, device=DEV)
        mask[torch.from_numpy(inner).to(DEV)] = 1
        d = A.diag()

        def M(r):
            u = A.scatter(r / d).view(-1, n ** 3)
            rms = u.square().mean(1, keepdim=True).sqrt()
            return r / d + A.gather((u / rms) @ L.T * mask * rms)
        return _cg(A, _vector(A.ng, seed, 0), c["iters"], precond=M, flexible=True)[0]
    X, T, W1, W2 = _pairs(c, seed)
    W = [torch.from_numpy(a.astype(np.float64)).to(DEV).requires_grad_() for a in (W1, W2)]
    opt = torch.optim.Adam(W, lr=1e-3)
    B, rows = c["batch"], X.shape[0]
    for t in range(c["steps"]):
        o = t * B % rows
        for g in opt.param_groups:
            g["lr"] = _rate(c, t)
        opt.zero_grad()
        loss = (torch.relu(X[o:o + B].double() @ W[0].T) @ W[1].T
                - T[o:o + B].double()).square().mean()
        loss.backward()
        opt.step()
    return loss.detach().view(1), tuple(w.detach() for w in W)
