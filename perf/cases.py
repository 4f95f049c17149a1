"""What a user of this framework has it do, as cases that can be timed.

Every case goes through the public binding (``paper_2211_11303_gb300.hlu``): the
residual product, H-LU preconditioned FGMRES on a held factor, a
factorisation with its solve, the whole path from the mesh, Algorithm 1's
Richardson iteration on the magnet, and a mix of requests factored in one launch
and stepped together.  The outputs are the solutions in FP64; the tolerances are
those of a solve whose answer is wanted to rounding, not to the preconditioner's
truncation.
"""
import itertools
import math

import numpy as np
import torch

from paper_2211_11303_gb300 import example3, hlu

TOL = 1e-11        # relative residual; the forward error is then far below 1e-9
EXACT_MAX_N = 12   # largest cube whose dense 64-bit solve takes a few seconds


def listed():
    return [
        # residual of one right-hand side on the smallest mesh in use: a launch
        {"name": "spmv_n6_1rhs", "kind": "spmv", "n": 6, "kappa": 4.0, "nrhs": 1},
        # residual product of a block of right-hand sides at the benchmark's size
        {"name": "spmv_n24_8rhs", "kind": "spmv", "n": 24, "kappa": 8.0, "nrhs": 8},
        # serving: one more right-hand side for a small cached factor
        {"name": "solve_n8_1rhs", "kind": "solve", "n": 8, "kappa": 8.0, "nrhs": 1,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # an ordinary block solve, odd column count, with a cached factor
        {"name": "solve_n16_5rhs", "kind": "solve", "n": 16, "kappa": 5.0, "nrhs": 5,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # the benchmark's mesh with a cached factor
        {"name": "solve_n24_8rhs", "kind": "solve", "n": 24, "kappa": 8.0, "nrhs": 8,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # a new wave number on a small mesh: the oracle's sample workload
        {"name": "factor_n8_1rhs", "kind": "factor", "n": 8, "kappa": 8.0, "nrhs": 1,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # a ragged mesh (no power of two anywhere), a finer truncation
        {"name": "factor_n13_3rhs", "kind": "factor", "n": 13, "kappa": 6.0, "nrhs": 3,
         "eps": 1e-5, "leaf": 32, "precision": "fp32"},
        # the benchmark: factorisation and FGMRES of 8 right-hand sides
        {"name": "factor_n24_8rhs", "kind": "factor", "n": 24, "kappa": 8.0, "nrhs": 8,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # the plain FP64 path
        {"name": "factor_n11_fp64_2rhs", "kind": "factor", "n": 11, "kappa": 8.0, "nrhs": 2,
         "eps": 1e-4, "leaf": 32, "precision": "fp64"},
        # everything from the mesh on: assembly, trees, load vector, H-LU, FGMRES
        {"name": "whole_n8_fp64_2rhs", "kind": "whole", "n": 8, "kappa": 1.0, "nrhs": 2,
         "eps": 1e-4, "leaf": 32, "precision": "fp64"},
        # Example 3's magnet: material coefficient, Richardson iteration
        {"name": "richardson_n16", "kind": "richardson", "n": 16, "kappa": math.sqrt(10.0), "nrhs": 1,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
        # serving: problems of several sizes in one factorisation launch, their
        # FGMRES states advanced together
        {"name": "served_n6_to_12", "kind": "served", "n": 6, "n_hi": 12, "count": 6, "kappa": 4.0, "nrhs": 3,
         "eps": 1e-4, "leaf": 32, "precision": "fp32"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["spmv", "solve", "solve", "factor", "factor", "fp64", "whole", "richardson", "served"])
    kappa = round(rng.uniform(2.0, 10.0), 3)
    if kind == "spmv":
        return {"kind": "spmv", "n": _log_int(rng, 4, 24), "kappa": kappa, "nrhs": rng.randint(1, 16)}
    c = {"kind": kind, "n": _log_int(rng, 4, 20), "kappa": kappa, "nrhs": rng.randint(1, 16),
         "eps": rng.choice([1e-3, 1e-4, 1e-4, 1e-5]), "leaf": rng.choice([16, 32, 32, 64]), "precision": "fp32"}
    if kind == "fp64":
        c.update(kind="factor", n=_log_int(rng, 4, 12), precision="fp64")
    elif kind == "whole":
        c.update(n=_log_int(rng, 4, 14), nrhs=rng.randint(2, 8))
    elif kind == "richardson":
        c.update(n=_log_int(rng, 6, 18), kappa=math.sqrt(10.0), nrhs=1, eps=1e-4)
    elif kind == "served":
        c.update(n=rng.randint(4, 6), n_hi=rng.randint(8, 12), count=rng.randint(2, 8), nrhs=rng.randint(1, 4))
    return c


def _normal(seed, k, N, nrhs):
    """Seeded N(0, 1) columns, column-major (N, nrhs)."""
    g = torch.Generator(device="cuda").manual_seed(7919 * seed + k)
    return torch.randn((nrhs, N), dtype=torch.float64, device="cuda", generator=g).t()


def _precision(case):
    return hlu.HLU_FP64 if case["precision"] == "fp64" else hlu.HLU_FP32


def _served_problems(case):
    """(n, kappa) of a served mix: sizes spread over [n, n_hi], a wave number each."""
    k = case["count"]
    return [(case["n"] + round(i * (case["n_hi"] - case["n"]) / max(1, k - 1)),
             case["kappa"] + 0.75 * (i % 5)) for i in range(k)]


class Handles:
    """The handles a program holds; destroyed with the state."""

    def __init__(self):
        self.hs = []

    def build(self, *args, **kw):
        self.hs.append(hlu.hlu_build(*args, **kw))
        return self.hs[-1]

    def __del__(self):
        for h in self.hs:
            hlu.hlu_destroy(h)


def prepare(case, seed):
    kind, n = case["kind"], case["n"]
    own = Handles()
    s = {"case": case, "own": own}
    if kind == "served":
        s["b"], s["x"] = [], []
        for i, (m, kappa) in enumerate(_served_problems(case)):
            N = hlu.hlu_n(own.build(m, kappa, case["leaf"], 2.0, case["eps"]))
            s["b"].append(_normal(seed, i, N, case["nrhs"]))
            s["x"].append(hlu.colmajor(N, case["nrhs"]))
        return s
    beta = example3.magnet_beta(n) if kind == "richardson" else None
    h = own.build(n, case["kappa"], case.get("leaf", 32), 2.0, case.get("eps", 1e-4), beta=beta)
    N = hlu.hlu_n(h)
    s["h"] = h
    s["x"] = hlu.colmajor(N, case["nrhs"])
    if kind == "richardson":
        g = np.random.default_rng(seed)
        s["b"] = hlu.colmajor(N, 1)
        hlu.hlu_rhs_constant_current(h, 10.0 * g.standard_normal(3), s["b"])
    else:
        s["b"] = _normal(seed, 0, N, case["nrhs"])
    if kind == "solve":
        hlu.hlu_factor(h, _precision(case))
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "spmv":
        hlu.hlu_spmv(s["h"], s["b"], s["x"])
    elif kind == "solve":
        hlu.gmres_solve(s["h"], s["b"], s["x"], restart=50, tol=TOL)
    elif kind == "factor":
        hlu.hlu_factor(s["h"], _precision(case))
        hlu.gmres_solve(s["h"], s["b"], s["x"], restart=50, tol=TOL)
    elif kind == "richardson":
        hlu.hlu_factor(s["h"], _precision(case))
        hlu.hlu_richardson(s["h"], s["b"], s["x"], tol=TOL)
    elif kind == "whole":
        b = s["b"].t().clone().t()
        with hlu.Problem(case["n"], case["kappa"], case["leaf"], 2.0, case["eps"]) as P:
            hlu.hlu_rhs_manufactured(P.h, b[:, 0])
            hlu.hlu_factor(P.h, _precision(case))
            hlu.gmres_solve(P.h, b, s["x"], restart=50, tol=TOL)
        return {"b": b, "x": s["x"]}
    else:
        hlu.hlu_factor_batch(s["own"].hs, _precision(case))
        gs = [hlu.hlu_gmres_begin(h, b, x, restart=50, tol=TOL) for h, b, x in zip(s["own"].hs, s["b"], s["x"])]
        while not all(hlu.hlu_gmres_status(g)[0] for g in gs):
            hlu.hlu_gmres_step_batch(gs)
        for g in gs:
            hlu.hlu_gmres_end(g)
    return s["x"]


def _size(n):
    """Unknowns and matrix entries of the Kuhn cube with n^3 sub-cubes."""
    return 7 * n**3 - 9 * n**2 + 3 * n, 115 * n**3 - 261 * n**2 + 195 * n - 48


def work(case):
    """The matrix and the right-hand sides read once, the solutions written
    once, and one product with the matrix (the least that shows a solution)."""
    ns = [m for m, _ in _served_problems(case)] if case["kind"] == "served" else [case["n"]]
    bytes_, flops = 0, 0
    for n in ns:
        N, nnz = _size(n)
        bytes_ += 12 * nnz + 8 * (N + 1) + 16 * N * case["nrhs"]
        flops += 2 * nnz * case["nrhs"]
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------- 64-bit answers
def _elements(n, beta=None):
    """Edge unknowns (T, 6) (-1 on the boundary), K_e and M_e (T, 6, 6), vertex
    coordinates (T, 4, 3) and local edges (6, 2) of the Kuhn cube."""
    i = torch.arange(n)
    base = torch.cartesian_prod(i, i, i).reshape(-1, 1, 1, 3)
    shape = torch.zeros(6, 4, 3, dtype=torch.int64)
    for t, perm in enumerate(itertools.permutations(range(3))):
        for k, a in enumerate(perm):
            shape[t, k + 1] = shape[t, k]
            shape[t, k + 1, a] += 1
    V = (base + shape).reshape(-1, 4, 3)  # the order of hlu_mesh_kuhn_cube
    vid = (V[..., 0] * (n + 1) + V[..., 1]) * (n + 1) + V[..., 2]
    pairs = torch.tensor(list(itertools.combinations(range(4), 2)))
    a, b = pairs[:, 0], pairs[:, 1]  # vertex ids grow along a Kuhn path: lo -> hi
    Va, Vb = V[:, a], V[:, b]
    boundary = (((Va == 0) & (Vb == 0)) | ((Va == n) & (Vb == n))).any(-1)
    key = vid[:, a] * (n + 1) ** 3 + vid[:, b]
    uniq = torch.unique(key[~boundary])
    dof = torch.where(boundary, torch.tensor(-1), torch.searchsorted(uniq, key.contiguous()))
    P = V.double() / n
    J = (P[:, 1:] - P[:, :1]).transpose(1, 2)
    G = torch.cat([torch.zeros(len(V), 1, 3, dtype=torch.float64), torch.linalg.inv(J)], 1)
    G[:, 0] = -G[:, 1:].sum(1)
    vol = torch.linalg.det(J).abs() / 6.0
    curl = 2.0 * torch.linalg.cross(G[:, a], G[:, b])
    K = vol[:, None, None] * curl @ curl.transpose(1, 2)
    if beta is not None:
        K = K / torch.from_numpy(beta)[:, None, None]
    S = vol[:, None, None] * (1.0 + torch.eye(4, dtype=torch.float64)) / 20.0
    D = G @ G.transpose(1, 2)

    def term(p, q, r, s):  # int l_p l_q (grad l_r . grad l_s) for every edge pair
        return S[:, p[:, None], q[None, :]] * D[:, r[:, None], s[None, :]]

    M = term(a, a, b, b) - term(a, b, b, a) - term(b, a, a, b) + term(b, b, a, a)
    return dof, K, M, P, (a, b), G, vol


def _manufactured(n, kappa):
    """Load vector of J = (2 pi^2 - kappa^2) E, 4-point rule."""
    dof, _, _, P, (a, b), G, vol = _elements(n)
    al, be = (5.0 - math.sqrt(5.0)) / 20.0, (5.0 + 3.0 * math.sqrt(5.0)) / 20.0
    rhs = torch.zeros(_size(n)[0] + 1, dtype=torch.float64)
    for q in range(4):
        lam = torch.full((4,), al, dtype=torch.float64)
        lam[q] = be
        s = torch.sin(math.pi * (lam @ P))
        E = torch.stack([s[:, 1] * s[:, 2], s[:, 2] * s[:, 0], s[:, 0] * s[:, 1]], 1)
        W = lam[a][:, None] * G[:, b] - lam[b][:, None] * G[:, a]
        v = (2 * math.pi**2 - kappa**2) * (vol / 4.0)[:, None] * (W @ E[:, :, None])[..., 0]
        rhs.index_add_(0, torch.where(dof < 0, _size(n)[0], dof).reshape(-1), v.reshape(-1))
    return rhs[:-1].cuda()


def _current(n, J):
    """Load vector of a constant current: int w_ab = |T|/4 (grad l_b - grad l_a)."""
    dof, _, _, _, (a, b), G, vol = _elements(n)
    v = (vol / 4.0)[:, None] * ((G[:, b] - G[:, a]) @ torch.from_numpy(J))
    rhs = torch.zeros(_size(n)[0] + 1, dtype=torch.float64)
    rhs.index_add_(0, torch.where(dof < 0, _size(n)[0], dof).reshape(-1), v.reshape(-1))
    return rhs[:-1].cuda()


def _matrix(n, kappa, beta=None):
    """(rows, columns, values) of K - kappa^2 M, duplicates to be summed."""
    dof, K, M = _elements(n, beta)[:3]
    A = K - kappa**2 * M
    r = dof[:, :, None].expand_as(A)
    c = dof[:, None, :].expand_as(A)
    keep = (r >= 0) & (c >= 0)
    return r[keep].cuda(), c[keep].cuda(), A[keep].cuda()


def _dense_solve(n, kappa, b, beta=None):
    r, c, v = _matrix(n, kappa, beta)
    N = _size(n)[0]
    A = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    A.index_put_((r, c), v, accumulate=True)
    LU, piv = torch.linalg.lu_factor(A)
    x = torch.linalg.lu_solve(LU, piv, b.contiguous())
    for _ in range(2):
        x = x + torch.linalg.lu_solve(LU, piv, b - A @ x)
    return x


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    N = _size(n)[0]
    if kind == "spmv":
        r, c, v = _matrix(n, case["kappa"])
        b = _normal(seed, 0, N, case["nrhs"])
        y = torch.zeros((N, case["nrhs"]), dtype=torch.float64, device="cuda")
        for j in range(case["nrhs"]):
            y[:, j].index_add_(0, r, v * b[c, j])
        return y
    if kind == "served":
        out = []
        for i, (m, kappa) in enumerate(_served_problems(case)):
            out.append(_dense_solve(m, kappa, _normal(seed, i, _size(m)[0], case["nrhs"])))
        return out
    if n > EXACT_MAX_N:
        return None
    if kind == "richardson":
        J = 10.0 * np.random.default_rng(seed).standard_normal(3)
        c = _elements(n)[3].mean(1).numpy()  # centroids; the magnet is 0.5 x 0.5 x 0.75, centred
        inside = (np.abs(c - 0.5) < (0.25, 0.25, 0.375)).all(1)
        return _dense_solve(n, case["kappa"], _current(n, J)[:, None], np.where(inside, 10.0, 1.0))
    b = _normal(seed, 0, N, case["nrhs"])
    if kind == "whole":
        b = b.contiguous()
        b[:, 0] = _manufactured(n, case["kappa"])
        return {"b": b, "x": _dense_solve(n, case["kappa"], b)}
    return _dense_solve(n, case["kappa"], b)
