"""Performance cases: what a program built on this package has it compute, over the range of sizes,
precisions and options it is used with.

A case is a plain dict; `kind` names the entry point:

  matvec    Solver.matvec            y = A x or A^T x (FP64), for programs with their own Krylov loop
  precond   Solver.precond_apply     z = P_tilde^{-1} r with the default FP64 preconditioner
  solve     Solver.solve             one forward solve from a source and initial data
  batch     solve_batched            independent problems of uneven size, one stream each
  gradient  heat_solve + backward    a tracking functional's gradient in f and the nodal kappa, states
                                     checkpointed

Grids are "n0xn1" or "n0xn1xn2" interior points on the unit square or cube.  Inputs follow the workloads of
`synth`: Gaussian random fields with a squared-exponential covariance in 2D, a sine product plus
noise in 3D, kappa = exp(Gaussian field).
"""
import math

import numpy as np
import torch

from paper_2609_16863_gb300 import Solver, solve_batched
from paper_2609_16863_gb300.autograd import heat_solve

DEV = "cuda:0"


def listed():
    return [
        # the smallest call: one product on the 32 x 32, s = 2, 16-step problem, launch latency above all
        dict(name="matvec_small", kind="matvec", grid="32x32", method="radau", s=2, nt=16, T=1.0, kappa=False,
             transpose=False),
        # the product at the benchmark's size, as in every outer iteration
        dict(name="matvec_large", kind="matvec", grid="256x256", method="radau", s=3, nt=128, T=1.0, kappa=False,
             transpose=False),
        # the adjoint's product on a ragged 3D grid with a diffusivity field
        dict(name="matvec_adjoint_3d", kind="matvec", grid="49x45x41", method="gauss", s=2, nt=24, T=0.5, kappa=True,
             transpose=True),
        # one application of the default (FP64) preconditioner, a building block for a caller's own Krylov method
        dict(name="precond_fp64", kind="precond", grid="64x64", method="radau", s=2, nt=32, T=1.0, kappa=False,
             mgrit=0),
        # the plain FP64 method on the small workload, with its tolerance of 1e-10
        dict(name="solve_small_fp64", kind="solve", grid="32x32", method="radau", s=2, nt=16, T=1.0, tol=1e-10,
             prec="fp64", disc="fd", mgrit=0),
        # the benchmark workload: FP32 preconditioner, the recurrence by MGRIT
        dict(name="solve_large_fp32", kind="solve", grid="256x256", method="radau", s=3, nt=128, T=1.0, tol=1e-8,
             prec="fp32", disc="fd", mgrit=9),
        # an odd grid with the default schedule (forward substitution)
        dict(name="solve_odd_fp32", kind="solve", grid="127x95", method="radau", s=3, nt=40, T=1.0, tol=1e-8,
             prec="fp32", disc="fd", mgrit=0),
        # low-precision storage in 3D on the 96^3 grid, a shorter horizon than the full workload's 32 steps
        dict(name="solve_3d_bf16", kind="solve", grid="96x96x96", method="gauss", s=2, nt=8, T=0.125, tol=1e-8,
             prec="bf16", disc="fd", mgrit=0),
        # the other 16-bit format on a ragged 3D grid, three stages
        dict(name="solve_3d_fp16_ragged", kind="solve", grid="47x39x43", method="radau", s=3, nt=12, T=0.1875,
             tol=1e-8, prec="fp16", disc="fd", mgrit=0),
        # Q1 finite elements, the paper's own discretisation
        dict(name="solve_q1_fp32", kind="solve", grid="80x72", method="radau", s=2, nt=24, T=1.0, tol=1e-8,
             prec="fp32", disc="q1", mgrit=0),
        # one gradient of the 128 x 128 diffusivity workload: handles built for this kappa, forward solve, adjoint
        # solve and the recomputed windows, as each step of an optimiser over kappa does
        dict(name="gradient_kappa", kind="gradient", grid="128x128", method="radau", s=3, nt=64, T=1.0, tol=1e-10,
             prec="fp32", mgrit=8, ckpt=8),
        # a batch of uneven problems from the batched workload's ranges of sizes, steps and stages
        dict(name="batch_fp32", kind="batch", tol=1e-8, prec="fp32",
             problems="32:16:2 48:64:3 64:32:2 96:128:3 128:16:2 192:32:3 256:16:3 64:64:3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "precond", "solve", "solve", "solve3d", "gradient", "batch"])
    method, s = rng.choice([("radau", 2), ("radau", 3), ("gauss", 2)])
    n0 = _log_int(rng, 32, 256)
    n1 = max(32, min(256, int(n0 * math.exp(rng.uniform(-0.5, 0.5)))))
    if kind == "matvec":
        transpose, kappa = rng.random() < 0.5, rng.random() < 0.5
        if rng.random() < 0.3:
            m0, m1, m2 = (_log_int(rng, 16, 96) for _ in range(3))
            return dict(kind=kind, grid="%dx%dx%d" % (m0, m1, m2), method=method, s=s, nt=_log_int(rng, 4, 16), T=0.25,
                        kappa=kappa, transpose=transpose)
        return dict(kind=kind, grid="%dx%d" % (n0, n1), method=method, s=s, nt=_log_int(rng, 16, 128), T=1.0,
                    kappa=kappa, transpose=transpose)
    if kind == "precond":
        n0, n1 = min(n0, 160), min(n1, 160)
        return dict(kind=kind, grid="%dx%d" % (n0, n1), method=method, s=s, nt=_log_int(rng, 8, 64), T=1.0,
                    kappa=rng.random() < 0.5, mgrit=rng.choice([0, 0, 4]))
    if kind == "solve":
        prec = rng.choice(["fp32", "fp32", "bf16", "fp16", "fp64"])
        disc = rng.choice(["fd", "fd", "fd", "q1"])
        nt = _log_int(rng, 12, 16 if prec == "fp64" or disc == "q1" else 48)
        if prec == "fp64" or disc == "q1":
            n0, n1 = min(n0, 120), min(n1, 120)
        return dict(kind=kind, grid="%dx%d" % (n0, n1), method=method, s=s, nt=nt, T=nt / 64.0, tol=1e-8, prec=prec,
                    disc=disc, mgrit=rng.choice([0, 0, 4, 5, 6]))
    if kind == "solve3d":
        m0, m1, m2 = (_log_int(rng, 24, 72) for _ in range(3))
        nt = _log_int(rng, 4, 8)
        return dict(kind="solve", grid="%dx%dx%d" % (m0, m1, m2), method=method, s=s, nt=nt, T=nt / 64.0, tol=1e-8,
                    prec=rng.choice(["bf16", "fp16", "fp32"]), disc="fd", mgrit=0)
    if kind == "gradient":
        nt = rng.choice([16, 24, 32])
        return dict(kind=kind, grid="%dx%d" % (min(n0, 128), min(n1, 128)), method=method, s=s, nt=nt, T=nt / 64.0,
                    tol=1e-10, prec="fp32", mgrit=rng.choice([0, 4, 8]), ckpt=rng.choice([0, 4, 8]))
    problems = []
    for _ in range(rng.randint(3, 6)):
        N = rng.choice([32, 48, 64, 96, 128, 192]) + rng.choice([0, 0, 1, -3])
        problems.append("%d:%d:%d" % (N, rng.choice([16, 32, 64]), rng.choice([2, 3])))
    return dict(kind="batch", tol=1e-8, prec=rng.choice(["fp32", "bf16"]), problems=" ".join(problems))


# ---------------------------------------------------------------------------------------- inputs

def _grid(text):
    return tuple(int(v) for v in text.split("x"))


def _nx(n):
    return int(np.prod(n))


def _n_st(n, s, nt):
    return _nx(n) * (nt + 1 + s * nt)


def _sqrt_cov(n, ell, boundary):
    x = np.arange(0, n + 2) / (n + 1.0) if boundary else np.arange(1, n + 1) / (n + 1.0)
    d = x[:, None] - x[None, :]
    w, q = np.linalg.eigh(np.exp(-d * d / (2.0 * ell * ell)))
    return (q * np.sqrt(np.clip(w, 0.0, None))) @ q.T


def _field(n, ell, sigma, rng, boundary=False):
    """A separable squared-exponential Gaussian field on the grid, x fastest, on the GPU."""
    roots = [_sqrt_cov(v, ell, boundary) for v in n]
    a = rng.standard_normal([r.shape[0] for r in roots[::-1]])
    for axis in range(len(n)):
        a = np.moveaxis(np.tensordot(roots[len(n) - 1 - axis], a, axes=([1], [axis])), 0, axis)
    return torch.from_numpy((sigma * a).reshape(-1).copy()).to(DEV)


def _kappa(n, rng):
    return torch.exp(_field(n, 0.15, 0.5, rng, boundary=True))


def _source_and_start(n, rng):
    if len(n) == 2:
        return _field(n, 0.1, 1.0, rng), _field(n, 0.1, 1.0, rng)
    u = 1.0
    for axis, v in enumerate(n):
        shape = [1, 1, 1]
        shape[2 - axis] = v
        u = u * np.sin(math.pi * np.arange(1, v + 1) / (v + 1.0)).reshape(shape)
    u0 = (u + 1e-2 * rng.standard_normal(u.shape)).reshape(-1)
    return torch.zeros(u0.size, dtype=torch.float64, device=DEV), torch.from_numpy(u0).to(DEV)


def _inner(prec):
    return dict(inner_maxit=5, inner_tol=1e-6) if prec == "fp64" else dict(inner_maxit=3, inner_tol=1e-3)


def _problems(case):
    return [tuple(int(v) for v in p.split(":")) for p in case["problems"].split()]


def _fields(case, seed):
    """The tensors of a case, from the seed alone."""
    rng = np.random.default_rng([int(seed), 17])
    kind = case["kind"]
    if kind == "batch":
        d = {}
        for k, (N, _, _) in enumerate(_problems(case)):
            d["f%d" % k], d["u%d" % k] = _source_and_start((N, N), rng)
        return d
    n = _grid(case["grid"])
    d = {}
    if kind == "gradient" or case.get("kappa"):
        d["kappa"] = _kappa(n, rng)
    if kind in ("matvec", "precond"):
        g = torch.Generator(device=DEV).manual_seed(int(seed))
        d["x"] = torch.randn(_n_st(n, case["s"], case["nt"]), dtype=torch.float64, device=DEV, generator=g)
    else:
        d["f"], d["u0"] = _source_and_start(n, rng)
        if kind == "gradient":
            d["target"] = _field(n, 0.1, 1.0, rng)
    return d


def prepare(case, seed):
    d = _fields(case, seed)
    kind = case["kind"]
    if kind == "batch":
        d["solvers"], d["streams"], d["out"] = [], [], []
        for N, nt, s in _problems(case):
            st = torch.cuda.Stream(device=DEV)
            d["streams"].append(st)
            d["solvers"].append(Solver((N, N), 1.0, nt, method="radau", s=s, prec_P=case["prec"], tol=case["tol"],
                                       stream=st.cuda_stream, mgrit_m=8 if nt >= 16 else 0, **_inner(case["prec"])))
            d["out"].append(torch.zeros(d["solvers"][-1].n_st, dtype=torch.float64, device=DEV))
        torch.cuda.synchronize()
        d["case"] = case
        return d
    n = _grid(case["grid"])
    if kind == "gradient":
        d["cfg"] = dict(n=n, T=case["T"], nt=case["nt"], method=case["method"], s=case["s"], prec_P=case["prec"],
                        tol=case["tol"], maxit=200, ckpt_every=case["ckpt"], mgrit_m=case["mgrit"],
                        **_inner(case["prec"]))
    else:
        kw = dict(method=case["method"], s=case["s"], kappa=d.get("kappa"))
        if kind == "matvec":
            kw.update(prec_P="fp32", restart=1)
        elif kind == "precond":
            kw.update(restart=1, mgrit_m=case["mgrit"])
        else:
            kw.update(prec_P=case["prec"], tol=case["tol"], disc=case["disc"], mgrit_m=case["mgrit"],
                      **_inner(case["prec"]))
        d["S"] = Solver(n, case["T"], case["nt"], **kw)
        d["out"] = torch.zeros(d["S"].n_st, dtype=torch.float64, device=DEV)
    d["case"] = case
    return d


def run(d):
    case = d["case"]
    kind = case["kind"]
    if kind == "matvec":
        return d["S"].matvec(d["x"], d["out"], transpose=case["transpose"])
    if kind == "precond":
        return d["S"].precond_apply(d["x"], d["out"])
    if kind == "solve":
        return d["S"].solve(d["f"], d["u0"], d["out"])[0]
    if kind == "batch":
        k = range(len(d["solvers"]))
        solve_batched(d["solvers"], [d["f%d" % i] for i in k], [d["u%d" % i] for i in k], d["out"])
        return d["out"]
    f = d["f"].clone().requires_grad_(True)
    kap = d["kappa"].clone().requires_grad_(True)
    x = heat_solve(f, d["u0"], kap, **d["cfg"])
    nx = d["u0"].numel()
    last = x[case["nt"] * nx:(case["nt"] + 1) * nx]
    J = 0.5 * ((last - d["target"]) ** 2).sum() + 0.5e-4 * (f ** 2).sum()
    J.backward()
    return {"J": J.detach(), "grad_f": f.grad, "grad_kappa": kap.grad}


def work(case):
    """Inputs read once and outputs written once; operations of one product with the space-time operator
    (a solve contains several, and its preconditioner)."""
    def product(n, s, nt):
        return float(_nx(n) * nt * ((s + 1) * (4 * len(n) + 1) + 2 * s * s + 2 * s + 2))
    if case["kind"] == "batch":
        p = [((N, N), s, nt) for N, nt, s in _problems(case)]
        return {"bytes": 8.0 * sum(_n_st(*q) + 2 * _nx(q[0]) for q in p), "flops": sum(product(*q) for q in p)}
    n, s, nt = _grid(case["grid"]), case["s"], case["nt"]
    nst, nk = _n_st(n, s, nt), _nx([v + 2 for v in n])
    read = nk if case["kind"] == "gradient" or case.get("kappa") else 0
    if case["kind"] in ("matvec", "precond"):
        return {"bytes": 8.0 * (2 * nst + read), "flops": product(n, s, nt)}
    if case["kind"] == "gradient":
        # f, u0, the target and kappa in, two gradients out; a forward and an adjoint product
        return {"bytes": 8.0 * (4 * _nx(n) + 2 * nk), "flops": 2.0 * product(n, s, nt)}
    return {"bytes": 8.0 * (nst + 2 * _nx(n)), "flops": product(n, s, nt)}


# ---------------------------------------------------------------------------------------- 64-bit values

class _Space:
    """K (and M) of a grid in plain torch, FP64, with the eigenvectors that diagonalise them: the
    type-I sine basis for constant coefficients, a dense symmetric eigensolver for a kappa field."""

    def __init__(self, n, kappa=None, disc="fd"):
        self.n, self.h2 = n, [float((v + 1) ** 2) for v in n]
        self.shape = tuple(n[::-1])
        d = len(n)
        self.face = None
        if kappa is not None:
            k = kappa.reshape([v + 2 for v in n[::-1]])
            self.face = []
            for a in range(d):
                ax = d - 1 - a
                k1 = k
                for b in range(d):      # interior nodes in the other directions
                    if b != ax:
                        k1 = k1.narrow(b, 1, n[d - 1 - b])
                m = n[a]
                self.face.append(0.5 * (k1.narrow(ax, 0, m + 1) + k1.narrow(ax, 1, m + 1)) * self.h2[a])
        self.Q = None
        if kappa is None:
            self.basis, k1, m1 = [], [], []
            for v in n:
                i = torch.arange(1, v + 1, dtype=torch.float64, device=DEV)
                self.basis.append(math.sqrt(2.0 / (v + 1)) * torch.sin(math.pi * torch.outer(i, i) / (v + 1)))
                c = torch.cos(math.pi * i / (v + 1))
                h = 1.0 / (v + 1)
                k1.append((2 - 2 * c) / h if disc == "q1" else (2 - 2 * c) / h ** 2)
                m1.append(h / 6 * (4 + 2 * c) if disc == "q1" else torch.ones_like(c))
            lam = torch.zeros(self.shape, dtype=torch.float64, device=DEV)
            mu = torch.ones(self.shape, dtype=torch.float64, device=DEV)
            for a in range(d):
                t = torch.ones(self.shape, dtype=torch.float64, device=DEV)
                for b in range(d):
                    view = [1] * d
                    view[d - 1 - b] = n[b]
                    t = t * (k1[b] if a == b else m1[b]).reshape(view)
                lam = lam + t
                view = [1] * d
                view[d - 1 - a] = n[a]
                mu = mu * m1[a].reshape(view)
            self.lam, self.mu = lam.reshape(-1), mu.reshape(-1)

    def diagonalise(self):
        """The eigenvectors of a kappa field's K (few unknowns only)."""
        nx = _nx(self.n)
        K = torch.empty(nx, nx, dtype=torch.float64, device=DEV)
        eye = torch.eye(nx, dtype=torch.float64, device=DEV)
        for i in range(0, nx, 256):
            K[i:i + 256] = self.K(eye[i:i + 256])
        self.lam, self.Q = torch.linalg.eigh(0.5 * (K + K.T))
        self.mu = torch.ones_like(self.lam)

    def K(self, u):
        """K applied to the rows of u (FD)."""
        d = len(self.n)
        w = u.reshape((-1,) + self.shape)
        out = torch.zeros_like(w)
        for a in range(d):
            ax = 1 + d - 1 - a
            pad = list(w.shape)
            pad[ax] = 1
            z = torch.zeros(pad, dtype=torch.float64, device=DEV)
            q = torch.cat([z, w, z], ax).diff(dim=ax)
            q = q * (self.h2[a] if self.face is None else self.face[a])
            out = out - q.diff(dim=ax)
        return out.reshape(u.shape)

    def modes(self, u):
        """Coefficients of the rows of u in the eigenbasis (its own inverse for the sine basis)."""
        if self.Q is not None:
            return u.reshape(-1, _nx(self.n)) @ self.Q
        return self._sines(u)

    def points(self, c):
        if self.Q is not None:
            return c.reshape(-1, _nx(self.n)) @ self.Q.T
        return self._sines(c)

    def _sines(self, u):
        d = len(self.n)
        w = u.reshape((-1,) + self.shape)
        for a in range(d):
            w = torch.movedim(torch.tensordot(w, self.basis[a], dims=([1 + d - 1 - a], [0])), -1, 1 + d - 1 - a)
        return w.reshape(-1, _nx(self.n))


def _tableau(case):
    """Closed forms of the methods used: Radau IIA with 2 and 3 stages, Gauss with 2."""
    q, r = math.sqrt(6.0), math.sqrt(3.0)
    A, b = {
        ("radau", 2): ([[5 / 12, -1 / 12], [3 / 4, 1 / 4]], [3 / 4, 1 / 4]),
        ("radau", 3): ([[(88 - 7 * q) / 360, (296 - 169 * q) / 1800, (-2 + 3 * q) / 225],
                        [(296 + 169 * q) / 1800, (88 + 7 * q) / 360, (-2 - 3 * q) / 225],
                        [(16 - q) / 36, (16 + q) / 36, 1 / 9]], [(16 - q) / 36, (16 + q) / 36, 1 / 9]),
        ("gauss", 2): ([[1 / 4, 1 / 4 - r / 6], [1 / 4 + r / 6, 1 / 4]], [1 / 2, 1 / 2]),
    }[(case["method"], case["s"])]
    return (torch.tensor(A, dtype=torch.float64, device=DEV), torch.tensor(b, dtype=torch.float64, device=DEV))


def _product(sp, A, b, tau, nt, x, transpose):
    nx, s = _nx(sp.n), len(b)
    v, V = x[:(nt + 1) * nx].reshape(nt + 1, nx), x[(nt + 1) * nx:].reshape(nt, s, nx)
    KV = sp.K(V)
    if not transpose:
        yv = torch.cat([v[:1], v[1:] - v[:-1] - tau * torch.einsum("i,nip->np", b, V)])
        yV = V + sp.K(v[:-1])[:, None] + tau * torch.einsum("ij,njp->nip", A, KV)
    else:
        yv = torch.cat([v[:-1] - v[1:] + KV.sum(1), v[-1:]])
        yV = V - tau * b[None, :, None] * v[1:, None] + tau * torch.einsum("ji,njp->nip", A, KV)
    return torch.cat([yv.reshape(-1), yV.reshape(-1)])


def _forward(sp, A, b, tau, nt, f, u0):
    """Every state and stage of the Runge--Kutta steps, mode by mode."""
    s = len(b)
    G = torch.linalg.inv(sp.mu[:, None, None] * torch.eye(s, dtype=torch.float64, device=DEV) +
                         tau * sp.lam[:, None, None] * A)
    fh, v = sp.modes(f)[0], sp.modes(u0)[0]
    vs, Vs = [v], []
    for _ in range(nt):
        V = (G @ (sp.mu * fh - sp.lam * v)[:, None, None].expand(-1, s, 1)).squeeze(-1)
        v = v + tau * (V @ b)
        vs.append(v)
        Vs.append(V.T)
    return sp.points(torch.stack(vs)), sp.points(torch.cat(Vs))


def exact(case, seed):
    kind = case["kind"]
    if kind == "precond":
        return None       # P_tilde^{-1} is defined by its own truncated iterations
    d = _fields(case, seed)
    if kind == "batch":
        out = []
        for k, (N, nt, s) in enumerate(_problems(case)):
            A, b = _tableau(dict(method="radau", s=s))
            v, V = _forward(_Space((N, N)), A, b, 1.0 / nt, nt, d["f%d" % k], d["u%d" % k])
            out.append(torch.cat([v.reshape(-1), V.reshape(-1)]))
        return out
    n, nt, tau = _grid(case["grid"]), case["nt"], case["T"] / case["nt"]
    A, b = _tableau(case)
    sp = _Space(n, d.get("kappa"), case.get("disc", "fd"))
    if kind == "matvec":
        return _product(sp, A, b, tau, nt, d["x"], case["transpose"])
    if kind == "solve":
        v, V = _forward(sp, A, b, tau, nt, d["f"], d["u0"])
        return torch.cat([v.reshape(-1), V.reshape(-1)])
    if _nx(n) > 4200:
        return None       # the dense eigensolver takes too long
    return _gradient(sp, A, b, tau, nt, d)


def _gradient(sp, A, b, tau, nt, d):
    sp.diagonalise()
    n, nx, s = sp.n, _nx(sp.n), len(b)
    dim = len(n)
    v, V = _forward(sp, A, b, tau, nt, d["f"], d["u0"])
    V = V.reshape(nt, s, nx)
    r = v[-1] - d["target"]
    J = 0.5 * (r ** 2).sum() + 0.5e-4 * (d["f"] ** 2).sum()
    G = torch.linalg.inv(torch.eye(s, dtype=torch.float64, device=DEV) + tau * sp.lam[:, None, None] * A.T)
    lv, lV = sp.modes(r)[0], [None] * nt
    for i in reversed(range(nt)):
        L = (G @ (tau * b[None, :, None] * lv[:, None, None])).squeeze(-1)
        lv = lv - sp.lam * L.sum(1)
        lV[i] = L.T
    lV = sp.points(torch.cat(lV)).reshape(nt, s, nx)
    W = v[:-1, None] + tau * torch.einsum("ij,njp->nip", A, V)
    gk = torch.zeros([m + 2 for m in n[::-1]], dtype=torch.float64, device=DEV)
    for a in range(dim):
        ax = dim - 1 - a

        def jumps(u):
            w = u.reshape((nt * s,) + sp.shape)
            pad = list(w.shape)
            pad[1 + ax] = 1
            z = torch.zeros(pad, dtype=torch.float64, device=DEV)
            return torch.cat([z, w, z], 1 + ax).diff(dim=1 + ax)
        part = -0.5 * sp.h2[a] * (jumps(lV) * jumps(W)).sum(0)
        g1 = gk
        for c in range(dim):
            if c != ax:
                g1 = g1.narrow(c, 1, n[dim - 1 - c])
        m = n[a] + 1
        g1.narrow(ax, 0, m).add_(part)
        g1.narrow(ax, 1, m).add_(part)
    return {"J": J, "grad_f": lV.sum((0, 1)) + 1e-4 * d["f"], "grad_kappa": gk.reshape(-1)}
