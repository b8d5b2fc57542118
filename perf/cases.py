"""The measured work of the library: its solves and their building blocks, through the Python binding.

A case is a dict of plain values.  ``prepare`` returns what a program holds before the call: the problem handle with
its hierarchy (built once per problem and kept, as a program that solves for many right-hand sides keeps it) and the
vectors of this call, drawn on the GPU from the seed.  ``run`` is one call of the public entry point.

Solves run to a relative residual of 1e-12, the tolerance of the repository's FP64 parity tests, so that the solution
is determined to about 1e-10 and two runs can be compared.  The sizes are those of the repository's workloads
(``synth.CONFIGS``, the batched recipe, the model problem) and ragged ones between them.
"""

from __future__ import annotations

import math
from functools import lru_cache

import numpy as np
import torch

import paper_2407_05930_gb300 as amg
from paper_2407_05930_gb300.autograd import SymPoisson

DEV = "cuda"
TOL = 1e-12
PREC = {"fp64": amg.PREC_FP64, "fp32": amg.PREC_MIXED_FP32, "bf16": amg.PREC_MIXED_BF16}


def listed():
    big = dict(nx=256, ny=256, nz=256, s=3, gamma=1.5, vark=True, nrhs=1)
    return [
        # the benchmark's workload: one right-hand side of the stretched variable-coefficient cube, mixed precision
        dict(big, name="solve mixed 256cube", kind="solve", prec="fp32"),
        # the preconditioner alone, for a caller with a Krylov method of its own
        dict(big, name="vcycle fp32 256cube", kind="vcycle", prec="fp32"),
        # the reduced operator alone (a residual check, a time step)
        dict(big, name="operator fp32 256cube", kind="apply", prec="fp32"),
        # the change of basis there and back
        dict(big, name="transforms 256cube", kind="transform"),
        # the adjoint workload: differentiable FP64 solve, gradients of the right-hand side and of log k
        dict(name="adjoint fp64 192cube", kind="adjoint", nx=192, ny=192, nz=192, s=3, gamma=1.5, vark=True, nrhs=1),
        # the multigrid reduction as preconditioner: the fewest iterations
        dict(name="solve amgr mixed 160cube", kind="solve", nx=160, ny=160, nz=160, s=3, gamma=1.5, vark=True, nrhs=1,
             prec="fp32", amgr=True),
        # several right-hand sides at once on the uniform cube
        dict(name="solve mixed 128cube 4rhs", kind="solve", nx=128, ny=128, nz=128, s=3, gamma=0.0, vark=False, nrhs=4,
             prec="fp32"),
        # ragged sizes, one unmirrored odd axis, an odd number of right-hand sides, FP64 throughout
        dict(name="solve fp64 ragged 3rhs", kind="solve", nx=90, ny=76, nz=51, s=2, gamma=1.5, vark=True, nrhs=3,
             prec="fp64"),
        # a batch of uneven problems with 16 right-hand sides each
        dict(name="batch 8 problems 16rhs", kind="batch", problems=8, nmin=32, nmax=96, sizes=7, nrhs=16, prec="fp32"),
        # the paper's model problem: Neumann walls, GMRES with the rank-8 correction
        dict(name="gmres lrc neumann 64cube", kind="gmres", nx=64, ny=64, nz=64, s=3, gamma=1.5, vark=False, nrhs=1,
             rank=8),
        # a small preconditioner application with a ragged column count: bound by latency
        dict(name="vcycle fp32 ragged 3rhs", kind="vcycle", nx=62, ny=50, nz=37, s=1, gamma=1.5, vark=True, nrhs=3,
             prec="fp32"),
        # the smallest workload: a 2D solve, launches and host work only
        dict(name="solve fp64 2d 64x64", kind="solve", nx=64, ny=64, nz=0, s=1, gamma=0.0, vark=False, nrhs=1,
             prec="fp64"),
    ]


def _even(v):
    return max(8, 2 * round(v / 2))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "vcycle", "vcycle", "apply", "transform", "adjoint", "batch", "gmres"])
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 10), nmin=rng.choice([20, 32]), nmax=rng.choice([48, 64, 96]),
                    sizes=rng.randint(0, 9999), nrhs=rng.choice([1, 4, 8, 16]), prec="fp32")
    two_d = kind in ("solve", "vcycle") and rng.random() < 0.15
    top = {"gmres": 80, "adjoint": 144, "solve": 176}.get(kind, 224)
    edge = math.exp(rng.uniform(math.log(40 if two_d else 20), math.log(400 if two_d else top)))
    s = rng.randint(1, 2) if two_d else rng.randint(1, 3)
    N = [edge * math.exp(rng.uniform(-0.25, 0.25)) for _ in range(2 if two_d else 3)]
    N = [_even(v) if a < s else max(8, round(v)) for a, v in enumerate(N)]
    vol = math.prod(N)
    nrhs = rng.choice([1, 1, 1, 2, 3, 4, 8])
    while nrhs > 1 and nrhs * vol > 6_000_000:
        nrhs -= 1
    c = dict(kind=kind, nx=N[0], ny=N[1], nz=0 if two_d else N[2], s=s, gamma=rng.choice([0.0, 1.5]),
             vark=rng.random() < 0.5, nrhs=nrhs)
    if kind == "gmres":
        c.update(vark=False, rank=rng.choice([0, 4, 8]), nrhs=min(nrhs, 2))
    elif kind == "adjoint":
        c.update(nrhs=1)
    elif kind == "solve":
        c.update(prec=rng.choice(["fp64", "fp32", "fp32", "bf16"]))
        if not two_d and rng.random() < 0.3:
            c.update(amgr=True)
    elif kind in ("vcycle", "apply"):
        c.update(prec=rng.choice(["fp64", "fp32", "fp32"]))
    return c


# ----------------------------------------------------------------------------
# problems

def _grid(case):
    return (case["nx"], case["ny"]) if not case["nz"] else (case["nx"], case["ny"], case["nz"])


def _log_k(N, s, corr=8.0):
    """A smooth random log-coefficient of unit variance, mirror-symmetric bit for bit: white noise on the base cells
    smoothed by a Gaussian of `corr` cells with reflecting ends, then reflected across the first s axes."""
    base = [n // 2 if a < s else n for a, n in enumerate(N)]
    f = np.random.default_rng(3000).standard_normal(base[::-1])
    for ax, n in enumerate(base[::-1]):
        i = np.arange(n)
        w = np.exp(-0.5 * ((i[:, None] - i[None, :]) / corr) ** 2) + np.exp(-0.5 * ((i[:, None] + i[None, :] + 1) / corr) ** 2)
        w += np.exp(-0.5 * ((2 * n - 1 - i[:, None] - i[None, :]) / corr) ** 2)
        f = np.moveaxis(np.tensordot(w / w.sum(1, keepdims=True), f, (1, ax)), 0, ax)
    f = (f - f.mean()) / f.std()
    for a in range(s):
        ax = len(N) - 1 - a
        f = np.concatenate([f, np.flip(f, ax)], ax)
    return np.ascontiguousarray(f).reshape(-1)


def _coefficient(N, s, vark):
    return _log_k(N, s) if vark else None


@lru_cache(maxsize=3)
def _problem(N, s, gamma, vark, bc, setup):
    return amg.Problem.structured(N, gamma, _coefficient(N, s, vark), s, bc).setup(**dict(setup))


@lru_cache(maxsize=1)
def _corrected(N, s, gamma, rank):
    P = amg.Problem.structured(N, gamma, None, s, "neumann").setup()
    return P.lrc_setup(rank) if rank else P


@lru_cache(maxsize=1)
def _differentiable(N, s, gamma, vark):
    g = _coefficient(N, s, vark)
    return SymPoisson(N, gamma, s, solve_kw=dict(tol=TOL)), np.zeros(math.prod(N)) if g is None else g


def _batch_specs(case):
    rng = np.random.default_rng(case["sizes"])
    evens = np.arange(case["nmin"], case["nmax"] + 1, 2)
    return tuple((int(rng.choice(evens)), int(rng.integers(1, 4))) for _ in range(case["problems"]))


@lru_cache(maxsize=1)
def _batch(specs, nrhs):
    return amg.Batch([amg.Problem.structured((n,) * 3, 0.0, None, s).setup(coarse_max=64) for n, s in specs],
                     [nrhs] * len(specs))


def _handle(case):
    setup = {}
    if case.get("amgr"):
        setup["amgr"] = 1
    if case.get("prec") == "bf16":
        setup["precisions"] = 7
    return _problem(_grid(case), case["s"], case["gamma"], case["vark"], "dirichlet", tuple(sorted(setup.items())))


def _rhs(case, seed, n, nrhs, index=0):
    gen = torch.Generator(device=DEV).manual_seed(1000 * seed + index)
    return torch.rand((nrhs, n), generator=gen, dtype=torch.float64, device=DEV).mul_(2.0).sub_(1.0)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        B = _batch(_batch_specs(case), case["nrhs"])
        bs = [_rhs(case, seed, p.n, case["nrhs"], i) for i, p in enumerate(B.problems)]
        return dict(kind=kind, B=B, bs=bs, xs=[torch.empty_like(b) for b in bs])
    N, nrhs = _grid(case), case["nrhs"]
    n = math.prod(N)
    if kind == "adjoint":
        op, g = _differentiable(N, case["s"], case["gamma"], case["vark"])
        b = _rhs(case, seed, n, 1)[0]
        return dict(kind=kind, op=op, b=b.requires_grad_(), g=torch.from_numpy(g).to(DEV).requires_grad_(),
                    target=_rhs(case, seed, n, 1, 1)[0])
    if kind == "gmres":
        P = _corrected(N, case["s"], case["gamma"], case["rank"])
        b = _rhs(case, seed, n, nrhs)
        return dict(kind=kind, P=P, b=b - b.mean(1, keepdim=True), lrc=case["rank"] > 0)
    P = _handle(case)
    st = dict(kind=kind, P=P, nrhs=nrhs)
    if kind == "solve":
        st.update(b=_rhs(case, seed, n, nrhs), x=torch.empty((nrhs, n), dtype=torch.float64, device=DEV),
                  kw=dict(tol=TOL, precision=PREC[case["prec"]],
                          preconditioner=amg.PC_AMGR if case.get("amgr") else amg.PC_AMG))
    elif kind == "transform":
        st.update(b=_rhs(case, seed, n, nrhs), x=torch.empty((nrhs, n), dtype=torch.float64, device=DEV),
                  xh=torch.empty((P.n_b, nrhs * P.nb), dtype=torch.float64, device=DEV))
    else:  # reduced vectors [n_b][nrhs * 2^s]
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        X = _rhs(case, seed, nrhs * P.nb, P.n_b).to(dt)
        st.update(X=X, Y=torch.empty_like(X), prec=PREC[case["prec"]])
    return st


def run(state):
    kind = state["kind"]
    if kind == "solve":
        x, info = state["P"].solve(state["b"], state["x"], **state["kw"])
        if not info.converged:
            raise RuntimeError(f"not converged: {info}")
        return x
    if kind == "vcycle":
        return state["P"].vcycle(state["X"], state["Y"], state["nrhs"], state["prec"])
    if kind == "apply":
        return state["P"].apply_reduced(state["X"], state["Y"], state["nrhs"], state["prec"])
    if kind == "transform":
        P = state["P"]
        P.transform_forward(state["b"], state["nrhs"], state["xh"])
        P.transform_backward(state["xh"], state["nrhs"], state["x"])
        return dict(reduced=state["xh"], natural=state["x"])
    if kind == "adjoint":
        u = state["op"](state["b"], state["g"])
        loss = (u - state["target"]).square().sum()
        gb, gg = torch.autograd.grad(loss, (state["b"], state["g"]))
        return dict(u=u.detach(), grad_b=gb, grad_logk=gg)
    if kind == "gmres":
        x, info = state["P"].solve_gmres(state["b"], restart=60, lrc=state["lrc"], tol=TOL)
        if not info.converged:
            raise RuntimeError(f"not converged: {info}")
        return x
    xs, infos = state["B"].solve(state["bs"], state["xs"], tol=TOL)
    if not all(i.converged for i in infos):
        raise RuntimeError("a problem of the batch did not converge")
    return xs


def work(case):
    """Inputs read once and outputs written once: the vectors of the call and one copy of the base block's operator
    (a solve cannot do without more than one pass, but how many is the method's choice)."""
    if case["kind"] == "batch":
        cells = [(n ** 3, n ** 3 >> s, 7) for n, s in _batch_specs(case)]
    else:
        N = _grid(case)
        cells = [(math.prod(N), math.prod(N) >> case["s"], 2 * len(N) + 1)]
    nrhs, size = case["nrhs"], 4 if case["kind"] in ("vcycle", "apply") and case["prec"] != "fp64" else 8
    bytes_, flops = 0, 0
    for n, n_b, pts in cells:
        if case["kind"] == "transform":
            bytes_ += 4 * 8 * n * nrhs + 2 * 4 * n  # there and back, and the permutation each way
            flops += 2 * case["s"] * n * nrhs
        elif case["kind"] == "adjoint":
            bytes_ += 8 * (6 * n + pts * n_b)
            flops += 4 * pts * n
        else:
            # symmetric stencil: the diagonal and one of each pair
            bytes_ += size * (2 * n * nrhs + (pts + 1) // 2 * n_b)
            flops += 2 * pts * n * nrhs
    return dict(bytes=bytes_, flops=flops)


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch

def _shape(N):
    return tuple(reversed(N))


def _widths(n, gamma):
    if gamma == 0.0:
        return np.full(n, 1.0 / n)
    x = np.tanh(gamma * (2.0 * np.arange(n + 1) / n - 1.0)) / (2.0 * math.tanh(gamma)) + 0.5
    h = np.diff(x)
    return 0.5 * (h + h[::-1])


def _faces(N, gamma, k):
    """Per grid axis: (interior face transmissibilities, low wall, high wall), arrays over the cells."""
    d = len(N)
    h = [torch.from_numpy(_widths(n, gamma)).to(DEV) for n in N]
    hb = [v.reshape([-1 if d - 1 - ax == a else 1 for ax in range(d)]) for a, v in enumerate(h)]
    out = []
    for a in range(d):
        ax = d - 1 - a
        area = torch.ones([1] * d, dtype=torch.float64, device=DEV)
        for b in range(d):
            if b != a:
                area = area * hb[b]
        r = hb[a] / (2.0 * k)
        n = N[a]
        t = area / (r.narrow(ax, 0, n - 1) + r.narrow(ax, 1, n - 1))
        out.append((t, area / r.narrow(ax, 0, 1), area / r.narrow(ax, n - 1, 1)))
    return out


def _apply_full(N, faces, v):
    """A v on the whole grid (homogeneous Dirichlet walls); v: [..., Nz, Ny, Nx]."""
    d = len(N)
    out = torch.zeros_like(v)
    for a, (t, lo, hi) in enumerate(faces):
        ax = v.dim() - 1 - a
        n = N[a]
        flux = t * (v.narrow(ax, 1, n - 1) - v.narrow(ax, 0, n - 1))
        out.narrow(ax, 0, n - 1).sub_(flux)
        out.narrow(ax, 1, n - 1).add_(flux)
        out.narrow(ax, 0, 1).add_(lo * v.narrow(ax, 0, 1))
        out.narrow(ax, n - 1, 1).add_(hi * v.narrow(ax, n - 1, 1))
    return out


def _mirror_copies(v, N, s):
    """The 2^s reflections of the base cells: [copies, ..., base shape]."""
    d = len(N)
    got = []
    for j in range(1 << s):
        w = v
        for a in range(s):
            if j >> a & 1:
                w = w.flip(v.dim() - 1 - a)
        for a in range(s):
            w = w.narrow(v.dim() - 1 - a, 0, N[a] // 2)
        got.append(w)
    return torch.stack(got)


def _hadamard(s):
    return torch.tensor([[(-1.0) ** bin(i & j).count("1") for j in range(1 << s)] for i in range(1 << s)],
                        dtype=torch.float64, device=DEV)


def _to_reduced(v, N, s):
    """[nrhs, grid] -> [n_b, nrhs * 2^s]: unnormalised butterfly over the mirror copies."""
    nrhs = v.shape[0]
    c = _mirror_copies(v.reshape(nrhs, *_shape(N)), N, s).reshape(1 << s, nrhs, -1)
    return torch.einsum("ij,jrl->lri", _hadamard(s), c).reshape(-1, nrhs << s).contiguous()


def _from_reduced(X, N, s):
    """The inverse of _to_reduced: [n_b, nrhs * 2^s] -> [nrhs, grid]."""
    d, nb = len(N), 1 << s
    nrhs = X.shape[1] // nb
    base = [n // 2 if a < s else n for a, n in enumerate(N)]
    c = torch.einsum("ji,lri->jrl", _hadamard(s), X.reshape(-1, nrhs, nb)) / nb
    c = c.reshape(nb, nrhs, *_shape(base))
    for a in range(s):  # axis a: copies with bit a clear are the lower half, the others its reflection
        ax = c.dim() - 1 - a
        step = c.reshape(c.shape[0] // 2, 2, *c.shape[1:])
        c = torch.cat([step[:, 0], step[:, 1].flip(ax)], ax)
    return c.reshape(nrhs, -1)


def _sine_solve(N, b):
    """The exact solution for k = 1 on the uniform grid: A is diagonal in the basis sin(pi m (i + 1/2) / N)."""
    d = len(N)
    v = b.reshape(b.shape[0], *_shape(N))
    lam = torch.zeros([1] * d, dtype=torch.float64, device=DEV)
    bases = []
    for a, n in enumerate(N):
        ax = d - 1 - a
        m = torch.arange(1, n + 1, dtype=torch.float64, device=DEV)
        i = torch.arange(n, dtype=torch.float64, device=DEV) + 0.5
        S = torch.sin(math.pi / n * m[:, None] * i[None, :]) * math.sqrt(2.0 / n)
        S[-1] *= math.sqrt(0.5)
        t = math.prod(1.0 / q for q in N) * n * n  # face area over cell width
        lam = lam + (t * (2.0 - 2.0 * torch.cos(math.pi * m / n))).reshape([-1 if x == ax else 1 for x in range(d)])
        bases.append(S)
        v = torch.movedim(torch.tensordot(v, S, ([ax + 1], [1])), -1, ax + 1)
    v = v / lam
    for a, S in enumerate(bases):
        ax = d - 1 - a
        v = torch.movedim(torch.tensordot(v, S, ([ax + 1], [0])), -1, ax + 1)
    return v.reshape(b.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_sine_solve((n,) * 3, _rhs(case, seed, n ** 3, case["nrhs"], i))
                for i, (n, _) in enumerate(_batch_specs(case))]
    N, s, nrhs = _grid(case), case["s"], case["nrhs"]
    n = math.prod(N)
    if kind == "solve":
        uniform = case["gamma"] == 0.0 and not case["vark"]
        return _sine_solve(N, _rhs(case, seed, n, nrhs)) if uniform else None
    if kind == "transform":
        b = _rhs(case, seed, n, nrhs)
        return dict(reduced=_to_reduced(b, N, s), natural=b)
    if kind == "apply":
        dt = torch.float64 if case["prec"] == "fp64" else torch.float32
        X = _rhs(case, seed, nrhs << s, n >> s).to(dt).double()
        g = _coefficient(N, s, case["vark"])
        k = torch.ones(n, dtype=torch.float64, device=DEV) if g is None else torch.from_numpy(np.exp(g)).to(DEV)
        faces = _faces(N, case["gamma"], k.reshape(_shape(N)))
        v = _from_reduced(X, N, s)
        return _to_reduced(_apply_full(N, faces, v.reshape(nrhs, *_shape(N))).reshape(nrhs, -1), N, s)
    return None
