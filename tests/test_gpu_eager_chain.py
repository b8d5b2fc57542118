"""Eager chains of launches, whose kernels may start while their predecessors
drain, against the same chains without that (marked gpu): captured by the
caller, where every launch is an ordinary one.  The kernels and their order are
the same, so the results are equal bit for bit.  And what a handle's first calls
rest on: setups and first solves of many new handles agree bit for bit."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from synth import gaussian_logk, rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


def _captured(call):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        call()
    g.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("N,s,nrhs", [((62, 50, 37), 1, 3), ((64, 48, 40), 3, 1), ((40, 36, 30), 2, 4), ((60, 44), 1, 1)])
@pytest.mark.parametrize("prec", [amg.PREC_FP64, amg.PREC_MIXED_FP32])
@pytest.mark.parametrize("form", ["vcycle", "vcycle_noalloc", "amgr_apply"])
def test_chains_equal_captured_ones(N, s, nrhs, prec, form):
    g = gaussian_logk(N, s, seed=33, corr=3.0)
    P = amg.Problem.structured(N, 1.5, g, s).setup(coarse_max=40, amgr=int(form == "amgr_apply"))
    apply = getattr(P, form)
    dt = torch.float64 if prec == amg.PREC_FP64 else torch.float32
    R = torch.from_numpy(np.random.default_rng(nrhs).uniform(-1.0, 1.0, (P.n_b, nrhs << s))).to(DEV, dt)
    Z = [torch.empty_like(R) for _ in range(8)]
    H = torch.empty_like(R)

    def chain():  # back to back, every second call on the result of the one before
        for z in Z:
            apply(R, H, nrhs, prec)
            apply(H, z, nrhs, prec)

    chain()
    torch.cuda.synchronize()
    eager = [z.clone() for z in Z]
    assert all(torch.isfinite(z).all() for z in eager)
    for z in Z:
        z.fill_(float("nan"))
    _captured(chain)
    assert all(torch.equal(a, z) for a, z in zip(eager, Z))


@pytest.mark.parametrize("prec", [amg.PREC_FP64, amg.PREC_MIXED_FP32])
@pytest.mark.parametrize("form", ["vcycle", "amgr_apply"])
def test_a_graph_behind_a_chain_sees_its_result(form, prec):
    N, s, nrhs = (64, 48, 40), 2, 2
    g = gaussian_logk(N, s, seed=36, corr=3.0)
    P = amg.Problem.structured(N, 1.5, g, s).setup(coarse_max=40, amgr=int(form == "amgr_apply"))
    apply = getattr(P, form)
    dt = torch.float64 if prec == amg.PREC_FP64 else torch.float32
    rng = np.random.default_rng(11)
    R = [torch.from_numpy(rng.uniform(-1.0, 1.0, (P.n_b, nrhs << s))).to(DEV, dt) for _ in range(4)]
    ref = [apply(r, torch.empty_like(r), nrhs, prec).clone() for r in R]
    Z, Y = torch.empty_like(R[0]), torch.empty_like(R[0])
    graph = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        Y.copy_(Z)
    for k in range(200):
        Z.fill_(float("nan"))
        apply(R[k % 4], Z, nrhs, prec)
        graph.replay()
        assert torch.equal(Y, ref[k % 4]), k


@pytest.mark.parametrize("N,s,nrhs,count", [((32, 28, 24), 3, 4, 60), ((64, 64, 64), 3, 1, 30)])
def test_new_handles_agree(N, s, nrhs, count):
    g = gaussian_logk(N, s, seed=34, corr=3.0)
    first = None
    for k in range(count):
        P = amg.Problem.structured(N, 1.5, g, s).setup(coarse_max=40)
        b = torch.from_numpy(rhs_uniform(P.n, nrhs, config=91)).to(DEV)
        x, info = P.solve(b, tol=1e-12, precision=amg.PREC_MIXED_FP32)
        assert info.converged
        omega = [P.level_info(l)["omega"] for l in range(P.num_levels() - 1)]
        if first is None:
            first = (omega, x, info.iters)
        assert omega == first[0] and info.iters == first[2] and torch.equal(x, first[1]), k
        P.close()


def test_damping_of_a_larger_hierarchy_matches_the_host_estimate():
    N, s = (128, 112, 96), 3
    g = gaussian_logk(N, s, seed=35, corr=4.0)
    P = amg.Problem.structured(N, 1.5, g, s).setup()
    H = amg.Problem.structured(N, 1.5, g, s).setup(host_only=1)
    assert P.num_levels() == H.num_levels() >= 4
    for l in range(P.num_levels() - 1):  # 30 power steps, each to rounding of sums of up to 172k terms
        w, wh = P.level_info(l)["omega"], H.level_info(l)["omega"]
        assert abs(w - wh) <= 1e-9 * wh, (l, w, wh)


def test_gmres_steps_repeat_bit_for_bit():
    N, s = (32, 32, 32), 3
    P = amg.Problem.structured(N, 1.5, None, s, "neumann").setup(coarse_max=40).lrc_setup(4)
    b = torch.from_numpy(rhs_uniform(P.n, 2, config=92)).to(DEV)
    b -= b.mean(1, keepdim=True)
    x, info = P.solve_gmres(b, restart=20, lrc=True, tol=1e-10)
    assert info.converged
    for _ in range(20):
        y, again = P.solve_gmres(b, restart=20, lrc=True, tol=1e-10)
        assert again.iters == info.iters and torch.equal(x, y)
