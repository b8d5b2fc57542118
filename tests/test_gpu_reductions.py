"""Column counts at the edges of the reductions (marked gpu): the fused dots of
the PCG, the multi-vector dots of the GMRES and the dense coarsest solve, with
one row slot per warp or many, slots that do and do not divide a warp, odd
counts and the largest.  Each solve is compared with the exact one: the error
of a solution of relative residual 1e-12 is at most kappa * 1e-12, and kappa =
4 (16^2 + 12^2 + 10^2) / (3 pi^2) = 68 on this grid."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from oracle import solvers  # noqa: E402
from synth import rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
N = (16, 12, 10)
BOUND = 68e-12

#: (s, nrhs): 1, 3, 5, 6, 12, 20, 24, 32, 64, 72, 136, 256 columns
COLUMNS = [(0, 1), (0, 3), (0, 5), (1, 3), (2, 3), (2, 5), (3, 3), (3, 4), (3, 8), (3, 9), (3, 17), (3, 32)]


def _worst(x, b):
    x = x.cpu().numpy()
    ref = solvers.dst_solve(N, b).reshape(x.shape)
    return max(np.linalg.norm(x[r] - ref[r]) / np.linalg.norm(ref[r]) for r in range(x.shape[0]))


@pytest.mark.parametrize("s,nrhs", COLUMNS)
@pytest.mark.parametrize("prec", [amg.PREC_FP64, amg.PREC_MIXED_FP32])
def test_pcg_column_counts(s, nrhs, prec):
    P = amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=40)
    b = rhs_uniform(P.n, nrhs, config=60 + s)
    x, info = P.solve(torch.from_numpy(b).to("cuda"), tol=1e-12, precision=prec)
    assert info.converged and _worst(x, b) <= BOUND


@pytest.mark.parametrize("s,nrhs", COLUMNS)
def test_gmres_column_counts(s, nrhs):
    P = amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=40)
    b = rhs_uniform(P.n, nrhs, config=70 + s)
    x, info = P.solve_gmres(torch.from_numpy(b).to("cuda"), restart=25, tol=1e-12, maxit=400)
    assert info.converged and _worst(x, b) <= BOUND


@pytest.mark.parametrize("nrhs", [1, 3, 16, 32])
@pytest.mark.parametrize("coarse_max", [20, 64, 300])
def test_batch_coarsest_solves(nrhs, coarse_max):
    probs = [amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=coarse_max) for s in (1, 2)]
    bs = [rhs_uniform(p.n, nrhs, config=80 + i) for i, p in enumerate(probs)]
    xs, res = amg.Batch(probs, [nrhs] * 2).solve([torch.from_numpy(b).to("cuda") for b in bs], tol=1e-12)
    assert all(r.converged for r in res)
    for x, b in zip(xs, bs):
        assert _worst(x, b) <= BOUND


@pytest.mark.parametrize("s,nrhs", [(0, 1), (2, 3), (3, 4)])
def test_pcg_large_magnitudes(s, nrhs):
    """FP32 partials of 2^90 and more (squares of residuals of 1e15) take the
    FP64 sums of the fused dots; the same bound holds."""
    P = amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=40)
    b = rhs_uniform(P.n, nrhs, config=90 + s) * 1e15
    x, info = P.solve(torch.from_numpy(b).to("cuda"), tol=1e-12, precision=amg.PREC_MIXED_FP32)
    assert info.converged and _worst(x, b) <= BOUND
