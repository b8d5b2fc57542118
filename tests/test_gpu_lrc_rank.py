"""GMRES restarts shorter than the correction's rank (marked gpu): the step's
coefficient buffer holds whichever is more."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from oracle import solvers  # noqa: E402
from synth import rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
N = (16, 12, 10)  # kappa = 68: a relative residual of 1e-12 is an error of at most 68e-12


@pytest.mark.parametrize("rank,restart,nrhs", [(16, 1, 1), (16, 4, 3), (11, 4, 1), (12, 4, 2), (24, 10, 1)])
def test_rank_above_the_restart(rank, restart, nrhs):
    P = amg.Problem.structured(N, 0.0, None, 2).setup(coarse_max=40).lrc_setup(rank)
    b = rhs_uniform(P.n, nrhs, config=97)
    x, info = P.solve_gmres(torch.from_numpy(b).to("cuda"), restart=restart, lrc=True, tol=1e-12, maxit=400)
    ref = solvers.dst_solve(N, b).reshape(b.shape)
    err = np.linalg.norm(x.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert info.converged and err.max() <= 68e-12
