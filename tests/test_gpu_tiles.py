"""Entry lanes and shared epilogues of the CSR products at the column counts
where the layout changes (marked gpu): slots that divide a warp and that do not
(3, 5, 6, 7, 12 column threads), one column per thread, few rows (many lanes)
and many.  A level's products run inside the V-cycle, so its linear action is
compared with the same cycle of the oracle-free host matrices in FP64: the
FP64 cycle to 1e-12 relative (a few hundred roundings of 1e-16 amplified by the
cycle's norm, below 10), the FP32 cycle to 1e-5 (the same count of 6e-8)."""

import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from synth import gaussian_logk  # noqa: E402

pytestmark = pytest.mark.gpu


def _mat(P, l, which):
    rp, ci, v, shape = P.level_matrix(l, which)
    return sp.csr_matrix((v, ci, rp), shape=shape)


def _vcycle(P, l, y):
    """V(1,1) of the hierarchy's host matrices, FP64."""
    A = _mat(P, l, "A")
    if l == P.num_levels() - 1:
        return np.linalg.solve(A.toarray(), y)
    G, Pm, w = _mat(P, l, "G"), _mat(P, l, "P"), P.level_info(l)["omega"]
    z = w * (G.T @ (G @ y))
    z = z + Pm @ _vcycle(P, l + 1, Pm.T @ (y - A @ z))
    return z + w * (G.T @ (G @ (y - A @ z)))


@pytest.mark.parametrize("N,s", [((24, 20, 18), 1), ((40, 36, 30), 0), ((60, 44), 1)])
@pytest.mark.parametrize("nrhs", [1, 3, 5, 7, 9, 12, 20, 24])
def test_vcycle_against_host_matrices(N, s, nrhs):
    g = gaussian_logk(N, s, seed=5, corr=3.0)
    P = amg.Problem.structured(N, 1.0, g, s).setup(coarse_max=40)
    C = nrhs << s
    R = np.random.default_rng(nrhs).uniform(-1.0, 1.0, (P.n_b, C))
    ref = _vcycle(P, 0, R)
    for prec, dt, tol in ((amg.PREC_FP64, torch.float64, 1e-12), (amg.PREC_MIXED_FP32, torch.float32, 1e-5)):
        Rt = torch.from_numpy(R).to("cuda", dt)
        Z = P.vcycle(Rt, torch.empty_like(Rt), nrhs, prec).double().cpu().numpy()
        assert np.linalg.norm(Z - ref) <= tol * np.linalg.norm(ref)
