"""The flagged (interface) rows taken by blocks of their own (marked gpu), over
the sizes where the split of the blocks changes: everything resident at once or
not, one, two and three mirror planes, few columns and many.  Against the
problem's own blocks A^_i (the oracle's differ from them by 1e-14 of a row sum,
from the rounding of the grid's widths): each value is a sum of at most 10 products, so FP64 agrees to
1e-14 and FP32 to 1e-6 of the sum of magnitudes, bounded here by the largest row
sum of |A^| times the largest input."""

import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from gpu_common import oracle_apply_hat, oracle_problem  # noqa: E402

pytestmark = pytest.mark.gpu


def _blocks(P):
    rp, ci, v = P.inner_block()
    shape = (P.n_b, P.n_b)
    row, col, val = P.interface()
    inner = sp.csr_matrix((v, ci, rp), shape=shape)
    return [inner + sp.csr_matrix((val[:, i], (row, col)), shape=shape) for i in range(P.nb)]


@pytest.mark.parametrize("N,s", [((16, 12, 10), 3), ((48, 40, 36), 1), ((48, 40, 36), 2), ((48, 40, 36), 3), ((120, 90), 1),
                                 ((120, 90), 2)])
@pytest.mark.parametrize("nrhs", [1, 3, 16, 32])
def test_reduced_product(N, s, nrhs):
    g = oracle_problem(N, s, gamma=1.5, vark=True)[0]
    P = amg.Problem.structured(N, 1.5, g, s).setup(coarse_max=64)
    hat = _blocks(P)
    X = np.random.default_rng(nrhs).uniform(-1.0, 1.0, (P.n_b, nrhs << s))
    for prec, dt, eps in ((amg.PREC_FP64, torch.float64, 1e-14), (amg.PREC_MIXED_FP32, torch.float32, 1e-6)):
        Xt = torch.from_numpy(X).to("cuda", dt)
        ref = oracle_apply_hat(hat, Xt.double().cpu().numpy(), P.nb)
        Y = P.apply_reduced(Xt, torch.full_like(Xt, float("nan")), nrhs, prec).double().cpu().numpy()
        mag = max(abs(B).sum(axis=1).max() for B in hat)
        assert np.abs(Y - ref).max() <= eps * mag
