"""Halo-staged products at column counts whose threads do not divide a warp
(marked gpu): 3, 5 and 6 column threads with several entry lanes.  The sums are
the CSR kernel's, so the V-cycles agree bit for bit, and the profile names the
kernel that ran."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from synth import gaussian_logk, rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.mark.parametrize("prec", [amg.PREC_FP64, amg.PREC_MIXED_FP32])
@pytest.mark.parametrize("s,nrhs", [(2, 1), (2, 3), (1, 5), (1, 6), (0, 5)])
def test_halo_at_ragged_column_counts(s, nrhs, prec):
    N = (128, 96, 96)
    g = gaussian_logk(N, s, seed=16, corr=3.0)
    kw = dict(coarse_max=64, sell=0)
    P = amg.Problem.structured(N, 1.5, g, s).setup(halo_kb=32, **kw)
    Q = amg.Problem.structured(N, 1.5, g, s).setup(halo_kb=0, **kw)
    dt = torch.float64 if prec == amg.PREC_FP64 else torch.float32
    R = torch.from_numpy(np.random.default_rng(7).uniform(-1.0, 1.0, (P.n_b, nrhs << s))).to(DEV, dt)
    Za, Zb = (H.vcycle(R, torch.empty_like(R), nrhs, prec) for H in (P, Q))
    assert torch.isfinite(Za).all() and torch.equal(Za, Zb)
    b = torch.from_numpy(rhs_uniform(P.n, nrhs, config=17)).to(DEV)
    used = [r for r in P.profile_step(b, torch.empty_like(b), nrhs, prec) if r["kernel"].startswith("spmm_halo_kernel")]
    assert any(r["role"].startswith("L1 A") or r["role"].startswith("L0 R") for r in used)
