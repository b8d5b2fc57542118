"""Vectors of the caller at every address its contract allows, a multiple of 16
bytes (marked gpu): the same results as at multiples of 32 or more."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from synth import gaussian_logk  # noqa: E402

pytestmark = pytest.mark.gpu


def _at(x, shift):
    """A copy of x `shift` bytes past a 256-byte boundary."""
    buf = torch.empty(x.numel() + 64, dtype=x.dtype, device="cuda")
    off = (-buf.data_ptr() % 256 + shift) // x.element_size()
    v = buf[off:off + x.numel()].view(x.shape)
    assert v.data_ptr() % 256 == shift
    return v.copy_(x)


@pytest.mark.parametrize("prec,dt", [(amg.PREC_FP64, torch.float64), (amg.PREC_MIXED_FP32, torch.float32)])
@pytest.mark.parametrize("zmarch", [0, 1])
@pytest.mark.parametrize("s,nrhs", [(3, 1), (2, 3), (3, 4)])
def test_vectors_at_multiples_of_16_bytes(prec, dt, zmarch, s, nrhs):
    N = (64, 64, 32)
    P = amg.Problem.structured(N, 1.5, gaussian_logk(N, s, seed=41, corr=3.0), s).setup(
        coarse_max=40, zmarch=zmarch, amgr=1 - zmarch)
    X = torch.from_numpy(np.random.default_rng(s).uniform(-1.0, 1.0, (P.n_b, nrhs << s))).to("cuda", dt)
    calls = [P.apply_reduced, P.vcycle, P.vcycle_noalloc] + ([] if zmarch else [P.amgr_apply])
    for call in calls:
        ref = call(X, torch.empty_like(X), nrhs, prec)
        for si, so in ((16, 0), (0, 16), (16, 16), (48, 80)):
            Y = call(_at(X, si), _at(torch.zeros_like(X), so), nrhs, prec)
            # column sums may be grouped otherwise: a few hundred roundings
            tol = 1e-12 if dt == torch.float64 else 1e-5
            assert (Y - ref).norm() <= tol * ref.norm(), (call.__name__, si, so)
