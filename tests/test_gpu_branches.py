"""Branches of the transforms and of the GMRES step that ordinary inputs do not
reach (marked gpu): reduced vectors at addresses that allow vectors of 32, 16 or
8 bytes, results the exponent arithmetic of 2^-s does not cover (zeros,
subnormals, infinities, NaN, the smallest normal numbers), and columns whose
next Krylov vector has no norm."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from oracle import solvers  # noqa: E402
from synth import rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
N = (16, 12, 10)


def _mirror(P, s):
    return torch.from_numpy(amg.mirror_perm(N, s).astype(np.int64)).to("cuda")  # [2^s][n_b]


def _butterfly(v):  # [2^s][...], the additions of the transform, stage by stage
    v = list(v)
    for st in range(len(v).bit_length() - 1):
        for i in range(len(v)):
            if not i >> st & 1:
                v[i], v[i | 1 << st] = v[i] + v[i | 1 << st], v[i] - v[i | 1 << st]
    return torch.stack(v)


def _forward(P, s, b):  # [nrhs][n] -> [n_b][nrhs 2^s]
    t = _butterfly(b[:, _mirror(P, s)].permute(1, 2, 0))
    return t.permute(1, 2, 0).reshape(P.n_b, -1)


def _backward(P, s, xh, nrhs):
    t = _butterfly(xh.reshape(P.n_b, nrhs, 1 << s).permute(2, 0, 1)) * 2.0 ** -s
    x = torch.empty((nrhs, P.n), dtype=torch.float64, device="cuda")
    for r in range(nrhs):
        x[r, _mirror(P, s).reshape(-1)] = t[:, :, r].reshape(-1)
    return x


def _same(a, b):  # bit for bit, any NaN for any NaN
    ok = ~torch.isnan(b)
    return torch.equal(~torch.isnan(a), ok) and torch.equal(a[ok].view(torch.int64), b[ok].view(torch.int64))


def _special(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    v = torch.randn(shape, generator=g, dtype=torch.float64, device="cuda")
    pick = torch.randint(0, 9, shape, generator=g, device="cuda")
    # of one cell's copies only some are special, so that sums mix them
    for k, val in enumerate((0.0, -0.0, 5e-324, 2.0 ** -1022, 2.0 ** -1020, 1e308, float("inf"))):
        v = torch.where(pick == k, torch.full_like(v, val) * torch.sign(v), v)
    v.view(-1)[3::101] = float("nan")
    return v


@pytest.mark.parametrize("shift", [0, 1, 2, 3])  # doubles past a 256-byte boundary
@pytest.mark.parametrize("s,nrhs", [(0, 1), (1, 3), (2, 2), (3, 1), (3, 5)])
@pytest.mark.parametrize("values", ["random", "special"])
def test_transforms_bit_for_bit(s, nrhs, shift, values):
    P = amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=40)
    C = nrhs << s
    make = _special if values == "special" else lambda shape, seed: torch.from_numpy(
        np.random.default_rng(seed).standard_normal(shape)).to("cuda")
    b, xin = make((nrhs, P.n), 1), make((P.n_b, C), 2)
    buf = torch.empty(P.n_b * C + 64, dtype=torch.float64, device="cuda")
    at = (-buf.data_ptr() % 256) // 8 + shift
    xh = buf[at:at + P.n_b * C].view(P.n_b, C)
    assert xh.data_ptr() % 256 == 8 * shift
    P.transform_forward(b, nrhs, xh)
    assert _same(xh, _forward(P, s, b))
    xh.copy_(xin)
    x = P.transform_backward(xh, nrhs, torch.empty((nrhs, P.n), dtype=torch.float64, device="cuda"))
    assert _same(x, _backward(P, s, xin, nrhs))


@pytest.mark.parametrize("zero", [0, 2])
def test_gmres_with_a_right_hand_side_of_zeros(zero):
    """Its columns have no Krylov vector at any step."""
    P = amg.Problem.structured(N, 0.0, None, 2).setup(coarse_max=40)
    b = rhs_uniform(P.n, 3, config=98)
    b[zero] = 0.0
    x, info = P.solve_gmres(torch.from_numpy(b).to("cuda"), restart=12, tol=1e-12, maxit=400)
    x = x.cpu().numpy()
    assert info.converged and not x[zero].any()
    for r in {0, 1, 2} - {zero}:
        ref = solvers.dst_solve(N, b[r])
        assert np.linalg.norm(x[r] - ref) <= 68e-12 * np.linalg.norm(ref)  # kappa = 68 on this grid


def test_gmres_with_an_exact_preconditioner():
    """A single dense level without symmetries: the first step's Krylov space is the whole one."""
    P = amg.Problem.structured(N, 0.0, None, 0).setup(coarse_max=4096)
    assert P.num_levels() == 1
    b = rhs_uniform(P.n, 2, config=99)
    x, info = P.solve_gmres(torch.from_numpy(b).to("cuda"), restart=12, tol=1e-12, maxit=40)
    ref = solvers.dst_solve(N, b).reshape(b.shape)
    err = np.linalg.norm(x.cpu().numpy() - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert info.converged and info.iters <= 3 and err.max() <= 68e-12
