"""A breakdown of the PCG says what was seen, and leaves the handle usable
(marked gpu): residuals of 1e30 have products that overflow FP32."""

import re

import pytest

torch = pytest.importorskip("torch")

import paper_2407_05930_gb300 as amg  # noqa: E402
from synth import rhs_uniform  # noqa: E402

pytestmark = pytest.mark.gpu
N, S = (16, 12, 10), 2
SEEN = re.compile(r"column (\d+), iteration 0, p\^T A p = -?(inf|nan), r\^T z = -?(inf|nan)")


def test_breakdown_of_a_solve():
    P = amg.Problem.structured(N, 0.0, None, S).setup(coarse_max=40)
    b = torch.from_numpy(rhs_uniform(P.n, 3, config=95)).to("cuda")
    x, _ = P.solve(b, tol=1e-12, precision=amg.PREC_MIXED_FP32)
    with pytest.raises(amg.AmgsymError, match="BREAKDOWN") as e:
        P.solve(b * 1e30, tol=1e-12, precision=amg.PREC_MIXED_FP32)
    m = SEEN.search(str(e.value))
    assert m and int(m.group(1)) < 3 << S
    y, info = P.solve(b, tol=1e-12, precision=amg.PREC_MIXED_FP32)
    assert info.converged and torch.equal(x, y)


def test_breakdown_of_a_batch():
    probs = [amg.Problem.structured(N, 0.0, None, s).setup(coarse_max=40) for s in (1, S)]
    bs = [torch.from_numpy(rhs_uniform(p.n, 2, config=96 + i)).to("cuda") for i, p in enumerate(probs)]
    B = amg.Batch(probs, [2, 2])
    xs, _ = B.solve(bs, tol=1e-12)
    with pytest.raises(amg.AmgsymError, match="problem 1, ") as e:
        B.solve([bs[0], bs[1] * 1e30], tol=1e-12)
    assert SEEN.search(str(e.value))
    ys, res = B.solve(bs, tol=1e-12)
    assert all(r.converged for r in res) and all(torch.equal(a, c) for a, c in zip(xs, ys))
