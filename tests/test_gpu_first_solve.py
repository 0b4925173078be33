"""A hierarchy's first solve, whose first iterations run by launches while the
iteration graph is built, against the same solve again, by the graph alone: same
bits, iteration counts and statuses, whether it ends within the launches or after.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


# more entries than the one-cluster solve takes; one right-hand side and several
@pytest.mark.parametrize("prec", [A.AMG_FP64, A.AMG_FP32])
@pytest.mark.parametrize("kw", [dict(rtol=1e-9), dict(rtol=1e-1), dict(rtol=0.0, itmax=3), dict(rtol=0.0, itmax=8),
                                dict(rtol=0.0, itmax=9), dict(rtol=1e-9, itmax=0)])
def test_first_solve_equals_the_second(kw, prec):
    q = I.poisson_box(2, 64, 4)
    F = torch.from_numpy(q.F).cuda()
    H = A.Hierarchy(q.rowptr, q.col, q.val, precision=prec)
    a, b = H.solve(F, **kw), H.solve(F, **kw)
    assert (a["iters"], a["status"], a["relres"]) == (b["iters"], b["status"], b["relres"])
    assert torch.equal(a["u"], b["u"])
    G = torch.stack([F, 2.0 * F, torch.zeros_like(F)])
    H = A.Hierarchy(q.rowptr, q.col, q.val, precision=prec)
    a, b = H.solve_multi(G, **kw), H.solve_multi(G, **kw)
    assert (a["iters"] == b["iters"]).all() and (a["relres"] == b["relres"]).all() and a["status"] == b["status"]
    assert torch.equal(a["u"], b["u"])


def test_first_solve_of_a_nan_right_hand_side():
    q = I.poisson_box(2, 64, 4)
    F = q.F.copy()
    F[5] = np.nan
    H = A.Hierarchy(q.rowptr, q.col, q.val)
    assert H.solve(torch.from_numpy(F).cuda())["status"] == A.AMG_ERR_NAN
    out = H.solve(torch.from_numpy(q.F).cuda(), rtol=1e-9)
    assert out["status"] == 0 and out["relres"] <= 1.0001e-9
