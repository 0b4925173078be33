"""A hierarchy's first solve of a system that is solved already (F = 0, a converged
guess): it builds no iteration graph; the solve after it does, and is as on a fresh
hierarchy, to the bit.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


@pytest.mark.parametrize("prec", [A.AMG_FP64, A.AMG_FP32])
@pytest.mark.parametrize("kind", ["one", "several", "batch"])
@pytest.mark.parametrize("start", ["zero", "converged"])
def test_first_solve_of_a_solved_system(prec, kind, start):
    q = I.poisson_box(2, 64, 4)  # more entries than the one-cluster solve takes
    K, F = (q.rowptr, q.col, q.val), torch.from_numpy(q.F).cuda()

    def fresh():
        if kind == "batch":
            H = A.BatchHierarchy([K, K], precision=prec)
            return H, lambda f, u, **kw: H.solve_batch([f, 2.0 * f], [u.clone(), 2.0 * u], **kw)
        H = A.Hierarchy(*K, precision=prec)
        if kind == "several":
            return H, lambda f, u, **kw: H.solve_multi(torch.stack([f, 2.0 * f]), torch.stack([u, 2.0 * u]), **kw)
        return H, lambda f, u, **kw: H.solve(f, u.clone(), **kw)

    zero = torch.zeros_like(F)
    u = A.Hierarchy(*K).solve(F, rtol=1e-10)["u"]
    f0, u0 = (zero, zero) if start == "zero" else (F, u)
    H, solve = fresh()
    out = solve(f0, u0, rtol=1e-8)
    assert out["status"] == 0 and max([out["iters"]] if kind == "one" else out["iters"]) == 0
    assert H.info.graph_build_ms == 0.0
    ref = fresh()[1](F, zero, rtol=1e-8)
    got = solve(F, zero, rtol=1e-8)
    assert (ref["iters"] == got["iters"]) if kind == "one" else (ref["iters"] == got["iters"]).all()
    assert H.info.graph_build_ms > 0.0
    for a, b in zip(ref["u"], got["u"]):
        assert torch.equal(a, b)
