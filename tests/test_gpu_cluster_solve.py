"""The FP64 solve of small systems as one kernel on one cluster, against the
oracle and against the solve by launches (which a hierarchy with kernel timing
switched on takes).

Solutions within 1e-10 of the oracle's at equal iterations, single iterates
within 1e-12, as for the solve by launches (only the summation order differs).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


def gpu(a):
    return torch.from_numpy(a).cuda()


# two to four levels; the smallest coarsest level (fewer rows than blocks); more
# iterations than one launch does (3-D p = 3); about 1e5 entries, and more than
# the cluster takes (2-D p = 4 n = 64, 3-D n = 14)
@pytest.mark.parametrize("flexible", [0, 1])
@pytest.mark.parametrize("d,n,p,coarse_max", [(2, 4, 2, 8), (2, 9, 2, 20), (2, 16, 2, 40), (2, 25, 3, 40),
                                              (2, 33, 2, 40), (2, 64, 2, 40), (2, 64, 4, 40), (3, 5, 2, 8),
                                              (3, 8, 3, 40), (3, 11, 2, 40), (3, 14, 2, 40)])
def test_small_solves_match_the_oracle(d, n, p, coarse_max, flexible):
    q = I.poisson_box_random_rhs(d, n, p, seed=n)
    H = A.Hierarchy(q.rowptr, q.col, q.val, coarse_max=coarse_max, flexible=flexible)
    Ho = O.Hierarchy(q.rowptr, q.col, q.val, coarse_max=coarse_max)
    F = gpu(q.F)
    for k in (1, 3):
        ref = Ho.pcg(q.F, rtol=0.0, itmax=k, flexible=bool(flexible))
        out = H.solve(F, rtol=0.0, itmax=k)
        assert out["status"] == A.AMG_ERR_NOT_CONVERGED and out["iters"] == k
        assert np.linalg.norm(out["u"].cpu().numpy() - ref["u"]) <= 1e-12 * np.linalg.norm(ref["u"])
    ref = Ho.pcg(q.F, rtol=1e-9, flexible=bool(flexible))
    out = H.solve(F, rtol=1e-9)
    assert out["status"] == 0 and out["relres"] <= 1.0001e-9 and abs(out["iters"] - ref["iters"]) <= 1
    if out["iters"] == ref["iters"]:
        assert np.linalg.norm(out["u"].cpu().numpy() - ref["u"]) <= 1e-10 * np.linalg.norm(ref["u"])
    again = H.solve(F, rtol=1e-9)
    assert torch.equal(again["u"], out["u"]) and again["iters"] == out["iters"]
    warm = H.solve(F, u=out["u"].clone(), rtol=1e-9)
    assert warm["iters"] <= 1 and warm["status"] == 0
    A.amg_profile_kernels(H._h, True)
    by_launches = H.solve(F, rtol=1e-9)
    assert by_launches["status"] == 0 and abs(by_launches["iters"] - out["iters"]) <= 1


@pytest.mark.parametrize("d,n,p", [(2, 32, 2), (3, 8, 3)])
def test_small_solves_end_like_the_solve_by_launches(d, n, p):
    q = I.poisson_box(d, n, p)
    H = A.Hierarchy(q.rowptr, q.col, q.val)
    L = A.Hierarchy(q.rowptr, q.col, q.val)
    A.amg_profile_kernels(L._h, True)
    inf, nan = q.F.copy(), q.F.copy()
    inf[3], nan[-1] = np.inf, np.nan
    for F, kw in ((q.F * 0, {}), (q.F, dict(itmax=0)), (q.F, dict(itmax=1)), (inf, {}), (nan, {}),
                  (q.F, dict(rtol=2.0)), (q.F, dict(rtol=0.0, itmax=64)), (q.F, dict(rtol=0.0, itmax=65)),
                  (q.F, {})):
        got, ref = [], []
        for h, into in ((H, got), (L, ref)):
            out = h.solve(gpu(F), **{"rtol": 1e-9, **kw})
            into += [out["status"], out["iters"]]
        assert got == ref or (kw == {} and got[0] == ref[0] == 0 and abs(got[1] - ref[1]) <= 1)


def test_rows_that_do_not_fit_one_block():
    """Few entries in all, but most of them in the rows of few coarse rows (a
    dense block beside a chain): the launches solve it, on every call."""
    m, c = 400, 2000
    rp, ci, v = [0], [], []
    for i in range(m):
        ci.append(np.arange(m))
        v.append(np.where(np.arange(m) == i, m + 0.5, -1.0))
        rp.append(rp[-1] + m)
    for i in range(c):
        col = [j for j in (i - 1, i, i + 1) if 0 <= j < c]
        ci.append(np.array(col) + m)
        v.append(np.array([2.01 if j == i else -1.0 for j in col]))
        rp.append(rp[-1] + len(col))
    rp, ci, v = np.array(rp, np.int64), np.concatenate(ci).astype(np.int32), np.concatenate(v)
    F = np.random.default_rng(2).normal(size=m + c)
    H = A.Hierarchy(rp, ci, v)
    assert H.num_levels > 1 and sum(H.level_nnz(l) for l in range(H.num_levels)) <= 200000
    ref = O.Hierarchy(rp, ci, v).pcg(F, rtol=1e-9)
    for _ in range(2):
        out = H.solve(gpu(F), rtol=1e-9)
        assert out["status"] == 0 and abs(out["iters"] - ref["iters"]) <= 1
        if out["iters"] == ref["iters"]:
            assert np.linalg.norm(out["u"].cpu().numpy() - ref["u"]) <= 1e-10 * np.linalg.norm(ref["u"])
