"""Row-group kernels at the edges of their row splits, and the kernels of
several right-hand sides and batches for all column counts and matrix forms.

FP64: V-cycles within 1e-12 of the oracle's and solutions within 1e-10 (only
the summation order differs).  Mixed precision: solutions to rtol 1e-8 within
1e-7 of the FP64 oracle's, as for single solves.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


def irregular(n, seed, longest=60):
    """Random SPD CSR with rows of 1 .. longest entries and no run structure."""
    rng = np.random.default_rng(seed)
    K = np.zeros((n, n))
    for i in range(1, n):
        k = int(rng.integers(0, min(i, longest // 2) + 1))
        j = rng.choice(i, size=k, replace=False)
        K[i, j] = -rng.uniform(0.1, 1.0, k)
    K = K + K.T
    K[np.arange(n), np.arange(n)] = np.abs(K).sum(1) * 1.1 + 0.5
    rp, ci, v = [0], [], []
    for i in range(n):
        c = np.flatnonzero(K[i])
        ci.append(c)
        v.append(K[i, c])
        rp.append(rp[-1] + len(c))
    return np.array(rp, np.int64), np.concatenate(ci).astype(np.int32), np.concatenate(v)


# rows: 576 (a warp per row), 625 (4 rows per warp from 608 on), 78,400 short
# rows (a lane per row from 77,824 on), 40,000 (4 short rows, many); 3-D: 3,375
# and 4,096 long rows (4 per warp from 3,648 on), 39,304 (8 per warp)
@pytest.mark.parametrize("d,n,p", [(2, 24, 2), (2, 25, 2), (2, 280, 2), (2, 200, 2), (3, 14, 3), (3, 15, 3),
                                   (3, 34, 2)])
def test_fp64_vcycle_at_the_edges_of_the_row_splits(d, n, p):
    prob = I.poisson_box(d, n, p)
    r = np.random.default_rng(n).normal(size=prob.n)
    H = A.Hierarchy(prob.rowptr, prob.col, prob.val, matrix_format=0)
    z = H.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    zo = O.Hierarchy(prob.rowptr, prob.col, prob.val).vcycle(r)
    assert np.linalg.norm(z - zo) <= 1e-12 * np.linalg.norm(zo)


@pytest.mark.parametrize("form", ["cubic", "ragged_2d", "irregular"])
@pytest.mark.parametrize("prec", [A.AMG_FP64, A.AMG_FP32, A.AMG_FP32_BF16FINE])
@pytest.mark.parametrize("R", [1, 2, 4, 6, 8, 13, 24, 32])
def test_multi_rhs_every_width_and_matrix_form(form, prec, R):
    if form == "irregular":
        rp, ci, v = irregular(331, 7)
    else:
        q = I.poisson_box(3, 7, 3) if form == "cubic" else I.poisson_box(2, 21, 4)
        rp, ci, v = q.rowptr, q.col, q.val
    n = len(rp) - 1
    F = np.random.default_rng(R).normal(size=(R, n))
    H = A.Hierarchy(rp, ci, v, coarse_max=20, precision=prec)
    Ho = O.Hierarchy(rp, ci, v, coarse_max=20)
    out = H.solve_multi(torch.from_numpy(F).cuda(), rtol=1e-8)
    assert out["status"] == 0 and (out["relres"] <= 1.0001e-8).all()
    U = out["u"].cpu().numpy()
    for c in range(R):
        ref = Ho.pcg(F[c], rtol=1e-8, flexible=prec != A.AMG_FP64)
        if prec == A.AMG_FP64 and out["iters"][c] != ref["iters"]:
            assert abs(int(out["iters"][c]) - ref["iters"]) <= 1
            continue
        tol = 1e-10 if prec == A.AMG_FP64 else 1e-7
        assert np.linalg.norm(U[c] - ref["u"]) <= tol * np.linalg.norm(ref["u"])


@pytest.mark.parametrize("prec", [A.AMG_FP64, A.AMG_FP32])
def test_multi_rhs_infinite_column_stays_alone(prec):
    q = I.poisson_box(3, 7, 3)
    F = np.random.default_rng(1).normal(size=(5, q.n))
    F[2, 17] = np.inf
    H = A.Hierarchy(q.rowptr, q.col, q.val, coarse_max=20, precision=prec)
    out = H.solve_multi(torch.from_numpy(F).cuda(), rtol=1e-8)
    assert out["status"] == A.AMG_ERR_NAN
    keep = [0, 1, 3, 4]
    good = H.solve_multi(torch.from_numpy(F[keep]).cuda(), rtol=1e-8)
    assert (out["relres"][keep] <= 1e-8).all() and (out["iters"][keep] == good["iters"]).all()


@pytest.mark.parametrize("prec", [A.AMG_FP64, A.AMG_FP32, A.AMG_FP32_BF16FINE])
def test_batch_of_very_different_systems(prec):
    one = (np.array([0, 1], np.int64), np.array([0], np.int32), np.array([3.0]))
    sysl = [one, irregular(150, 3), *[(q.rowptr, q.col, q.val) for q in (I.poisson_box(3, 8, 3),
            I.poisson_box(2, 40, 2), I.poisson_box(2, 3, 4))], one, irregular(33, 5)]
    rng = np.random.default_rng(4)
    us = [rng.normal(size=len(s[0]) - 1) for s in sysl]
    Fs = [torch.from_numpy(I.csr_apply(*s, u)).cuda() for s, u in zip(sysl, us)]
    B = A.BatchHierarchy(sysl, coarse_max=20, precision=prec)
    out = B.solve_batch(Fs, rtol=1e-10)
    assert out["status"] == 0 and (out["relres"] <= 1.0001e-10).all()
    for u, g in zip(us, out["u"]):
        # the residual bounds the error by the condition number (below 1e5 here)
        assert np.linalg.norm(g.cpu().numpy() - u) <= 1e-5 * np.linalg.norm(u)
