"""The down sweep with its restriction in one kernel, for aggregates of 2 to 16
members, levels that are plain CSR or run-encoded, few and many rows.

V-cycles within 1e-12 of the oracle's in FP64 (only the summation order differs)
and 1e-5 in mixed precision (FP32 V-cycle; a few hundred roundings of 6e-8);
solutions of several right-hand sides within 1e-10 at equal iterations.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


# long rows (a warp each) and short ones (8 lanes), coarse levels of any size;
# one coarse row per block (4 passes) up to 16 (1 pass, 4 rows per warp)
@pytest.mark.parametrize("passes", [1, 2, 3, 4])
@pytest.mark.parametrize("fmt", [0, 2])
@pytest.mark.parametrize("d,n,p", [(2, 7, 2), (2, 31, 3), (2, 60, 2), (3, 6, 2), (3, 13, 3)])
def test_vcycle_of_every_aggregate_size(d, n, p, fmt, passes):
    q = I.poisson_box(d, n, p)
    r = np.random.default_rng(n).normal(size=q.n)
    zo = O.Hierarchy(q.rowptr, q.col, q.val, match_passes=passes, coarse_max=12).vcycle(r)
    for prec, tol in ((A.AMG_FP64, 1e-12), (A.AMG_FP32, 1e-5)):
        H = A.Hierarchy(q.rowptr, q.col, q.val, match_passes=passes, coarse_max=12, matrix_format=fmt,
                        precision=prec)
        z = H.vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
        assert np.linalg.norm(z - zo) <= tol * np.linalg.norm(zo)


# several right-hand sides: levels with a warp for every row and larger ones
@pytest.mark.parametrize("passes", [1, 2, 3, 4])
@pytest.mark.parametrize("d,n,p", [(2, 9, 2), (2, 31, 3), (3, 24, 2)])
def test_multi_rhs_of_every_aggregate_size(d, n, p, passes):
    q = I.poisson_box(d, n, p)
    F = np.random.default_rng(n).normal(size=(3, q.n))
    H = A.Hierarchy(q.rowptr, q.col, q.val, match_passes=passes, coarse_max=12)
    out = H.solve_multi(torch.from_numpy(F).cuda(), rtol=1e-9)
    assert out["status"] == 0
    Ho = O.Hierarchy(q.rowptr, q.col, q.val, match_passes=passes, coarse_max=12)
    for c in range(3):
        ref = Ho.pcg(F[c], rtol=1e-9)
        assert abs(int(out["iters"][c]) - ref["iters"]) <= 1
        if out["iters"][c] == ref["iters"]:
            u = out["u"][c].cpu().numpy()
            assert np.linalg.norm(u - ref["u"]) <= 1e-10 * np.linalg.norm(ref["u"])
