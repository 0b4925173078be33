"""The down sweep with its restriction in one kernel, for aggregates of 2 to 16
members, levels that are plain CSR or run-encoded, few and many rows.

V-cycles within 1e-12 of the oracle's in FP64 (only the summation order differs)
and 1e-5 in mixed precision (FP32 V-cycle; a few hundred roundings of 6e-8).
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
