"""Row-group kernels at the edges of their row splits: FP64 V-cycles within
1e-12 of the oracle's (only the summation order differs)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


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
