"""FP64 levels of short rows with one or a few long ones among them, at the lines
where the row splits change (128 and 320 entries), against the oracle; and no
slower than a split that gives a long row a whole warp.

V-cycles within 1e-12 of the oracle's (only the summation order differs).
"""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402


def lattice_with_hubs(m, hubs, length):
    """5-point matrix of an m x m lattice whose rows m (m + 1) k, k < hubs, have
    `length` entries: weak couplings to rows spread over the whole lattice."""
    T = sp.diags([-1.0, 2.0, -1.0], [-1, 0, 1], (m, m))
    K = (sp.kron(T, sp.identity(m)) + sp.kron(sp.identity(m), T)).tocsr()
    n, r, c = m * m, [], []
    for k in range(hubs):
        i = m * (m + 1) * (k + 1) // (hubs + 1)
        have = K.indices[K.indptr[i]:K.indptr[i + 1]]
        free = np.setdiff1d(np.arange(n), have)
        j = free[np.linspace(0, len(free) - 1, length - len(have)).astype(int)]
        r.append(np.full(len(j), i))
        c.append(j)
    r, c = np.concatenate(r), np.concatenate(c)
    W = sp.coo_matrix((np.ones(len(r)), (r, c)), (n, n)).tocsr()
    W = W.maximum(W.T) * 1e-3
    K = (K - W + sp.diags(np.asarray(W.sum(1)).ravel() + 1e-3)).tocsr()
    K.sort_indices()
    return K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data.astype(np.float64)


# 78,400 rows: a lane per row from 77,824 on; 3,600: 8 lanes per row
@pytest.mark.parametrize("m", [60, 280])
@pytest.mark.parametrize("length", [128, 129, 320, 321, 2500])
def test_vcycle_with_one_long_row(m, length):
    rp, ci, v = lattice_with_hubs(m, 1, length)
    assert np.diff(rp).max() == length
    r = np.random.default_rng(length).normal(size=m * m)
    z = A.Hierarchy(rp, ci, v).vcycle(torch.from_numpy(r).cuda()).cpu().numpy()
    zo = O.Hierarchy(rp, ci, v).vcycle(r)
    assert np.linalg.norm(z - zo) <= 1e-12 * np.linalg.norm(zo)


def test_a_few_very_long_rows_do_not_hold_the_fp64_vcycle_up():
    """The FP32 V-cycle gives every row of this matrix a warp's 32 lanes, and
    FP64 has twice its bytes: a time above four times its is a chain of single
    lanes (eleven times, 160,000 rows with five of 20,000 entries)."""
    mat = lattice_with_hubs(400, 5, 20000)
    r = torch.ones(160000, dtype=torch.float64, device="cuda")
    sec = []
    for prec in (A.AMG_FP32, A.AMG_FP64):
        H = A.Hierarchy(*mat, precision=prec)
        ts = []
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            H.vcycle(r)
            torch.cuda.synchronize()
            ts.append(time.perf_counter() - t)
        sec.append(min(ts[1:]))
    assert sec[1] <= 4.0 * sec[0], sec
