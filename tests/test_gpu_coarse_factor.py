"""Coarsest level's dense factorisation at the sizes where its kernels change:
one cluster of 16 blocks (rows per block 0, 1, several; up to its shared
memory), of 8, one block; the inverse with a block per column (128 and 256
rows) and with a warp per column.

The factor equals the oracle's bit for bit (same operations in the same
order, each correctly rounded).  The inverse is compared with numpy's: the
matrices B B^T / n + I have condition numbers below 10, so both errors are
below about n eps cond = 660 x 1.1e-16 x 10 < 1e-12 of the largest entry.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402


def dense_csr(K):
    n = len(K)
    return (np.arange(n + 1, dtype=np.int64) * n, np.tile(np.arange(n, dtype=np.int32), n), K.ravel().copy())


def spd(n, seed=3):
    B = np.random.default_rng(seed + n).normal(size=(n, n))
    K = B @ B.T / n + np.eye(n)
    return np.tril(K) + np.tril(K, -1).T


@pytest.mark.parametrize("n,scale", [(1, 0), (2, 0), (15, 0), (16, 0), (17, 0), (33, 600), (33, -600), (128, 0),
                                     (129, 0), (240, 0), (256, 0), (257, 0), (460, 0), (660, 0)])
def test_factor_bit_exact_and_inverse(n, scale):
    K = spd(n) * 2.0 ** scale  # exact scaling; 2^+-600 leaves the range of the fast square root and division
    opts = dict(coarse_max=1000)
    H = A.Hierarchy(*dense_csr(K), **opts)
    assert H.num_levels == 1
    L, Ai = H.export_coarse()
    Lo = O.Hierarchy(*dense_csr(K), **opts).coarse_chol()
    assert np.array_equal(L.view(np.uint64), Lo.view(np.uint64))
    inv = np.linalg.inv(spd(n)) * 2.0 ** -scale
    assert np.abs(Ai - inv).max() <= 1e-12 * np.abs(inv).max()


@pytest.mark.parametrize("n", [2, 40, 300])
def test_indefinite_matrix_is_refused(n):
    K = np.eye(n)
    K[n - 1, n - 2] = K[n - 2, n - 1] = 2.0  # positive diagonal, negative last pivot
    with pytest.raises(A.AmgError) as e:
        A.Hierarchy(*dense_csr(K), coarse_max=1000)
    assert e.value.code == A.AMG_ERR_NOT_SPD
