"""Kernels whose dynamic shared memory grows with the matrix: hierarchies and
assemblies of different size side by side, one after the other and from two host
threads.  A kernel's limit is one of the process, so a smaller hierarchy must not
take it away from a larger one.  Same bits as alone.
"""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


# more than 48 KB of vector window per block for the larger one, in each layout
@pytest.mark.parametrize("opts", [dict(precision=A.AMG_FP64), dict(precision=A.AMG_FP32),
                                  dict(precision=A.AMG_FP32_BF16FINE), dict(precision=A.AMG_FP64, cheb_degree=3)])
def test_larger_hierarchy_solves_after_a_smaller_setup(opts):
    def mat(n):
        return I.assemble_kron(3, n, 3)

    F = torch.from_numpy(I.poisson_box(3, 30, 3).F).cuda()
    with A.Hierarchy(*mat(30), **opts) as H:
        alone = H.solve(F, rtol=1e-6)
    large = A.Hierarchy(*mat(30), **opts)
    small = A.Hierarchy(*mat(20), **opts)
    out = large.solve(F, rtol=1e-6)
    assert out["status"] == 0 and out["iters"] == alone["iters"] and torch.equal(out["u"], alone["u"])
    assert small.solve(torch.from_numpy(I.poisson_box(3, 20, 3).F).cuda(), rtol=1e-6)["status"] == 0


def in_two_threads(a, b):
    """Results of a() and b(), each called over and over by its own thread."""
    res, err = [None, None], []

    def work(k, f):
        try:
            for _ in range(60):
                r = f()
                assert res[k] is None or all(np.array_equal(x, y) for x, y in zip(res[k], r))
                res[k] = r
        except BaseException as e:  # noqa: BLE001
            err.append(e)

    ts = [threading.Thread(target=work, args=(k, f)) for k, f in enumerate((a, b))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not err, err[0]
    return res


def test_coarsest_levels_of_different_size_in_two_threads():
    def dense(n):
        B = np.random.default_rng(n).normal(size=(n, n))
        K = B @ B.T / n + np.eye(n)
        K = np.tril(K) + np.tril(K, -1).T
        return np.arange(n + 1, dtype=np.int64) * n, np.tile(np.arange(n, dtype=np.int32), n), K.ravel().copy()

    def setup(K):
        with A.Hierarchy(*K, coarse_max=1000) as H:
            return H.export_coarse()

    big, small = dense(195), dense(40)
    alone = setup(big), setup(small)
    for ref, got in zip(alone, in_two_threads(lambda: setup(big), lambda: setup(small))):
        assert all(np.array_equal(x, y) for x, y in zip(ref, got))


def test_assemblies_of_different_size_in_two_threads():
    def assemble(n, p, nq):  # the contractions stage 32 n nq doubles per block
        s = A.iga_assemble(n, p, nq=nq, geometry=A.AMG_GEOM_ANNULUS)
        return s["val"].cpu().numpy(), s["F"].cpu().numpy()

    alone = assemble(25, 2, 8), assemble(5, 2, 0)
    for ref, got in zip(alone, in_two_threads(lambda: assemble(25, 2, 8), lambda: assemble(5, 2, 0))):
        assert all(np.array_equal(x, y) for x, y in zip(ref, got))
