"""Which small FP64 systems are solved by the one-cluster kernel and which by
launches, seen by the iteration graph that only the launches build and by the
number of kernels launched; solutions to the tolerance asked for on both.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu

from paper_2511_21268_gb300 import amg as A  # noqa: E402
from paper_2511_21268_gb300 import inputs as I  # noqa: E402


def csr(K):
    K = K.tocsr()
    K.sort_indices()
    return K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data.astype(np.float64)


def lattice(*dims):
    """Second differences in each direction: 3, 5, 7 entries per row."""
    K = sp.csr_matrix((1, 1))
    for m in dims:
        T = sp.diags([-1.0, 2.0, -1.0], [-1, 0, 1], (m, m))
        K = sp.kron(K, sp.identity(m)) + sp.kron(sp.identity(K.shape[0]), T)
    return csr(K)


def hub(m, length):
    """5-point matrix of m x m points, one row coupled weakly to `length` others."""
    rp, ci, v = lattice(m, m)
    n = m * m
    K = sp.csr_matrix((v, ci, rp), (n, n))
    j = np.linspace(0, n - 2, length).astype(int)
    W = sp.coo_matrix((np.full(length, 1e-3), (np.full(length, n - 1), j)), (n, n)).tocsr()
    W = W + W.T
    return csr(K - W + sp.diags(np.asarray(W.sum(1)).ravel()))


def solve(H, rtol=1e-8):
    """First solve of H: (graph built, kernels launched, iterations)."""
    F = torch.from_numpy(np.random.default_rng(5).normal(size=H.level_n(0))).cuda()
    before = A.lib().amg_kernel_launches()
    out = H.solve(F, rtol=rtol)
    count = A.lib().amg_kernel_launches() - before
    assert out["status"] == 0 and out["relres"] <= 1.0001 * rtol
    return H.info.graph_build_ms > 0.0, count, out["iters"]


@pytest.mark.parametrize("make,opts", [
    (lambda: I.assemble_kron(2, 32, 2), {}), (lambda: I.assemble_kron(2, 64, 2), {}),
    (lambda: I.assemble_kron(3, 8, 3), {}), (lambda: I.assemble_kron(3, 12, 2), {}),
    (lambda: lattice(2000), {}), (lambda: lattice(64, 64), {}), (lambda: lattice(16, 16, 16), {}),
    (lambda: lattice(32, 32), dict(coarse_max=400)), (lambda: hub(30, 300), {})])
def test_the_cluster_takes_what_it_is_faster_at(make, opts):
    graph, count, its = solve(A.Hierarchy(*make(), **opts))
    # a launch per 64 iterations, and the final residual's few
    assert not graph and count <= its // 64 + 6


@pytest.mark.parametrize("make,opts", [
    # entries; rows; a large coarsest level; a long row
    (lambda: I.assemble_kron(2, 64, 4), {}), (lambda: I.assemble_kron(3, 14, 2), {}),
    (lambda: lattice(6000), {}), (lambda: lattice(80, 80), {}), (lambda: lattice(20, 20, 20), {}),
    (lambda: lattice(12000), dict(coarse_max=3000)), (lambda: lattice(64, 64), dict(coarse_max=2000)),
    (lambda: I.assemble_kron(2, 48, 2), dict(coarse_max=1000)), (lambda: hub(50, 400), {})])
def test_the_launches_take_the_rest(make, opts):
    graph, _, _ = solve(A.Hierarchy(*make(), **opts))
    assert graph


def test_rows_that_do_not_fit_are_found_once():
    """A dense block beside a chain, within the rule's lines: the blocks that own
    its coarse rows would need more shared memory than they have.  The first solve
    launches the cluster kernel for nothing, the second knows."""
    m, c = 250, 1500
    D = sp.identity(m) * (m + 0.5) - sp.csr_matrix(np.ones((m, m)))
    T = sp.diags([-1.0, 2.01, -1.0], [-1, 0, 1], (c, c))
    H = A.Hierarchy(*csr(sp.block_diag([D, T])))
    levels = range(H.num_levels)
    assert H.num_levels > 1 and sum(H.level_nnz(k) for k in levels) <= 200000
    assert sum(H.level_n(k) for k in levels) + H.level_n(H.num_levels - 1) ** 2 // 100 + 9 * m <= 6000
    graph, first, its = solve(H)
    _, second, again = solve(H)
    assert graph and its == again and first == second + 1
