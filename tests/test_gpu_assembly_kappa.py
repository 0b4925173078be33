"""The coefficient's fixed-point product at the edges of its tiles: numbers of
features around multiples of 16 (columns padded to 32), Gauss points that are
no multiple of 64, more features than one piece of the plane holds; K's
exact symmetry; and values that are not finite.  Entries within 1e-12 of the oracle's element loop
(relative to the largest), as in test_gpu_assembly.py."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from oracle import iga  # noqa: E402
from paper_2511_21268_gb300 import amg as A  # noqa: E402


def features(M, ell=0.4, seed=5):
    rng = np.random.default_rng(seed + M)
    return rng.normal(size=(M, 3)) / ell, rng.uniform(0, 2 * math.pi, M)


def gpu(n, p, nq, om, ph, sigma):
    return A.iga_assemble(n, p, nq=nq, geometry=A.AMG_GEOM_ANNULUS, source=A.AMG_SRC_SINE,
                          kappa=(torch.from_numpy(om).cuda(), torch.from_numpy(ph).cuda(), sigma))


@pytest.mark.parametrize("n,p,nq,M", [(2, 2, 0, 1), (3, 2, 5, 15), (4, 3, 0, 16), (3, 3, 7, 17), (5, 2, 13, 33),
                                      (4, 2, 16, 257), (6, 2, 6, 6000)])
def test_values_match_the_element_loop(n, p, nq, M):
    om, ph = features(M)
    g = gpu(n, p, nq, om, ph, 1.0)
    P = iga.Patch(n, p, nq=nq or p + 1, geom="annulus", omega=om, phi=ph, sigma=1.0, src="sine")
    K, F = P.assemble()
    rp, ci, v = (g[k].cpu().numpy() for k in ("rowptr", "col", "val"))
    D = np.zeros((g["n"], g["n"]))
    for i in range(g["n"]):
        D[i, ci[rp[i]:rp[i + 1]]] = v[rp[i]:rp[i + 1]]
    assert np.abs(D - K).max() <= 1e-12 * np.abs(K).max()
    assert np.array_equal(D, D.T)  # each pair of entries is computed once
    assert np.abs(g["F"].cpu().numpy() - F).max() <= 1e-12 * np.abs(F).max()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("axis", [0, 2])
def test_a_frequency_that_is_not_finite_shows(bad, axis):
    om, ph = features(20)
    om[7, axis] = bad
    g = gpu(3, 2, 0, om, ph, 1.0)
    assert torch.isnan(g["val"]).all()
