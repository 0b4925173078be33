"""Few right-hand sides in FP64: the vectors of a solve have as many columns as
right-hand sides, rounded up to two (a row is whole 16-byte pieces).
"""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# device memory that a solve of R right-hand sides takes from the device, after the setup
PROBE = """
import numpy as np, scipy.sparse as sp, torch
from paper_2511_21268_gb300 import amg as A
m, R = 2000, {R}
T = sp.diags([-1.0, 2.0, -1.0], [-1, 0, 1], (m, m))
K = (sp.kron(T, sp.identity(m)) + sp.kron(sp.identity(m), T)).tocsr()
K.sort_indices()
H = A.Hierarchy(K.indptr.astype(np.int64), K.indices.astype(np.int32), K.data)
F = torch.ones(R, m * m, dtype=torch.float64, device="cuda")
U = torch.zeros_like(F)
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
A.amg_pcg_solve_multi(H._h, F, U, 0.0, 2)
torch.cuda.synchronize()
print(free - torch.cuda.mem_get_info()[0], sum(H.level_n(l) for l in range(H.num_levels)))
"""


@pytest.mark.parametrize("R,cols", [(1, 2), (2, 2), (5, 6)])
def test_workspace_of_few_right_hand_sides(R, cols):
    # a process of its own: the library keeps freed memory in its pool
    out = subprocess.run([sys.executable, "-c", PROBE.format(R=R)], cwd=ROOT, capture_output=True, text=True,
                         timeout=300, check=True).stdout.split()
    taken, rows = int(out[0]), int(out[1])
    n = 2000 * 2000
    # six CG vectors and the staging copy; x and t of every level, f of the coarse ones
    need = 8 * (6 * cols + R) * n + 8 * cols * (3 * rows - n)
    assert taken <= need + (128 << 20)  # the pool grows in pieces; four columns for one: 650 MB more
