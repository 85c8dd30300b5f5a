"""Edges of the solver variants' ranges (GPU): restart lengths at the bucket and
instantiation limits, and grids whose CTAs hold one tile, ragged tiles or many.

Tolerance: the solves stop at a true relative residual of 1e-10 and the error is
at most that times the condition number over its smooth part; the stated bound
for rtol 1e-10 is 1e-7 against the exact (DST-I) solution.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import direct
from synthetic import MovingGaussians2D

pytestmark = pytest.mark.gpu


def _solve_2d(n, **opt):
    from paper_2103_10975_gb300 import Solver
    b = MovingGaussians2D(n, 77, 50).rhs(3)
    s = Solver(n, rtol=1e-10, **opt)
    x, r = s.solve(torch.as_tensor(b).cuda())
    xe = direct.dst_solve_2d(n, b)
    assert r["status"] == 0 and r["relres_true"] <= 1e-10, r
    err = np.linalg.norm(x.cpu().numpy() - xe) / np.linalg.norm(xe)
    assert err <= 1e-7, (n, opt, err)


@pytest.mark.parametrize("n,m", [(2, 3), (6, 7), (11, 8), (23, 16), (32, 31), (33, 32), (33, 33),
                                 (45, 24), (90, 40), (130, 32), (129, 50)])
def test_fp64_shared_variants(n, m):
    _solve_2d(n, m=m, precision="fp64")
