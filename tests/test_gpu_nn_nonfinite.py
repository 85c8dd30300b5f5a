"""A target value that is not finite spoils the gradient entries it is a term of, and no
others (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from test_gpu_nn import unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n", [(2, 33), (2, 40), (2, 300), (3, 9), (3, 20)])
def test_infinite_target_on_the_last_row(dim, n):
    """dW[c][tap] of the output convolution is the sum over points p of gy[p] t[p + off]:
    for p on the last row of the y axis the taps one row further reach outside the grid
    and take no part.  Sides with ragged segments (rows of a segment past the grid) and
    without."""
    from paper_2103_10975_gb300 import Solver
    s = Solver(n, dim=dim, m=5, batch=2)
    rng = np.random.default_rng(n)
    u = rng.standard_normal((2,) + (n,) * dim)
    t = rng.standard_normal((2,) + (n,) * dim)
    t[(1,) + (n // 2,) * (dim - 2) + (n - 1, n // 2)] = np.inf
    f = lambda v: torch.as_tensor(v.reshape(2, -1), dtype=torch.float32).cuda()
    loss, g = s.nn_loss_grad(f(u), f(t))
    assert not np.isfinite(loss)
    w = unpack(g, n, dim=dim)["out.w"].reshape((32,) + (3,) * dim)
    assert np.isfinite(w[..., 2, :]).all()
    assert not np.isfinite(w[..., :2, :]).any()
