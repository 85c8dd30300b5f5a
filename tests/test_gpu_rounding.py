"""Rounding of FP64 results against extended precision (GPU)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _sweeps_by_differences(n, b, x, sweeps, omega, dtype):
    """Damped Jacobi as written in the paper's notation, x + omega/d (b - A x), A x from
    the differences to the four neighbours, in `dtype`."""
    h = 2.0 / (n + 1)
    s2 = 1.0 / (h * h)
    f, s2 = dtype(omega / (4.0 * s2)), dtype(s2)
    b, x = b.reshape(n, n).astype(dtype), x.reshape(n, n).astype(dtype)
    for _ in range(sweeps):
        p = np.pad(x, 1)
        ax = s2 * (((x - p[1:-1, :-2]) + (x - p[1:-1, 2:])) + ((x - p[:-2, 1:-1]) + (x - p[2:, 1:-1])))
        x = x + f * (b - ax)
    return x.reshape(-1)


@pytest.mark.parametrize("n,sweeps", [(64, 16), (100, 32), (256, 8), (256, 32), (321, 12)])
def test_smooth_rounds_no_worse_than_differences(n, sweeps):
    """mlgmres_smooth on a smooth iterate: no further from extended precision than the
    plain formula by differences in FP64.  The kernel may contract multiply-adds, which
    only drops roundings; 1.15 leaves room for the scatter of a norm over n^2 roundings.
    (A weighted sum of the five points is about 1.5 to 1.9 times as far.)"""
    from paper_2103_10975_gb300 import Solver
    rng = np.random.default_rng(n + sweeps)
    t = -1.0 + 2.0 / (n + 1) * np.arange(1, n + 1)
    x0, b = np.zeros((n, n)), np.zeros((n, n))
    for _ in range(3):
        (cx, cy), a = rng.uniform(-0.6, 0.6, 2), rng.uniform(0.5, 1.5)
        for out, w in ((x0, 0.4), (b, 0.1)):
            out += a * np.outer(np.exp(-(t - cy) ** 2 / (2 * w * w)), np.exp(-(t - cx) ** 2 / (2 * w * w)))
    x0, b = x0.reshape(-1), b.reshape(-1)
    omega = float(np.float32(0.8))
    s = Solver(n, m=10, guess_omega=omega)
    xd = s.smooth(torch.as_tensor(b).cuda(), torch.as_tensor(x0.copy()).cuda(), sweeps)
    ref = _sweeps_by_differences(n, b, x0, sweeps, omega, np.longdouble)
    plain = _sweeps_by_differences(n, b, x0, sweeps, omega, np.float64)

    def err(v):
        return np.linalg.norm((v - ref).astype(np.float64)) / np.linalg.norm(ref.astype(np.float64))

    assert err(xd.cpu().numpy()) <= 1.15 * err(plain), (err(xd.cpu().numpy()), err(plain))


@pytest.mark.parametrize("at", ["corner", "edge"])
def test_fp64_norm_is_the_rounded_root(at):
    """The first subdiagonal entry of the Hessenberg matrix from a unit vector at a corner
    (or edge) point: A e leaves -1/h^2 at its 2 (3) neighbours, every sum on the way is
    exact or rounded once, so ||w|| is the correctly rounded root of 2 (3) / h^4."""
    from paper_2103_10975_gb300 import Solver
    for n in range(3, 17):
        h = 2.0 / (n + 1)
        s2 = 1.0 / (h * h)
        a = s2 * s2
        e = torch.zeros(n * n, dtype=torch.float64)
        e[0 if at == "corner" else 1] = 1.0
        _, H, _ = Solver(n, m=4).arnoldi(e.cuda(), 2)
        assert H[1, 0] == np.sqrt(2.0 * a if at == "corner" else 2.0 * a + a), n


@pytest.mark.parametrize("n", [5, 33, 130, 321, 384, 390, 450])
def test_sweeps_in_one_call_or_one_by_one(n):
    """Several sweeps per launch (small grids), one per launch (large ones) and the
    remainders of one or two sweeps: the same operations per point, so at most a rounding
    or two per sweep apart if a compiler contracts them differently."""
    from paper_2103_10975_gb300 import Solver
    s = Solver(n, m=5, guess_omega=0.75)
    rng = np.random.default_rng(n)
    b = torch.as_tensor(rng.standard_normal(n * n)).cuda()
    x0 = torch.as_tensor(rng.standard_normal(n * n)).cuda()
    one = x0.clone()
    for k in range(1, 12):
        s.smooth(b, one, 1)
        many = s.smooth(b, x0.clone(), k)
        assert float((many - one).norm()) <= k * 2.3e-16 * float(one.norm()), k
