"""Launch shapes: the tuner's cache and the untuned choices (GPU)."""

import pytest

torch = pytest.importorskip("torch")

from synthetic import MovingGaussians2D

pytestmark = pytest.mark.gpu


def test_tuning_cache_keeps_options_apart():
    """A shape found under one set of options is not taken over by a handle that times
    other candidates: two CTAs per SM (compact = 1) would be more than a handle without
    the compact variant can launch, and a fixed CTA count is no choice at all."""
    from paper_2103_10975_gb300 import Solver
    n, m = 660, 28
    bd = torch.as_tensor(MovingGaussians2D(n, 77, 50).rhs(3)).cuda()
    for opt in ({"compact": 1}, {"grid_blocks": 100}, {"compact": 0}, {"v_stages": 0},
                {"compact": 0, "v_stages": 4}, {}):
        for again in (0, 1):
            s = Solver(n, m=m, rtol=1e-10, precision="fp32_refine", max_iters=2 * m, **opt)
            t = s.autotune(bd)
            assert t["from_cache"] == again, (opt, t)
            if again == 0:
                first = t
            assert all(t[k] == first[k] for k in ("grid_blocks", "v_stages", "compact")), (opt, t)
            _, r = s.solve(bd, check=False)
            assert r["status_code"] == 1 and r["iters"] == 2 * m, (opt, r, s.error())
            s.close()
