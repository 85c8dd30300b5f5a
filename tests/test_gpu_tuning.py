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


@pytest.mark.parametrize("n,free", [(256, True), (300, True), (380, True), (512, False), (660, False)])
def test_untuned_learned_handles_leave_sms_free(n, free):
    """Without tuning, a handle that trains beside its solves leaves an eighth of the SMs
    free where the basis stays in shared memory all the same (GMRES(30): not at 512^2, and
    660^2 streams).  The CTA count shows in the order of the sums: the iterate after
    a capped first solve has the bits of a plain handle's on the expected count."""
    from paper_2103_10975_gb300 import Solver
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    bd = torch.as_tensor(MovingGaussians2D(n, 77, 50).rhs(3)).cuda()

    def first(**kw):
        s = Solver(n, m=30, rtol=1e-10, precision="fp32_refine", max_iters=90, **kw)
        x, r = s.solve(bd, check=False)
        assert r["status_code"] == 1, s.error()
        s.close()
        return x

    x = first(guess="learned", replay_cap=2, batch=1)
    if n == 256:
        assert torch.equal(x, first(grid_blocks=128))
    elif free:
        assert torch.equal(x, first(grid_blocks=sms - sms // 8))
        assert not torch.equal(x, first(grid_blocks=sms))
    else:
        assert torch.equal(x, first())
