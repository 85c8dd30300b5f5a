"""The schedule of 2D FP32 batches whose bases stay in shared memory (host logic behind
mlgmres_solve_batch), through the C ABI with no GPU."""
import random

import pytest

from paper_2103_10975_gb300 import MLGMRESError, batch_plan_slices

CTAS, STREAM = 152, 304  # one and two CTAs per SM


def tiles(n):
    return (n * n + 31) // 32


def max_tiles(m):
    # 213 KB (m <= 32) or about 165 KB of shared memory, 32-point rows of pairs of vectors
    return (213 if m <= 32 else 165) * 1024 // (128 * (m + (m & 1)))


def check(sides, ctas, most, gc, go):
    assert 1 <= len(gc) <= ctas and sum(gc) <= ctas and min(gc) >= 1
    assert len(go) == len(sides) and set(go) == set(range(len(gc)))
    for n, g in zip(sides, go):
        assert -(-tiles(n) // gc[g]) <= most, (n, gc[g], most)


@pytest.mark.parametrize("seed", range(12))
def test_every_slice_fits(seed):
    r = random.Random(seed)
    m = r.choice([1, 2, 8, 20, 30, 33, 47, 64])
    lo = r.randint(1, 120)
    sides = [r.randint(lo, lo + r.choice([0, 20, 150])) for _ in range(r.choice([1, 2, 7, 40, 400]))]
    ctas = r.choice([1, 5, 40, CTAS])
    most = max_tiles(m)
    gc, go, _ = batch_plan_slices(sides, m, ctas, 2 * ctas, most)
    if max(-(-tiles(n) // ctas) for n in sides) > most:
        assert gc == [] and go == []
        return
    check(sides, ctas, most, gc, go)
    assert batch_plan_slices(sides, m, ctas, 2 * ctas, most)[:2] == (gc, go)


def test_limits_of_the_fit():
    # a system of exactly ctas * max_tiles tiles takes every CTA; one tile more fits nothing
    assert tiles(80) == 200
    assert batch_plan_slices([80], 30, 10, 20, 20)[:2] == ([10], [0])
    assert batch_plan_slices([80], 30, 10, 20, 19)[:2] == ([], [])
    # two of them share the one group there can be
    assert batch_plan_slices([80, 80], 30, 10, 20, 20)[:2] == ([10], [0, 0])


def test_preferred_where_it_was_faster_and_only_there():
    """Batches timed with either placement (GB300; slices against streamed, ms)."""
    def preferred(count, lo, hi, m, **kw):
        step = (hi - lo) / max(1, count - 1)
        sides = [round(lo + i * step) for i in range(count)]
        return batch_plan_slices(sides, m, CTAS, STREAM if m <= 47 else CTAS, max_tiles(m), **kw)[2]
    assert preferred(42, 76, 102, 30)        # 8.1 / 12.6
    assert preferred(19, 109, 207, 16)       # 41 / 63
    assert preferred(19, 51, 89, 64)         # 6.2 / 8.4
    assert preferred(40, 24, 160, 30)        # 36 / 55
    assert not preferred(356, 39, 75, 64)    # 26 / 17
    assert not preferred(290, 9, 119, 50)    # 65 / 32
    assert not preferred(231, 132, 161, 40)  # 642 / 302
    assert not preferred(102, 30, 140, 40)   # 41 / 22
    assert not preferred(46, 16, 160, 40)    # 55 / 44


def test_step_budget_counts():
    """Under a budget that every system uses up, the large ones do not take n^2 times
    as long: the groups differ from those of converging solves."""
    sides = list(range(64, 200, 2))
    a = batch_plan_slices(sides, 4, CTAS, STREAM, max_tiles(4))
    b = batch_plan_slices(sides, 4, CTAS, STREAM, max_tiles(4), max_iters=500)
    check(sides, CTAS, max_tiles(4), *a[:2])
    check(sides, CTAS, max_tiles(4), *b[:2])
    assert a[0] != b[0]


@pytest.mark.parametrize("args", [([], 30, 8, 8, 50), ([10], 0, 8, 8, 50), ([10], 30, 0, 8, 50),
                                  ([10], 30, 8, 0, 50), ([10], 30, 8, 8, 0), ([0], 30, 8, 8, 50),
                                  ([32769], 30, 8, 8, 50)])
def test_bad_arguments(args):
    with pytest.raises((MLGMRESError, ValueError)):
        batch_plan_slices(*args)


@pytest.mark.parametrize("kw", [{"rtol": 0.0}, {"rtol": 1.0}, {"max_iters": 0}])
def test_bad_stopping_rule(kw):
    with pytest.raises(MLGMRESError):
        batch_plan_slices([10], 30, 8, 8, 50, **kw)
