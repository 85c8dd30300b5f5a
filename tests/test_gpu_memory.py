"""Device memory that a handle takes (GPU)."""

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _taken(**kw):
    from paper_2103_10975_gb300 import Solver
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    s = Solver(**kw)
    free1 = torch.cuda.mem_get_info()[0]
    s.close()
    return free0 - free1


@pytest.mark.parametrize("dim,n,prec,vectors", [(2, 512, "fp32_refine", 3), (2, 512, "fp64", 2),
                                                (3, 64, "fp32_refine", 2), (3, 64, "fp64", 2)])
def test_batch_workspace(dim, n, prec, vectors):
    """Per reserved group a basis of m + 1 vectors (rounded up to pairs) and two work
    vectors, three in 2D FP32 (w' with tags); 24 MB for the rest and the allocator's
    granularity."""
    m, slots = 5, 100
    kw = dict(dim=dim, n=n, m=m, precision=prec)
    vec = n ** dim * (8 if prec == "fp64" else 4)  # (n^dim is a multiple of 64)
    extra = _taken(batch_slots=slots, **kw) - _taken(**kw)
    assert extra <= slots * vec * (m + 1 + vectors) + (24 << 20), extra / (slots * vec)


@pytest.mark.parametrize("prec", ["fp64", "fp32_refine"])
def test_small_handles_stay_small(prec):
    """Four handles at n = 32, m = 20: each needs about 0.2 MB of vectors and 0.6 MB of
    partial sums (rows of at most 304 CTAs), in FP32 7 MB of triangles for the compact
    variants; with rows for 1 024 CTAs the sums take 1.8 MB."""
    from paper_2103_10975_gb300 import Solver
    keep = Solver(32, m=20, precision=prec)  # (the library's own first allocations)
    free0 = torch.cuda.mem_get_info()[0]
    hs = [Solver(32, m=20, precision=prec) for _ in range(4)]
    taken = free0 - torch.cuda.mem_get_info()[0]
    for h in hs + [keep]:
        h.close()
    assert taken <= (4 << 20) + (4 * (8 << 20) if prec == "fp32_refine" else 0), taken
