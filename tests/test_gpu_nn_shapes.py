"""The network's kernels at the edges of their tiles, segments and levels (GPU):
one-level grids, odd sides (dropped pooling rows), rows around the segment length
and past the staged row's limit, several samples.  Bounds as in test_gpu_nn: BF16
operands, 3e-2 on the outputs and 4e-2 per gradient tensor against the FP64
oracle at the BF16-rounded weights."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import nn as onn
from test_gpu_nn import (bf16_params_3d, bf16_round, check_grads, sample_batch,
                         sample_batch_3d, unpack)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,n,B", [(2, 8, 1), (2, 9, 3), (2, 15, 2), (2, 31, 1), (2, 67, 3),
                                     (2, 130, 2), (2, 257, 1), (2, 385, 1), (3, 9, 1), (3, 17, 2),
                                     (3, 21, 1)])
def test_forward_and_gradients_at_odd_shapes(dim, n, B):
    from paper_2103_10975_gb300 import Solver
    s = Solver(n, dim=dim, m=10, batch=B)
    if dim == 2:
        P = unpack(s.get_params(), n)
        for k in P:
            if k.startswith("level") and k.endswith(".w") or k == "dil.w":
                P[k] = bf16_round(P[k])
        u, t = sample_batch(n, B, 11)
    else:
        P = bf16_params_3d(s, n)
        u, t = sample_batch_3d(n, B, 11)
    ud = torch.as_tensor(u, dtype=torch.float32).cuda()
    y = s.nn_forward(ud).cpu().numpy()
    for b in range(B):
        yr = onn.forward(P, u[b], n, dim=dim)
        assert np.linalg.norm(y[b] - yr) <= 3e-2 * np.linalg.norm(yr), b
    loss, g = s.nn_loss_grad(ud, torch.as_tensor(t, dtype=torch.float32).cuda())
    lr, gr = onn.loss_and_grads(P, u, t, n, dim=dim)
    assert abs(loss - lr) <= 2e-2 * lr
    check_grads(unpack(g, n, dim=dim), gr, "%dD n=%d" % (dim, n))


@pytest.mark.parametrize("dim,n,B", [(2, 100, 4), (2, 127, 3), (3, 8, 1), (3, 13, 2), (3, 30, 2),
                                     (3, 52, 1)])
def test_packed_tiles_give_the_row_tiles_bits(dim, n, B, monkeypatch):
    """Tiles over several padded rows against a tile per row segment
    (MLGMRES_TC_MIN_ROW = 1): the same MMAs per output in the same order, so the
    forward pass is the same bits; the weight gradients' FP32 sums are split
    differently (relative 1e-6 of each tensor's norm: about sqrt(tiles) roundings)."""
    from paper_2103_10975_gb300 import Solver
    s = Solver(n, dim=dim, m=10, batch=B)
    rng = np.random.default_rng(n)
    u = torch.as_tensor(rng.standard_normal((B, n ** dim)), dtype=torch.float32).cuda()
    t = torch.as_tensor(rng.standard_normal((B, n ** dim)), dtype=torch.float32).cuda()
    out = []
    for rows in (None, "1"):
        if rows:
            monkeypatch.setenv("MLGMRES_TC_MIN_ROW", rows)
        out.append((s.nn_forward(u).cpu().numpy(), s.nn_loss_grad(u, t)[1]))
    assert np.array_equal(out[0][0], out[1][0])
    d = np.linalg.norm(out[0][1] - out[1][1])
    assert d <= 1e-6 * np.linalg.norm(out[1][1]), d
