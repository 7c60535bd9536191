"""The network kernels at the edges of their 128-row tiles: fewer rows than a
tile, one row more than a whole wave of tiles, and inputs that are only 4-byte
aligned, against the FP64 oracle with BF16 operands."""
import numpy as np
import pytest

from oracle import wall_oracle as w
from tests import seeded

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,offset", [(1, 0), (127, 1), (128, 0), (129, 3), (300, 2), (152 * 128 + 1, 1)])
def test_forward_and_gradient_at_tile_edges(rows, offset):
    import torch

    from paper_1701_02005_gb300.wallmodel import MLP

    net = MLP(rows, seed=25)
    r = seeded.rng(26 + rows)
    norm = [r.normal(size=40).astype(np.float32), r.uniform(0.5, 2, 40).astype(np.float32),
            r.normal(size=5).astype(np.float32), r.uniform(0.5, 2, 5).astype(np.float32)]
    net.set_normalization(*norm)
    p = net.params()
    p[-5:] = 0.1   # output biases too
    net.set_params(p)
    X = r.standard_normal((rows, 40)).astype(np.float32)
    T = r.standard_normal((rows, 5)).astype(np.float32)

    def device(a):   # contiguous, `offset` floats behind an aligned address
        buf = torch.zeros(a.size + 4, device="cuda")
        v = buf[offset:offset + a.size].view(a.shape)
        v.copy_(torch.from_numpy(a))
        return v

    Xd, Td = device(X), device(T)
    # a BF16 operand whose rounding flips between the two GELU evaluations moves by
    # 2^-8; one flip per hidden layer on the way to a value bounds the difference
    # where few rows average it
    tol = 4 * 2.0 ** -8
    Y = net.forward(Xd).cpu().numpy()
    Yr, _ = w.forward(p, X, norm, bf16=True, bf16_act=True)
    Yr = np.clip((Yr - norm[2]) * norm[3], -6, 6) / norm[3] + norm[2]
    assert np.max(np.abs(Y - Yr)) <= tol * np.max(np.abs(Yr))
    g, loss = net.gradient(Xd, Td)
    lr, gr = w.loss_and_grad(p, X, T, norm, bf16=True, bf16_act=True)
    assert abs(loss - lr) <= tol * lr
    sl, _ = w.param_slices()
    for ws, bs, _, _ in sl:
        for s_ in (ws, bs):
            assert np.max(np.abs(g[s_] - gr[s_])) <= tol * np.max(np.abs(gr[s_]))
    g2, loss2 = net.gradient(Xd, Td)   # fixed-order sums
    assert np.array_equal(g, g2) and loss == loss2
    assert net.status() == 0
    net.close()
