"""The gradient of batches of several tiles per CTA, with the labels of one tile's rows
so far off that they make up the gradient: a row of that tile that is dropped, taken
twice or mixed with another tile's shows in every layer."""
import numpy as np
import pytest

from oracle import wall_oracle as w
from tests import seeded

pytestmark = pytest.mark.gpu

TILE = 128


# tile of the one that matters: the last of the first turn, the first of the second, one
# in the third, and the rest of the batch (77 rows, or a single one) in the turn after
@pytest.mark.parametrize("turns,rest,turn,cta", [(1, 1, 1, 0), (3, 77, 0, -1), (3, 77, 1, 0), (3, 77, 2, 60),
                                                 (3, 77, 3, 0)])
def test_one_tile_makes_the_gradient(turns, rest, turn, cta):
    import torch

    from paper_1701_02005_gb300.wallmodel import MLP

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    rows = turns * sms * TILE + rest
    first = (turn * sms + cta % sms) * TILE
    hot = slice(first, min(first + TILE, rows))
    net = MLP(rows, seed=25)
    r = seeded.rng(27 + turn)
    norm = [r.normal(size=40).astype(np.float32), r.uniform(0.5, 2, 40).astype(np.float32),
            r.normal(size=5).astype(np.float32), r.uniform(0.5, 2, 5).astype(np.float32)]
    net.set_normalization(*norm)
    p = net.params()
    p[-5:] = 0.1
    net.set_params(p)
    X = r.standard_normal((rows, 40)).astype(np.float32)
    Y, _ = w.forward(p, X, norm, bf16=True, bf16_act=True)
    T = Y.astype(np.float32)   # the other rows' labels: the network's own outputs
    T[hot] += 1e3 * r.standard_normal(T[hot].shape).astype(np.float32)
    g, loss = net.gradient(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    lr, gr = w.loss_and_grad(p, X, T, norm, bf16=True, bf16_act=True)
    # a BF16 operand whose rounding flips between the two GELU evaluations moves by
    # 2^-8: one flip per hidden layer on the way to a value, as where a batch is one
    # row.  The other rows' errors (2^-8 of outputs of order 1, signs mixed) stay below
    # 2^-8 sqrt(rows) = 1 beside the 1e3 of each row that matters.
    tol = 4 * 2.0 ** -8
    assert abs(loss - lr) <= tol * lr
    sl, _ = w.param_slices()
    for ws, bs, _, _ in sl:
        for s_ in (ws, bs):
            assert np.max(np.abs(g[s_] - gr[s_])) <= tol * np.max(np.abs(gr[s_]))
    assert net.status() == 0
    net.close()
