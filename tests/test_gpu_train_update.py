"""The training step's one update launch against the gradient, Adam and copies
made one by one: widths that are no multiple of the 32 x 32 tiles, one row,
batches that end inside a tile, and a network of more layers than one launch
takes.  The float32 sums run in the same order and Adam is the same formula, so
parameters agree to its rounding (an update is at most lr = 1e-3 in size).
"""
import numpy as np
import pytest

import meshgen

torch = pytest.importorskip("torch")
import paper_2510_12053_gb300 as cc  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d_in,hidden,layers,d_out,batch", [(30, 64, 2, 24, 77), (9, 40, 1, 8, 1), (258, 72, 3, 40, 33),
                                                            (17, 24, 10, 16, 96), (64, 256, 2, 576, 1000)])
def test_training_equals_gradient_and_adam_steps(d_in, hidden, layers, d_out, batch):
    rows, steps, ldx = 200, 3, (d_in + 7) // 8 * 8
    X = torch.zeros((rows, ldx), dtype=torch.bfloat16)
    X[:, :d_in] = torch.from_numpy(meshgen.normal(3, np.arange(rows * d_in)).reshape(rows, d_in)).to(torch.bfloat16)
    T = torch.from_numpy((0.3 * meshgen.normal(4, np.arange(rows * d_out))).reshape(rows, d_out).astype(np.float32))
    idx = torch.from_numpy(meshgen.batch_indices(5, 0, steps, batch, rows))
    X, T = X.cuda(), T.cuda()
    shape = dict(d_in=d_in, hidden=hidden, layers=layers, d_out=d_out, max_batch=batch)
    a, b = cc.MLP(**shape), cc.MLP(**shape)
    p = (0.1 * meshgen.normal(6, np.arange(a.param_count))).astype(np.float32)
    a.set_params(p)
    b.set_params(p)
    losses = a.train(X, T, idx.cuda(), batch, lr=1e-3)
    for t in range(steps):
        rows_t = idx[t].long().cuda()
        loss, g = b.loss_grad(X[rows_t].contiguous(), T[rows_t].contiguous())
        b.adam_step(g, lr=1e-3)
        assert abs(losses[t] - loss) <= 1e-6 * loss
    np.testing.assert_allclose(a.get_params(), b.get_params(), rtol=0, atol=3 * 1e-6)
    assert np.abs(a.get_params() - p).max() > 1e-4
    a.close()
    b.close()
