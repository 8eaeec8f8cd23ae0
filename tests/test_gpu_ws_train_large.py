"""GPU test of the trainer's gradient on a minibatch above 2048 rows per SM, where the number of
blocks follows the rows (a block sums at most 2048) instead of the SMs, the grid takes several waves
and a block runs tens of chunks.

Bound: as over the smaller splits, the gradient in 64 bits within 1e-4 of each tensor's largest
entry; the FP32 sums over rows are no longer than there (2048 rows a block, then the blocks)."""
import numpy as np
import pytest

import oracle.warmstart as W

pytestmark = pytest.mark.gpu


def test_gradient_of_a_minibatch_of_several_waves():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1009_6039_gb300 as ot
    B, n, part = 400000, 50021, 25000  # B > 2048 x 152, a last block that is not full
    rng = np.random.default_rng(7)
    p = np.concatenate([a.reshape(-1) for a in (
        rng.standard_normal((W.H, W.K)) / 4, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal((W.H, W.H)) / 11, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal((W.H, W.H)) / 11, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal(W.H) / 11, 0.1 * rng.standard_normal(1))]).astype(np.float32)
    X = rng.standard_normal((n, W.K)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    idx = rng.integers(0, n, B)
    dX, dt, di = (torch.from_numpy(v).cuda() for v in (X, t, idx))
    tr = ot.Trainer(B, p)
    loss, g = tr.grad(dX, dt, di)
    loss2, g2 = tr.grad(dX, dt, di)
    tr.close()
    assert loss2 == loss and np.array_equal(g2, g)
    # the mean over the rows as the mean over equal parts of them
    p64, loss_ref, g_ref = p.astype(np.float64), 0.0, 0.0
    for b in range(0, B, part):
        r = idx[b:b + part]
        a, d = W.loss_and_grad(p64, X[r].astype(np.float64), t[r].astype(np.float64))
        loss_ref, g_ref = loss_ref + a * part / B, g_ref + d * (part / B)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    o = 0
    for size in (W.H * W.K, W.H, W.H * W.H, W.H, W.H * W.H, W.H, W.H, 1):
        a, b = g[o:o + size], g_ref[o:o + size]
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max() + 1e-12, o
        o += size
