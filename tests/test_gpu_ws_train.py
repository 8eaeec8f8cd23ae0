"""GPU tests of the trainer's gradient kernel (csrc/ws_train.cu) over its splits of a minibatch:
two, four and seven rows per warp pair, one chunk and several per block, a last chunk and a last
block that are not full, fewer rows than one block holds.

Bound: the oracle's gradient in 64 bits, within 1e-4 of each tensor's largest entry (the bound of
the other gradient test): three layers of 128-term FP32 dot products forward and two backward, each
within 128 x 2^-24 = 8e-6 of the sum of its terms' sizes, and the sums over rows on top."""
import numpy as np
import pytest

import oracle.warmstart as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1009_6039_gb300 as m
    return m


@pytest.mark.parametrize("B", [64, 192, 1024, 2496, 4864, 8512, 20032])
def test_gradient_over_batch_splits(ot, B):
    import torch
    rng = np.random.default_rng(B)
    p = np.concatenate([a.reshape(-1) for a in (
        rng.standard_normal((W.H, W.K)) / 4, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal((W.H, W.H)) / 11, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal((W.H, W.H)) / 11, 0.1 * rng.standard_normal(W.H),
        rng.standard_normal(W.H) / 11, 0.1 * rng.standard_normal(1))]).astype(np.float32)
    n = B + 37
    X = rng.standard_normal((n, W.K)).astype(np.float32)
    t = rng.standard_normal(n).astype(np.float32)
    idx = rng.integers(0, n, B)
    tr = ot.Trainer(B, p)
    loss, g = tr.grad(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda(),
                      torch.from_numpy(idx).cuda())
    loss_ref, g_ref = W.loss_and_grad(p.astype(np.float64), X[idx].astype(np.float64),
                                      t[idx].astype(np.float64))
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    o = 0
    for size in (W.H * W.K, W.H, W.H * W.H, W.H, W.H * W.H, W.H, W.H, 1):
        a, b = g[o:o + size], g_ref[o:o + size]
        assert np.abs(a - b).max() <= 1e-4 * np.abs(b).max() + 1e-12, o
        o += size
    # the same rows again: the same bits (fixed summation order)
    loss2, g2 = tr.grad(torch.from_numpy(X).cuda(), torch.from_numpy(t).cuda(),
                        torch.from_numpy(idx).cuda())
    assert loss2 == loss and np.array_equal(g2, g)
    tr.close()
