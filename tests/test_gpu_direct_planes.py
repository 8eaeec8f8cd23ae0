"""GPU tests of calls that use the caller's memory as the passes' own operands: planes 16 bytes
aligned and 8 bytes off, results over an input, refused inputs, a gradient without its loss.

Every path runs the same kernels on the same values, so they agree bit for bit."""
import ctypes

import numpy as np
import pytest

import ot_inputs as I
from gpu_util import dev, ptr

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


def off8(a):
    """a on the device, 8 bytes past a 16-byte boundary"""
    import torch
    t = torch.zeros(a.size + 1, dtype=torch.float64, device="cuda")[1:]
    t.copy_(dev(a).view(-1))
    assert t.data_ptr() % 16 == 8
    return t


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("N,M", [(16, 24), (96, 64), (256, 512)])
def test_planes_where_they_lie(ot, N, M, prec):
    rng = np.random.default_rng(N + M)
    P = N * M
    x = rng.standard_normal((N, M))
    coef = rng.standard_normal((5, N, M))
    abar = np.array([1.1, 0.9, 0.05, 0.0, 0.0])
    ab = ctypes.c_void_p(abar.ctypes.data)
    p = ot.Plan(N, M, precision=prec)
    get = lambda t, n=P: t.view(-1)[:n].cpu().numpy()
    calls = {
        "fwd": lambda a, o, c: ot.ot_fft_forward(p.h, ptr(a), ptr(o)),
        "inv": lambda a, o, c: ot.ot_fft_inverse(p.h, ptr(a), ptr(o)),
        "lbar": lambda a, o, c: ot.ot_apply_lbar_inverse(p.h, ab, ptr(a), ptr(o)),
        "op": lambda a, o, c: ot.ot_apply_operator(p.h, ptr(c), ab, ptr(a), ptr(o)),
    }
    for name, call in calls.items():
        a, o, c = dev(x), dev(np.zeros((N, M))), dev(coef)
        assert call(a, o, c) == 0
        ref = get(o)
        assert np.abs(ref).max() > 0 and np.array_equal(get(a), x.ravel())
        assert np.array_equal(get(c, 5 * P), coef.ravel())
        a, o, c = off8(x), off8(np.zeros((N, M))), off8(coef)
        assert call(a, o, c) == 0 and np.array_equal(get(o), ref), name
        a, c = dev(x), dev(coef)
        assert call(a, a, c) == 0 and np.array_equal(get(a), ref), name
        if name == "op":  # the result over a coefficient plane
            a, c = dev(x), dev(coef)
            assert call(a, c[2], c) == 0 and np.array_equal(get(c[2]), ref)
    p.close()


def test_refused_inputs_leave_the_rows(ot):
    import torch
    N, M = 64, 96
    f, g = I.blob_pair(N, M, s=3)
    p = ot.Plan(N, M, precision="mixed")
    for bad in (np.nan, np.inf, -1e6):
        X = torch.full((N * M, 16), 7.0, dtype=torch.float32, device="cuda")
        t = torch.full((N * M,), 7.0, dtype=torch.float32, device="cuda")
        fb = f.copy()
        fb[5, 7] = bad
        with pytest.raises(ot.OTError):
            p.ws_features(dev(fb), dev(g), X, t, phi_star=dev(np.zeros((N, M))))
        assert bool((X == 7.0).all()) and bool((t == 7.0).all())
    p.ws_features(dev(f), dev(g), X, t, phi_star=dev(np.zeros((N, M))))
    assert not bool((X == 7.0).any()) and bool(torch.isfinite(t).all())
    p.close()


def test_gradient_and_loss_on_their_own(ot):
    import torch
    rng = np.random.default_rng(2)
    X = torch.tensor(rng.standard_normal((256, 16)), dtype=torch.float32, device="cuda")
    t = torch.tensor(rng.standard_normal(256), dtype=torch.float32, device="cuda")
    idx = torch.arange(128, dtype=torch.int64, device="cuda")
    tr = ot.Trainer(128, I.ws_init_params(4))
    loss, grad = tr.grad(X, t, idx)
    g2, l2 = np.zeros_like(grad), ctypes.c_double()
    args = (ptr(X), ptr(t), ptr(idx))
    assert ot.ot_ws_trainer_grad(tr.h, *args, ctypes.c_void_p(g2.ctypes.data), None) == 0
    assert ot.ot_ws_trainer_grad(tr.h, *args, None, ctypes.byref(l2)) == 0
    assert np.array_equal(g2, grad) and l2.value == loss
    assert tr.step(X, t, idx, 1e-3, want_loss=True) == loss
    assert tr.step(X, t, idx, 1e-3) is None
    assert tr.grad(X, t, idx)[0] < loss
    tr.close()
