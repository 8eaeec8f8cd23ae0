"""GPU tests of the FP64 residual's scalars with a NaN in f.

Expected values: res_inf is the largest |F| over the points whose F is a number.  The kernel forms
it as max(|max(f - f_n) + shift|, |min(f - f_n) + shift|) and F as (f - f_n) + shift, and rounding
is monotone, so the two agree bit for bit."""
import numpy as np
import pytest

import oracle as O
from gpu_util import dev, hptr, ptr

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


def residual(ot, f, c, u, plan=None):
    N, M = u.shape
    F, coef, scal = dev(np.zeros((N, M))), dev(np.zeros((5, N, M))), np.zeros(10)
    planes = [dev(v) for v in (f, c, u)] + [F, coef]
    a = [ptr(v) for v in planes] + [hptr(scal)]
    rc = ot.ot_eval_residual(plan.h, *a) if plan else ot.ot_eval_residual_noalloc(N, M, *a)
    assert rc == 0
    return F.cpu().numpy(), coef.cpu().numpy(), scal


# 4-, 8- and 32-row tiles; the finite points' largest |F| above or below zero
@pytest.mark.parametrize("N,M", [(40, 40), (512, 520), (801, 803)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("side", [1.0, -1.0])
def test_nan_in_f_leaves_the_other_points_maximum(ot, N, M, sign, side):
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    u = 1e-4 * np.cos(2 * np.pi * (x + y))
    f = 1 + 0.3 * np.cos(2 * np.pi * x)
    f[N - 1, M // 2] += 5 * side
    f[3, 5] = np.copysign(np.nan, sign)
    f[N // 2, M - 1] = np.copysign(np.nan, sign)
    c = 1 + 0.1 * np.sin(2 * np.pi * (x + 2 * y))
    F, _, scal = residual(ot, f, c, u)
    assert np.array_equal(np.isnan(F), np.isnan(f))
    assert scal[1] == np.nanmax(np.abs(F)) > 4
    assert scal[4] == O.residual(f, c, u)[2]["nonfinite"] == 0
    # f_n, its mean and the determinant do not see f
    clean = residual(ot, np.where(np.isnan(f), 1.0, f), c, u)[2]
    assert scal[0] == clean[0] and scal[3] == clean[3]


def test_nan_in_f_with_a_plan(ot):
    N, M = 64, 96
    f, c, u = np.ones((N, M)), np.ones((N, M)), np.zeros((N, M))
    f[1, 2], f[40, 50] = np.nan, 7.0
    p = ot.Plan(N, M)
    F, _, scal = residual(ot, f, c, u, p)
    p.close()
    assert np.array_equal(np.isnan(F), np.isnan(f))
    assert scal[1] == np.nanmax(np.abs(F)) > 5
