"""GPU tests of the FP64 residual kernel (csrc/residual_f64.cu) over its tile forms: 4, 8 and 32
rows, ragged last tiles on both axes, odd sizes (the plan-free entry point), the smallest grid,
displacements over many cells and across the period, and values that are not finite.

Bound: as the other residual tests, 32 eps max|u| max(N, M)^2 max|g| for the stencils plus 1e-13
for the gather and the products."""
import numpy as np
import pytest

import oracle as O
import ot_inputs as I
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


def noalloc(ot, f, c, u):
    N, M = u.shape
    F, coef, scal = dev(np.zeros((N, M))), dev(np.zeros((5, N, M))), np.zeros(10)
    assert ot.ot_eval_residual_noalloc(N, M, ptr(dev(f)), ptr(dev(c)), ptr(dev(u)), ptr(F),
                                       ptr(coef), hptr(scal)) == 0
    return F.cpu().numpy(), coef.cpu().numpy(), scal


# (8, 8) .. (333, 250): 4-row tiles; (512, 520) and (1000, 260): 8-row tiles; (801, 803): 32-row
# tiles with ragged edges
@pytest.mark.parametrize("N,M", [(8, 8), (9, 11), (66, 34), (333, 250), (512, 520), (1000, 260),
                                 (801, 803)])
@pytest.mark.parametrize("amp", [1e-3, 0.2])
def test_residual_over_tile_forms(ot, N, M, amp):
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    # amp 0.2: displacements of more than a period (|grad u| up to 2.5), det of any sign
    u = amp * (np.cos(2 * np.pi * (x + y)) + 0.5 * np.sin(2 * np.pi * (x - y)))
    f = 1 + 0.5 * np.cos(2 * np.pi * x)
    c = 1 + 0.3 * np.sin(2 * np.pi * (x + 2 * y))
    F_ref, coef_ref, s = O.residual(f, c, u)
    F, coef, scal = noalloc(ot, f, c, u)
    # det reaches (4 pi^2 amp)^2: the determinant's own rounding scales with it
    big = max(1.0, np.abs(coef_ref).max())
    tol = 32 * np.finfo(float).eps * amp * max(N, M) ** 2 * big + 1e-13 * big ** 2
    assert np.abs(F - F_ref).max() <= tol
    assert np.abs(coef - coef_ref).max() <= tol * max(N, M)  # b: gradients of g in grid units
    for k, name in enumerate(("mean_fn", "res_inf", "res_l2", "min_det")):
        assert abs(scal[k] - s[name]) <= tol
    assert scal[4] == 0
    abar = np.array([O.simpson_mean(coef_ref[q]) for q in range(5)])
    assert np.abs(scal[5:] - abar).max() <= tol * max(N, M)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_values_that_are_not_finite_are_counted(ot, bad):
    N = M = 40
    f, c = np.ones((N, M)), 1 + 0.1 * np.cos(2 * np.pi * np.arange(M) / M)[None, :] * np.ones((N, 1))
    u = np.zeros((N, M))
    u[7, 9] = bad
    s = O.residual(f, c, u)[2]
    F, _, scal = noalloc(ot, f, c, u)
    # every point whose stencils reach it: the 5 x 5 neighbourhood
    reach = np.zeros((N, M), bool)
    reach[5:10, 7:12] = True
    assert scal[4] == s["nonfinite"] == 25
    assert np.array_equal(np.isfinite(F), ~reach)
    # the others keep their values, up to the shift by the mean (of the finite f_n only)
    F0 = O.residual(f, c, np.zeros((N, M)))[0]
    assert np.ptp((F - F0)[~reach]) <= 1e-13


def test_coefficients_into_planes_that_overlap_an_input(ot):
    N = M = 64
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    u = 1e-3 * np.cos(2 * np.pi * (x + y))
    f, c = I.blob_density(N, M, 5), O.bspline_coeffs(I.blob_density(N, M, 6))
    p = ot.Plan(N, M)
    F, coef, scal = dev(np.zeros((N, M))), dev(np.zeros((5, N, M))), np.zeros(10)
    assert ot.ot_eval_residual(p.h, ptr(dev(f)), ptr(dev(c)), ptr(dev(u)), ptr(F), ptr(coef),
                               hptr(scal)) == 0
    # u is the third of the five output planes: read before it is overwritten
    both = dev(np.zeros((5, N, M)))
    both[2].copy_(dev(u))
    F2, scal2 = dev(np.zeros((N, M))), np.zeros(10)
    assert ot.ot_eval_residual(p.h, ptr(dev(f)), ptr(dev(c)), ptr(both[2]), ptr(F2), ptr(both),
                               hptr(scal2)) == 0
    assert (F2 == F).all() and (both == coef).all() and np.array_equal(scal, scal2)
    p.close()
