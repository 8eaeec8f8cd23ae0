"""GPU tests of the mixed mode's residual on packed point pairs: each of its three tile forms, rows
that have no partner, grids smaller than a tile, and non-finite points, against the FP64 mode.

Bounds: F 2^-44 of the largest stencil term times the largest |G det| factor (2^-48 per double-float
operation, some ten of them in a row); the coefficients G (1 + u_xx) and so on 2^-20 of each plane's
largest value (FP32 products), those with the gradient 8 2^-24 max|c| det times N or M (FP32 weights
of at most 2 in absolute sum and the sums' own rounding); counts exactly."""
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


def evaluate(ot, prec, f, g, u):
    N, M = f.shape
    p = ot.Plan(N, M, precision=prec)
    c, F, coef = dev(np.zeros((N, M))), dev(np.zeros((N, M))), dev(np.zeros((5, N, M)))
    scal = np.zeros(10)
    assert ot.ot_prefilter(p.h, ptr(dev(g)), ptr(c)) == 0
    assert ot.ot_eval_residual(p.h, ptr(dev(f)), ptr(c), ptr(dev(u)), ptr(F), ptr(coef),
                               ctypes.c_void_p(scal.ctypes.data)) == 0
    p.close()
    return F.cpu().numpy(), coef.cpu().numpy(), scal, c.cpu().numpy()


# 1, 1, 2, 6, 144 tiles; 384 and 576; 1024 and 1536
@pytest.mark.parametrize("N,M", [(8, 16), (12, 24), (24, 48), (96, 64), (384, 384), (512, 768),
                                 (768, 768), (1024, 1024), (1536, 1024)])
@pytest.mark.parametrize("broken", [False, True])
def test_pairs_against_fp64(ot, N, M, broken):
    f, g = I.blob_density(N, M, 31), I.blob_density(N, M, 32)
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    u = 1e-3 * (np.cos(2 * np.pi * (x + y)) + np.sin(2 * np.pi * (2 * x - y)))
    if broken:
        u[N - 1, M // 3] = np.nan
        u[N // 3, 0] = np.inf
    F, coef, s, _ = evaluate(ot, "mixed", f, g, u)
    R, cref, r, c = evaluate(ot, "fp64", f, g, u)
    assert s[4] == r[4] and (s[4] > 0) == broken
    ok = np.isfinite(R)
    assert np.array_equal(np.isfinite(F), ok)
    if broken:
        assert not ok.all()
        return
    d = np.abs(f - F).max()  # f_n
    big = 62.0 / 12.0 * (M * M + N * N) * np.abs(u).max() * max(d, 1.0)
    assert np.abs(F - R).max() <= 2.0 ** -44 * max(big, 1.0)
    assert abs(s[1] - r[1]) <= 2.0 ** -43 * max(big, 1.0)
    assert abs(s[0] - r[0]) <= 2.0 ** -44 * max(big, 1.0)
    assert abs(s[3] - r[3]) <= 2.0 ** -44 * max(big, 1.0)
    for k in range(5):
        if k < 3:
            bound = 2.0 ** -20 * np.abs(cref[k]).max()
        else:  # det <= 1 + 2 |D^2 u| + ..: below 2 for this u
            bound = 8 * 2.0 ** -24 * np.abs(c).max() * 2.0 * (M if k == 3 else N)
        assert np.abs(coef[k] - cref[k]).max() <= bound
        assert abs(s[5 + k] - r[5 + k]) <= bound
