"""GPU tests of the FP64 spectral passes (csrc/spectral_f64.cu) at the sizes where their launch
forms change: the smallest lengths, several rows per block, five or three transforms side by
side and one after the other, lengths with a factor 3 whose first stage leaves threads idle, and
the longest rows and columns.

Bounds: the passes are FP64 transforms with the spectral multiplies; 1e-12 of the result's
scale, the bound of the other FP64 operator tests (a few hundred ulps: ~20 butterfly levels over
the forward and inverse transforms, each within a few ulps of the data's scale, times the
growth of the symbols)."""
import numpy as np
import pytest

import oracle as O
import ot_inputs as I
from gpu_util import dev, hptr, pack_spectrum, ptr, unpack_spectrum

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


@pytest.mark.parametrize("N,M", [(8, 16), (8, 24), (12, 16), (2048, 64), (2048, 16), (16, 2048),
                                 (48, 1536), (1536, 24), (96, 192), (512, 256), (1024, 512)])
def test_fp64_operator_theta_and_transforms(ot, N, M):
    rng = np.random.default_rng(100 * N + M)
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    u = 1e-3 * (np.cos(2 * np.pi * (x + y)) + np.sin(2 * np.pi * (2 * x - y)))
    _, coef, _ = O.residual(I.blob_density(N, M, 31), O.bspline_coeffs(I.blob_density(N, M, 32)), u)
    abar = np.array([O.simpson_mean(coef[q]) for q in range(5)])
    sigma = rng.standard_normal((N, M))
    w_ref, th_ref = O.apply_op(coef, abar, sigma), O.apply_lbar_inv(abar, sigma)
    half_ref = O.fft2(sigma)[:, :M // 2 + 1]
    p = ot.Plan(N, M)
    cd, sd = dev(coef), dev(sigma)
    wd, td, zd, bd = (dev(np.zeros((N, M))) for _ in range(4))
    assert ot.ot_apply_operator(p.h, ptr(cd), hptr(abar), ptr(sd), ptr(wd)) == 0
    assert ot.ot_apply_lbar_inverse(p.h, hptr(abar), ptr(sd), ptr(td)) == 0
    assert ot.ot_fft_forward(p.h, ptr(sd), ptr(zd)) == 0
    assert ot.ot_fft_inverse(p.h, ptr(dev(pack_spectrum(half_ref, N, M))), ptr(bd)) == 0
    for got, ref in ((wd.cpu().numpy(), w_ref), (td.cpu().numpy(), th_ref),
                     (unpack_spectrum(zd.cpu().numpy(), N, M), half_ref),
                     (bd.cpu().numpy() / (N * M), sigma)):
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
    p.close()
