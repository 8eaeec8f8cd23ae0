"""GPU tests of the pair passes (two rows or columns side by side) over every length they take:
powers of two and three times them, single problems (operator, theta, the fused update) and
batched launches (a plan set against single-problem solves).

Bounds: the operator as the other FP32 variants (5e-6 of the scale, 2e-6 in the 2-norm); theta by
the solve's residual, which a wrong theta would not bring below the tolerance; solves by the root
(two roots with max|F| < tol are within ||J^-1|| 2 tol, 1e-6 as the other mixed solves)."""
import numpy as np
import pytest

import oracle as O
import ot_inputs as I
from gpu_util import dev, hptr, ptr

pytestmark = pytest.mark.gpu
PAIRS = 63 + 256 + 512 + 1024  # every pass on pairs where the size allows it


@pytest.fixture(scope="module")
def ot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1009_6039_gb300 as m
    return m


# (columns, 2 x rows): every column length and every row length once, with the shortest and
# longest counterparts
@pytest.mark.parametrize("N,M", [(96, 128), (128, 192), (192, 256), (256, 384), (384, 512),
                                 (512, 768), (768, 1024), (1024, 1536), (1536, 64), (2048, 16),
                                 (8, 2048), (12, 1536), (96, 16)])
def test_operator_on_pairs(ot, N, M):
    rng = np.random.default_rng(N + 7 * M)
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    u = 1e-3 * (np.cos(2 * np.pi * (x + y)) + np.sin(2 * np.pi * (2 * x - y)))
    _, coef, _ = O.residual(I.blob_density(N, M, 31), O.bspline_coeffs(I.blob_density(N, M, 32)), u)
    abar = np.array([O.simpson_mean(coef[q]) for q in range(5)])
    sigma = rng.standard_normal((N, M))
    w_ref = O.apply_op(coef, abar, sigma)
    p = ot.Plan(N, M, precision="mixed", fft_variant=PAIRS)
    wd = dev(np.zeros((N, M)))
    assert ot.ot_apply_operator(p.h, ptr(dev(coef)), hptr(abar), ptr(dev(sigma)), ptr(wd)) == 0
    w = wd.cpu().numpy()
    assert np.abs(w - w_ref).max() <= 5e-6 * np.abs(w_ref).max()
    assert np.linalg.norm(w - w_ref) <= 2e-6 * np.linalg.norm(w_ref)
    p.close()


# theta's double-float passes and the warm start's Poisson solve, bit for bit the scalar kernels'
# arithmetic after the FP32 forward transform: P(src) against the oracle's at the double-float
# bound of the forward transform (FP32, 2e-6 of the scale)
@pytest.mark.parametrize("N,M", [(96, 128), (128, 192), (192, 256), (384, 384), (768, 768),
                                 (1536, 64)])
@pytest.mark.parametrize("lowpass", [False, True])
def test_poisson_on_pairs(ot, N, M, lowpass):
    rng = np.random.default_rng(N * 3 + M)
    src = rng.standard_normal((N, M))
    src -= src.mean()
    p = ot.Plan(N, M, precision="mixed")
    u = dev(np.zeros((N, M)))
    p.ws_poisson(dev(src), u, lowpass=lowpass)
    ref = O.fd_poisson(src, lowpass=lowpass)
    assert np.abs(u.cpu().numpy() - ref).max() <= 2e-6 * np.abs(ref).max()
    p.close()


@pytest.mark.parametrize("N,M", [(96, 192), (192, 192), (384, 384), (128, 128), (192, 256)])
def test_solves_on_pairs_fused_and_batched(ot, N, M):
    import torch
    f, g = I.noise_blob_pair(N, M, s=3711)
    opts = dict(tau=1.0, tol=1e-8, eta=1e-2, symbols=1)
    ref = ot.Plan(N, M, **opts)  # FP64
    u = torch.zeros((N, M), dtype=torch.float64, device="cuda")
    rc, st = ref.solve(dev(f), dev(g), u)
    assert rc == 0
    ref.close()
    out = []
    for fused in (1, 0):
        p = ot.Plan(N, M, precision="mixed", fft_variant=PAIRS, fused_update=fused, **opts)
        phi = torch.zeros_like(u)
        rc, st = p.solve(dev(f), dev(g), phi)
        assert rc == 0 and st["res_inf"] < 1e-8
        assert float((phi - u).abs().max()) <= 1e-6
        out.append(phi)
        p.close()
    assert torch.equal(out[0], out[1])  # fused and separate launches agree bit for bit
    # the same pair twice in a set, next to one of another size (a generic-kernel size)
    f2, g2 = I.noise_blob_pair(48, 40 + 8, s=3712)
    ps = ot.PlanSet([(N, M), (48, 48), (N, M)], **{k: v for k, v in opts.items()})
    phis = [torch.zeros_like(u), torch.zeros((48, 48), dtype=torch.float64, device="cuda"),
            torch.zeros_like(u)]
    rc, sts = ps.solve([dev(f), dev(f2), dev(f)], [dev(g), dev(g2), dev(g)], phis)
    assert rc == 0 and all(s["res_inf"] < 1e-8 for s in sts)
    assert torch.equal(phis[0], phis[2])
    assert float((phis[0] - u).abs().max()) <= 1e-6
    ps.close()


@pytest.mark.parametrize("N,M", [(96, 768), (128, 1024), (192, 768), (256, 1024), (384, 768),
                                 (512, 768), (768, 768), (1024, 768)])
def test_two_column_pairs_per_block(ot, N, M):
    # more than 152 column pairs: blocks of two (the same bounds)
    test_operator_on_pairs(ot, N, M)
    test_poisson_on_pairs(ot, N, M, False)
