"""GPU tests of the chunked B-spline prefilter (csrc/prefilter.cu): lengths below and above its
64-point tile and 32-point halo (periods that wrap into the halo several times), lengths that are
not multiples of the 8-point chunk, ragged groups of lines, FP64 and double-float.

Bound: 1e-13 as the other prefilter test (|c| ~ 1.5; FP64 recursions or unit round-off 2^-48 with
three roundings per step, damped by 0.27)."""
import numpy as np
import pytest

import oracle as O
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


@pytest.mark.parametrize("N,M", [(8, 16), (12, 24), (24, 2048), (48, 96), (64, 64), (96, 192),
                                 (2048, 16), (384, 768)])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_prefilter_lengths(ot, N, M, prec):
    rng = np.random.default_rng(N + M)
    g = 1 + 0.5 * rng.random((N, M))
    g[0, 0] = g[-1, -1] = 3.0  # corners: what the periodic halo carries
    p = ot.Plan(N, M, precision=prec)
    c = dev(np.zeros((N, M)))
    assert ot.ot_prefilter(p.h, ptr(dev(g)), ptr(c)) == 0
    assert np.abs(c.cpu().numpy() - O.bspline_coeffs(g)).max() <= 1e-13
    both = dev(g)  # in place
    assert ot.ot_prefilter(p.h, ptr(both), ptr(both)) == 0
    assert (both == c).all()
    p.close()
