"""Double-float planes at the ends of the FP64 range: the integer splitting of the wire format.

The transport outputs (and a mixed plan's prefilter) read FP64 planes as (hi, lo) float pairs.  The pair holds
the value to 2^-48 relative to it wherever both parts are normal floats, and whatever the plane
holds beyond (zeros of either sign, denormals, infinities, NaN) takes the conversion
instructions.
"""

import numpy as np
import pytest

from gpu_util import dev

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


@pytest.mark.parametrize("scale", [2.0 ** -40, 2.0 ** -20, 1.0, 2.0 ** 40, 2.0 ** 100])
def test_transport_divergence_scales_exactly(ot, scale):
    # div = D_xx phi + D_yy phi is linear: a power of two on phi is a power of two on div, as long
    # as no product leaves the normal range of a float (the stencils' factors are below 2^20)
    N, M = 64, 96
    rng = np.random.default_rng(5)
    phi = rng.standard_normal((N, M))
    phi[3, 5] = 0.0
    phi[7, 9] = -0.0
    # mantissas that end on a tie of the high part, and one bit to each side of it
    phi[11, 13] = 1.0 + 2.0 ** -24
    phi[11, 14] = 1.0 + 2.0 ** -24 + 2.0 ** -52
    phi[11, 15] = -(1.0 + 2.0 ** -24 - 2.0 ** -52)
    f = np.ones((N, M))
    p = ot.Plan(N, M, precision="mixed")
    out = []
    for s in (1.0, scale):
        div = dev(np.zeros((N, M)))
        p.transport_outputs(dev(f), dev(phi * s), div)
        out.append(div.cpu().numpy())
    p.close()
    assert np.array_equal(out[1], out[0] * scale)
    # against FP64 stencils: 2^-44 of the largest term covers the pair's 2^-48 per operation
    w = np.array([-1, 16, -30, 16, -1]) / 12.0
    ref = sum(w[k + 2] * (M * M * np.roll(phi, -k, 1) + N * N * np.roll(phi, -k, 0))
              for k in range(-2, 3))
    big = np.abs(phi).max() * 62.0 / 12.0 * (M * M + N * N)
    assert np.abs(out[0] - ref).max() <= 2.0 ** -44 * big


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 1e300])
def test_transport_keeps_values_beyond_floats(ot, value):
    # no finite pair holds these: the points whose stencils read them are not finite, all others
    # are untouched
    N, M = 32, 64
    phi = np.zeros((N, M))
    phi[10, 20] = value
    p = ot.Plan(N, M, precision="mixed")
    div = dev(np.zeros((N, M)))
    p.transport_outputs(dev(np.ones((N, M))), dev(phi), div)
    d = div.cpu().numpy()
    p.close()
    hit = np.zeros((N, M), bool)
    hit[8:13, 20] = True
    hit[10, 18:23] = True
    assert not np.isfinite(d[hit]).any()
    assert (d[~hit] == 0.0).all()
