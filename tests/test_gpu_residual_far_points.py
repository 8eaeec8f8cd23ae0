"""GPU tests of the FP64 residual kernel at finite displacements of more cells than an int holds
(the iterates of a diverging outer iteration): the cell is the displaced position's floor modulo
the period, also for lengths that do not divide a power of two, and the fraction lies in [0, 1).

u is one value U, elsewhere 0, with N^2 / 12 and M^2 / 12 of few binary digits, so that differences
and displacements are exact and the expected position j + M u_x is one rounding away, as in the
kernel.  Bound: the weights (six values below 1, of up to eight roundings), the 16 taps (two roundings
each, all terms below max|c|, a gradient tap below 2 max|c|) and a handful of products after that:
fewer than 100 roundings of the coefficient's largest term, so 1e-13 of it."""
import numpy as np
import pytest

from gpu_util import dev, hptr, ptr

pytestmark = pytest.mark.gpu

N, M = 33, 27  # N^2 / 12 = 90.75, M^2 / 12 = 60.75


@pytest.fixture(scope="module")
def ot():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1009_6039_gb300 as m
    return m


def taps(t):
    """Cubic B-spline weights and their derivatives at t, taps -1 .. 2."""
    s = 1 - t
    return (np.stack([s ** 3, 3 * t ** 3 - 6 * t ** 2 + 4, 3 * s ** 3 - 6 * s ** 2 + 4, t ** 3]) / 6,
            np.stack([-s * s, t * (3 * t - 4), -s * (3 * s - 4), t * t]) / 2)


def cells(x, L):
    """Index floor(x) modulo L (in Python's integers) and fraction."""
    fl = np.floor(x)
    return np.array([int(v) % L for v in fl.flat]).reshape(x.shape), x - fl


def expected(c, u):
    """The coefficient planes and their scales."""
    r = lambda ax, k: np.roll(u, -k, ax)  # noqa: E731
    d1 = lambda ax: -r(ax, 2) + 8 * r(ax, 1) - 8 * r(ax, -1) + r(ax, -2)  # noqa: E731
    d2 = lambda ax: -r(ax, 2) + 16 * r(ax, 1) - 30 * u + 16 * r(ax, -1) - r(ax, -2)  # noqa: E731
    dy = d1(0)
    uxy = (-np.roll(dy, -2, 1) + 8 * np.roll(dy, -1, 1) - 8 * np.roll(dy, 1, 1) +
           np.roll(dy, 2, 1)) * (M * N / 144.0)
    axx, ayy = 1 + d2(1) * (M * M / 12.0), 1 + d2(0) * (N * N / 12.0)
    det = axx * ayy - uxy * uxy
    j, tx = cells(np.arange(M)[None, :] + d1(1) * (M * M / 12.0), M)
    i, ty = cells(np.arange(N)[:, None] + dy * (N * N / 12.0), N)
    (wx, dwx), (wy, dwy) = taps(tx), taps(ty)
    G, gx, gy = np.zeros((3, N, M))
    for b in range(4):
        for a in range(4):
            v = c[(i + b - 1) % N, (j + a - 1) % M]
            G += v * wx[a] * wy[b]
            gx += v * dwx[a] * wy[b] * M
            gy += v * wx[a] * dwy[b] * N
    scale = np.stack([np.abs(ayy), np.abs(uxy), np.abs(axx), 2 * M * np.abs(det),
                      2 * N * np.abs(det)]) * np.abs(c).max()
    return np.stack([G * ayy, -G * uxy, G * axx, det * gx, det * gy]), scale


def coefficients(ot, f, c, u):
    F, coef, scal = dev(np.zeros((N, M))), dev(np.zeros((5, N, M))), np.zeros(10)
    planes = [dev(v) for v in (f, c, u)] + [F, coef]
    rc = ot.ot_eval_residual_noalloc(N, M, *[ptr(v) for v in planes], hptr(scal))
    assert rc == 0
    return coef.cpu().numpy(), scal


# cells beyond 2^31 with a fraction; beyond 2^51, where the position is still a multiple of 1/4;
# beyond 2^53 and 2^63 (whole numbers, M and N do not divide their powers of two)
@pytest.mark.parametrize("U", [2.0 ** 23 + 2.0 ** -4, 2.0 ** 42 + 2.0 ** -8, 2.0 ** 46, 2.0 ** 60])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_cells_beyond_the_range_of_int(ot, U, sign):
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    c = 1 + 0.3 * np.sin(2 * np.pi * (x + 2 * y)) + 0.2 * np.cos(2 * np.pi * (3 * x - y))
    u = np.zeros((N, M))
    u[9, 14] = sign * U
    f = np.ones((N, M))
    got, scal = coefficients(ot, f, c, u)
    want, scale = expected(c, u)
    assert np.isfinite(got).all() and scal[4] == 0
    bad = np.abs(got - want) > 1e-13 * scale
    assert not bad.any(), (np.argwhere(bad)[:5], (np.abs(got - want) / (scale + 1e-300)).max())


# neighbouring doubles are many periods apart: any cell, but the weights stay those of a point
@pytest.mark.parametrize("U", [2.0 ** 120, -2.0 ** 400])
def test_displacements_without_a_cell(ot, U):
    y, x = np.meshgrid(np.arange(N) / N, np.arange(M) / M, indexing="ij")
    c = 1 + 0.3 * np.sin(2 * np.pi * (x + 2 * y))
    u = np.zeros((N, M))
    u[9, 14] = U
    got, scal = coefficients(ot, np.ones((N, M)), c, u)
    scale = expected(c, u)[1]
    assert np.isfinite(got).all() and scal[4] == 0
    assert (np.abs(got) <= (1 + 1e-13) * scale).all()
