"""GPU test of the FP64 transforms' rounding (csrc/spectral_f64.cu) on image-like densities, whose
energy is in the lowest frequencies: a butterfly that takes the rounding of its sum a + w b into the
difference a - w b carries the large entries' rounding into the small ones.

Bound: 1.1 times what radix-8 butterflies with separate products, sums and differences (each rounded
once at its own size) left on the same inputs, summed over them: 3.60e-15 forward, 3.68e-15 inverse.
(The form that takes 2 a - (a + w b) left 4.21e-15 and 4.49e-15.)"""
import numpy as np
import pytest

from gpu_util import dev, ptr

pytestmark = pytest.mark.gpu

if np.finfo(np.longdouble).eps >= np.finfo(np.float64).eps:
    pytest.skip("long double is double here", allow_module_level=True)


def density(N, M, seed):
    rng = np.random.default_rng(seed)
    y, x = np.arange(N)[:, None] / N, np.arange(M)[None, :] / M
    d = np.full((N, M), 0.25)
    for _ in range(8):
        cx, cy, s, w = rng.random(4)
        s = 2 * (0.03 + 0.09 * s) ** 2
        d += (0.5 + 1.5 * w) * sum(np.exp(-(y - cy + p) ** 2 / s) for p in (-1, 0, 1)) * sum(
            np.exp(-(x - cx + p) ** 2 / s) for p in (-1, 0, 1))
    return d / d.mean()


def error(got, want):
    return float(np.sqrt((np.abs(got - want) ** 2).sum() / (np.abs(want) ** 2).sum()))


def packed(h):
    """The library's packed spectrum of a half spectrum: column 0 holds columns 0 and M / 2 as A + i B
    (in h's precision)."""
    z = h[:, :-1].copy()
    z[:, 0] = h[:, 0] + 1j * h[:, -1]
    return z


def unpacked(z):
    h = np.concatenate([z, z[:, :1]], 1)
    m = np.conj(z[-np.arange(len(z)) % len(z), 0])
    h[:, 0], h[:, -1] = (z[:, 0] + m) / 2, (z[:, 0] - m) / 2j
    return h


def test_rounding_of_the_transforms():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_1009_6039_gb300 as ot
    here = np.zeros(2)
    for N, M in ((64, 64), (96, 96), (128, 512), (384, 256), (512, 512)):
        p = ot.Plan(N, M)
        for seed in range(3):
            x = density(N, M, seed)
            want = np.fft.rfft2(x.astype(np.longdouble))
            X, d = dev(np.zeros((N, M))), dev(x)
            assert ot.ot_fft_forward(p.h, ptr(d), ptr(X)) == 0
            here[0] += error(X.cpu().numpy().view(np.complex128), packed(want))
            Z = np.ascontiguousarray(packed(want).astype(np.complex128))
            half = unpacked(Z.astype(np.clongdouble))
            want = np.fft.irfft2(half, s=(N, M)) * (N * M)
            dz, y = dev(Z.view(np.float64)), dev(np.zeros((N, M)))
            assert ot.ot_fft_inverse(p.h, ptr(dz), ptr(y)) == 0
            here[1] += error(y.cpu().numpy(), want)
        p.close()
    assert (here <= 1.1 * np.array([3.60e-15, 3.68e-15])).all(), here
