"""GPU tests of the learned start's tiled kernels where they can go wrong: grids smaller than a tile,
tiles of 8 and of 32 rows with ragged edges, feature rows that cannot take 16-byte stores, a target
over the potential, inputs used as given.

Bounds: features and target as against the oracle elsewhere (1e-5 of a feature's largest value; the
two with log det weighted by the clamped det); one path against another bit for bit.  Divergence:
2^-44 of the largest term a stencil can hold (2^-48 per double-float operation)."""
import numpy as np
import pytest

import oracle.warmstart as W
import ot_inputs as I
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


@pytest.mark.parametrize("N,M", [(8, 16), (16, 16), (96, 48), (768, 512)])
def test_feature_rows_by_every_path(ot, N, M):
    import torch
    P = N * M
    f, g = I.blob_pair(N, M, s=21)
    fn, gn = W.normalise(f, g)
    x, y = I.grid(N, M)
    phi = 1e-3 * np.cos(2 * np.pi * x) * np.sin(4 * np.pi * y)
    X_ref, h, _ = W.features(fn, gn)
    t_ref = W.target(phi, h)

    def check(X, t):
        det = np.clip(1.0 + X_ref[:, 4] + X_ref[:, 7], 1e-3, 1.0)
        for k in range(16):
            wk = det if k in (3, 14) else 1.0
            scale = max(np.abs(X_ref[:, k]).max(), 1e-3)
            assert np.max(np.abs(X[:, k] - X_ref[:, k]) * wk) <= 1e-5 * scale, k
        assert np.abs(t - t_ref).max() <= 1e-5 * np.abs(t_ref).max()

    f32 = dict(dtype=torch.float32, device="cuda")
    p = ot.Plan(N, M, precision="mixed")
    X, t = torch.zeros((P, 16), **f32), torch.zeros(P, **f32)
    p.ws_features(dev(f), dev(g), X, t, phi_star=dev(phi))
    X0, t0 = X.cpu().numpy(), t.cpu().numpy()
    check(X0, t0)
    # rows that start 4 bytes off
    flat = torch.zeros(P * 16 + 1, **f32)
    p.ws_features(dev(f), dev(g), flat[1:].view(P, 16), t, phi_star=dev(phi))
    assert np.array_equal(flat[1:].view(P, 16).cpu().numpy(), X0) and float(flat[0]) == 0.0
    # the target over the potential
    d = dev(phi)
    p.ws_features(dev(f), dev(g), X, d.view(torch.float32).view(-1)[:P], phi_star=d)
    assert np.array_equal(d.view(torch.float32).view(-1)[:P].cpu().numpy(), t0)
    p.close()
    # inputs used as given
    p = ot.Plan(N, M, precision="mixed", translate=0)
    p.ws_features(dev(fn), dev(gn), X, t, phi_star=dev(phi))
    check(X.cpu().numpy(), t.cpu().numpy())
    p.close()


@pytest.mark.parametrize("N,M", [(8, 16), (24, 48), (384, 384), (512, 384)])
def test_divergence_tiles(ot, N, M):
    phi = np.random.default_rng(N + M).standard_normal((N, M))
    p = ot.Plan(N, M, precision="mixed")
    div = dev(np.zeros((N, M)))
    p.transport_outputs(dev(np.ones((N, M))), dev(phi), div)
    p.close()
    w = np.array([-1, 16, -30, 16, -1]) / 12.0
    ref = sum(w[k + 2] * (M * M * np.roll(phi, -k, 1) + N * N * np.roll(phi, -k, 0))
              for k in range(-2, 3))
    big = np.abs(phi).max() * 62.0 / 12.0 * (M * M + N * N)
    assert np.abs(div.cpu().numpy() - ref).max() <= 2.0 ** -44 * big
