"""The work that is timed: what programs have this library do, through its public entry
points, from the smallest calls to the largest.

A case is a dict with its "kind" and sizes.  The kinds:

  solve        ot.Plan.solve: one optimal-transport problem, FP64 or mixed precision
  set          ot.PlanSet.solve: many problems of uneven sizes in one call
  residual     ot_eval_residual (FP64): residual and linearised coefficients of an iterate
  noalloc      ot_eval_residual_noalloc: the same without a plan, any size of 8..2048
  operator     ot_apply_operator (FP64): the preconditioned product L Lbar^{-1} sigma
  fft          ot_fft_forward and ot_fft_inverse (FP64): the 2-D real transform both ways
  transport    ot.Plan.transport_outputs: distance and divergence of a computed map
  features     ot.Plan.ws_features (mixed): a pair's training rows of the learned start
  network      ot.Plan.ws_mlp_forward: the learned start's network on rows
  grad         ot.Trainer.grad: loss and gradient of one training minibatch
"""
import ctypes
import math

import numpy as np
import torch

import paper_1009_6039_gb300 as ot

DEV = "cuda"
F8 = torch.float64
TWO_PI = 2.0 * math.pi
K, H = 16, 128  # the network's inputs and hidden units
N_WEIGHTS = H * K + 2 * H * H + H


def listed():
    return [
        # one small problem in the plan's default precision: interactive use and the tests'
        # sizes; launches and latency count
        {"name": "solve_64_fp64", "kind": "solve", "N": 64, "M": 64, "precision": "fp64"},
        # the library's main workload: one image-sized pair in mixed precision
        {"name": "solve_1024_mixed", "kind": "solve", "N": 1024, "M": 1024,
         "precision": "mixed"},
        # a batch of image pairs of uneven sizes, each the size that its source happens to have
        {"name": "set_24_uneven", "kind": "set",
         "sizes": "128,384,192,512,256,192,128,512,384,256,192,512,128,256,384,256,512,128,"
                  "192,384,512,128,256,192"},
        # one residual evaluation of a program that runs its own outer iteration
        {"name": "residual_1024", "kind": "residual", "N": 1024, "M": 1024},
        # the same from a program whose memory is all its own, on an odd-shaped grid
        {"name": "noalloc_250x333", "kind": "noalloc", "N": 250, "M": 333},
        # one operator product of such a program's own Krylov method, with a factor 3 in both
        # transform lengths
        {"name": "operator_384x768", "kind": "operator", "N": 384, "M": 768},
        # the transforms alone, at the largest size that the library takes
        {"name": "fft_2048", "kind": "fft", "N": 2048, "M": 2048},
        # what is read off a computed map: transport distance and divergence
        {"name": "transport_512x1024", "kind": "transport", "N": 512, "M": 1024},
        # training rows of the learned start, one per grid point of a solved pair
        {"name": "features_512", "kind": "features", "N": 512, "M": 512},
        # the network over all grid points of a 1024 x 1024 problem
        {"name": "network_1M", "kind": "network", "rows": 1048576},
        # a training minibatch as the benchmark's network takes it, and a small one
        {"name": "grad_32768", "kind": "grad", "batch": 32768},
        {"name": "grad_1024", "kind": "grad", "batch": 1024},
    ]


def _length(rng, lo, hi):
    """A supported transform length 2^a or 3 * 2^a of [lo, hi], even in its logarithm."""
    ok = sorted(v for a in range(1, 12) for v in (1 << a, 3 << a) if lo <= v <= hi)
    return rng.choice(ok)


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "set", "residual", "noalloc", "operator", "fft",
                       "transport", "features", "network", "grad"])
    c = {"kind": kind}
    if kind == "solve":
        c["precision"] = rng.choice(["fp64", "mixed"])
        lo, hi = (32, 128) if c["precision"] == "fp64" else (128, 1024)
        c["N"], c["M"] = _length(rng, lo, hi), _length(rng, lo, hi)
        # the densities' blobs and noise are made for grids that are not far from square
        while not c["N"] / 2 <= c["M"] <= 2 * c["N"]:
            c["M"] = _length(rng, lo, hi)
    elif kind == "set":
        n = rng.randint(3, 24)
        c["sizes"] = ",".join(str(rng.choice([128, 192, 256, 384, 512])) for _ in range(n))
    elif kind == "noalloc":
        c["N"], c["M"] = _log_int(rng, 16, 1024), _log_int(rng, 16, 1024)
    elif kind in ("residual", "transport", "operator"):
        c["N"], c["M"] = _length(rng, 32, 1024), _length(rng, 32, 1024)
    elif kind == "fft":
        c["N"], c["M"] = _length(rng, 32, 2048), _length(rng, 32, 2048)
    elif kind == "features":
        c["N"], c["M"] = _length(rng, 64, 512), _length(rng, 64, 512)
    elif kind == "network":
        c["rows"] = _log_int(rng, 1000, 1048576)
    else:
        c["batch"] = 64 * _log_int(rng, 1, 512)
    return c


# ---- inputs ------------------------------------------------------------------------------
def _grids(N, M):
    y = torch.arange(N, dtype=F8, device=DEV) / N
    x = torch.arange(M, dtype=F8, device=DEV) / M
    return y, x


def _blobs(N, M, rng, count):
    """Sum of `count` periodic Gaussians: widths 0.03 to 0.12, weights 0.5 to 2."""
    y, x = _grids(N, M)
    out = torch.zeros(N, M, dtype=F8, device=DEV)
    for _ in range(count):
        cx, cy, s, w = rng.random_sample(4)
        s = 2.0 * (0.03 + 0.09 * s) ** 2
        gx = sum(torch.exp(-((x - cx + p) ** 2) / s) for p in (-1, 0, 1))
        gy = sum(torch.exp(-((y - cy + p) ** 2) / s) for p in (-1, 0, 1))
        out += (0.5 + 1.5 * w) * gy[:, None] * gx[None, :]
    return out


def _blob_density(N, M, seed):
    """Smooth image-like density, mean 1 (the batched workload's blobs on a floor)."""
    d = 0.25 + _blobs(N, M, np.random.RandomState(seed % 2 ** 32), 8)
    return d / d.mean()


def _noise_density(N, M, seed):
    """Smoothed noise (8 pixels) plus 16 blobs, max / min = 10, mean 1: the main workload."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    z = torch.rand(N, M, dtype=F8, device=DEV, generator=gen)
    k2 = torch.fft.fftfreq(N, dtype=F8, device=DEV)[:, None]
    k1 = torch.fft.rfftfreq(M, dtype=F8, device=DEV)[None, :]
    z = torch.fft.irfft2(torch.fft.rfft2(z) * torch.exp(-2 * math.pi ** 2 * 64 *
                                                        (k2 ** 2 + k1 ** 2)), s=(N, M))
    z = (z - z.min()) / (z.max() - z.min())
    v = z + 0.5 * _blobs(N, M, np.random.RandomState(seed % 2 ** 32), 16)
    d = 1.0 + 9.0 * (v - v.min()) / (v.max() - v.min())
    return (d / d.mean()).contiguous()


def _pair(case, seed):
    make = _noise_density if case["kind"] == "solve" else _blob_density
    return (make(case["N"], case["M"], 2 * seed + 1), make(case["N"], case["M"], 2 * seed + 2))


def _set_pairs(case, seed):
    sizes = [int(s) for s in case["sizes"].split(",")]
    return [(_blob_density(n, n, 100 * seed + 2 * k), _blob_density(n, n, 100 * seed + 2 * k + 1))
            for k, n in enumerate(sizes)]


def _stencil_symbol(L, n, dtype=F8):
    """(first, second) derivative symbols of the 4th-order stencils at indices 0..n-1."""
    t = TWO_PI * torch.arange(n, dtype=dtype, device=DEV) / L
    s1 = (8 * torch.sin(t) - torch.sin(2 * t)) * L / 6
    s2 = (-2 * torch.cos(2 * t) + 32 * torch.cos(t) - 30) * L * L / 12
    return s1, s2


def _poisson(src):
    """Mean-zero inverse of the 4th-order stencil Laplacian."""
    N, M = src.shape
    lam = _stencil_symbol(N, N)[1][:, None] + _stencil_symbol(M, M // 2 + 1)[1][None, :]
    lam[0, 0] = 1.0
    s = torch.fft.rfft2(src) / lam
    s[0, 0] = 0.0
    return torch.fft.irfft2(s, s=(N, M)).contiguous()


def _spline(g):
    """Coefficients of the periodic cubic B-spline interpolant."""
    N, M = g.shape
    ey = (4 + 2 * torch.cos(TWO_PI * torch.arange(N, dtype=F8, device=DEV) / N)) / 6
    ex = (4 + 2 * torch.cos(TWO_PI * torch.arange(M // 2 + 1, dtype=F8, device=DEV) / M)) / 6
    s = torch.fft.rfft2(g) / (ey[:, None] * ex[None, :])
    return torch.fft.irfft2(s, s=(N, M)).contiguous()


def _iterate(case, seed):
    """(f, spline coefficients of g, u): a problem at an iterate of the solver's kind, half
    the linearised potential."""
    f, g = _pair(case, seed)
    return f, _spline(g), 0.5 * _poisson(torch.log(f) - torch.log(g))


def _operator_inputs(case, seed):
    """(coefficient planes, their averages on the host, sigma) of a Newton step."""
    F, coef, scal, _ = _linearise(*_iterate(case, seed))
    return coef.contiguous(), np.ascontiguousarray(scal[5:].cpu().numpy()), F.contiguous()


def _weights(rng):
    """Network parameters at the size of a trained network's."""
    parts = []
    for o, i in ((H, K), (H, H), (H, H)):
        parts += [rng.uniform(-1, 1, o * i) * 1.5 / math.sqrt(i), 0.1 * rng.standard_normal(o)]
    parts += [rng.uniform(-1, 1, H) / math.sqrt(H), 0.1 * rng.standard_normal(1)]
    return np.concatenate(parts).astype(np.float32)


def _rows(n, seed):
    """Feature rows as the solver makes them: O(1) values, the last one zero."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    X = torch.randn(n, K, device=DEV, generator=gen)
    X[:, 15] = 0.0
    t = torch.sin(X[:, 0]) * X[:, 1] + 0.3 * X[:, 2]
    return X, t.contiguous()


def _p(t):
    return ctypes.c_void_p(t.data_ptr())


def _hp(a):
    return ctypes.c_void_p(a.ctypes.data)


def prepare(case, seed):
    kind, s = case["kind"], {"kind": case["kind"]}
    new = lambda *shape: torch.empty(shape, dtype=F8, device=DEV)  # noqa: E731
    if kind == "solve":
        s["f"], s["g"] = _pair(case, seed)
        s["phi"] = torch.zeros_like(s["f"])
        # the main workload's settings
        s["plan"] = ot.Plan(case["N"], case["M"], tau=1.0, tol=1e-8, eta=1e-2, symbols=1,
                            precision=case["precision"])
    elif kind == "set":
        pairs = _set_pairs(case, seed)
        s["f"], s["g"] = [p[0] for p in pairs], [p[1] for p in pairs]
        s["phi"] = [torch.zeros_like(f) for f in s["f"]]
        # the batched workload's settings with the main workload's inner tolerance
        s["set"] = ot.PlanSet([tuple(f.shape) for f in s["f"]], tau=1.0, tol=1e-8, eta=1e-2,
                              symbols=1, max_newton=1000, tau_retry=2)
    elif kind in ("residual", "noalloc"):
        N, M = case["N"], case["M"]
        s["f"], s["c"], s["u"] = _iterate(case, seed)
        s["F"], s["coef"], s["scal"] = new(N, M), new(5, N, M), np.zeros(10)
        if kind == "residual":
            s["plan"] = ot.Plan(N, M)
    elif kind == "operator":
        s["coef"], s["abar"], s["sigma"] = _operator_inputs(case, seed)
        s["w"] = new(case["N"], case["M"])
        s["plan"] = ot.Plan(case["N"], case["M"])
    elif kind == "fft":
        s["x"], y = _pair(case, seed)
        s["z"] = _packed(torch.fft.fft2(y))
        s["X"], s["y"] = new(case["N"], case["M"]), new(case["N"], case["M"])
        s["plan"] = ot.Plan(case["N"], case["M"])
    elif kind == "transport":
        s["f"], _, s["u"] = _iterate(case, seed)
        s["div"] = new(case["N"], case["M"])
        s["plan"] = ot.Plan(case["N"], case["M"])
    elif kind == "features":
        s["f"], s["g"], s["phi"] = _solved(case, seed)
        n = case["N"] * case["M"]
        s["X"] = torch.empty(n, K, dtype=torch.float32, device=DEV)
        s["t"] = torch.empty(n, dtype=torch.float32, device=DEV)
        s["plan"] = ot.Plan(case["N"], case["M"], precision="mixed")
    elif kind == "network":
        s["X"] = _rows(case["rows"], seed)[0]
        s["out"] = torch.empty(case["rows"], dtype=torch.float32, device=DEV)
        s["plan"] = ot.Plan(32, 32, precision="mixed").set_weights(
            _weights(np.random.RandomState(seed % 2 ** 32)))
    else:
        s.update(_minibatch(case, seed))
        s["trainer"] = ot.Trainer(case["batch"], s["params"])
    return s


def _solved(case, seed):
    """(f, g, phi): a pair and a potential near its solution."""
    f, g = _blob_density(case["N"], case["M"], 2 * seed + 1), _blob_density(
        case["N"], case["M"], 2 * seed + 2)
    h = _poisson(torch.log(f) - torch.log(g))
    return f, g, 0.9 * h + 0.02 * _poisson(f - g)


def _minibatch(case, seed):
    """A training set of four minibatches, row indices of one and the current parameters."""
    n = 4 * case["batch"]
    X, t = _rows(n, seed)
    gen = torch.Generator(device=DEV).manual_seed(seed + 1)
    idx = torch.randint(0, n, (case["batch"],), device=DEV, generator=gen)
    return {"X": X, "t": t, "idx": idx,
            "params": _weights(np.random.RandomState(seed % 2 ** 32))}


# ---- one pass ----------------------------------------------------------------------------
def _ok(rc):
    if rc != ot.OT_OK:
        raise RuntimeError(ot.ot_strerror(rc))


def run(s):
    kind = s["kind"]
    if kind == "solve":
        s["plan"].solve(s["f"], s["g"], s["phi"])
        return s["phi"]
    if kind == "set":
        s["set"].solve(s["f"], s["g"], s["phi"])
        return s["phi"]
    if kind == "residual":
        _ok(ot.ot_eval_residual(s["plan"].h, _p(s["f"]), _p(s["c"]), _p(s["u"]), _p(s["F"]),
                                _p(s["coef"]), _hp(s["scal"])))
        return s["F"], s["coef"], s["scal"]
    if kind == "noalloc":
        N, M = s["f"].shape
        _ok(ot.ot_eval_residual_noalloc(N, M, _p(s["f"]), _p(s["c"]), _p(s["u"]), _p(s["F"]),
                                        _p(s["coef"]), _hp(s["scal"])))
        return s["F"], s["coef"], s["scal"]
    if kind == "operator":
        _ok(ot.ot_apply_operator(s["plan"].h, _p(s["coef"]), _hp(s["abar"]), _p(s["sigma"]),
                                 _p(s["w"])))
        return s["w"]
    if kind == "fft":
        _ok(ot.ot_fft_forward(s["plan"].h, _p(s["x"]), _p(s["X"])))
        _ok(ot.ot_fft_inverse(s["plan"].h, _p(s["z"]), _p(s["y"])))
        return s["X"], s["y"]
    if kind == "transport":
        return s["plan"].transport_outputs(s["f"], s["u"], s["div"]), s["div"]
    if kind == "features":
        s["plan"].ws_features(s["f"], s["g"], s["X"], s["t"], phi_star=s["phi"])
        return s["X"], s["t"]
    if kind == "network":
        s["plan"].ws_mlp_forward(s["X"], s["out"])
        return s["out"]
    loss, grad = s["trainer"].grad(s["X"], s["t"], s["idx"])
    return np.float32(loss), grad  # the trainer computes in FP32


def work(case):
    kind = case["kind"]
    if kind == "network":
        return {"bytes": 68 * case["rows"], "flops": 2 * N_WEIGHTS * case["rows"]}
    if kind == "grad":
        # rows, targets and indices in, parameters in, gradient out; forward, data gradients
        # of the upper layers and weight gradients
        B = case["batch"]
        return {"bytes": 76 * B + 8 * (N_WEIGHTS + 3 * H + 1),
                "flops": (6 * N_WEIGHTS - 2 * H * K) * B}
    if kind == "set":
        return {k: sum(_solve_work(n, n, 9, 100)[k] for n in map(int, case["sizes"].split(",")))
                for k in ("bytes", "flops")}
    N, M = case["N"], case["M"]
    P, lN, lM = N * M, math.log2(N), math.log2(M)
    if kind == "solve":
        # Newton steps and Krylov steps as such pairs take them
        return _solve_work(N, M, *((11, 80) if case["precision"] == "mixed" else (7, 50)))
    if kind in ("residual", "noalloc"):
        return {"bytes": 72 * P, "flops": 190 * P}
    if kind == "operator":
        return {"bytes": 56 * P, "flops": _operator_flops(P, lN, lM)}
    if kind == "fft":
        return {"bytes": 32 * P, "flops": 5 * P * (lN + lM)}
    if kind == "transport":
        return {"bytes": 24 * P, "flops": 60 * P}
    return {"bytes": 92 * P, "flops": 5 * P * (lN + lM) + 260 * P}  # features


def _operator_flops(P, lN, lM):
    # one forward transform, three inverse column transforms, five inverse row transforms,
    # the symbols and the coefficients
    return P * (2.5 * (lN + lM) + 3 * 2.5 * lN + 5 * 2.5 * lM + 30)


def _solve_work(N, M, newton, krylov):
    P, lN, lM = N * M, math.log2(N), math.log2(M)
    return {"bytes": 24 * P,
            "flops": krylov * (_operator_flops(P, lN, lM) + 24 * P) + newton * 190 * P}


# ---- the same in 64 bits, in plain torch ---------------------------------------------------
def _packed(z):
    """The library's packed half spectrum of a full 2-D transform (N x M, (re, im) pairs):
    column 0 holds A + i B, A and B the transforms of the real row coefficients k1 = 0, M/2."""
    M = z.shape[1]
    h = z[:, :M // 2].clone()
    h[:, 0] = z[:, 0] + 1j * z[:, M // 2]
    return torch.view_as_real(h).reshape(z.shape[0], M).contiguous()


def _d1(u, ax):
    r = lambda k: torch.roll(u, -k, ax)  # noqa: E731
    return (r(-2) - 8 * r(-1) + 8 * r(1) - r(2)) * u.shape[ax] / 12


def _d2(u, ax):
    r = lambda k: torch.roll(u, -k, ax)  # noqa: E731
    return (-r(-2) + 16 * r(-1) - 30 * u + 16 * r(1) - r(2)) * u.shape[ax] ** 2 / 12


def _sample(c, x, y):
    """Value and gradient of the spline interpolant at grid positions (x, y)."""
    N, M = c.shape

    def weights(t):
        w = [(1 - t) ** 3 / 6, (3 * t ** 3 - 6 * t ** 2 + 4) / 6,
             (-3 * t ** 3 + 3 * t ** 2 + 3 * t + 1) / 6, t ** 3 / 6]
        d = [-(1 - t) ** 2 / 2, (3 * t * t - 4 * t) / 2, (-3 * t * t + 2 * t + 1) / 2, t * t / 2]
        return w, d

    j0, i0 = torch.floor(x), torch.floor(y)
    (wx, dx), (wy, dy) = weights(x - j0), weights(y - i0)
    j0, i0 = j0.long(), i0.long()
    v, gx, gy = (torch.zeros_like(x) for _ in range(3))
    for b in range(4):
        row = torch.remainder(i0 + b - 1, N) * M
        for a in range(4):
            cv = c.reshape(-1)[row + torch.remainder(j0 + a - 1, M)]
            v += cv * wx[a] * wy[b]
            gx += cv * dx[a] * wy[b]
            gy += cv * wx[a] * dy[b]
    return v, gx * M, gy * N


def _positions(u):
    N, M = u.shape
    i = torch.arange(N, dtype=F8, device=DEV)[:, None]
    j = torch.arange(M, dtype=F8, device=DEV)[None, :]
    ux, uy = _d1(u, 1), _d1(u, 0)
    return ux, uy, j + M * ux, i + N * uy


def _linearise(f, c, u):
    """(F, coefficient planes, the 10 scalars, min det) at the iterate u."""
    N, M = u.shape
    ux, uy, x, y = _positions(u)
    uxx, uyy, uxy = _d2(u, 1), _d2(u, 0), _d1(ux, 0)
    G, gx, gy = _sample(c, x, y)
    det = (1 + uxx) * (1 + uyy) - uxy * uxy
    fn = G * det
    F = f - (fn - fn.mean() + 1)
    coef = torch.stack([G * (1 + uyy), -G * uxy, G * (1 + uxx), det * gx, det * gy])
    wy = (2.0 + 2.0 * (torch.arange(N, device=DEV) % 2).to(F8)) / (3 * N)
    wx = (2.0 + 2.0 * (torch.arange(M, device=DEV) % 2).to(F8)) / (3 * M)
    avg = (coef * (wy[:, None] * wx[None, :])).sum((1, 2))
    scal = torch.stack([fn.mean(), F.abs().max(), (F * F).mean().sqrt(), det.min(),
                        torch.zeros((), dtype=F8, device=DEV)])
    return F, coef, torch.cat([scal, avg]), det.min()


def _symbols(N, M, stencil):
    if stencil:
        (y1, y2), (x1, x2) = _stencil_symbol(N, N), _stencil_symbol(M, M // 2 + 1)
    else:
        k2 = torch.fft.fftfreq(N, 1.0 / N, dtype=F8, device=DEV)
        k1 = torch.arange(M // 2 + 1, dtype=F8, device=DEV)
        y1, x1 = TWO_PI * k2, TWO_PI * k1
        y2, x2 = -y1 * y1, -x1 * x1
    y1, x1 = y1.clone(), x1.clone()
    y1[N // 2] = 0.0
    x1[M // 2] = 0.0
    return x1[None, :], x2[None, :], y1[:, None], y2[:, None]


def _lbar_inverse(abar, sigma, sym):
    """The spectrum of theta = Lbar^{-1} sigma."""
    x1, x2, y1, y2 = sym
    den = torch.complex(abar[0] * x2 - 2 * abar[1] * x1 * y1 + abar[2] * y2,
                        abar[3] * x1 + abar[4] * y1)
    zero = den == 0
    return torch.where(zero, torch.zeros_like(den), torch.fft.rfft2(sigma) /
                       torch.where(zero, torch.ones_like(den), den))


def _apply(coef, abar, sigma, sym):
    x1, x2, y1, y2 = sym
    th = _lbar_inverse(abar, sigma, sym)
    back = lambda z: torch.fft.irfft2(z, s=sigma.shape)  # noqa: E731
    return (coef[0] * back(x2 * th) - 2 * coef[1] * back(x1 * y1 * th) +
            coef[2] * back(y2 * th) + coef[3] * back(1j * x1 * th) +
            coef[4] * back(1j * y1 * th))


def _gmres(op, b, m=30, tol=1e-6):
    beta = b.norm()
    V, Hm = [(b / beta).reshape(-1)], np.zeros((m + 1, m))
    for j in range(m):
        w = op(V[j].reshape(b.shape)).reshape(-1)
        A = torch.stack(V)
        h = A @ w
        w = w - h @ A
        h2 = A @ w
        w = w - h2 @ A
        Hm[:j + 1, j] = (h + h2).cpu().numpy()
        Hm[j + 1, j] = float(w.norm())
        e = np.zeros(j + 2)
        e[0] = float(beta)
        y, *_ = np.linalg.lstsq(Hm[:j + 2, :j + 1], e, rcond=None)
        if np.linalg.norm(Hm[:j + 2, :j + 1] @ y - e) <= tol * float(beta) or Hm[j + 1, j] == 0:
            break
        V.append(w / w.norm())
    return (torch.stack(V[:len(y)]).T @ torch.from_numpy(y).to(DEV)).reshape(b.shape)


def _root(f, g):
    """The mean-zero potential with F = 0, by Newton's method with halved steps."""
    f, c = f - f.mean() + 1, _spline(g - g.mean() + 1)
    u, sym, step = torch.zeros_like(f), _symbols(*f.shape, stencil=True), 1.0
    F, coef, scal, _ = _linearise(f, c, u)
    for _ in range(100):
        if float(F.abs().max()) < 1e-12:
            break
        abar = scal[5:]
        sigma = _gmres(lambda v: _apply(coef, abar, v, sym), F)
        theta = torch.fft.irfft2(_lbar_inverse(abar, sigma, sym), s=f.shape)
        before = float(F.norm())
        while True:
            cand = u + step * theta
            F, coef, scal, det = _linearise(f, c, cand)
            if float(det) > 0 or step < 1e-6:
                break
            step *= 0.5
        u, step = cand, min(1.0, 2 * step)
        if step == 1.0 and float(F.norm()) > 0.5 * before and float(F.abs().max()) < 1e-10:
            break  # round-off
    return u - u.mean()


def _network(w, X):
    o, layers = 0, []
    for rows, cols in ((H, K), (H, H), (H, H), (1, H)):
        layers.append((w[o:o + rows * cols].reshape(rows, cols),
                       w[o + rows * cols:o + rows * cols + rows]))
        o += rows * cols + rows
    a = X
    for k, (W, b) in enumerate(layers):
        a = a @ W.T + b
        if k < 3:
            a = a * torch.sigmoid(a)
    return a[:, 0]


def _features(f, g, phi):
    f, g = f - f.mean() + 1, g - g.mean() + 1
    h = _poisson(torch.log(f) - torch.log(g))
    hx, hy, x, y = _positions(h)
    hxx, hyy, hxy = _d2(h, 1), _d2(h, 0), _d1(hx, 0)
    G, gx, gy = _sample(_spline(g), x, y)
    Gc = G.clamp(min=1e-3)
    det = ((1 + hxx) * (1 + hyy) - hxy * hxy).clamp(min=1e-3)
    lf, lg = torch.log(f), torch.log(Gc)
    r = lf - lg - torch.log(det)
    X = torch.stack([lf, torch.log(g), lg, r, hxx + hyy, hxx - hyy, 2 * hxy,
                     hxx * hyy - hxy * hxy, 10 * hx, 10 * hy, 0.1 * gx / Gc, 0.1 * gy / Gc,
                     (gx * hx + gy * hy) / Gc, (hxx - hyy) ** 2 + 4 * hxy ** 2,
                     r * (hxx + hyy), torch.zeros_like(r)], -1)
    d = phi - h
    return X.reshape(-1, K), (_d2(d, 1) + _d2(d, 0)).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "solve":
        return _root(*_pair(case, seed))
    if kind == "set":
        pairs = _set_pairs(case, seed)
        return [_root(f, g) for f, g in pairs] if len(pairs) <= 6 else None  # else too long
    if kind in ("residual", "noalloc"):
        F, coef, scal, _ = _linearise(*_iterate(case, seed))
        return F, coef, scal
    if kind == "operator":
        coef, abar, sigma = _operator_inputs(case, seed)
        return _apply(coef, torch.from_numpy(abar).to(DEV), sigma,
                      _symbols(case["N"], case["M"], stencil=False))
    if kind == "fft":
        x, y = _pair(case, seed)
        return _packed(torch.fft.fft2(x)), y * (case["N"] * case["M"])
    if kind == "transport":
        f, _, u = _iterate(case, seed)
        ux, uy = _d1(u, 1), _d1(u, 0)
        return float(((ux * ux + uy * uy) * f).mean()), _d2(u, 1) + _d2(u, 0)
    if kind == "features":
        return _features(*_solved(case, seed))
    if kind == "network":
        w = torch.from_numpy(_weights(np.random.RandomState(seed % 2 ** 32))).to(DEV, F8)
        return _network(w, _rows(case["rows"], seed)[0].to(F8))
    b = _minibatch(case, seed)
    w = torch.from_numpy(b["params"]).to(DEV, F8).requires_grad_(True)
    loss = ((_network(w, b["X"][b["idx"]].to(F8)) - b["t"][b["idx"]].to(F8)) ** 2).mean()
    loss.backward()
    return np.float64(loss.item()), w.grad
