"""The framework's work as its users have it done, through its public entry points.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare` makes a case's
inputs on the GPU with the context and output buffers a program keeps, `run` is one pass, `work`
its bytes and operations, `exact` its floating results in 64 bits from plain torch.

Every state has a context of its own, all on one stream that is not the legacy default stream, as a
program does that calls again with buffers it keeps.  The launch-shape autotuner is off where the
sums run in split-BF16: a shape it picks by timing sets the pixel ranges the FP32 partial sums run
over, so two runs of one program would differ in their last digits.
"""
import math
import random

import numpy as np
import torch

import paper_2412_02246_gb300 as absm

DEV = "cuda:0"
_streams = []


def _stream():
    if not _streams:
        _streams.append(torch.cuda.Stream(DEV))
    return _streams[0]


# ------------------------------------------------------------------------------- cases


def _estimate(**kw):
    c = {"kind": "estimate", "lo": 46.0, "hi": 1320.0, "log": True, "layout": "array", "u_min": 7.0, "u_max": 220.0,
         "n_time": 1, "n_src": 0, "gridder": "gauss", "sigma": 1.0, "radius": 3, "weights": "mean",
         "precision": "fp32", "n_real": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a tiny grid, where launches and latency count (a test or a teaching run)
        _estimate(name="tiny-fp32", n_grid=64, du=2.0, lo=25.0, hi=375.0, log=False, n_bins=8, n_vis=5000,
                  layout="annulus", u_min=4.0, u_max=60.0),
        # one MWA snapshot set (128 antennas x 120 samples), the paper's own shape, plain FP32
        _estimate(name="mwa-fp32", n_grid=512, du=2.3, n_bins=20, n_vis=8128 * 120, n_time=120),
        # an ensemble over one baseline set with its (l1, mu, t) statistics: the paper's error bars
        _estimate(name="ensemble-16-fp32", kind="ensemble", n_grid=512, du=2.3, n_bins=20, n_vis=8128 * 120,
                  n_time=120, n_real=16),
        # fine bins on a larger grid, split-BF16 sums
        _estimate(name="precision-split", n_grid=2048, du=1.15, n_bins=64, n_vis=4_000_000, precision="split_bf16"),
        # one channel of a wide-band data set at 139 MHz (point sources in the sky, holes in the outer rings)
        _estimate(name="channel-split", n_grid=4096, du=0.6, n_bins=128, n_vis=10_000_000, precision="split_bf16",
                  u_min=7.0 * 139.0 / 154.25, u_max=220.0 * 139.0 / 154.25, n_src=2000),
        # many estimates of uneven size in one call
        {"name": "batch-16-split", "kind": "batch", "items": 16, "shapes": 2412, "precision": "split_bf16"},
        # a multi-frequency cube: every channel gridded, delay bins, voxel sums
        {"name": "cube-32ch-split", "kind": "cube", "n_grid": 512, "du": 2.3, "lo": 46.0, "hi": 1320.0, "n_bins": 20,
         "n_vis": 8128 * 120, "n_time": 120, "n_chan": 32, "tau": "0,1,4,8,16", "precision": "split_bf16"},
        # gridding alone (a program that goes on from the gridded data itself), an odd number of visibilities
        {"name": "grid-1024", "kind": "grid", "n_grid": 1024, "du": 1.15, "n_vis": 1_000_003, "n_time": 1,
         "gridder": "gauss", "sigma": 1.0, "radius": 3},
        # the ring fields alone, from gridded data
        {"name": "fields-1024-fp32", "kind": "fields", "n_grid": 1024, "du": 1.15, "lo": 46.0, "hi": 1320.0,
         "n_bins": 33, "n_fft": 0, "precision": "fp32"},
        # sums and exact counts alone, from a caller's fields, mask and triplet list
        {"name": "triple-512-fp32", "kind": "triple", "n_grid": 512, "du": 2.3, "lo": 46.0, "hi": 1320.0, "n_bins": 24,
         "n_fft": 0, "precision": "fp32", "fill": 0.97},
        # the discretely sampled analytic prediction the estimate is compared with
        {"name": "predict-512", "kind": "predict", "n_grid": 512, "du": 2.3, "lo": 46.0, "hi": 1320.0, "n_bins": 20,
         "n_fft": 0, "precision": "fp32", "fill": 0.97},
        # simulated visibilities of a 256 x 256 map through the MWA tile beam
        {"name": "simulate-256", "kind": "simulate", "m": 256, "dtheta": math.radians(0.029), "n_vis": 100_000,
         "beam": "tile", "beam_param": 2.058},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _shape(rng, r_max, n_max):
    """Grid side, spacing and rings: the outer edge 210 wavelengths out at `R` cells."""
    R = _logint(rng, 30, r_max)
    du = 1320.0 / (2.0 * math.pi) / R
    n = 2 * rng.randint(int(1.05 * R) + 4, min(n_max // 2, int(3.2 * R)))
    nb = _logint(rng, 6, max(8, min(128, int(0.37 * R))))
    return {"n_grid": n, "du": du, "lo": 46.0, "hi": 1320.0, "n_bins": nb}


def draw(rng):
    kind = rng.choice(["estimate"] * 6 + ["ensemble", "batch", "cube", "grid", "grid", "fields", "triple", "predict",
                                          "simulate"])
    if kind in ("estimate", "ensemble"):
        c = _estimate(kind=kind, **_shape(rng, 300 if kind == "estimate" else 120, 4096))
        c["n_vis"] = _logint(rng, 5000, 8_000_000 if kind == "estimate" else 1_000_000)
        if rng.random() < 0.3:
            c["n_time"] = rng.randint(8, 150)
            c["n_vis"] -= c["n_vis"] % c["n_time"]
        c["precision"] = rng.choice(["fp32", "split_bf16"])
        # the FP32 sums of a fine grid with fine bins cost more than any listed case: those run in split-BF16
        if c["n_bins"] > 40:
            c["precision"] = "split_bf16"
        c["gridder"] = rng.choice(["gauss"] * 4 + ["ngp"])
        c["sigma"], c["radius"] = rng.choice([(1.0, 3)] * 4 + [(0.7, 2), (1.5, 3), (0.5, 1)])
        c["weights"] = rng.choice(["mean"] * 6 + ["noise", "literal"])
        c["u_max"] = rng.choice([220.0, 220.0, 205.0])
        if kind == "ensemble":
            c["n_real"] = rng.randint(2, 24)
            c["n_bins"] = min(c["n_bins"], 32)
        return c
    if kind == "batch":
        return {"kind": "batch", "items": rng.randint(3, 16), "shapes": rng.randrange(1 << 30), "precision": "split_bf16"}
    if kind == "cube":
        n_chan = rng.randint(9, 32)
        top = rng.randint(3, min(16, (n_chan - 1) // 2))
        c = {"kind": "cube", **_shape(rng, 90, 600), "n_vis": _logint(rng, 20_000, 900_000), "n_time": 1,
             "n_chan": n_chan, "tau": rng.choice(["0,1,%d" % top, "0,1,2,%d" % top, "1,%d" % top]),
             "precision": "split_bf16"}
        c["n_bins"] = min(c["n_bins"], 18)
        return c
    if kind == "grid":
        n = 2 * _logint(rng, 32, 1500)
        s, r = rng.choice([(1.0, 3)] * 3 + [(0.7, 2)])
        return {"kind": "grid", "n_grid": n, "du": 440.0 / n * rng.uniform(0.9, 1.3), "n_vis": _logint(rng, 5000, 6_000_000),
                "n_time": rng.choice([1, 1, 60]), "gridder": rng.choice(["gauss", "gauss", "gauss", "ngp"]), "sigma": s,
                "radius": r}
    if kind in ("fields", "triple", "predict"):
        c = {"kind": kind, **_shape(rng, 200 if kind == "fields" else 100, 2048), "n_fft": 0,
             "precision": rng.choice(["fp32", "fp32", "split_bf16"]) if kind != "predict" else "fp32"}
        c["n_bins"] = min(c["n_bins"], 48 if kind == "fields" else 30)
        if rng.random() < 0.3:   # a larger sky grid than the smallest one, odd ones among them
            q, N = _rings(c)
            c["n_fft"] = rng.choice([x for x in _smooth(2 * N) if x > N])
        if kind != "fields":
            c["fill"] = rng.uniform(0.85, 0.999)
        return c
    return {"kind": "simulate", "m": _logint(rng, 48, 300), "dtheta": math.radians(0.029) * rng.uniform(0.5, 2.0),
            "n_vis": _logint(rng, 2000, 110_000), "beam": rng.choice(["none", "tile", "gauss"]),
            "beam_param": rng.uniform(0.1, 2.1)}


def _items(case):
    """The estimates of a batch: grids of 256, 512 or 1024 cells a side, 1e5 to 1e6 visibilities, 16 to 48 bins."""
    r, out = random.Random(case["shapes"]), []
    for _ in range(case["items"]):
        n = r.choice([256, 512, 1024])
        out.append(_estimate(n_grid=n, du=2.3 * 512.0 / n, n_vis=r.randint(100_000, 1_000_000), n_bins=r.randint(16, 48),
                             precision=case["precision"]))
    return out


# ------------------------------------------------------------------------------- geometry (host)


def _edges(c):
    f = np.geomspace if c.get("log", True) else np.linspace
    return np.asarray(f(c["lo"], c["hi"], c["n_bins"] + 1), np.float64)


def _smooth(most):
    return sorted(2 ** a * 3 ** b * 5 ** d for a in range(13) for b in range(9) for d in range(6)
                  if 2 ** a * 3 ** b * 5 ** d <= most)


def _rings(c):
    """The thresholds of |g|^2 between rings and the side of the sky grid."""
    du = float(np.float32(c["du"]))
    q = [math.ceil((e / (2.0 * math.pi * du)) ** 2) for e in _edges(c)]
    half, R = c["n_grid"] // 2 - 1, 0
    for x in range(min(half, math.isqrt(max(q[-1] - 1, 0))), -1, -1):
        y_lo = math.isqrt(max(q[0] - x * x - 1, 0)) + 1 if q[0] > x * x else 0
        if y_lo <= min(half, math.isqrt(q[-1] - 1 - x * x)):
            R = x
            break
    least = max(3 * R + 1, 8)
    return q, c.get("n_fft") or next(v for v in _smooth(2 * least + 8) if v >= least)


def _triplets(q):
    """i <= j <= k that can close, in lexicographic order."""
    nb = len(q) - 1
    q = np.asarray(q, np.int64)
    i, j, k = np.meshgrid(np.arange(nb), np.arange(nb), np.arange(nb), indexing="ij")
    a, b = q[i + 1] - 1, q[j + 1] - 1
    left = q[k] - a - b
    ok = (i <= j) & (j <= k) & (a >= 0) & (b >= 0) & ((left <= 0) | (left * left <= 4 * a * b))
    return np.stack([i[ok], j[ok], k[ok]], 1).astype(np.int32)


def _tau(c):
    return [int(x) for x in c["tau"].split(",")]


def _delay_counts(tau):
    """Ordered delays (t1, t2, t3) with t1 + t2 + t3 = 0, one in each of three bins of |t|."""
    top, na = tau[-1] - 1, len(tau) - 1

    def of(t):
        return next((a for a in range(na) if tau[a] <= abs(t) < tau[a + 1]), -1)

    T = np.zeros((na, na, na), np.int64)
    for a in range(-top, top + 1):
        for b in range(-top, top + 1):
            x = of(a), of(b), of(a + b) if abs(a + b) <= top else -1
            if min(x) >= 0:
                T[x] += 1
    return T


def _bin_triplets(q, tau):
    """u <= v <= w (bin = ring * delay bins + delay bin) whose rings and delays both can close."""
    nb, na = len(q) - 1, len(tau) - 1
    ring = np.zeros((nb, nb, nb), bool)
    t = _triplets(q)
    for p in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        ring[t[:, p[0]], t[:, p[1]], t[:, p[2]]] = True
    u, v, w = np.meshgrid(*[np.arange(nb * na)] * 3, indexing="ij")
    ok = (u <= v) & (v <= w) & ring[u // na, v // na, w // na] & (_delay_counts(tau) > 0)[u % na, v % na, w % na]
    return np.stack([u[ok], v[ok], w[ok]], 1).astype(np.int32)


# ------------------------------------------------------------------------------- inputs (on the GPU)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _baselines(c, g, layout="array"):
    """Antenna pairs with areal density ~ |U|^-1.5, each tracked over n_time samples of a 7.5 degree turn, or
    points uniform in an annulus."""
    nt = c.get("n_time", 1)
    n = c["n_vis"] // nt
    lo, hi = c.get("u_min", 7.0), c.get("u_max", 220.0)
    s = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    if layout == "annulus":
        r = torch.sqrt(lo * lo + s * (hi * hi - lo * lo))
    else:
        r = (math.sqrt(lo) + s * (math.sqrt(hi) - math.sqrt(lo))) ** 2
    phi = 2.0 * math.pi * torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    turn = math.radians(7.5) * torch.arange(nt, device=DEV, dtype=torch.float64) / nt
    a = (phi[:, None] + turn[None, :]).reshape(-1)
    r = r.repeat_interleave(nt)
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], 1)


def _power(m, z=1):
    """|k|^-2.5 on an m x m (x z) grid, summing to the number of its cells."""
    k = torch.fft.fftfreq(m, 1.0 / m, device=DEV, dtype=torch.float64)
    kk = k[:, None] ** 2 + k[None, :] ** 2
    if z > 1:
        kz = torch.fft.fftfreq(z, 1.0 / z, device=DEV, dtype=torch.float64)
        kk = kk[None] + kz[:, None, None] ** 2
    p = torch.where(kk > 0, kk, 1.0) ** -1.25
    p = torch.where(kk > 0, p, 0.0)
    return p * (p.numel() / p.sum())


def _sky(m, g, n_src=0, z=1):
    """Fourier modes of a local quadratic transform of a Gaussian sky (one map per channel for z > 1), with
    point sources of dN/dS ~ S^-1.6 if asked for."""
    dim = (-2, -1) if z == 1 else (-3, -2, -1)
    white = torch.randn((m, m) if z == 1 else (z, m, m), generator=g, device=DEV, dtype=torch.float64)
    f = torch.fft.ifftn(torch.fft.fftn(white, dim=dim) * torch.sqrt(_power(m, z)), dim=dim).real
    f = f + 0.3 * (f * f - 1.0)
    if n_src:
        x = torch.rand(n_src, generator=g, device=DEV, dtype=torch.float64)
        flux = (1.0 + x * (1000.0 ** -0.6 - 1.0)) ** (-1.0 / 0.6)
        at = torch.randint(0, m * m, (n_src,), generator=g, device=DEV)
        f.view(-1).index_add_(0, at, flux)
    return torch.fft.ifft2(f) * (m * m)


def _observe(modes, uv, du, g):
    """The modes read at the baselines (bilinear, periodic) with 5 % complex noise, float32 [n][2]."""
    m = modes.shape[-1]
    x, y = uv[:, 0].double() / du, uv[:, 1].double() / du
    x0, y0 = torch.floor(x), torch.floor(y)
    tx, ty = x - x0, y - y0
    i0, j0 = x0.long() % m, y0.long() % m
    i1, j1 = (i0 + 1) % m, (j0 + 1) % m
    f = modes.reshape(-1)
    v = ((1 - tx) * (1 - ty)) * f[j0 * m + i0]
    v += (tx * (1 - ty)) * f[j0 * m + i1]
    v += ((1 - tx) * ty) * f[j1 * m + i0]
    v += (tx * ty) * f[j1 * m + i1]
    s = 0.05 * torch.sqrt((v.real ** 2 + v.imag ** 2).mean()) / math.sqrt(2.0)
    v += s * torch.randn(v.shape, generator=g, device=DEV, dtype=torch.complex128) * math.sqrt(2.0)
    return torch.view_as_real(v).float().contiguous()


def _config(c, **kw):
    prec = absm.ABS_SPLIT_BF16 if c.get("precision") == "split_bf16" else absm.ABS_FP32
    w = {"mean": absm.ABS_W_MEAN_UNITMASK, "literal": absm.ABS_W_PAPER_LITERAL, "noise": absm.ABS_W_NOISE}
    return absm.Config(n_grid=c["n_grid"], du=c["du"], ell_edges=_edges(c) if "lo" in c else np.array([46.0, 1320.0]),
                       kernel=absm.ABS_KERNEL_NGP if c.get("gridder") == "ngp" else absm.ABS_KERNEL_GAUSS,
                       sigma_cells=c.get("sigma", 1.0), radius_cells=c.get("radius", 3), n_fft=c.get("n_fft", 0),
                       precision=prec, weight_mode=w[c.get("weights", "mean")], **kw)


def _context(c):
    ctx = absm.Context(0, _stream())
    if c.get("precision") == "split_bf16":
        ctx.autotune(False)
    return ctx


def _visibilities(c, seed):
    """uv float32 [n][2] and vis float32 [n_real][n][2]."""
    g = _gen(seed)
    uv = _baselines(c, g, c.get("layout", "array")).float().contiguous()
    m = c["n_grid"] + c["n_grid"] % 2
    vis = [_observe(_sky(m, g, c.get("n_src", 0)), uv, c["du"], g) for _ in range(c.get("n_real", 1))]
    return uv, torch.stack(vis) if len(vis) > 1 else vis[0]


def _cube_data(c, seed):
    g = _gen(seed)
    base = _baselines(c, g)
    sky = _sky(c["n_grid"], g, z=c["n_chan"])
    uv, vis = [], []
    for k, nu in enumerate(np.linspace(139.0, 169.0, c["n_chan"])):
        uv.append((base * (nu / 154.25)).float())
        vis.append(_observe(sky[k], uv[-1], c["du"], g))
    return torch.stack(uv).contiguous(), torch.stack(vis).contiguous()


def _mirror(a):
    """a at -g, for grids in FFT order."""
    return torch.roll(torch.flip(a, (0, 1)), (1, 1), (0, 1))


def _gridded(c, seed):
    """Gridded data as abs_grid leaves it: grid float32 [n][n][2] Hermitian, weight sums, filled mask."""
    n, g = c["n_grid"], _gen(seed)
    on = torch.ones(n, device=DEV, dtype=torch.bool)
    on[n // 2] = False
    hole = torch.rand((n, n), generator=g, device=DEV) > c.get("fill", 0.98)
    mask = ~(hole | _mirror(hole)) & on[:, None] & on[None, :]
    w = 0.05 + 40.0 * torch.rand((n, n), generator=g, device=DEV, dtype=torch.float64) ** 3
    w = ((w + _mirror(w)) * mask).float()
    v = torch.sqrt(_power(n)) * n * torch.randn((n, n), generator=g, device=DEV, dtype=torch.complex128)
    v = (v + _mirror(v).conj()) * w
    return torch.view_as_real(v).float().contiguous(), w.contiguous(), mask.to(torch.uint8).contiguous()


def _ring_map(c, q):
    """The ring of every cell, -1 outside."""
    n = c["n_grid"]
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=torch.float64).round().long()
    ok = k.abs() <= n // 2 - 1
    r2 = k[None, :] ** 2 + k[:, None] ** 2
    ring = torch.bucketize(r2, torch.tensor(q, device=DEV, dtype=torch.int64), right=True) - 1
    ring[(ring >= len(q) - 1) | ~(ok[:, None] & ok[None, :])] = -1
    return ring, r2


def _fields(x, ring, nb, N):
    """FFT of every ring of x on the N x N sky grid, FP64 [nb][N * N] (the real part; complex x is Hermitian)."""
    n = x.shape[0]
    k = torch.fft.fftfreq(n, 1.0 / n, device=DEV, dtype=torch.float64).round().long()
    out = torch.empty((nb, N * N), device=DEV, dtype=torch.float64)
    for m in range(nb):
        y, xx = torch.nonzero(ring == m, as_tuple=True)
        z = torch.zeros((N, N), device=DEV, dtype=torch.complex128)
        z[k[y] % N, k[xx] % N] = x[y, xx].to(torch.complex128)
        out[m] = torch.fft.fft2(z).real.reshape(-1)
    return out


def _sums(D, ijk, fields=None):
    """sum over points of D_i D_j D_k for every listed triplet, FP64."""
    nb = D.shape[0]
    S = torch.zeros((nb, nb, nb), device=DEV, dtype=torch.float64)
    for j in range(nb):
        S[: j + 1, j, j:] = D[: j + 1] @ (D[j] * D[j:]).T
    t = torch.from_numpy(ijk.astype(np.int64)).to(DEV)
    return S[t[:, 0], t[:, 1], t[:, 2]]


def _out(n, dtype=torch.float64):
    return torch.zeros(n, dtype=dtype, device=DEV)


def prepare(case, seed):
    c, kind = case, case["kind"]
    ctx, cfg, s = _context(c), None, {"kind": kind, "weighted": c.get("weights", "mean") != "mean"}
    if kind in ("estimate", "ensemble"):
        cfg = _config(c)
        s["uv"], s["vis"] = _visibilities(c, seed)
        nt, nb = len(absm.abs_triplets(cfg)), c["n_bins"]
        s.update(nt=nt, B=_out((c["n_real"], nt)) if kind == "ensemble" else _out(nt), T=_out(nt, torch.int64), E=_out(nb))
        if kind == "ensemble":
            s.update(mean=_out((nb, 5, 5)), sigma=_out((nb, 5, 5)), weight=_out((nb, 5, 5)))
    elif kind == "batch":
        s["items"] = []
        for i, it in enumerate(_items(c)):
            f = _config(it)
            uv, vis = _visibilities(it, seed * 64 + i)
            nt = len(absm.abs_triplets(f))
            s["items"].append((f, uv, vis, nt, None, _out(nt), _out(nt, torch.int64), _out(it["n_bins"])))
    elif kind == "cube":
        cfg = absm.Config3D(_config(c), c["n_chan"], np.asarray(_tau(c), np.int32))
        s["uv"], s["vis"] = _cube_data(c, seed)
        nt = len(absm.abs_triplets_3d(cfg))
        s.update(nt=nt, B=_out(nt), T=_out(nt, torch.int64), E=_out(c["n_bins"]))
    elif kind == "grid":
        cfg, n = _config(c), c["n_grid"]
        s["uv"], s["vis"] = _visibilities(c, seed)
        s.update(grid=_out((n, n, 2), torch.float32), wsum=_out((n, n), torch.float32), mask=_out((n, n), torch.uint8))
    elif kind == "fields":
        cfg = _config(c)
        s["grid"], s["wsum"], s["mask"] = _gridded(c, seed)
        s["fields"] = _out((c["n_bins"], cfg.N, cfg.N), torch.float32)
    elif kind == "triple":
        cfg = _config(c)
        q, N = _rings(c)
        grid, w, s["mask"] = _gridded(c, seed)
        x = torch.view_as_complex(grid.double()) / torch.where(w > 0, w.double(), 1.0)
        s["fields"] = _fields(x, _ring_map(c, q)[0], c["n_bins"], N).float().reshape(c["n_bins"], N, N).contiguous()
        s["ijk"] = torch.from_numpy(_triplets(q)).to(DEV)
        s.update(S=_out(len(s["ijk"])), T=_out(len(s["ijk"]), torch.int64))
    elif kind == "predict":
        cfg = _config(c)
        s["C"], s["mask"], s["T"], ijk = _prediction_inputs(c, seed)
        s["out"] = _out(len(ijk))
    else:
        g = _gen(seed)
        m = c["m"]
        f = torch.fft.ifft2(torch.fft.fft2(torch.randn((m, m), generator=g, device=DEV, dtype=torch.float64))
                            * torch.sqrt(_power(m))).real
        s["sky"] = (f + 0.3 * (f * f - 1.0)).float().contiguous()
        s["uv"] = _baselines(c, g).float().contiguous()
        s["vis"] = _out((c["n_vis"], 2), torch.float32)
        s["beam"] = {"none": absm.ABS_BEAM_NONE, "tile": absm.ABS_BEAM_MWA_TILE, "gauss": absm.ABS_BEAM_GAUSS}[c["beam"]]
        s.update(dtheta=c["dtheta"], beam_param=c["beam_param"] if c["beam"] != "none" else 0.0)
    s.update(ctx=ctx, cfg=cfg)
    return s


def _prediction_inputs(c, seed):
    """A per-cell angular power spectrum, the filled mask and the triangle counts of that mask."""
    q, N = _rings(c)
    mask = _gridded(c, seed)[2]
    ring, r2 = _ring_map(c, q)
    C = torch.where(r2 > 0, r2.double(), 1.0) ** -1.25 * (1.0 + 0.3 * (seed % 97) / 97.0)
    ijk = _triplets(q)
    T = torch.round(_sums(_fields(mask.double(), ring, c["n_bins"], N), ijk) / (N * N)).long()
    return C.contiguous(), mask, T, ijk


def _with_triangles(s):
    """B; in the weighted forms, whose quotient means nothing for a triplet without triangles, NaN there."""
    if not s["weighted"]:
        return s["B"]
    with torch.cuda.stream(_stream()):
        return torch.where(s["T"] > 0, s["B"], float("nan"))


def run(state):
    s, ctx = state, state["ctx"]
    kind = s["kind"]
    if kind == "estimate":
        ctx.abs_estimate(s["cfg"], s["uv"], s["vis"], s["nt"], None, s["B"], s["T"], s["E"])
        return {"B": _with_triangles(s), "T": s["T"], "ell": s["E"]}
    if kind == "ensemble":
        ctx.abs_estimate_many(s["cfg"], s["uv"], s["vis"], s["nt"], None, s["B"], s["T"], s["E"])
        if s["weighted"]:
            return {"B": _with_triangles(s), "T": s["T"], "ell": s["E"]}
        ctx.abs_rebin(s["cfg"], s["B"], s["T"], s["E"], mean=s["mean"], sigma=s["sigma"], weight=s["weight"])
        return {"B": s["B"], "T": s["T"], "ell": s["E"], "mean": s["mean"], "sigma": s["sigma"], "weight": s["weight"]}
    if kind == "batch":
        ctx.abs_estimate_batched(s["items"])
        return [x for it in s["items"] for x in it[5:8]]
    if kind == "cube":
        ctx.abs_estimate_3d(s["cfg"], s["uv"], s["vis"], s["nt"], None, s["B"], s["T"], s["E"])
        return {"B": s["B"], "T": s["T"], "ell": s["E"]}
    if kind == "grid":
        ctx.abs_grid(s["cfg"], s["uv"], s["vis"], s["grid"], s["wsum"], s["mask"])
        return {"grid": s["grid"], "wsum": s["wsum"], "mask": s["mask"]}
    if kind == "fields":
        ctx.abs_filter_fft(s["cfg"], s["grid"], s["wsum"], s["mask"], s["fields"])
        return s["fields"]
    if kind == "triple":
        ctx.abs_triple(s["cfg"], s["fields"], s["mask"], s["ijk"], s["S"], s["T"])
        return {"S": s["S"], "T": s["T"]}
    if kind == "predict":
        ctx.abs_bana_d(s["cfg"], s["C"], s["mask"], s["T"], s["out"])
        return s["out"]
    ctx.abs_simulate_vis(s["sky"], s["dtheta"], s["uv"], s["vis"], s["beam"], s["beam_param"])
    return s["vis"]


# ------------------------------------------------------------------------------- work and exact values


def _work_estimate(c):
    q, N = _rings(c)
    nt, nb, nv, nr = len(_triplets(q)), c["n_bins"], c["n_vis"], c["n_real"]
    cells = 1 if c["gridder"] == "ngp" else (2 * c["radius"] + 1) ** 2
    one = 6.0 * cells * nv + _work_fields(nb, N) + (2.0 * nt + nb * (nb + 1) / 2) * N * N
    return {"bytes": 8.0 * nv + nr * (8.0 * nv + 8.0 * nt) + 8.0 * nt + 8.0 * nb, "flops": nr * one}


def _work_fields(nb, N):
    return nb / 2 * 5.0 * N * N * math.log2(N * N)


def work(case):
    c, kind = case, case["kind"]
    if kind in ("estimate", "ensemble"):
        return _work_estimate(c)
    if kind == "batch":
        w = [_work_estimate(i) for i in _items(c)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    if kind == "cube":
        q, N = _rings(c)
        tau = _tau(c)
        nt, nu, nz, t1 = len(_bin_triplets(q, tau)), c["n_bins"] * (len(tau) - 1), 3 * tau[-1] - 2, tau[-1]
        P = N * N * nz
        flops = 294.0 * c["n_vis"] * c["n_chan"] + 2.0 * t1 * _work_fields(c["n_bins"], N) + 4.0 * t1 * c["n_bins"] * P \
            + (2.0 * nt + nu * (nu + 1) / 2) * P
        return {"bytes": 16.0 * c["n_vis"] * c["n_chan"] + 16.0 * nt, "flops": flops}
    if kind == "grid":
        cells = 1 if c["gridder"] == "ngp" else (2 * c["radius"] + 1) ** 2
        return {"bytes": 16.0 * c["n_vis"] + 13.0 * c["n_grid"] ** 2, "flops": 6.0 * cells * c["n_vis"]}
    if kind == "simulate":
        return {"bytes": 16.0 * c["n_vis"] + 4.0 * c["m"] ** 2, "flops": 4.0 * c["n_vis"] * c["m"] ** 2}
    q, N = _rings(c)
    nb, nt = c["n_bins"], len(_triplets(q))
    if kind == "fields":
        return {"bytes": 13.0 * math.pi * q[-1] + 4.0 * nb * N * N, "flops": _work_fields(nb, N)}
    if kind == "triple":
        return {"bytes": 4.0 * nb * N * N + math.pi * q[-1] + 28.0 * nt, "flops": (2.0 * nt + nb * (nb + 1) / 2) * N * N}
    return {"bytes": 9.0 * math.pi * q[-1] + 16.0 * nt,
            "flops": 2 * _work_fields(nb, N) + (6.0 * nt + nb * (nb + 1) / 2) * N * N}


def _exact_grid(c, uv, vis):
    """FP64 gridded sums with the mirror: V, sum w, sum w^2 and the number of visibilities, flat in FFT order."""
    n, half = c["n_grid"], c["n_grid"] // 2 - 1
    du32 = torch.tensor(c["du"], dtype=torch.float32, device=DEV)
    acc = torch.zeros((5, n * n), device=DEV, dtype=torch.float64)
    r = 0 if c["gridder"] == "ngp" else c["radius"]
    for a in range(0, len(uv), 1 << 20):
        p, v = uv[a:a + (1 << 20)], vis[a:a + (1 << 20)].double()
        cell = torch.floor(p / du32 + 0.5).long()
        f = p.double() / du32.double() - cell
        w1 = torch.ones((len(p), 2, 1), device=DEV, dtype=torch.float64)
        if c["gridder"] != "ngp":
            d = torch.arange(-r, r + 1, device=DEV, dtype=torch.float64)
            w1 = torch.exp(-(d - f[:, :, None]) ** 2 / (2.0 * c["sigma"] ** 2))
        for dy in range(-r, r + 1):
            for dx in range(-r, r + 1):
                gx, gy = cell[:, 0] + dx, cell[:, 1] + dy
                ok = (gx.abs() <= half) & (gy.abs() <= half)
                at = ((gy % n) * n + gx % n)[ok]
                w = (w1[:, 0, dx + r] * w1[:, 1, dy + r])[ok]
                for k, x in enumerate((w * v[ok, 0], w * v[ok, 1], w, w * w, torch.ones_like(w))):
                    acc[k].index_add_(0, at, x)
    acc = acc.view(5, n, n)
    m = torch.stack([_mirror(x) for x in acc])
    return torch.complex(acc[0] + m[0], acc[1] - m[1]), acc[2] + m[2], acc[3] + m[3], acc[4] + m[4]


def _ell(c, ring, r2, filled):
    x = 2.0 * math.pi * float(np.float32(c["du"])) * torch.sqrt(r2.double())
    return torch.stack([x[(ring == m) & filled].mean() for m in range(c["n_bins"])])


def _exact_estimate(c, uv, vis):
    """B (FP64 [n_real][n_trip]), its counts and the mean l of every ring."""
    q, N = _rings(c)
    ring, r2 = _ring_map(c, q)
    ijk, nb = _triplets(q), c["n_bins"]
    B, T, den = [], None, None
    for v in (vis if vis.dim() == 3 else vis[None]):
        G, w, w2, cnt = _exact_grid(c, uv, v)
        filled = cnt > 0
        if den is None:
            T = torch.round(_sums(_fields(filled.double(), ring, nb, N), ijk) / (N * N))
        one = torch.where(filled, w, 1.0)
        if c["weights"] == "mean":
            x, den = G / one, T
        else:
            wg = 1.0 / torch.where(filled, cnt, 1.0) if c["weights"] == "literal" else w / torch.where(filled, w2, 1.0)
            i = wg if c["weights"] == "literal" else wg * w
            if den is None:
                den = _sums(_fields(i * filled, ring, nb, N), ijk) / (N * N)
            x = G * wg
        s = _sums(_fields(x * filled, ring, nb, N), ijk) / (N * N)
        B.append(torch.where(T > 0, s / den, float("nan")))
    return torch.stack(B), T, _ell(c, ring, r2, filled)


def _exact_rebin(c, B, T, ell):
    q, _ = _rings(c)
    ijk, nb = _triplets(q), c["n_bins"]
    ok = T > 0
    t = torch.from_numpy(ijk.astype(np.int64)).to(DEV)[ok]
    l3, l2, l1 = ell[t[:, 0]], ell[t[:, 1]], ell[t[:, 2]]
    mu = ((l1 * l1 + l2 * l2) - l3 * l3) / (2.0 * l1 * l2)
    at = [torch.floor((x - 0.5) * 10.0).clamp(0, 4).long() for x in (mu, l2 / l1)]
    cell = (t[:, 2] * 5 + at[0]) * 5 + at[1]
    w = torch.zeros(nb * 25, device=DEV, dtype=torch.float64).index_add_(0, cell, T[ok])
    r = torch.stack([torch.zeros_like(w).index_add_(0, cell, T[ok] * b[ok]) / w for b in B])
    mean = r.mean(0)
    sig = torch.sqrt(((r * r).mean(0) - mean * mean).clamp_min(0))
    return [x.view(nb, 5, 5) for x in (mean, sig, w)]


def _exact_cube(c, uv, vis):
    q, N = _rings(c)
    ring, r2 = _ring_map(c, q)
    tau, nb = _tau(c), c["n_bins"]
    na, t1, nz = len(tau) - 1, tau[-1], 3 * tau[-1] - 2
    cc = dict(c, gridder="gauss", sigma=1.0, radius=3)
    X, common = [], torch.ones_like(ring, dtype=torch.bool)
    for k in range(c["n_chan"]):
        G, w, _, cnt = _exact_grid(cc, uv[k], vis[k])
        common &= cnt > 0
        X.append(G / torch.where(cnt > 0, w, 1.0))
    X = torch.fft.fft(torch.stack(X) * common, dim=0)[:t1]
    k = torch.fft.fftfreq(c["n_grid"], 1.0 / c["n_grid"], device=DEV, dtype=torch.float64).round().long()
    F = torch.zeros((nb, t1, N * N), device=DEV, dtype=torch.complex128)
    for m in range(nb):
        y, x = torch.nonzero(ring == m, as_tuple=True)
        z = torch.zeros((t1, N, N), device=DEV, dtype=torch.complex128)
        z[:, k[y] % N, k[x] % N] = X[:, y, x]
        F[m] = torch.fft.fft2(z).reshape(t1, -1)
    ijk = _bin_triplets(q, tau)
    S = torch.zeros(len(ijk), device=DEV, dtype=torch.float64)
    for z in range(nz):
        D = torch.zeros((nb, na, N * N), device=DEV, dtype=torch.float64)
        for a in range(na):
            for t in range(tau[a], tau[a + 1]):
                w = 2.0 * math.pi * ((t * z) % nz) / nz
                D[:, a] += (1.0 if t == 0 else 2.0) * (F[:, t].real * math.cos(w) + F[:, t].imag * math.sin(w))
        S += _sums(D.view(nb * na, -1), ijk)
    r = np.sort(ijk // na, 1)
    T2 = torch.round(_sums(_fields(common.double(), ring, nb, N), r) / (N * N))
    T = T2 * torch.from_numpy(_delay_counts(tau)[tuple((ijk % na).T)]).to(DEV)
    return torch.where(T > 0, S / (N * N * nz) / T, float("nan")), _ell(c, ring, r2, common)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("estimate", "ensemble"):
        B, T, ell = _exact_estimate(c, *_visibilities(c, seed))
        if kind == "estimate":
            return {"B": B[0], "T": None, "ell": ell}
        if c["weights"] != "mean":
            return {"B": B, "T": None, "ell": ell}
        mean, sigma, weight = _exact_rebin(c, B, T, ell)
        return {"B": B, "T": None, "ell": ell, "mean": mean, "sigma": sigma, "weight": weight}
    if kind == "batch":
        out = []
        for i, it in enumerate(_items(c)):
            B, _, ell = _exact_estimate(it, *_visibilities(it, seed * 64 + i))
            out += [B[0], None, ell]
        return out
    if kind == "cube":
        B, ell = _exact_cube(c, *_cube_data(c, seed))
        return {"B": B, "T": None, "ell": ell}
    if kind == "grid":
        G, w, _, _ = _exact_grid(c, *_visibilities(c, seed))
        return {"grid": torch.view_as_real(G), "wsum": w, "mask": None}
    if kind == "fields":
        q, N = _rings(c)
        grid, w, mask = _gridded(c, seed)
        x = torch.view_as_complex(grid.double()) / torch.where(mask > 0, w.double(), 1.0) * mask
        return _fields(x, _ring_map(c, q)[0], c["n_bins"], N).view(c["n_bins"], N, N)
    if kind == "triple":
        s = prepare(c, seed)
        N = s["fields"].shape[-1]
        return {"S": _sums(s["fields"].double().view(c["n_bins"], -1), _triplets(_rings(c)[0])) / (N * N), "T": None}
    if kind == "predict":
        C, mask, T, ijk = _prediction_inputs(c, seed)
        q, N = _rings(c)
        ring = _ring_map(c, q)[0]
        P, I = (_fields(x, ring, c["n_bins"], N) for x in (C * mask, mask.double()))
        t = torch.from_numpy(ijk.astype(np.int64)).to(DEV)
        S = torch.zeros((c["n_bins"],) * 3, device=DEV, dtype=torch.float64)
        for j in range(c["n_bins"]):
            S[:, j, :] = P @ (P[j] * I).T + I @ (P[j] * P).T + P @ (I[j] * P).T
        S = S[t[:, 0], t[:, 1], t[:, 2]] / (N * N)
        return torch.where(T > 0, 0.6 * S / T, float("nan"))
    m, dth, uv = c["m"], c["dtheta"], None
    s = prepare(c, seed)
    th = (torch.arange(m, device=DEV, dtype=torch.float64) - m // 2) * dth
    if c["beam"] == "tile":
        b = torch.sinc(c["beam_param"] * th) ** 2
        A = b[:, None] * b[None, :]
    elif c["beam"] == "gauss":
        A = torch.exp(-(th[:, None] ** 2 + th[None, :] ** 2) / c["beam_param"] ** 2)
    else:
        A = torch.ones((m, m), device=DEV, dtype=torch.float64)
    W = (dth * dth * A * s["sky"].double()).to(torch.complex128)
    ex = torch.exp(2j * math.pi * s["uv"][:, :1].double() * th)
    ey = torch.exp(2j * math.pi * s["uv"][:, 1:].double() * th)
    return torch.view_as_real(((ey @ W) * ex).sum(1))
