"""The row pass of the ring transforms over sky grids of one, two, three and more radix passes, of every first
radix, odd and even, up to the largest that takes two rows a CTA: fields against the FP64 oracle, and the
split planes that the pass writes itself against those made from its FP32 fields."""
import numpy as np
import pytest

import oracle
import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [16, 18, 20, 24, 25, 27, 30, 36, 45, 50, 64, 75, 81, 90, 100, 125, 144, 160, 225, 256, 375, 486, 540]
N_GRID = 32
# double-float transforms: one FP32 rounding of every value, of the grid and of the result; plain FP32
# transforms: at most 2^-24 a butterfly level and value, fewer than 20 levels with the radix constants
TOL = {"fp32": 2e-7, "split": 2e-6}


def _config(precision, N):
    edges = 2 * np.pi * np.array([0.9, 2.1, 3.3, 4.9])
    return absmod.Config(n_grid=N_GRID, du=1.0, ell_edges=edges, n_fft=N,
                         precision=absmod.ABS_SPLIT_BF16 if precision == "split" else absmod.ABS_FP32)


def _fields(precision, N):
    absbuild.build()
    cfg = _config(precision, N)
    rng = np.random.default_rng(N)
    X = rng.standard_normal((N_GRID, N_GRID)) + 1j * rng.standard_normal((N_GRID, N_GRID))
    m = rng.random((N_GRID, N_GRID)) < 0.9
    neg = (-np.arange(N_GRID)) % N_GRID
    X = (X + np.conj(X[neg][:, neg])) / 2
    m &= m[neg][:, neg]
    g = np.stack([X.real, X.imag], -1).astype(np.float32)
    dev = torch.device("cuda:0")
    out = torch.full((3, N, N), float("nan"), dtype=torch.float32, device=dev)
    ctx = absmod.Context(0)
    ctx.abs_filter_fft(cfg, torch.from_numpy(g).to(dev), torch.ones((N_GRID, N_GRID), device=dev),
                       torch.from_numpy(m.astype(np.uint8)).to(dev), out)
    ctx.sync()
    got = out.cpu().numpy().astype(np.float64)
    ctx.close()
    r = np.fft.fftfreq(N_GRID, 1 / N_GRID).astype(int)
    r2 = r[:, None] ** 2 + r[None] ** 2
    q = oracle.ring_q(cfg.ell_edges, 1.0)
    keep = m & (np.abs(r)[:, None] < N_GRID // 2) & (np.abs(r)[None] < N_GRID // 2)
    Xd = g[..., 0].astype(np.float64) + 1j * g[..., 1]
    for i in range(3):
        Z = np.zeros((N, N), complex)
        y, x = np.nonzero(keep & (r2 >= q[i]) & (r2 < q[i + 1]))
        Z[r[y] % N, r[x] % N] = Xd[y, x]
        ref = np.fft.fft2(Z)
        assert np.abs(ref.imag).max() <= 1e-12 * np.abs(ref.real).max()
        assert np.linalg.norm(got[i] - ref.real) <= TOL[precision] * np.linalg.norm(ref.real), (N, i)


@pytest.mark.parametrize("precision", ["fp32", "split"])
@pytest.mark.parametrize("N", SIZES)
def test_fields(precision, N):
    _fields(precision, N)


@pytest.mark.parametrize("precision,N", [("fp32", 3600), ("split", 3600), ("split", 4096)])
def test_lines_as_long_as_shared_memory(precision, N):
    _fields(precision, N)


@pytest.mark.parametrize("N", SIZES)
def test_planes(N):
    absbuild.build()
    cfg = _config("split", N)
    ijk = absmod.abs_triplets(cfg)
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(N)
    uv = (torch.rand((3000, 2), generator=g, device=dev) - 0.5) * 12
    vis = torch.randn((3000, 2), generator=g, device=dev)
    ctx = absmod.Context(0)
    ctx.autotune(False)
    B = [torch.full((len(ijk),), float("nan"), dtype=torch.float64, device=dev) for _ in range(2)]
    ctx.abs_estimate(cfg, uv, vis, len(ijk), None, B[0])
    ctx.abs_estimate(cfg, uv, vis, len(ijk), torch.from_numpy(ijk).to(dev), B[1])
    ctx.sync()
    a, b = (x.cpu().numpy() for x in B)
    ctx.close()
    # the same fields and products; the sums' ranges may differ (FP32 partial sums)
    assert np.linalg.norm(a - b) <= 1e-5 * np.linalg.norm(b)
