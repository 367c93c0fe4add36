"""Gridding at the edges of its plan and accumulation: visibility counts around the sort's chunk (4,096),
the accumulation's segments (64, 128) and warps (32), grids whose cell key takes one, two and three radix
passes, long runs of one cell, and positions that are skipped, against the FP64 oracle."""
import numpy as np
import pytest

import oracle
import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild
from paper_2412_02246_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-6   # normwise, per cell: the gridding tolerance of the parity tests


def _check(n, du, uv, vis, kernel="gauss", sigma=1.0, radius=3):
    absbuild.build()
    oracle.build()
    cfg = absmod.Config(n_grid=n, du=du, ell_edges=np.array([2 * np.pi * du, 4 * np.pi * du]),
                        kernel=absmod.ABS_KERNEL_NGP if kernel == "ngp" else absmod.ABS_KERNEL_GAUSS,
                        sigma_cells=sigma, radius_cells=radius)
    ctx = absmod.Context(0)
    dev = torch.device("cuda:0")
    g = torch.empty((n, n, 2), dtype=torch.float32, device=dev)
    w = torch.empty((n, n), dtype=torch.float32, device=dev)
    m = torch.empty((n, n), dtype=torch.uint8, device=dev)
    ctx.abs_grid(cfg, torch.from_numpy(uv).to(dev), torch.from_numpy(synth.vis_as_float2(vis)).to(dev), g, w, m)
    ctx.sync()
    ok = np.isfinite(uv).all(1)
    ref = oracle.grid(n, du, uv[ok], vis[ok], kernel, sigma, radius)
    bound = oracle.grid(n, du, uv[ok], np.abs(vis[ok]).astype(np.complex64), kernel, sigma, radius).grid.real
    G = g.cpu().numpy().astype(np.float64)
    G = G[..., 0] + 1j * G[..., 1]
    assert np.array_equal(m.cpu().numpy(), (ref.ncontrib > 0).astype(np.uint8))
    on = bound > 0
    assert np.max(np.abs(G - ref.grid)[on] / bound[on], initial=0.0) <= TOL
    W, ws = w.cpu().numpy(), ref.wsum > 0
    assert np.max(np.abs(W[ws] - ref.wsum[ws]) / ref.wsum[ws], initial=0.0) <= TOL
    assert np.all(G[~on] == 0) and np.all(W[~ws] == 0)


def _vis(rng, n):
    return (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)


@pytest.mark.parametrize("n_vis", [1, 31, 33, 63, 65, 127, 128, 129, 511, 513, 4095, 4096, 4097, 12293])
@pytest.mark.parametrize("n_grid", [8, 66, 600])
def test_counts_of_visibilities(n_grid, n_vis):
    rng = np.random.default_rng(n_vis + n_grid)
    uv = (rng.uniform(-0.55, 0.55, (n_vis, 2)) * n_grid * 1.3).astype(np.float32)
    uv[rng.random(n_vis) < 0.02] = np.nan
    _check(n_grid, 1.3, uv, _vis(rng, n_vis))


@pytest.mark.parametrize("n_grid", [2030, 2048, 8192])   # two radix passes of 11 bits, three
def test_wide_keys(n_grid):
    rng = np.random.default_rng(n_grid)
    uv = (rng.uniform(-0.51, 0.51, (20011, 2)) * n_grid * 0.7).astype(np.float32)
    _check(n_grid, 0.7, uv, _vis(rng, len(uv)))


@pytest.mark.parametrize("kernel,sigma,radius", [("gauss", 1.0, 3), ("gauss", 0.7, 2), ("gauss", 0.5, 1),
                                                 ("gauss", 0.6, 0), ("ngp", 1.0, 3)])
def test_runs_of_one_cell(kernel, sigma, radius):
    """Runs of 1 to 300 visibilities of a cell, in and out of input order, over the grid's edges and axes."""
    rng = np.random.default_rng(5)
    n = 48
    cells = rng.integers(-25, 26, (160, 2))
    runs = [np.repeat(c[None], k, 0) for c, k in zip(cells, rng.integers(1, 301, 160))]
    c = np.concatenate(runs)
    if radius == 2:
        c = c[rng.permutation(len(c))]
    uv = ((c + rng.uniform(-0.5, 0.5, c.shape)) * 2.0).astype(np.float32)
    _check(n, 2.0, uv, _vis(rng, len(uv)), kernel, sigma, radius)


@pytest.mark.parametrize("n_vis", [60_000, 120_001, 240_003])   # units of 128, 256 and 512 visibilities
def test_units(n_vis):
    rng = np.random.default_rng(n_vis)
    uv = (rng.uniform(-0.5, 0.5, (n_vis, 2)) * 90).astype(np.float32)
    _check(90, 1.0, uv, _vis(rng, n_vis))


@pytest.mark.parametrize("n_grid", [16, 66, 600])   # keys of two and of three passes
@pytest.mark.parametrize("n_vis", [1023, 1025, 5119, 5120, 5121])   # rows and the largest set of the one-CTA plan
def test_one_cta_plan(n_grid, n_vis):
    rng = np.random.default_rng(n_vis + n_grid)
    uv = (rng.uniform(-0.52, 0.52, (n_vis, 2)) * n_grid * 0.9).astype(np.float32)
    uv[::97] = np.inf
    _check(n_grid, 0.9, uv, _vis(rng, n_vis))
