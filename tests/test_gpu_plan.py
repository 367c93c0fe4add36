"""The gridding plan where its slices hold several chunks of 4,096 records (from 1.2e6 visibilities on), with keys of
one, two and three radix passes, and the nearest cells it takes from a reciprocal: nearest-grid-point gridding of
integer visibilities, whose sums are exact, against integer sums over the cells of the FP32 division."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _check(n, du, uv, seed):
    absbuild.build()
    rng = np.random.default_rng(seed)
    vis = rng.integers(-3, 4, uv.shape).astype(np.float32)
    half = n // 2 - 1
    d = np.float32(du)
    with np.errstate(invalid="ignore", over="ignore"):
        c = np.floor((uv / d).astype(np.float32) + np.float32(0.5))
    on = np.isfinite(c).all(1) & (np.abs(c) <= half).all(1)
    k = c[on].astype(np.int64) % n
    cell = k[:, 1] * n + k[:, 0]
    plane = [np.bincount(cell, w, n * n).reshape(n, n) for w in (vis[on, 0], vis[on, 1], np.ones(on.sum()))]
    mirror = [np.roll(p[::-1, ::-1], (1, 1), (0, 1)) for p in plane]
    want = [plane[0] + mirror[0], plane[1] - mirror[1], plane[2] + mirror[2]]
    assert max(np.abs(w).max() for w in want) < 1 << 24   # exact in FP32
    cfg = absmod.Config(n_grid=n, du=du, ell_edges=2 * np.pi * float(d) * np.array([1.0, 2.0]),
                        kernel=absmod.ABS_KERNEL_NGP)
    dev = torch.device("cuda:0")
    g = torch.empty((n, n, 2), dtype=torch.float32, device=dev)
    w = torch.empty((n, n), dtype=torch.float32, device=dev)
    m = torch.empty((n, n), dtype=torch.uint8, device=dev)
    ctx = absmod.Context(0)
    ctx.abs_grid(cfg, torch.from_numpy(uv).to(dev), torch.from_numpy(vis).to(dev), g, w, m)
    ctx.sync()
    ctx.close()
    got = [g[..., 0].cpu().numpy(), g[..., 1].cpu().numpy(), w.cpu().numpy()]
    for a, b in zip(got, want):
        assert np.array_equal(a.astype(np.float64), b)
    assert np.array_equal(m.cpu().numpy(), (want[2] > 0).astype(np.uint8))


# records of a slice (whole rows of 512), and how many the last slice lacks: chunks of 4,096 just not full, full and
# begun, and a last chunk of one record
@pytest.mark.parametrize("per_slice,short", [(3584, 511), (4096, 0), (4096, 4095), (4608, 1), (8192, 8191), (8704, 511)])
@pytest.mark.parametrize("n_grid", [8, 66, 600])
def test_slices_of_several_chunks(n_grid, per_slice, short):
    n_vis = 2 * torch.cuda.get_device_properties(0).multi_processor_count * per_slice - short
    rng = np.random.default_rng(per_slice + short + n_grid)
    uv = ((rng.random((n_vis, 2), dtype=np.float32) - np.float32(0.5)) * np.float32(1.04 * n_grid * 1.3))
    uv[n_vis // 3:n_vis // 2] = uv[n_vis // 3]        # one cell for many chunks
    uv[rng.integers(0, n_vis, 1000)] = np.nan
    _check(n_grid, 1.3, uv, n_vis)


@pytest.mark.parametrize("n_grid", [64, 2048])
@pytest.mark.parametrize("du", [0.6, 1.15, 2.3, 1.0 / 3.0, 1.0, 1e-3, 7e4,
                                float(np.float32(2.0) - np.float32(2.0 ** -23)),    # a significand of ones: divided
                                float(np.float32(2.0) - np.float32(2.0 ** -22)),
                                float(np.float32(1.0) + np.float32(2.0 ** -23))])
def test_nearest_cells(n_grid, du):
    """Positions within two units in the last place of every cell boundary."""
    d = np.float32(du)
    b = (np.arange(-n_grid // 2, n_grid // 2).astype(np.float32) + np.float32(0.5)) * d
    near = [b]
    for to in (np.float32(-np.inf), np.float32(np.inf)):
        x = b
        for _ in range(2):
            x = np.nextafter(x, to)
            near.append(x)
    u = np.concatenate(near)
    rng = np.random.default_rng(n_grid)
    _check(n_grid, du, np.stack([u, u[rng.permutation(len(u))]], 1), n_grid)
