"""Exact triangle counts over fills from none to all: both routes of the count kernel (direct and
holes), masks with holes in every ring, symmetric classes on the axes and diagonals, a byte map in
shared memory and one too large for it, against unit-mask fields transformed in FP64 (rounded to the
integers they are)."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ring_of(cfg):
    n, q = cfg.n_grid, absmod.abs_ring_q(cfg)
    k = np.fft.fftfreq(n, 1.0 / n).round().astype(np.int64)
    r2 = k[:, None] ** 2 + k[None, :] ** 2
    ring = np.searchsorted(q, r2, side="right") - 1
    ring[(ring >= cfg.n_bins) | (np.abs(k)[:, None] > n // 2 - 1) | (np.abs(k)[None, :] > n // 2 - 1)] = -1
    return ring, k, r2


def _fft_counts(mask, ring, k, N, ijk, nb):
    D = torch.zeros((nb, N, N), dtype=torch.float64, device="cuda:0")
    for m in range(nb):
        y, x = np.nonzero((ring == m) & (mask > 0))
        u = np.zeros((N, N))
        u[k[y] % N, k[x] % N] = 1.0
        D[m] = torch.fft.fft2(torch.from_numpy(u).to("cuda:0")).real
    D = D.view(nb, -1)
    S = torch.zeros((nb, nb, nb), dtype=torch.float64, device="cuda:0")
    for j in range(nb):
        S[: j + 1, j, j:] = D[: j + 1] @ (D[j] * D[j:]).T
    T = (S / (N * N)).cpu().numpy()[ijk[:, 0], ijk[:, 1], ijk[:, 2]]
    assert np.max(np.abs(T - np.round(T)), initial=0.0) < 0.2
    return np.round(T).astype(np.int64)


# grid side, spacing, outer edge in cells, rings
SHAPES = [(8, 1.0, 3.2, 1), (16, 1.0, 7.9, 3), (64, 1.0, 31.5, 7), (98, 1.0, 40.0, 13), (500, 1.0, 235.0, 6),
          (600, 1.0, 260.0, 40)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("fill", [0.0, 0.3, 0.62, 0.9, 0.997, 1.0])
def test_counts_every_fill(shape, fill):
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    absbuild.build()
    n, du, top, nb = shape
    cfg = absmod.Config(n_grid=n, du=du, ell_edges=2 * np.pi * du * np.linspace(0.6, top, nb + 1))
    ring, k, r2 = _ring_of(cfg)
    rng = np.random.default_rng(int(1000 * fill) + n)
    h = rng.random((n, n)) >= fill
    if fill > 0.95:
        h &= (r2 > 0.8 * top * top) | (rng.random((n, n)) < 0.1)   # holes mostly in the outer rings
    h |= np.roll(h[::-1, ::-1], (1, 1), (0, 1))
    on = np.abs(k) <= n // 2 - 1
    mask = (~h & on[:, None] & on[None, :]).astype(np.uint8)
    ijk = absmod.abs_triplets(cfg)
    want = _fft_counts(mask, ring, k, cfg.N, ijk, nb)
    ctx = absmod.Context(0)
    d_ijk, d_mask = torch.from_numpy(ijk).to("cuda:0"), torch.from_numpy(mask).to("cuda:0")
    for call in range(2):   # the first call also makes the full-annulus counts
        T = torch.full((len(ijk),), -1, dtype=torch.int64, device="cuda:0")
        ell = torch.zeros(nb, dtype=torch.float64, device="cuda:0")
        ctx.abs_triple(cfg, None, d_mask, d_ijk, None, T)
        S = torch.ones(len(ijk), dtype=torch.float64, device="cuda:0")
        B = torch.empty_like(S)
        ctx.abs_normalise(cfg, S, T, B, d_mask, ell)
        ctx.sync()
        assert np.array_equal(T.cpu().numpy(), want), f"call {call}"
        for m in range(nb):
            r = np.sqrt(r2[(ring == m) & (mask > 0)].astype(np.float64))
            e = ell[m].item()
            assert np.isnan(e) if r.size == 0 else abs(e / (2 * np.pi * float(np.float32(du)) * r.mean()) - 1) < 1e-12
