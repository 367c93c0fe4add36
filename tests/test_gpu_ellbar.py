"""Mean l of every ring against sums in extended precision: the sums over a ring's cells carry FP64's accuracy."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# rms over the rings.  FP64 sums of a ring's partial sums: a dozen additions of 2^-53 each, the terms' own
# errors averaged over hundreds of cells, three roundings of the scale: 4e-16; twice that.
TOL_RMS = 8e-16


@pytest.mark.parametrize("n,du,top,nb", [(704, 1.0, 350.0, 128), (704, 1.0, 350.0, 20), (400, 0.7, 190.0, 20)])
@pytest.mark.parametrize("fill", [0.6, 1.0])
def test_mean_ell(n, du, top, nb, fill):
    absbuild.build()
    cfg = absmod.Config(n_grid=n, du=du, ell_edges=2 * np.pi * float(np.float32(du)) * np.linspace(0.6, top, nb + 1))
    q = absmod.abs_ring_q(cfg)
    k = np.fft.fftfreq(n, 1.0 / n).round().astype(np.int64)
    r2 = k[:, None] ** 2 + k[None, :] ** 2
    on = np.abs(k) <= n // 2 - 1
    hole = np.random.default_rng(n + nb).random((n, n)) >= fill
    hole |= np.roll(hole[::-1, ::-1], (1, 1), (0, 1))
    mask = ~hole & on[:, None] & on[None, :]
    ell = torch.zeros(nb, dtype=torch.float64, device="cuda:0")
    S = torch.ones(1, dtype=torch.float64, device="cuda:0")
    ctx = absmod.Context(0)
    ctx.abs_normalise(cfg, S, torch.ones(1, dtype=torch.int64, device="cuda:0"), torch.empty_like(S),
                      torch.from_numpy(mask.astype(np.uint8)).to("cuda:0"), ell)
    ctx.sync()
    r = np.sqrt(r2.astype(np.longdouble))
    rel = []
    for m in range(nb):
        c = r[(r2 >= q[m]) & (r2 < q[m + 1]) & mask]
        want = 2 * np.longdouble(np.pi) * np.longdouble(np.float32(du)) * c.sum() / c.size
        rel.append(float(np.longdouble(ell[m].item()) / want - 1))
    assert np.sqrt(np.mean(np.square(rel))) <= TOL_RMS
