"""bench.count_kernel_visits, which the count kernel's roofline rests on, against the kernel's enumeration written
out pair by pair on small masks (no GPU)."""
import numpy as np
import pytest

import bench
import oracle


def _enumerate(mask, q, n):
    half = n // 2 - 1
    ring = lambda x, y: int(np.searchsorted(q, x * x + y * y, side="right")) - 1
    cells = [(x, y) for y in range(0, half + 1) for x in range(-half, half + 1)
             if (y > 0 or x > 0) and q[0] <= x * x + y * y < q[-1]]
    nb = len(q) - 1
    up = [[c for c in cells if ring(*c) == m] for m in range(nb)]
    F = [[c for c in up[m] if mask[c[1] % n, c[0] % n]] for m in range(nb)]
    H = [[c for c in up[m] if not mask[c[1] % n, c[0] % n]] for m in range(nb)]
    orb = [sorted({(max(abs(x), abs(y)), min(abs(x), abs(y))) for x, y in H[m]}) for m in range(nb)]
    low = [min(((max(abs(x), abs(y)), min(abs(x), abs(y))) for x, y in up[m]), default=None) for m in range(nb)]
    direct = sum(len(F[a]) * 2 * len(F[b]) for a in range(nb) for b in range(a, nb))
    two = 2 * sum(len(H[a]) * 2 * len(H[b]) for a in range(nb) for b in range(a, nb))
    if not two + sum(map(len, orb)) * len(cells) < direct:
        return direct, "direct"
    one = 0
    for a in range(nb):
        for _ in orb[a]:   # u above half the ring's lowest orbit (y, x): row-major order of 2 u - h
            one += sum((2 * y - low[a][0], 2 * x - low[a][1]) > (0, 0) for b in range(nb) for x, y in up[b])
    return two + one, "holes"


@pytest.mark.parametrize("top", [7.5, 11.0, 13.0])
@pytest.mark.parametrize("fill,route", [(1.0, "holes"), (0.98, "holes"), (0.9, None), (0.3, "direct")])
def test_visits_of_the_kernel(top, fill, route):
    n = 24
    q = np.asarray(oracle.ring_q(2 * np.pi * np.linspace(1.5, top, 5), 1.0))
    rng = np.random.default_rng(int(100 * fill + top))
    hole = rng.random((n, n)) >= fill
    hole |= np.roll(hole[::-1, ::-1], (1, 1), (0, 1))
    mask = (~hole).astype(np.uint8)
    got = bench.count_kernel_visits(mask, q, n)
    assert got == _enumerate(mask, q, n)
    assert route is None or got[1] == route
    if fill == 1.0:
        assert got[0] == 0
    if got[1] == "holes" and fill < 1.0:   # below the plain enumeration's unit
        assert got[0] < bench.count_route_visits(*bench.ring_census(mask, q, n))
