"""Ensembles on a device short of memory: a lane without room for its workspaces hands its realisations back and
gives what it took back to the device, and a context that finds no room takes its lanes' workspaces back."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-6   # the order of the accumulators' FP64 atomics can move an FP32 rounding of a transform's input
N_REAL = 7


class Case:
    def __init__(self, n, st, dev, n_vis=20_000):
        self.cfg = absmod.Config(n_grid=n, du=1.0, ell_edges=2 * np.pi * np.linspace(2.0, 0.4 * n, 9))
        self.nt, self.dev = absmod.abs_triplets(self.cfg).shape[0], dev
        g = torch.Generator(device=dev).manual_seed(n)
        self.uv = (torch.rand((n_vis, 2), generator=g, device=dev) - 0.5) * 0.9 * n
        self.vis = torch.randn((N_REAL, n_vis, 2), generator=g, device=dev)
        st.wait_stream(torch.cuda.current_stream(dev))
        one = absmod.Context(0, st)
        self.want = self.out()
        for r in range(N_REAL):
            one.abs_estimate(self.cfg, self.uv, self.vis[r].contiguous(), self.nt, None, self.want[0][r], self.want[1])
        one.sync()
        one.close()

    def out(self):
        return (torch.full((N_REAL, self.nt), float("nan"), dtype=torch.float64, device=self.dev),
                torch.zeros(self.nt, dtype=torch.int64, device=self.dev))

    def check(self, ctx):
        B, T = self.out()
        ctx.abs_estimate_many(self.cfg, self.uv, self.vis, self.nt, None, B, T)
        ctx.sync()
        assert torch.equal(T, self.want[1])
        for r in range(N_REAL):
            d = torch.nan_to_num(B[r] - self.want[0][r])
            assert torch.equal(torch.isnan(B[r]), torch.isnan(self.want[0][r]))
            assert d.norm() <= TOL * torch.nan_to_num(self.want[0][r]).norm()


def _case(n):
    absbuild.build()
    dev = torch.device("cuda:0")
    st = torch.cuda.Stream(dev)
    return st, dev, Case(n, st, dev)


@pytest.mark.parametrize("failures", [1, 2, 9])
def test_lane_without_room(failures):
    st, dev, c = _case(512)
    with torch.cuda.stream(st):
        ctx = absmod.Context(0, st)
        B, T = c.out()
        ctx.abs_estimate(c.cfg, c.uv, c.vis[0].contiguous(), c.nt, None, B[0], T)   # the context's own workspaces
        ctx.sync()
        before = torch.cuda.mem_get_info(dev)[0]
        ctx.inject_alloc_failures(failures)
        c.check(ctx)
        ctx.inject_alloc_failures(0)
        # four lanes' accumulators, transforms and fields are over 200 MB here
        assert torch.cuda.mem_get_info(dev)[0] > before - (32 << 20)
        for _ in range(3):   # without lanes from here on: eager, captured, replayed
            c.check(ctx)
        assert torch.cuda.mem_get_info(dev)[0] > before - (64 << 20)
        ctx.close()


def test_context_takes_its_lanes_workspaces_back():
    st, dev, small = _case(96)
    big = Case(192, st, dev)
    with torch.cuda.stream(st):
        ctx = absmod.Context(0, st)
        for _ in range(3):
            small.check(ctx)
        ctx.inject_alloc_failures(1)
        big.check(ctx)      # its first workspace finds no room until the lanes' are freed
        ctx.inject_alloc_failures(0)
        for _ in range(3):
            small.check(ctx)
            big.check(ctx)
        ctx.close()
