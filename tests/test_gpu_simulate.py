"""Visibility simulator at the edges of its column blocks (32), row groups (4) and row passes (32), and in slabs:
where the partial sums of all visibilities do not fit, on a device without room and in a stream that is being
captured after a call with fewer visibilities, against the direct DFT in FP64."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-6   # of sum |dtheta^2 T|, the direct DFT's bound in the parity tests


def _inputs(m, n_vis, seed):
    absbuild.build()
    g = torch.Generator(device="cuda:0").manual_seed(seed)
    dth = 1.1 / m
    sky = torch.randn((m, m), generator=g, device="cuda:0")
    uv = (torch.rand((n_vis, 2), generator=g, device="cuda:0") - 0.5) * 440.0
    return dth, sky, uv


def _check(m, dth, sky, uv, vis):
    torch.cuda.synchronize()
    if len(uv) == 0:
        return
    th = (torch.arange(m, device="cuda:0", dtype=torch.float64) - m // 2) * dth
    ex = torch.exp(2j * np.pi * uv[:, :1].double() * th)
    ey = torch.exp(2j * np.pi * uv[:, 1:].double() * th)
    W = dth * dth * sky.double()
    ref = ((ex @ W.T.to(torch.complex128)) * ey).sum(1)
    assert (torch.view_as_complex(vis.double()) - ref).abs().max().item() <= TOL * W.abs().sum().item()


def _vis(n):
    return torch.full((n, 2), float("nan"), device="cuda:0")


@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 36, 63, 65, 100, 257])
@pytest.mark.parametrize("n_vis", [0, 1, 127, 129, 255, 257, 1030])
def test_sizes(m, n_vis):
    dth, sky, uv = _inputs(m, n_vis, 97 * m + n_vis)
    vis = _vis(n_vis)
    ctx = absmod.Context(0)
    ctx.abs_simulate_vis(sky, dth, uv, vis)
    ctx.sync()
    _check(m, dth, sky, uv, vis)
    ctx.close()


@pytest.mark.parametrize("m,n_vis,failures", [(64, 100, 1), (65, 3000, 1), (65, 3000, 4), (130, 3000, 8)])
def test_without_room(m, n_vis, failures):
    """The partial sums' allocation fails `failures` times: a shorter slab does."""
    dth, sky, uv = _inputs(m, n_vis, m)
    vis = _vis(n_vis)
    ctx = absmod.Context(0)
    ctx.abs_simulate_vis(sky, dth, uv[:1], vis[:1])   # the weighted map has its room
    ctx.inject_alloc_failures(failures)
    ctx.abs_simulate_vis(sky, dth, uv, vis)
    ctx.sync()
    ctx.inject_alloc_failures(0)
    _check(m, dth, sky, uv, vis)
    ctx.close()


@pytest.mark.parametrize("m,warm,n_vis", [(64, 1, 300), (65, 300, 3000), (257, 20, 2049)])
def test_callers_capture_of_more_visibilities(m, warm, n_vis):
    dth, sky, uv = _inputs(m, n_vis, m + warm)
    vis = _vis(n_vis)
    st = torch.cuda.Stream("cuda:0")
    st.wait_stream(torch.cuda.default_stream("cuda:0"))
    with torch.cuda.stream(st):
        ctx = absmod.Context(0, st)
        ctx.abs_simulate_vis(sky, dth, uv[:warm], vis[:warm])
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            ctx.abs_simulate_vis(sky, dth, uv, vis)
        vis.fill_(float("nan"))
        graph.replay()
        _check(m, dth, sky, uv, vis)
    ctx.close()
