"""Ensembles whose realisations run on several streams: every realisation against an estimate of its own, for
fewer and more realisations than streams, on the first call, the captured one and its replay with other
visibilities, and in a caller's own capture before and after the streams have their workspaces."""
import numpy as np
import pytest

import paper_2412_02246_gb300 as absmod
from paper_2412_02246_gb300 import build as absbuild

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# the same kernels on the same inputs; only the order of the FP64 atomics of the accumulators differs, which
# can move an FP32 rounding of a transform's input by one unit (6e-8)
TOL = 1e-6


def _setup(precision, n=96, n_vis=20_000):
    absbuild.build()
    dev = torch.device("cuda:0")
    st = torch.cuda.Stream(dev)
    edges = 2 * np.pi * np.linspace(2.0, 0.4 * n, 9)
    cfg = absmod.Config(n_grid=n, du=1.0, ell_edges=edges,
                        precision=absmod.ABS_SPLIT_BF16 if precision == "split" else absmod.ABS_FP32)
    g = torch.Generator(device=dev).manual_seed(7)
    uv = (torch.rand((n_vis, 2), generator=g, device=dev) - 0.5) * 0.9 * n
    ctx, one = absmod.Context(0, st), absmod.Context(0, st)
    for c in (ctx, one):
        c.autotune(False)
    return dev, st, cfg, g, uv, ctx, one, absmod.abs_triplets(cfg).shape[0]


def _fill(vis, g):
    vis.copy_(torch.randn(vis.shape, generator=g, device=vis.device))


def _each(one, cfg, uv, vis, nt):
    B = torch.empty((vis.shape[0], nt), dtype=torch.float64, device=uv.device)
    T = torch.empty(nt, dtype=torch.int64, device=uv.device)
    E = torch.empty(cfg.n_bins, dtype=torch.float64, device=uv.device)
    for r in range(vis.shape[0]):
        one.abs_estimate(cfg, uv, vis[r].contiguous(), nt, None, B[r], T, E)
    return B, T, E


def _close(got, ref):
    torch.cuda.synchronize()
    for r in range(ref[0].shape[0]):
        a, b = got[0][r].cpu().numpy(), ref[0][r].cpu().numpy()
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.linalg.norm(np.nan_to_num(a - b)) <= TOL * np.linalg.norm(np.nan_to_num(b))
    assert torch.equal(got[1], ref[1])
    np.testing.assert_allclose(got[2].cpu().numpy(), ref[2].cpu().numpy(), rtol=1e-12)


def _out(n_real, nt, cfg, dev):
    return (torch.full((n_real, nt), float("nan"), dtype=torch.float64, device=dev),
            torch.zeros(nt, dtype=torch.int64, device=dev),
            torch.zeros(cfg.n_bins, dtype=torch.float64, device=dev))


@pytest.mark.parametrize("precision", ["fp32", "split"])
@pytest.mark.parametrize("n_real", [2, 5, 6, 11])
def test_every_realisation(precision, n_real):
    dev, st, cfg, g, uv, ctx, one, nt = _setup(precision)
    with torch.cuda.stream(st):
        vis = torch.empty((n_real, uv.shape[0], 2), device=dev)
        out = _out(n_real, nt, cfg, dev)
        st.wait_stream(torch.cuda.default_stream(dev))
        for _ in range(4):
            _fill(vis, g)
            ctx.abs_estimate_many(cfg, uv, vis, nt, None, *out)
            _close(out, _each(one, cfg, uv, vis, nt))
    ctx.close()
    one.close()


@pytest.mark.parametrize("warm", [1, 6])
def test_callers_capture(warm):
    n_real = 6
    dev, st, cfg, g, uv, ctx, one, nt = _setup("fp32")
    with torch.cuda.stream(st):
        vis = torch.empty((n_real, uv.shape[0], 2), device=dev)
        first, out = _out(n_real, nt, cfg, dev), _out(n_real, nt, cfg, dev)
        st.wait_stream(torch.cuda.default_stream(dev))
        _fill(vis, g)
        ctx.abs_estimate_many(cfg, uv, vis[:warm], nt, None, first[0][:warm], *first[1:])
        st.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=st):
            ctx.abs_estimate_many(cfg, uv, vis, nt, None, *out)
        _fill(vis, g)
        graph.replay()
        _close(out, _each(one, cfg, uv, vis, nt))
    ctx.close()
    one.close()
