"""Long lists without a host wait: captured in a graph, with buffers that are too
small, and after a call that a capture refuses."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_forward

pytestmark = pytest.mark.gpu


def _scene():
    rng = np.random.default_rng(2)
    T = 5000   # lists of up to about 5,000 triangles
    verts = (rng.uniform(-0.1, 0.1, (T, 1, 3)) + rng.uniform(-0.5, 0.5, (T, 3, 3))).astype(np.float32)
    tex = I.logits(T, 2, 4, rng)
    tex[..., 3] -= 2.0
    sc = I.Scene(verts, tex, 2, [I.look_at([0.0, 0.0, 2.0], 45, 40)], I.mask_seeds(3, 1), 1, np.zeros(3, np.float32))
    return sc, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg)


@pytest.fixture(scope="module")
def scene():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    return _scene()


def _result(N, g, col):
    tri, bary, depth = N.split_gbuf(g[0])
    return [dict(tri_id=tri.cpu().numpy(), bary=bary.cpu().numpy(), depth=depth.cpu().numpy(), color=col[0].cpu().numpy(),
                 n_front=None)]


def test_captured(scene):
    import torch
    from paper_2603_27151_gb300 import native as N
    sc, ref = scene
    ctx = N.Context(0)
    sid, _, _ = gpu_forward(ctx, sc)
    pairs, _ = ctx.plan_stats()
    ctx.reserve(2 * pairs)
    g, col, _ = N.alloc_outputs(sc.cams, 1, 4, "cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        ctx.raster_forward(sid, sc.cams, sc.seeds, 1, N.DS_NO_SYNC, sc.bg, g, col)
        graph.capture_end()
        for _ in range(3):
            g[0].fill_(-7)
            graph.replay()
            s.synchronize()
            assert_forward_equal(_result(N, g, col), ref)
    ctx.status()
    ctx.close()


@pytest.mark.parametrize("pairs", [100, 2500, 9000])
def test_buffers_too_small(scene, pairs):
    import torch
    from paper_2603_27151_gb300 import native as N
    sc, ref = scene
    ctx = N.Context(0)
    ctx.reserve(pairs)
    sid = ctx.soup_upload(torch.from_numpy(sc.verts).cuda(), torch.from_numpy(sc.tex).cuda(), sc.grid_n)
    g, col, _ = N.alloc_outputs(sc.cams, 1, 4, "cuda")
    ctx.raster_forward(sid, sc.cams, sc.seeds, 1, N.DS_NO_SYNC, sc.bg, g, col)
    torch.cuda.synchronize()
    with pytest.raises(N.DsError):
        ctx.status()
    ctx.raster_forward(sid, sc.cams, sc.seeds, 1, 0, sc.bg, g, col)
    torch.cuda.synchronize()
    assert ctx.plan_stats()[0] > 1.25 * pairs + 64
    assert_forward_equal(_result(N, g, col), ref)
    ctx.close()


def test_without_allocation(scene):
    """The allocation-free forward on the same lists, twice on its scratch."""
    import torch
    from paper_2603_27151_gb300 import native as N
    sc, ref = scene
    v, t = torch.from_numpy(sc.verts).cuda(), torch.from_numpy(sc.tex).cuda()
    g, col, _ = N.alloc_outputs(sc.cams, 1, 4, "cuda")
    for _ in range(2):
        g[0].fill_(-7)
        N.raster_forward_noalloc(v, t, sc.grid_n, sc.cams, sc.seeds, 1, 0, sc.bg, g, col)
        torch.cuda.synchronize()
        assert_forward_equal(_result(N, g, col), ref)


def _refused_capture():
    import torch
    from paper_2603_27151_gb300 import native as N
    sc, ref = _scene()
    ctx = N.Context(0)
    sid, _, _ = gpu_forward(ctx, sc)
    g, col, _ = N.alloc_outputs(sc.cams, 1, 4, "cuda")
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        graph = torch.cuda.CUDAGraph()
        graph.capture_begin()
        with pytest.raises(N.DsError):
            ctx.raster_forward(sid, sc.cams, sc.seeds, 1, 0, sc.bg, g, col)
        with pytest.raises(RuntimeError):
            graph.capture_end()
    torch.cuda.synchronize()
    ctx.raster_forward(sid, sc.cams, sc.seeds, 1, 0, sc.bg, g, col)
    torch.cuda.synchronize()
    assert_forward_equal(_result(N, g, col), ref)
    ctx.close()


def test_waiting_call_is_refused_under_capture(scene):
    """A call that waits for the host ends the capture with an error, and the
    context goes on.  In a process of its own: torch's random generators stay in
    the state of the failed capture."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = "from tests.test_lists_capture_gpu import _refused_capture as f; f()"
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
