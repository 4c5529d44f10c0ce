"""Triangles over many tiles, whose boxes a warp or a whole CTA walks, alone and
among small ones, more of them in a row than a CTA's list holds: the forward
matches the oracle bit for bit; and few large triangles keep the chip busy."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_forward

pytestmark = pytest.mark.gpu
W, H = 640, 512   # 1,280 tiles of 16 x 16


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_27151_gb300 import native as N
    c = N.Context(0)
    yield c
    c.set_tuning()
    c.close()


def _scene(T, wide, rng):
    """T small triangles but for those at `wide`, of up to the whole view."""
    verts = I.box_soup(T, 0.05, rng)
    n = len(wide)
    ang = rng.uniform(0, 2 * np.pi, (n, 1)) + np.array([0.0, 2.1, 4.2])
    r = rng.choice([0.5, 1.0, 4.0], (n, 1))
    verts[wide] = np.stack([r * np.cos(ang), rng.uniform(-0.5, 0.5, (n, 3)), r * np.sin(ang)], -1)
    tex = I.logits(T, 1, 4, rng)
    cams = [I.look_at([0.0, 3.0, 0.1], W, H), I.look_at([0.2, -3.0, 0.3], 333, 300)]
    return I.Scene(verts, tex, 1, cams, I.mask_seeds(3, 2), 1, np.zeros(3, np.float32))


@pytest.mark.parametrize("T,first,n,bits", [(1, 0, 1, -1), (40, 0, 40, 0), (2000, 900, 50, -1), (10000, 777, 150, 0)])
def test_forward(ctx, T, first, n, bits):
    sc = _scene(T, np.arange(first, first + n), np.random.default_rng(T))
    ctx.set_tuning(depth_bits=bits)
    _, got, _ = gpu_forward(ctx, sc)
    assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg))


@pytest.mark.parametrize("T,n,limit", [(500, 500, 1.0), (20000, 64, 2.5)])
def test_few_wide_triangles_do_not_wait_for_a_warp(ctx, T, n, limit):
    """Full-screen triangles at 1280 x 720: finding their tiles (3,600 each) takes
    less time than drawing them, or 2.5 times that for 64 in a row among
    small ones (one warp after the other: 1.4 and 4.6 times)."""
    import torch
    from paper_2603_27151_gb300 import native as N
    rng = np.random.default_rng(4)
    verts = I.box_soup(T, 0.05, rng)
    verts[:n] = I.box_soup(n, 8.0, rng, 0.5)
    tex = torch.randn((T, 3, 4), device="cuda")
    ctx.set_tuning()
    sid = ctx.soup_upload(torch.from_numpy(verts).cuda(), tex, 1)
    cams = [I.look_at([0.0, 0.0, 3.0], 1280, 720)]
    g, col, _ = N.alloc_outputs(cams, 1, 4, "cuda")
    ms = {}
    for _ in range(5):   # the first one sizes the buffers
        ctx.profile_reset()
        ctx.profile(True)
        ctx.raster_forward(sid, cams, I.mask_seeds(3, 1), 1, 0, np.zeros(3, np.float32), g, col)
        torch.cuda.synchronize()
        ctx.profile(False)
        ms = {k: min(ms.get(k, 1e30), v[1]) for k, v in ctx.profile_read().items()}
    assert ctx.plan_stats()[0] > 1000 * n
    assert ms["setup"] + ms["emit"] < limit * ms["raster_fwd"], ms
