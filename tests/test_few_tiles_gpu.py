"""Binning with few tiles, whose counters are split: views of 1,023 to 1,025
tiles match the oracle bit for bit, and many triangles on few tiles are counted
and emitted as fast as on many."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_forward

pytestmark = pytest.mark.gpu


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


@pytest.mark.parametrize("cols,rows", [(33, 31), (32, 32), (41, 25)])
def test_forward_around_the_split(ctx, cols, rows):
    rng = np.random.default_rng(cols)
    T = 2500
    verts, tex = I.box_soup(T, 0.1, rng), I.logits(T, 1, 4, rng)
    sc = I.Scene(verts, tex, 1, [I.look_at([0.5, 0.4, 2.5], 16 * cols, 16 * rows - 3)], I.mask_seeds(3, 1), 1,
                 np.zeros(3, np.float32))
    ctx.set_tuning()
    _, got, _ = gpu_forward(ctx, sc)
    assert ctx.plan_stats()[1] == cols * rows
    assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg))


def test_few_tiles_are_not_waited_for(ctx):
    """200,000 triangles: set-up and emission in a view of 256 tiles take at most
    1.2 times what they take in one of 8,160 (one counter per tile, side by
    side: twice)."""
    import torch
    from paper_2603_27151_gb300 import native as N
    T = 200_000
    verts = torch.from_numpy(I.box_soup(T, 0.02, np.random.default_rng(1))).cuda()
    tex = torch.randn((T, 3, 4), device="cuda")
    ctx.set_tuning()
    sid = ctx.soup_upload(verts, tex, 1, borrow=True)
    ms = {}
    for w, h in ((256, 256), (1920, 1080)):
        cams = [I.look_at([0.0, 0.0, 3.0], w, h)]
        g, col, _ = N.alloc_outputs(cams, 1, 4, "cuda")
        for _ in range(6):   # the first one sizes the buffers
            ctx.profile_reset()
            ctx.profile(True)
            ctx.raster_forward(sid, cams, I.mask_seeds(3, 1), 1, 0, np.zeros(3, np.float32), g, col)
            torch.cuda.synchronize()
            ctx.profile(False)
            st = ctx.profile_read()
            ms[w] = min(ms.get(w, 1e30), st["setup"][1] + st["emit"][1])
    assert ms[256] < 1.2 * ms[1920], ms
