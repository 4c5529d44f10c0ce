"""The autotuner times staging chunks only for calls that stage by them: forwards
of one and two samples alone do not."""
import numpy as np
import pytest

from paper_2603_27151_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,candidates", [(1, 6), (2, 6), (4, 9)])
def test_forward_alone(S, candidates):
    """The tuning at the start (the first tile width, no candidate chunk), `candidates`
    others, then the chosen one once more; two runs each."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_27151_gb300 import native as N
    sc = I.plain_small()
    ctx = N.Context(0)
    sid = ctx.soup_upload(torch.from_numpy(sc.verts).cuda(), torch.from_numpy(sc.tex).cuda(), sc.grid_n)
    g, col, _ = N.alloc_outputs(sc.cams, S, sc.C, "cuda")
    ctx.set_tuning(tile_w=8, chunk=96)
    ctx.raster_forward(sid, sc.cams, sc.seeds, S, 0, sc.bg, g, col)
    n0 = N.kernel_launches()
    ctx.raster_forward(sid, sc.cams, sc.seeds, S, 0, sc.bg, g, col)
    n1 = N.kernel_launches()
    best, _ = ctx.autotune(sid, sc.cams, sc.seeds, S, 0, np.zeros(3, np.float32), g, col, reps=1)
    torch.cuda.synchronize()
    assert N.kernel_launches() - n1 == (n1 - n0) * 2 * (1 + candidates + 1)
    assert S == 4 or best["chunk"] == 96
    ctx.close()
