"""The profiler's stages keep their names and indices."""
import numpy as np
import pytest

from paper_2603_27151_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_stage_names():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_27151_gb300 import native as N
    sc = I.plain_small()
    ctx = N.Context(0)
    sid = ctx.soup_upload(torch.from_numpy(sc.verts).cuda(), torch.from_numpy(sc.tex).cuda(), sc.grid_n)
    g, col, _ = N.alloc_outputs(sc.cams, 1, sc.C, "cuda")
    ctx.profile(True)
    ctx.raster_forward(sid, sc.cams, sc.seeds, 1, 0, np.zeros(3, np.float32), g, col)
    ctx.profile(False)
    st = ctx.profile_read()
    assert list(st) == ["activate", "setup", "scan", "emit", "sort", "ranges", "raster_fwd", "count", "geom",
                        "raster_bwd", "edge_bwd", "finish", "train"]
    ran = [k for k, (n, ms) in st.items() if n]
    assert ran == ["activate", "setup", "scan", "emit", "sort", "raster_fwd"] and all(st[k][1] > 0 for k in ran)
    ctx.close()
