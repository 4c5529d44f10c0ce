"""The forward of one- and two-sample groups (a warp per 8 x 4 pixel block) at
the edges of its blocks and rounds: ragged views down to one pixel, every tile
shape, lists with more survivors than a round stages, both modes.  Bit for bit
against the oracle, fragment counts included."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_forward

pytestmark = pytest.mark.gpu
SIZES = [(1, 1), (7, 3), (9, 5), (33, 31), (70, 41)]


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
    c.close()


@pytest.mark.parametrize("tile,bits", [(8, 0), (16, -1), (32, 3)])
@pytest.mark.parametrize("S", [1, 2])
@pytest.mark.parametrize("T,C,mode", [(12, 5, 0), (500, 4, 0), (90, 16, 1)])
def test_forward_blocks(ctx, tile, bits, S, T, C, mode):
    rng = np.random.default_rng(T)
    verts = (rng.uniform(-0.2, 0.2, (T, 1, 3)) + rng.uniform(-0.7, 0.7, (T, 3, 3))).astype(np.float32)
    tex = I.logits(T, 3, C, rng)
    tex[..., -1] -= 1.5   # deep layers are reached
    cams = [I.look_at(e, w, h) for e, (w, h) in zip(I.sphere_eyes(len(SIZES), 3.0, rng), SIZES)]
    sc = I.Scene(verts, tex, 3, cams, I.mask_seeds(8, len(SIZES)), 1, np.linspace(0.1, 0.9, C - 1).astype(np.float32))
    ctx.set_tuning(tile_w=tile, depth_bits=bits)
    _, got, _ = gpu_forward(ctx, sc, S=S, mode=mode)
    ctx.set_tuning()
    assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, S=S, mode=mode, bg=sc.bg))
