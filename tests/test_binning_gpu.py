"""Binning: tile lists of every length class of the depth sort (a warp's
registers, shared memory, passes in global memory), boxes above and below the
size that a warp shares, with and without depth bits.  The forward must match
the oracle bit for bit whatever the lists' order."""
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
    c.close()


def _scene(T, seed=0):
    """T triangles around the middle of two views (9 and 130 tiles of 16 x 16)."""
    rng = np.random.default_rng(seed)
    c = rng.uniform(-0.12, 0.12, (T, 1, 3))
    verts = (c + rng.uniform(-0.35, 0.35, (T, 3, 3))).astype(np.float32)
    verts[: max(1, T // 50)] *= 4.0   # some cover most of the view
    tex = I.logits(T, 2, 4, rng)
    tex[..., 3] -= 1.0
    cams = [I.look_at([0.0, 0.0, 3.0], 48, 40), I.look_at([1.5, 2.0, 1.5], 200, 150)]
    return I.Scene(verts, tex, 2, cams, I.mask_seeds(3, 2), 1, np.zeros(3, np.float32))


@pytest.mark.parametrize("bits", [-1, 5, 0])
@pytest.mark.parametrize("T", [1, 31, 33, 64, 65, 128, 200, 1500, 4000])
def test_forward_lists(ctx, T, bits):
    sc = _scene(T, T)
    ctx.set_tuning(depth_bits=bits)
    _, got, _ = gpu_forward(ctx, sc)
    ctx.set_tuning()
    assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg))


def test_lists_grow_and_shrink(ctx):
    """Calls of different sizes on one context: the lists built with the
    buffers of the call before are built again when those are too small."""
    from paper_2603_27151_gb300 import native as N
    c = N.Context(0)
    for T in (3, 700, 40, 2500, 5):
        sc = _scene(T, 7)
        _, got, _ = gpu_forward(c, sc)
        assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg))
    c.close()


def test_many_tiles(ctx):
    """More tiles than one block of the scan holds (4,096): 64 views."""
    rng = np.random.default_rng(2)
    verts, tex = I.box_soup(50, 0.5, rng), I.logits(50, 2, 4, rng)
    eyes = I.sphere_eyes(64, 3.0, rng)
    sc = I.Scene(verts, tex, 2, [I.look_at(e, 170, 150) for e in eyes], I.mask_seeds(4, 64), 1, np.zeros(3, np.float32))
    _, got, _ = gpu_forward(ctx, sc)
    views = [0, 1, 37, 62, 63]
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, [sc.cams[v] for v in views], sc.seeds[views], bg=sc.bg)
    assert_forward_equal([got[v] for v in views], ref)
