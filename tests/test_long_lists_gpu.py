"""Lists around the lengths at which the depth sort changes hands (a warp's
registers, a CTA's shared memory, chunks of 2,048 merged by several CTAs),
with depth keys and without: the forward matches the oracle bit for bit and
the opacity gradients within the parity tests' tolerance."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_backward, gpu_forward, grad_mismatch, upstream

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


def _scene(T):
    """T triangles that all cover the middle tile (24 x 24 pixels, tiles of 16 x 16)."""
    rng = np.random.default_rng(T)
    ang = rng.uniform(0, 2 * np.pi, (T, 1)) + np.array([0.0, 2.0, 4.0]) + rng.uniform(-0.3, 0.3, (T, 3))
    z = rng.uniform(-0.5, 0.5, (T, 1)) + rng.uniform(-0.1, 0.1, (T, 3))
    r = rng.uniform(2.5, 4.0, (T, 3))
    verts = np.stack([r * np.cos(ang), r * np.sin(ang), z], -1).astype(np.float32)
    tex = I.logits(T, 2, 4, rng)
    tex[..., 3] -= 4.0   # deep layers are reached
    return I.Scene(verts, tex, 2, [I.look_at([0.0, 0.0, 3.0], 24, 24)], I.mask_seeds(3, 1), 1, np.zeros(3, np.float32))


@pytest.mark.parametrize("bits", [-1, 3, 0])
@pytest.mark.parametrize("T", [128, 129, 256, 257, 2047, 2048, 2049, 4096, 4097, 7000])
def test_lists_of_every_length(ctx, T, bits):
    sc = _scene(T)
    ctx.set_tuning(depth_bits=bits)
    sid, got, (g, col, verts, tex) = gpu_forward(ctx, sc)
    pairs, tiles = ctx.plan_stats()
    assert tiles == 4 and pairs > 3 * T   # every list holds nearly all of them
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg)
    assert_forward_equal(got, ref)
    gc, sw = upstream(ref, 1)
    gt, _ = gpu_backward(ctx, sid, sc, 1, g, col, gc, sw, 2, verts, tex)
    gt_ref, _ = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, 1, ref, gc, sw, flags=2)
    assert not grad_mismatch(gt, gt_ref).any()


def test_few_long_lists_are_sorted_side_by_side(ctx):
    """200,000 triangles in a view of 16 tiles take no longer to sort than a few
    times what the same triangles take in a view of 1,024 tiles (sorted by
    two CTAs: more than ten times)."""
    import torch
    from paper_2603_27151_gb300 import native as N
    rng = np.random.default_rng(1)
    T = 200_000
    verts = torch.from_numpy(I.box_soup(T, 0.1, rng)).cuda()
    tex = torch.randn((T, 3, 4), device="cuda")
    ctx.set_tuning()
    sid = ctx.soup_upload(verts, tex, 1, borrow=True)
    ms = {}
    for px in (64, 512):
        cams = [I.look_at([0.0, 0.0, 3.0], px, px)]
        g, col, _ = N.alloc_outputs(cams, 1, 4, "cuda")
        for _ in range(5):   # the first one sizes the buffers
            ctx.profile_reset()
            ctx.profile(True)
            ctx.raster_forward(sid, cams, I.mask_seeds(3, 1), 1, 0, np.zeros(3, np.float32), g, col)
            torch.cuda.synchronize()
            ctx.profile(False)
            ms[px] = min(ms.get(px, 1e30), ctx.profile_read()["sort"][1])
    assert ms[64] < 4 * ms[512], ms
