"""Triangles around the sizes where the tile kernels change the arithmetic of
the covered fragment: |2 area| below and from 2^31 (in 1/256-pixel units), and
edge values beyond 2^38.  Visibility must match the oracle bit for bit, the
gradients within the parity tests' 1e-4."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_backward, gpu_forward, grad_mismatch, upstream

pytestmark = pytest.mark.gpu
W, H = 221, 203


def _scene():
    """Screen-space corners (pixels, depth): right triangles of w x h pixels
    with 2 area = 65536 w h just below, at and above 2^31 = 65536 * 32768, and
    triangles out to the guard band."""
    rng = np.random.default_rng(5)
    tri = []
    for k, (w, h) in enumerate([(180, 182), (128, 256), (182, 182), (200, 190), (16, 2048), (15, 2184)]):
        x, y, z = 3.0 * k, 2.0 * k, 1.0 + 0.05 * k
        tri.append([(x, y, z), (x + w, y, z), (x, y + h, z + 0.3)])
    for k, far in enumerate([16000.0, 15000.0, 9000.0]):
        z = 1.4 + 0.1 * k
        tri.append([(-far, -far + 50 * k, z), (far, -far, z + 0.2), (-0.2 * far, far, z + 0.1)])
    for _ in range(20):
        c = rng.uniform(0, 200, 2)
        tri.append([(*(c + rng.uniform(-40, 40, 2)), rng.uniform(0.9, 2.0)) for _ in range(3)])
    tri += [[a, c, b] for a, b, c in tri[:9]]   # the other screen orientation, a little behind
    t = np.array(tri)
    t[29:, :, 2] += 0.02
    cam = I.Camera(W, H, 64.0, 64.0, 0.0, 0.0, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    verts = np.stack([t[..., 0] * t[..., 2] / 64.0, t[..., 1] * t[..., 2] / 64.0, t[..., 2]], -1).astype(np.float32)
    s = np.round(t[..., :2] * 256).astype(np.int64)
    area = np.abs((s[:, 1, 0] - s[:, 0, 0]) * (s[:, 2, 1] - s[:, 0, 1]) - (s[:, 2, 0] - s[:, 0, 0]) * (s[:, 1, 1] - s[:, 0, 1]))
    assert (area[:9] < 2 ** 31).sum() >= 2 and (area[:9] >= 2 ** 31).sum() >= 4 and (area[6:9] > 2 ** 41).all()
    tex = I.logits(len(verts), 8, 4, rng)
    return I.Scene(verts, tex, 8, [cam], I.mask_seeds(9, 1), 1, np.zeros(3, np.float32))


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


@pytest.mark.parametrize("S,mode,tile,bits", [(1, 0, 16, -1), (2, 0, 16, -1), (4, 0, 8, 0), (1, 1, 32, 0), (1, 0, 8, 4)])
def test_forward_matches_oracle(ctx, S, mode, tile, bits):
    sc = _scene()
    ctx.set_tuning(tile_w=tile, depth_bits=bits)
    _, got, _ = gpu_forward(ctx, sc, S=S, mode=mode)
    ctx.set_tuning()
    assert_forward_equal(got, O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, S=S, mode=mode, bg=sc.bg))


@pytest.mark.parametrize("S", [1, 4])
def test_backward_matches_oracle(ctx, S):
    sc = _scene()
    sid, _, (g, col, verts, tex) = gpu_forward(ctx, sc, S=S)
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, S=S, bg=sc.bg)
    gc, sw = upstream(ref, S)
    gt, _ = gpu_backward(ctx, sid, sc, S, g, col, gc, sw, 3, verts, tex)   # texture and score terms
    gt_ref, _ = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, S, ref, gc, sw, flags=3)
    assert not grad_mismatch(gt, gt_ref).any()


@pytest.mark.parametrize("S", [1, 2, 4])
def test_edge_gradients_around_the_int32_limit(ctx, S):
    """Edge terms of triangles below and above the size up to which boundary
    tests run in int32 (edges of 63 pixels), with |2 area| around 2^30 and
    edges around 2^21 (in 1/256 pixels); two views."""
    rng = np.random.default_rng(11)
    tri = []
    for k, (w, h) in enumerate([(128, 127), (128, 128), (130, 128), (64, 256), (24, 8180), (24, 8200), (30, 40)]):
        x, y, z = 5.0 + 11.0 * k, -30.0 * (h > 1000) + 9.0 * k, 1.0 + 0.04 * k
        tri.append([(x, y, z), (x + w, y + 3, z + 0.1), (x + 4, y + h, z + 0.2)])
    tri += [[a, c, b] for a, b, c in tri]
    t = np.array(tri)
    t[7:, :, 2] += 0.03
    cams = [I.Camera(w, h, 64.0, 64.0, cx, 0.0, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
            for w, h, cx in ((150, 140, 0.0), (97, 61, 12.25))]
    verts = np.stack([t[..., 0] * t[..., 2] / 64.0, t[..., 1] * t[..., 2] / 64.0, t[..., 2]], -1).astype(np.float32)
    s = np.round(t[..., :2] * 256).astype(np.int64)
    area = np.abs((s[:, 1, 0] - s[:, 0, 0]) * (s[:, 2, 1] - s[:, 0, 1]) - (s[:, 2, 0] - s[:, 0, 0]) * (s[:, 1, 1] - s[:, 0, 1]))
    assert (area < 2 ** 30).any() and (area >= 2 ** 30).any()
    tex = I.logits(len(verts), 8, 4, rng)
    sc = I.Scene(verts, tex, 8, cams, I.mask_seeds(3, 2), 1, np.zeros(3, np.float32))
    sid, got, (g, col, vd, td) = gpu_forward(ctx, sc, S=S)
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, S=S, bg=sc.bg)
    assert_forward_equal(got, ref)
    gc, sw = upstream(ref, S)
    _, gv = gpu_backward(ctx, sid, sc, S, g, col, gc, sw, 8, vd, td)   # edge terms
    _, gv_ref = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, S, ref, gc, sw, flags=8)
    assert not grad_mismatch(gv, gv_ref).any()
