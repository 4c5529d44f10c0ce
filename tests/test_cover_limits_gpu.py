"""Boundary tests in 32 bits: triangles whose longest edge is just below, at and
above the 63 pixels up to which they run in 32 bits, the first vertex in the
cells of 64 x 64 pixels left of and above the view, on cell borders and far
from the triangle's other corners, so that covered pixels lie at the far edges
of the nine cells around it.

The depth of a pixel's winner, taken again in the backward, decides which
fragments lie in front: the score terms match the oracle as closely as in the
parity tests (visibility is exact).  The boundary terms compare in FP32 what
the oracle compares in FP64, so that a pair in a hundred thousand may fall on
the other side of an edge; such a pair is one of the 60 or more along its
triangle's boundary.  Three triangles may be off by up to 2% of their largest
gradient, every other by the parity tests' 1e-4."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import assert_forward_equal, gpu_backward, gpu_forward, grad_mismatch, upstream

W, H, F = 200, 180, 64.0
LIMIT = 63 * 256


def _scene():
    """(scene, snapped corners [T, 3, 2] in 1/256 pixel)."""
    rng = np.random.default_rng(63)
    tri = []
    for k in range(96):
        ext = (62.0, 62.99, 63.0, 63.01, 64.0, 65.5)[k % 6]      # longest extent, along x or y
        other = rng.uniform(20.0, 62.0)
        w, h = (ext, other) if (k // 6) % 2 == 0 else (other, ext)
        # the first corner, on either side of the cell borders and outside the view
        x = rng.choice([-60.0, -33.0, -0.5, 0.5, 63.9, 64.1, 127.9, 128.1]) + rng.uniform(-0.2, 0.2)
        y = rng.choice([-60.0, -17.0, -0.4, 0.6, 63.8, 64.2, 127.8, 128.2]) + rng.uniform(-0.2, 0.2)
        sx = 1.0 if x < 40 else rng.choice([-1.0, 1.0])          # the triangle reaches right or left, down or up
        sy = 1.0 if y < 40 else rng.choice([-1.0, 1.0])
        z = rng.uniform(0.9, 1.6)
        c = [(x, y, z), (x + sx * w, y + sy * rng.uniform(0.1, 0.4) * h, z + rng.uniform(0, 0.2)),
             (x + sx * rng.uniform(0.0, 0.5) * w, y + sy * h, z + rng.uniform(0, 0.2))]
        tri.append(c if rng.random() < 0.5 else [c[0], c[2], c[1]])
    t = np.array(tri)
    verts = np.stack([t[..., 0] * t[..., 2] / F, t[..., 1] * t[..., 2] / F, t[..., 2]], -1).astype(np.float32)
    snap = np.round((verts[..., :2].astype(np.float64) / verts[..., 2:] * F) * 256).astype(np.int64)
    cam = I.Camera(W, H, F, F, 0.0, 0.0, np.eye(3, dtype=np.float32), np.zeros(3, np.float32))
    tex = I.logits(len(verts), 8, 4, rng)
    return I.Scene(verts, tex, 8, [cam], I.mask_seeds(9, 1), 1, np.zeros(3, np.float32)), snap


def test_scene_reaches_the_limits():
    sc, s = _scene()
    longest = np.abs(s - np.roll(s, 1, 1)).max((1, 2))
    near = np.abs(longest - LIMIT) <= 8
    assert ((longest <= LIMIT) & near).sum() >= 3 and ((longest > LIMIT) & near).sum() >= 3
    assert (longest < LIMIT - 100).sum() >= 10 and (longest > LIMIT + 100).sum() >= 20
    small = longest <= LIMIT
    cell = s[:, 0] >> 14
    assert (small & (cell[:, 0] < 0)).sum() >= 8 and (small & (cell[:, 1] < 0)).sum() >= 8
    # corners (and with them covered pixels) in the cells on both sides of the first corner's
    for axis in (0, 1):
        reach = (s[..., axis] >> 14) - cell[:, None, axis]
        assert (small & (reach.max(1) == 1)).sum() >= 5 and (small & (reach.min(1) == -1)).sum() >= 3
        assert small[np.abs(reach).max(1) > 1].sum() == 0


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


@pytest.mark.gpu
@pytest.mark.parametrize("S", [1, 2, 4])
def test_score_and_boundary_terms(ctx, S):
    sc, _ = _scene()
    sid, got, (g, col, verts, tex) = gpu_forward(ctx, sc, S=S)
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, S=S, bg=sc.bg)
    assert_forward_equal(got, ref)
    gc, sw = upstream(ref, S)
    gt, _ = gpu_backward(ctx, sid, sc, S, g, col, gc, sw, 2, verts, tex)   # score terms
    gt_ref, _ = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, S, ref, gc, sw, flags=2)
    assert not grad_mismatch(gt, gt_ref).any()
    _, gv = gpu_backward(ctx, sid, sc, S, g, col, gc, sw, 8, verts, tex)   # boundary terms
    _, gv_ref = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, S, ref, gc, sw, flags=8)
    off = grad_mismatch(gv, gv_ref).reshape(sc.T, -1).any(1)
    err = np.abs(gv - gv_ref).reshape(sc.T, -1).max(1) / np.abs(gv_ref).reshape(sc.T, -1).max(1).clip(1e-30)
    assert off.sum() <= 3 and np.all(err[off] <= 0.02), (np.flatnonzero(off), err[off])
