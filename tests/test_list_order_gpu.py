"""Every tile's list has one order, by (depth key, triangle), with and without
depth bits and at every list length: the opacity gradients, whose terms are
summed in FP32 over neighbouring list entries, come out the same in repeated
calls.

What may differ is the order of the FP64 atomics: a gradient of n addends moves
by at most n 2^-53 of their magnitudes, which reaches the rounding to FP32
(2^-24) for about one entry in 2^29 / n; n stays below 2^14 here, so fewer than
1e-4 of the entries, by one FP32 spacing.  Regrouped FP32 sums move most of
the entries that have more than a few terms."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I
from tests.gpu_helpers import gpu_backward, gpu_forward, grad_mismatch, upstream

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
    """T triangles, most of them over the same few tiles of two views."""
    rng = np.random.default_rng(T)
    c = rng.uniform(-0.1, 0.1, (T, 1, 3))
    verts = (c + rng.uniform(-0.4, 0.4, (T, 3, 3))).astype(np.float32)
    tex = I.logits(T, 2, 4, rng)
    tex[..., 3] -= 2.0
    cams = [I.look_at([0.0, 0.0, 3.0], 48, 40), I.look_at([1.5, 2.0, 1.5], 72, 56)]
    return I.Scene(verts, tex, 2, cams, I.mask_seeds(3, 2), 1, np.zeros(3, np.float32))


@pytest.mark.parametrize("S", [1, 4])
@pytest.mark.parametrize("T,bits", [(60, 0), (200, 0), (1200, 0), (4000, 0), (4000, 2), (4000, -1)])
def test_score_gradients_repeat(ctx, T, bits, S):
    sc = _scene(T)
    ctx.set_tuning(depth_bits=bits)
    ref = None
    for _ in range(4):
        sid, got, (g, col, verts, tex) = gpu_forward(ctx, sc, S=S, n_front=False)
        if ref is None:
            gc, sw = upstream(got, S)
        gt, _ = gpu_backward(ctx, sid, sc, S, g, col, gc, sw, 2, verts, tex)   # score terms alone
        if ref is None:
            ref = gt
            continue
        differ = gt != ref
        assert differ.mean() <= 1e-4, "%d of %d entries differ" % (differ.sum(), differ.size)
        assert np.all(np.abs(gt - ref) <= np.spacing(np.abs(ref)))


@pytest.mark.parametrize("bits", [0, 2, -1])
def test_score_gradients_of_long_lists_match_the_oracle(ctx, bits):
    """Lists of about 3,000 triangles, with many equal depth keys at two bits."""
    sc = _scene(4000)
    ctx.set_tuning(depth_bits=bits)
    sid, _, (g, col, verts, tex) = gpu_forward(ctx, sc)
    ref = O.forward(sc.verts, sc.tex, sc.grid_n, sc.cams, sc.seeds, bg=sc.bg)
    gc, sw = upstream(ref, 1)
    gt, _ = gpu_backward(ctx, sid, sc, 1, g, col, gc, sw, 2, verts, tex)
    gt_ref, _ = O.backward(sc.verts, sc.tex, sc.grid_n, sc.cams, 1, ref, gc, sw, flags=2)
    assert not grad_mismatch(gt, gt_ref).any()
