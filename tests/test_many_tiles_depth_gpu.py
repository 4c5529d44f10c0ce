"""The depth key's bits do not depend on the number of tiles: a view within a
call of more than 65,536 tiles has the lists that it has by itself, and with
them the groups in which the opacity terms are summed in FP32 (see
test_list_order_gpu.py for the share of entries that may differ)."""
import numpy as np
import pytest

from paper_2603_27151_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_view_among_many_tiles():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_27151_gb300 import native as N
    T, W, H, n, view = 3000, 528, 512, 64, 41   # 33 x 32 tiles a view, 67,584 in all
    rng = np.random.default_rng(3)
    verts = torch.from_numpy((rng.uniform(-0.3, 0.3, (T, 1, 3)) + rng.uniform(-0.1, 0.1, (T, 3, 3))).astype(np.float32)).cuda()
    tex = torch.from_numpy(I.logits(T, 2, 4, rng)).cuda() - 2.0
    cams = [I.look_at(e, W, H) for e in I.sphere_eyes(n, 3.0, rng)]
    seeds = I.mask_seeds(5, n)
    gen = torch.Generator(device="cuda").manual_seed(1)
    sw = torch.rand((1, H, W), device="cuda", generator=gen) + 0.1
    ctx = N.Context(0)
    sid = ctx.soup_upload(verts, tex, 2)
    grads, outs = [], []
    for pick in (list(range(n)), [view]):
        cc, ss = [cams[k] for k in pick], seeds[pick]
        g, col, _ = N.alloc_outputs(cc, 1, 4, "cuda")
        ctx.raster_forward(sid, cc, ss, 1, 0, np.zeros(3, np.float32), g, col)
        assert ctx.plan_stats()[1] == 1056 * len(pick)
        sws = [sw if k == view else torch.zeros_like(sw) for k in pick]
        gt, gv = torch.zeros_like(tex), torch.zeros_like(verts)
        ctx.raster_backward(sid, cc, 1, g, col, [torch.zeros_like(c) for c in col], sws, N.DS_G_SCORE, gv, gt)
        torch.cuda.synchronize()
        grads.append(gt.cpu().numpy())
        outs.append((g[pick.index(view)].cpu().numpy(), col[pick.index(view)].cpu().numpy()))
        del g, col
    assert np.array_equal(outs[0][0], outs[1][0]) and np.array_equal(outs[0][1], outs[1][1])
    differ = grads[0] != grads[1]
    assert np.abs(grads[1]).max() > 0 and differ.mean() <= 1e-4, "%d of %d entries differ" % (differ.sum(), differ.size)
    ctx.close()
