"""The marching L1 + SSIM kernel at every segment length (2 to 9 steps of 16
rows): views whose last segment is one row, one short of full and full, with
widths around the strips of 118 columns, in calls that the dispatch gives to
the march (its rule is restated here).  Against the oracle (tolerances as in
the other loss tests), and bit for bit against the tile kernel, which takes the
same views alone."""
import numpy as np
import pytest

from tests.test_ssim_gpu import _check, dev  # noqa: F401

pytestmark = pytest.mark.gpu
STRIP, TILE_W, TILE_H = 118, 64, 16


def _rows(steps):
    return 16 * steps - 20


def _route(sizes, S, sms):
    """The march's steps per segment, or 0 for the tile kernel."""
    best, steps = 1e300, 0
    for k in range(2, 10):
        ctas = sum(S * -(-w // STRIP) * -(-h // _rows(k)) for w, h in sizes)
        cost = -(-ctas // sms) * (k + 0.5)
        if cost < best:
            best, steps = cost, k
    tiles = sum(S * -(-w // TILE_W) * -(-h // TILE_H) for w, h in sizes)
    left = tiles % (2 * sms)
    return 0 if 2.3 * (tiles // (2 * sms)) + (0 if left == 0 else 1.6 if left <= sms else 2.6) <= best else steps


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def _call(c, t, scale, grads=True, sws=True):
    import torch
    from paper_2603_27151_gb300 import native as N
    g = [torch.full_like(x, 7.0) for x in c] if grads else None
    sw = [torch.full((x.shape[0], x.shape[2], x.shape[3]), 7.0, device="cuda") for x in c] if sws else None
    loss = torch.zeros(1, device="cuda")
    N.loss_l1_ssim(c, t, g, sw, loss, scale=scale)
    torch.cuda.synchronize()
    return g, sw, float(loss)


def _sizes(steps, S):
    """Views to look at, and as many full ones beside them as make the call march
    with `steps` steps."""
    r = _rows(steps)
    look = [(117, 1), (118, r - 1), (119, r), (1, r + 1), (236, r + 1), (237, 2 * r - 1), (235, 2 * r)]
    for n in range(1, 58):
        for w in (237, 118, 354):
            sizes = look + [(w, r)] * n
            if _route(sizes, S, _sms()) == steps:
                return look, sizes
    raise AssertionError("no call of %d steps" % steps)


@pytest.mark.parametrize("steps", range(2, 10))
def test_every_segment_length(dev, steps):  # noqa: F811
    import torch
    S, Co, scale = 2, 3, 0.5
    look, sizes = _sizes(steps, S)
    gen = torch.Generator(device="cuda").manual_seed(steps)
    c = [torch.rand((S, Co, h, w), device="cuda", generator=gen) for w, h in sizes]
    t = [torch.rand((Co, h, w), device="cuda", generator=gen) for w, h in sizes]
    g, sw, loss = _call(c, t, scale)
    host = lambda xs: [x.cpu().numpy() for x in xs[:len(look)]]
    _check(host(g), host(sw), host(c), host(t), scale)
    assert abs(loss - sum(float(x.double().sum()) for x in sw)) <= 1e-4 * abs(loss)
    for v, size in enumerate(look):
        assert _route([size], S, _sms()) == 0
        g1, sw1, _ = _call([c[v]], [t[v]], scale)
        assert torch.equal(g1[0], g[v]) and torch.equal(sw1[0], sw[v]), size


@pytest.mark.parametrize("grads,sws", [(False, False), (True, False), (False, True)])
def test_outputs_left_out(dev, grads, sws):  # noqa: F811
    """NULL gradients or score weights: the others and the loss are the same."""
    import torch
    S, n = 2, 6
    assert _route([(250, 331)] * n, S, _sms()) > 0
    gen = torch.Generator(device="cuda").manual_seed(1)
    c = [torch.rand((S, 3, 331, 250), generator=gen, device="cuda") for _ in range(n)]
    t = [torch.rand((3, 331, 250), generator=gen, device="cuda") for _ in range(n)]
    g, sw, loss = _call(c, t, 0.5)
    g1, sw1, loss1 = _call(c, t, 0.5, grads, sws)
    assert abs(loss1 - loss) <= 1e-5 * abs(loss)
    assert not grads or all(torch.equal(a, b) for a, b in zip(g, g1))
    assert not sws or all(torch.equal(a, b) for a, b in zip(sw, sw1))
