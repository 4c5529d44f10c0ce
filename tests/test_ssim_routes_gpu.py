"""The L1 + SSIM loss of many images that are low or narrow against the strips
and segments of the marching kernel: values against the oracle (tolerances as
in the other loss tests), and a time in proportion to the pixels."""
import numpy as np
import pytest

from tests.test_ssim_gpu import _check, _run, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h,n", [(512, 16, 64), (1, 700, 64), (40, 515, 30), (125, 33, 64), (192, 33, 64), (320, 17, 40)])
def test_values(dev, w, h, n):  # noqa: F811
    rng = np.random.default_rng(w + h)
    colors = [rng.uniform(0, 1, (1, 3, h, w)) for _ in range(n)]
    targets = [rng.uniform(0, 1, (3, h, w)) for _ in range(n)]
    g, sw, loss = _run(colors, targets, 0.5)
    pick = lambda a: [a[0], a[n // 2], a[-1]]
    _check(pick(g), pick(sw), pick(colors), pick(targets), 0.5)
    assert abs(loss - sum(float(x.astype(np.float64).sum()) for x in sw)) <= 1e-4 * abs(loss)


def test_low_images_cost_their_pixels(dev):  # noqa: F811
    """64 images of 1920 x 16 take at most 1.4 times as long as one of 1920 x 1080,
    which has as many pixels (strips and segments for the low ones: 1.7)."""
    import torch
    from paper_2603_27151_gb300 import native as N
    us = {}
    for w, h, n in ((1920, 16, 64), (1920, 1080, 1)):
        c = [torch.rand((1, 3, h, w), device="cuda") for _ in range(n)]
        t = [torch.rand((3, h, w), device="cuda") for _ in range(n)]
        g, sw = [torch.empty_like(x) for x in c], [torch.empty((1, h, w), device="cuda") for _ in range(n)]
        loss = torch.zeros(1, device="cuda")
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            N.loss_l1_ssim(c, t, g, sw, loss)
            s.synchronize()
            graph = torch.cuda.CUDAGraph()   # the device's time without the host's
            graph.capture_begin()
            for _ in range(5):
                N.loss_l1_ssim(c, t, g, sw, loss)
            graph.capture_end()
            best = 1e30
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(s)
                graph.replay()
                b.record(s)
                s.synchronize()
                best = min(best, a.elapsed_time(b) * 200)
        us[n] = best
    assert us[64] < 1.4 * us[1], us
