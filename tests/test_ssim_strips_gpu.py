"""The marching L1 + SSIM kernel at the edges of its strips (118 columns) and
segments (16 n - 20 rows): images one pixel below, at and above them, thinner
than the window, and calls large enough for every segment length.  Tolerances
as in the other loss tests."""
import numpy as np
import pytest

from tests.test_ssim_gpu import _check, _run, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 20, 150])   # views: more of them, longer segments
@pytest.mark.parametrize("w,h", [(117, 11), (118, 12), (119, 13), (1, 1), (3, 140), (236, 28), (237, 29), (128, 125)])
def test_strips(dev, n, w, h):  # noqa: F811
    n = min(n, 64)
    rng = np.random.default_rng(w * 1000 + h)
    S = 3 if n > 20 else 1
    colors = [rng.uniform(0, 1, (S, 2, h, w)) for _ in range(n)]
    targets = [rng.uniform(0, 1, (2, h, w)) for _ in range(n)]
    g, sw, loss = _run(colors, targets, 0.5)
    keep = [0, n - 1] if n > 1 else [0]
    pick = lambda a: [a[k] for k in keep]
    _check(pick(g), pick(sw), pick(colors), pick(targets), 0.5)
    assert abs(loss - sum(float(x.astype(np.float64).sum()) for x in sw)) <= 1e-4 * abs(loss)


def test_no_outputs_but_loss(dev):  # noqa: F811
    """NULL gradients and score weights: the loss alone is the same."""
    import torch
    from paper_2603_27151_gb300 import native as N
    gen = torch.Generator(device="cuda").manual_seed(1)
    c = [torch.rand((2, 3, 131, 250), generator=gen, device="cuda")]
    t = [torch.rand((3, 131, 250), generator=gen, device="cuda")]
    g, sw = [torch.empty_like(c[0])], [torch.empty((2, 131, 250), device="cuda")]
    a, b = torch.zeros(1, device="cuda"), torch.zeros(1, device="cuda")
    N.loss_l1_ssim(c, t, g, sw, a, scale=0.5)
    N.loss_l1_ssim(c, t, None, None, b, scale=0.5)
    assert abs(float(a) - float(b)) <= 1e-5 * abs(float(a))
    assert abs(float(a) - float(sw[0].double().sum())) <= 1e-5 * abs(float(a))
