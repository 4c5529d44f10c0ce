"""The shading backward takes blocks of 256 pixels, two per thread (p and
p + 128): views that end around those lines, against the FP64 oracle.

Tolerances as for the shading pass at other sizes: feature gradient
|d| <= 1e-5 (1 + |ref|) (three layers of at most 16 terms in FP32), parameter
gradient |d| <= 1e-4 (|ref| + 1e-2 max|ref|) (FP32 sums over a CTA's pixels).
"""
import numpy as np
import pytest

from oracle import shading as SH
from paper_2603_27151_gb300 import inputs as I

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


@pytest.mark.parametrize("sizes", [[(1, 1)], [(127, 1), (128, 1), (129, 1)], [(51, 5), (64, 4), (257, 1), (385, 1), (641, 3)]])
@pytest.mark.parametrize("S", [1, 2])
def test_backward_around_the_pixel_pairs(ctx, sizes, S):
    import torch
    rng = np.random.default_rng(31)
    eyes = I.sphere_eyes(len(sizes), 3.0, rng)
    cams = [I.look_at(e, w, h) for e, (w, h) in zip(eyes, sizes)]
    W1, b1, W2, b2, W3, b3 = SH.unpack(SH.xavier_params(5))
    params = SH.pack(W1, rng.normal(0, 0.3, 16), W2, rng.normal(0, 0.3, 16), W3, rng.normal(0, 0.3, 3)).astype(np.float32)
    feats = [rng.uniform(0, 1, (S, 7, h, w)).astype(np.float32) for w, h in sizes]
    grads = [rng.normal(size=(S, 3, h, w)).astype(np.float32) for w, h in sizes]
    dev = lambda x: torch.from_numpy(x).cuda()
    for want_feat in (True, False):
        gf = [torch.full(x.shape, 7.0, device="cuda") for x in feats] if want_feat else None
        gp = torch.full((SH.N_PARAMS,), 7.0, device="cuda")
        ctx.shade_backward(cams, dev(params), [dev(x) for x in feats], [dev(x) for x in grads], gf, gp, overwrite=True)
        gp_ref = np.zeros(SH.N_PARAMS)
        for v, c in enumerate(cams):
            f_ref, p_ref = SH.shade_backward(feats[v], c, params.astype(np.float64), grads[v])
            gp_ref += p_ref
            if want_feat:
                assert np.all(np.abs(gf[v].cpu().numpy() - f_ref) <= 1e-5 * (1 + np.abs(f_ref))), v
        assert np.all(np.abs(gp.cpu().numpy() - gp_ref) <= 1e-4 * (np.abs(gp_ref) + 1e-2 * np.abs(gp_ref).max()))
