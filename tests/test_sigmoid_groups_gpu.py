"""The composition evaluates the sigmoid of four channels at a time, on a short
path when all four lie within +-80: bit for bit the oracle's activation for
groups on both sides of that line, infinities and NaN, and for a dense sweep."""
import numpy as np
import pytest

import oracle as O
from paper_2603_27151_gb300 import inputs as I

pytestmark = pytest.mark.gpu

EDGES = np.float32([79.99999, 80.0, 80.00001, 87.3, 88.0, 88.8, 89.0, 103.9, 104.0, 200.0, np.inf, np.nan, 0.0, 1e-30, 1e-45, 3e38])


@pytest.mark.parametrize("C", [4, 8])
@pytest.mark.parametrize("what", ["sweep", "edges"])
def test_activation_bit_exact(what, C):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2603_27151_gb300 import native as N
    rng = np.random.default_rng(C)
    T, r_min, r_max = 500, 1, 3
    lv = [np.zeros_like(l) for l in I.level_logits(T, r_min, r_max, C, rng)]
    n = lv[-1].size
    if what == "sweep":
        fine = np.linspace(-90.0, 90.0, n, dtype=np.float32)
    else:   # about one edge value in every second group of four
        fine = rng.normal(0, 8, n).astype(np.float32)
        at = rng.random(n) < 0.15
        fine[at] = rng.choice(np.concatenate([EDGES, -EDGES]), at.sum())
    lv[-1] = fine.reshape(lv[-1].shape)
    out = torch.empty((T, N.level_V(r_max), C), device="cuda")
    tex = torch.from_numpy(np.concatenate([l.reshape(-1) for l in lv])).cuda()
    N.levels_compose(tex, T, r_min, r_max, C, out, activate=True)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), O.activate(O.compose(lv, r_min, r_max)), equal_nan=True)
