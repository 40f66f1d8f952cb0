"""DeepFlow of images with a NaN or an infinity in one pixel: the flow is not finite exactly where the FP32 oracle's is
not (a neighbour that does not exist adds nothing, so nothing passes from one border to the other), and has its bits
elsewhere.  One level, few sweeps, the pixel at a border: a level of the one-CTA kernel with even and odd rows, and
levels in tiles that end inside, at and one past a 32x16 block."""
import numpy as np
import pytest

import oracle
from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu

SIZES = [(40, 32), (39, 31), (100, 40), (97, 33), (64, 48)]


@pytest.mark.parametrize("W,H", SIZES)
@pytest.mark.parametrize("where", ["right", "left", "top left", "bottom"])
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_reach(W, H, where, value):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    pr = synth.make_pair_smooth(W, H, seed=W, max_disp=2.0)
    a, b = pr.img1.copy(), pr.img2.copy()
    y, x = {"right": (H // 2, W - 1), "left": (H // 2, 0), "top left": (0, 0), "bottom": (H - 1, W // 2)}[where]
    a[y, x] = value
    kw = dict(n_fixed=2, n_sor=2, eta=0.9, min_size=min(W, H))
    want = oracle.deepflow(a, b, None, "f32", **kw)
    ctx = dm.Context(dm.DM_FP32)
    try:
        got = [t.cpu().numpy() for t in ctx.deepflow(a, b, None, **kw)]
    finally:
        ctx.close()
    spoiled = ~np.isfinite(want[0])
    assert spoiled.any() and not spoiled.all()
    for g, w in zip(got, want):
        np.testing.assert_array_equal(np.isfinite(g), np.isfinite(w))
        np.testing.assert_array_equal(g[np.isfinite(w)], w[np.isfinite(w)])
