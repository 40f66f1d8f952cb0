"""The fused descriptor kernel where its split changes: images inside one tile, at, just
below and just past tiles of 16x8 and (from 77824 pixels) of 32x16, single rows and
columns, whose every tap is clamped; widths of radius 3 with other weights and widths that
take the pass-by-pass kernels.  Bit for bit against the FP32 oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (1, 37), (40, 1), (3, 5), (16, 8), (15, 9), (17, 7), (33, 40), (64, 48), (319, 243), (320, 256), (321, 257),
         (2432, 32), (31, 2511)]


def _torch():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build
    build.build()
    return torch


@pytest.mark.parametrize("widths", [{}, {"nu1": 0.7, "nu2": 0.8, "nu3": 0.9}, {"nu2": 1.3}, {"nu3": 0.5}])
@pytest.mark.parametrize("W,H", SIZES)
def test_bit_exact(W, H, widths):
    torch = _torch()
    from paper_1506_07656_gb300 import dm
    img = np.random.default_rng(W + 7 * H).random((H, W)).astype(np.float32)
    ctx = dm.Context(dm.DM_FP32, **widths)
    try:
        out = torch.full((H, W, 9), -1.0, dtype=torch.float32, device="cuda")
        tmp = torch.empty(W * H * 16 * 4 + 512, dtype=torch.uint8, device="cuda")
        dm.dm_descriptors(ctx.ctx, torch.from_numpy(img).cuda(), out, tmp)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        ctx.close()
    want = oracle.descriptors(img, "f32", **{k: float(np.float32(v)) for k, v in widths.items()})
    np.testing.assert_array_equal(got.view(np.uint32), want.astype(np.float32).view(np.uint32))
