"""Backtracking over argmax codes that no pooling writes, as a level kernel that gave up can
leave them: every code the same value, also one that leads out of the map at its border.
The call returns well-formed matches inside image 2."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("code", [0, 2, 6, 8, 9, 255])
@pytest.mark.parametrize("W,H", [(64, 48), (37, 29)])
def test_stale_codes_stay_inside(W, H, code):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    rng = np.random.default_rng(5)
    d = [torch.from_numpy(rng.random((H, W, 9), dtype=np.float32)).cuda() for _ in range(2)]
    ctx = dm.Context(dm.DM_FP32)
    try:
        sizes = dm.dm_workspace_bytes(ctx.ctx, W, H, W, H)
        ws = torch.empty(sizes["pyramid"], dtype=torch.uint8, device="cuda")
        h = dm.dm_correlate_pyramid(ctx.ctx, d[0], d[1], ws)
        g = dm.dm_geometry(W, H, W, H)
        for l in range(g["L"]):
            info = dm.dm_pyramid_level(h, l)
            o = info["argmax"] - ws.data_ptr()
            ws[o:o + info["n"] * info["mh"] * info["pitch"]] = code
        out = torch.zeros((g["n_patch0"], 5), device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        wsb = torch.empty(sizes["backtrack"], dtype=torch.uint8, device="cuda")
        dm.dm_backtrack(ctx.ctx, h, wsb, out, cnt)
        torch.cuda.synchronize()
        m = out[:int(cnt.item())].cpu().numpy()
        dm.dm_pyramid_free(h)
    finally:
        ctx.close()
    assert ((m[:, 2] >= 0) & (m[:, 2] < W) & (m[:, 3] >= 0) & (m[:, 3] < H)).all()
    assert (len(m) > 0) == (code <= 8)
