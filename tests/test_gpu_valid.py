"""The existence flags of all levels in one launch: wide, tall and square lattices, borders
where columns or rows drop out, more patches than one CTA has threads, and a lattice whose
columns and rows exceed the kernel's shared memory (level by level); against the oracle."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W1,H1", [(5, 4), (6, 5), (7, 64), (64, 48), (65, 13), (200, 30), (31, 257), (160, 161), (1030, 9),
                                   (9, 4096), (32740, 12), (32800, 7)])
def test_flags(W1, H1):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    W2, H2 = 12, 8
    rng = np.random.default_rng(1)
    d1 = torch.from_numpy(rng.random((H1, W1, 9), dtype=np.float32)).cuda()
    d2 = torch.from_numpy(rng.random((H2, W2, 9), dtype=np.float32)).cuda()
    ctx = dm.Context(dm.DM_FP32)
    try:
        ws = torch.full((dm.dm_workspace_bytes(ctx.ctx, W1, H1, W2, H2)["pyramid"],), 0xA5, dtype=torch.uint8, device="cuda")
        h = dm.dm_correlate_pyramid(ctx.ctx, d1, d2, ws)
        torch.cuda.synchronize()
        got = []
        for l in range(dm.dm_geometry(W1, H1, W2, H2)["L"] + 1):
            info = dm.dm_pyramid_level(h, l)
            o = info["valid"] - ws.data_ptr()
            got.append(ws[o:o + info["n"]].cpu().numpy())
        dm.dm_pyramid_free(h)
    finally:
        ctx.close()
    want = oracle.valid_flags(W1, H1, W2, H2)
    assert len(got) == len(want)
    for l, (a, b) in enumerate(zip(got, want)):
        np.testing.assert_array_equal(a, b, err_msg=f"level {l}")
