"""The reciprocal step's split over a cluster: patch counts at and past a warp, at one warp
of every CTA, and between (larger counts: the full-size checks); the matches, their order
and what an output that is too small keeps, against the FP32 oracle."""
import numpy as np
import pytest

import oracle
from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W1,H1", [(32, 16), (44, 12), (41, 13), (128, 128), (120, 124)])
def test_order_and_capacity(W1, H1):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    W2, H2 = 52, 40
    a = synth.make_pair_smooth(W1, H1, 3).img1.astype(np.float32)
    b = synth.make_pair_smooth(W2, H2, 4).img2.astype(np.float32)
    want = oracle.match(a, b, "f32")[0].astype(np.float32)
    assert len(want) > 3
    ctx = dm.Context(dm.DM_FP32)
    try:
        ws = torch.empty(dm.dm_workspace_bytes(ctx.ctx, W1, H1, W2, H2)["match"], dtype=torch.uint8, device="cuda")
        cnt = torch.zeros(1, dtype=torch.int32, device="cuda")
        for cap in (len(want), len(want) - 3):
            out = torch.full((len(want), 5), -1.0, dtype=torch.float32, device="cuda")
            dm.dm_match(ctx.ctx, torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), ws, out[:cap], cnt)
            torch.cuda.synchronize()
            assert int(cnt.item()) == len(want)
            got = out.cpu().numpy()
            np.testing.assert_array_equal(got[:cap], want[:cap])
            assert (got[cap:] == -1.0).all()
    finally:
        ctx.close()
