"""A tensor-core level-0 kernel whose wait runs out with copies and MMAs in flight (dm_inject_fault): every CTA stops
after its first tile, ends what it has started, gives shared memory and TMEM back, and reports it; the same context and
workspace then compute the pyramid they computed before.  The fields are large enough for many tiles per CTA."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

W, H = 320, 240


@pytest.mark.parametrize("prec", ["bf16", "fp8"])
def test_wait_that_runs_out(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    g = torch.Generator(device="cuda").manual_seed(2)
    d = [torch.rand((H, W, 9), device="cuda", generator=g) for _ in range(2)]
    ctx = dm.Context({"bf16": dm.DM_BF16, "fp8": dm.DM_FP8_E4M3}[prec])
    try:
        ws = torch.empty(dm.dm_workspace_bytes(ctx.ctx, W, H, W, H)["pyramid"], dtype=torch.uint8, device="cuda")

        def levels():
            ws.fill_(0xA5)
            h = dm.dm_correlate_pyramid(ctx.ctx, d[0], d[1], ws)
            torch.cuda.synchronize()
            st, _ = dm.dm_read_status(ctx.ctx, ws, 1)
            out = [dm.read_level(ws, dm.dm_pyramid_level(h, l)) for l in (0, dm.dm_geometry(W, H, W, H)["L"])]
            dm.dm_pyramid_free(h)
            return st, out

        st, want = levels()
        assert st == 0
        for _ in range(3):
            dm.dm_inject_fault(ctx.ctx, dm.DM_FAULT_WAIT, 2000)
            try:
                st, got = levels()
            finally:
                dm.dm_inject_fault(ctx.ctx, dm.DM_FAULT_WAIT, 0)
            assert st & dm.DM_DEV_TIMEOUT
            assert (got[0][1] == 0xA5).mean() > 0.25          # most tiles of level 0 were never computed
            st, again = levels()
            assert st == 0
            for (v, a, e), (wv, wa, we) in zip(again, want):
                np.testing.assert_array_equal(e, we)
                np.testing.assert_array_equal(v[we != 0], wv[we != 0])
                if a is not None:
                    np.testing.assert_array_equal(a, wa)
    finally:
        ctx.close()
