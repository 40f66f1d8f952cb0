"""The chains of programmatically dependent launches under capture: one dm_match and one
dm_match_star in a CUDA graph, replayed on other images in the same buffers and several
times in a row, equal the direct calls."""
import numpy as np
import pytest

from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["DM_FP32", "DM_BF16"])
@pytest.mark.parametrize("star", [False, True])
@pytest.mark.parametrize("W,H", [(64, 48), (130, 70)])
def test_replay_equals_call(W, H, star, prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    pairs = [synth.make_pair_smooth(W, H, s) for s in (1, 2)]
    imgs = [[torch.from_numpy(np.ascontiguousarray(i, dtype=np.float32)).cuda() for i in (p.img1, p.img2)] for p in pairs]
    ctx = dm.Context(getattr(dm, prec))
    try:
        sizes = dm.dm_star_workspace_bytes(ctx.ctx, W, H, W, H) if star else dm.dm_workspace_bytes(ctx.ctx, W, H, W, H)
        call = dm.dm_match_star if star else dm.dm_match
        ws = torch.empty(sizes["match"], dtype=torch.uint8, device="cuda")
        n0 = dm.dm_geometry(W, H, W, H)["n_patch0"]
        out, cnt = torch.zeros((n0, 5), device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
        want = []
        for a, b in imgs:
            call(ctx.ctx, a, b, ws, out, cnt)
            torch.cuda.synchronize()
            want.append(out[:int(cnt.item())].cpu().numpy().copy())
        i1, i2 = imgs[0][0].clone(), imgs[0][1].clone()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            call(ctx.ctx, i1, i2, ws, out, cnt)
        for k in (1, 0, 1):
            i1.copy_(imgs[k][0])
            i2.copy_(imgs[k][1])
            for _ in range(3):
                graph.replay()
            torch.cuda.synchronize()
            np.testing.assert_array_equal(out[:int(cnt.item())].cpu().numpy(), want[k])
    finally:
        ctx.close()
