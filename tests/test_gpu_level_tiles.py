"""The tiled level kernel at sizes whose levels it takes: more than 2048 lattice patches, and stored maps of 40 and 20
columns, which fill none of the row-streaming kernel's strips."""
import numpy as np
import pytest

from paper_1506_07656_gb300 import synth

pytestmark = pytest.mark.gpu

W1, H1, W2, H2 = 300, 124, 160, 96


@pytest.fixture(scope="module")
def dm_mod():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    return dm


def _images(seed):
    a = synth.value_noise(W1, H1, np.random.default_rng(seed)).astype(np.float32)
    return a, np.ascontiguousarray(a[14:14 + H2, 60:60 + W2])


@pytest.mark.parametrize("rows,ring", [(16, 3), (16, 2), (8, 3)])
def test_waves_of_both_child_sums(dm_mod, rows, ring):
    """Cross-pair waves in one process with compensated and plain child sums (two kernels of one type, each with
    its own shared-memory limit; 16 rows with a ring of 3 need more than 48 KB): every pair as dm_match alone."""
    import torch
    dm = dm_mod
    imgs = [_images(s) for s in (1, 2)]
    for comp in (1, 0, 1):
        ctx = dm.Context(dm.DM_FP32, compensated=comp)
        try:
            dm.dm_set_tuned_config(ctx.ctx, W1, H1, W2, H2, {"m_chunk": 1, "level_tile_rows": rows, "bt_ctas_per_sm": 8,
                                                             "level_ring": ring})
            n0 = dm.dm_geometry(W1, H1, W2, H2)["n_patch0"]
            items = [(torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda(), torch.zeros((n0, 5), device="cuda"),
                      torch.zeros(1, dtype=torch.int32, device="cuda")) for a, b in imgs]
            pairs = dm.make_pairs(items)
            dm.dm_set_batch_wave(ctx.ctx, 2)
            dm.dm_set_batch_lanes(ctx.ctx, 1)
            ws = torch.empty(dm.dm_batch_workspace_bytes(ctx.ctx, pairs), dtype=torch.uint8, device="cuda")
            dm.dm_match_batch(ctx.ctx, pairs, ws)
            torch.cuda.synchronize()
            for (a, b), (_, _, out, cnt) in zip(imgs, items):
                want = ctx.match(a, b).cpu().numpy()
                assert len(want) > 0
                np.testing.assert_array_equal(out[:int(cnt.item())].cpu().numpy(), want)
        finally:
            ctx.close()
