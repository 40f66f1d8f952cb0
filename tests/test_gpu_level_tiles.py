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


def _check_levels(dm, ws, h, pyr):
    for l in range(1, pyr.geom.L + 1):
        vals, codes, valid = dm.read_level(ws, dm.dm_pyramid_level(h, l))
        np.testing.assert_array_equal(valid, pyr.valid[l])
        keep = valid.astype(bool)
        np.testing.assert_array_equal(vals[keep], (pyr.pooled[l] if l < pyr.geom.L else pyr.top)[keep], err_msg=f"level {l}")
        if l < pyr.geom.L:
            np.testing.assert_array_equal(codes[keep], pyr.argmax[l][keep], err_msg=f"level {l} codes")


@pytest.mark.parametrize("compensated", [True, False])
@pytest.mark.parametrize("size", [(W1, H1, W2, H2), (130, 70, 133, 71)])
def test_every_tile_bit_exact(dm_mod, oracle_mod, size, compensated):
    """Every tile and ring, the default's too, against the FP32 oracle at every level >= 1 (tests/test_level_routes.py
    says which levels of these sizes are tiled: two, with the default tile only at the first size)."""
    import torch
    dm = dm_mod
    w1, h1, w2, h2 = size
    rng = np.random.default_rng(7)
    d1 = oracle_mod.descriptors(synth.value_noise(w1, h1, rng).astype(np.float32), "f32")
    d2 = oracle_mod.descriptors(synth.value_noise(w2, h2, rng).astype(np.float32), "f32")
    pyr = oracle_mod.pyramid(d1, d2, "f32", compensated=compensated)
    t1, t2 = torch.from_numpy(d1).cuda(), torch.from_numpy(d2).cuda()
    ctx = dm.Context(dm.DM_FP32, compensated=int(compensated))
    try:
        ws = torch.empty(dm.dm_workspace_bytes(ctx.ctx, *size)["pyramid"], dtype=torch.uint8, device="cuda")
        for rows in (16, 8, 4):
            for ring in (2, 3):
                ws.fill_(0xA5)
                dm.dm_set_tuned_config(ctx.ctx, *size, {"m_chunk": 1, "level_tile_rows": rows, "bt_ctas_per_sm": 8,
                                                        "level_ring": ring})
                h = dm.dm_correlate_pyramid(ctx.ctx, t1, t2, ws)
                try:
                    _check_levels(dm, ws, h, pyr)
                finally:
                    dm.dm_pyramid_free(h)
    finally:
        ctx.close()


@pytest.mark.parametrize("compensated", [True, False])
def test_approximate_form_bit_exact(dm_mod, oracle_mod, compensated):
    """The tiled instances that read level 0 through the prototype index (level 1), against the FP32 oracle's chain on
    the patches replaced by their prototypes."""
    import torch
    dm = dm_mod
    a, b = _images(3)
    rng = np.random.default_rng(4)
    vecs = oracle_mod.patch_vectors(oracle_mod.descriptors(a, "f32"))
    protos = np.ascontiguousarray(vecs[rng.choice(len(vecs), 37, replace=False)])
    assign = rng.integers(0, 37, len(vecs)).astype(np.int32)
    _, pyr, _ = oracle_mod.approx_match(a, b, protos, assign, "f32", compensated=compensated)
    d2 = torch.from_numpy(oracle_mod.descriptors(b, "f32")).cuda()
    tp, ta = torch.from_numpy(protos).cuda(), torch.from_numpy(assign).cuda()
    ctx = dm.Context(dm.DM_FP32, compensated=int(compensated))
    try:
        ws = torch.full((dm.dm_workspace_bytes(ctx.ctx, W1, H1, W2, H2)["pyramid"],), 0xA5, dtype=torch.uint8, device="cuda")
        h = dm.dm_correlate_pyramid_approx(ctx.ctx, tp, ta, W1, H1, d2, ws)
        try:
            _check_levels(dm, ws, h, pyr)
        finally:
            dm.dm_pyramid_free(h)
    finally:
        ctx.close()
