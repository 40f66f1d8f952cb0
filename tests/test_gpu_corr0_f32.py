"""The FP32 level-0 kernel where its split changes: bands of 2, 4 and 8 pooled rows, maps
that end inside, at and just past a tile of 32 pooled columns, ranges that begin in the
middle of a band (whose first window needs a column of the tile before) and more CTAs than
fit at once.  Pooled values and argmax codes of sampled patches, bit for bit against the
FP32 oracle; the fields take few values, so that windows hold equal maxima."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

# lattice image, target image
SIZES = [((20, 20), (64, 48)), ((64, 48), (65, 37)), ((101, 77), (66, 80)), ((97, 75), (31, 129)),
         ((161, 121), (331, 77)), ((130, 190), (257, 101)), ((400, 300), (160, 158)), ((16, 16), (16, 16))]


@pytest.mark.parametrize("levels", [2, 0])
@pytest.mark.parametrize("one,two", SIZES)
def test_level0_bit_exact(one, two, levels):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1506_07656_gb300 import build, dm
    build.build()
    (W1, H1), (W2, H2) = one, two
    rng = np.random.default_rng(W1 * 7 + W2)

    def field(W, H):
        d = rng.integers(0, levels, (H, W, 9)) if levels else rng.random((H, W, 9))
        return (np.asarray(d, dtype=np.float32) * np.float32(0.3125)).astype(np.float32)

    d1, d2 = field(W1, H1), field(W2, H2)
    g = dm.dm_geometry(W1, H1, W2, H2)
    n0 = g["n_patch0"]
    sel = np.unique(np.concatenate([[0, n0 - 1], rng.choice(n0, size=min(n0, 10), replace=False)]))
    ctx = dm.Context(dm.DM_FP32)
    try:
        ws = torch.empty(dm.dm_workspace_bytes(ctx.ctx, W1, H1, W2, H2)["pyramid"], dtype=torch.uint8, device="cuda")
        h = dm.dm_correlate_pyramid(ctx.ctx, torch.from_numpy(d1).cuda(), torch.from_numpy(d2).cuda(), ws)
        torch.cuda.synchronize()
        v, a, e = dm.read_level(ws, dm.dm_pyramid_level(h, 0), sel)
        dm.dm_pyramid_free(h)
    finally:
        ctx.close()
    want, codes, ex = oracle.levels_sampled(d1, d2, 0, sel, "f32")
    np.testing.assert_array_equal(e, ex)
    np.testing.assert_array_equal(a, codes)
    np.testing.assert_array_equal(v.view(np.uint32), np.asarray(want, dtype=np.float32).view(np.uint32))


# narrow maps and remainders: bands side by side in one row of tiles, each followed by an empty lane
@pytest.mark.parametrize("levels", [2, 0])
@pytest.mark.parametrize("one,two", [((256, 130), (24, 200)), ((130, 70), (5, 90)), ((257, 121), (62, 41)), ((300, 124), (64, 66)),
                                     ((300, 124), (66, 64)), ((97, 75), (9, 7)), ((196, 193), (127, 60)), ((64, 48), (4, 301)),
                                     ((220, 170), (200, 33))])
def test_dense_bands_bit_exact(one, two, levels):
    test_level0_bit_exact(one, two, levels)
