"""Which kernel takes a level (tiled or row-streaming), by the library's own rule: small images and filled maps stream, a
tile that was set is taken, and a small image 1 does not pull the wide maps of a larger image 2 along."""
import ctypes as C

import pytest

SMALL, SET = (8, 2), (8, 3)             # (rows, ring): the default tile, another one


@pytest.fixture(scope="module")
def tiled():
    from paper_1506_07656_gb300 import build, dm
    build.build()
    lib = dm.load()
    geom, rule = lib._Z12dm_make_geomiiiiP6DmGeom, lib._Z14dm_level_tiledRK6DmGeomiRK6DmTune
    rule.restype = C.c_bool

    def levels(W1, H1, W2, H2, tile):
        g = C.create_string_buffer(4096)
        assert geom(W1, H1, W2, H2, g) == 0
        tune = (C.c_int * 4)(1, tile[0], 8, tile[1])
        top = dm.dm_geometry(W1, H1, W2, H2)["L"]
        return [l for l in range(1, top) if rule(g, l, tune)]

    return levels


@pytest.mark.parametrize("pair,tile,want", [
    # maps of 33 and 17 columns (25, then 13), small images: streaming, unless a tile is set
    ((130, 70, 133, 71), SET, [1, 2]), ((300, 124, 160, 96), (16, 3), [1, 2]),
    ((130, 70, 130, 70), SMALL, []), ((130, 70, 130, 70), SET, [1, 2]), ((130, 70, 130, 70), (16, 2), [1, 2]),
    ((97, 61, 97, 61), SMALL, []), ((97, 61, 97, 61), (4, 3), [1]),
    ((64, 48, 64, 48), SMALL, []), ((130, 70, 130, 70), (0, 2), []),
    # image 1 of 144 and 1936 patches, maps of 160, 80, 40 and 20 columns
    ((48, 48, 640, 480), SMALL, [1, 2]), ((176, 176, 640, 480), SMALL, [1, 2]), ((48, 48, 320, 240), SMALL, [1]),
    ((48, 48, 640, 480), (0, 2), []),
    # filled maps of 311, 256 and 128 columns: streaming with twice as many patches
    ((48, 48, 1242, 375), SMALL, [1, 2, 3]), ((96, 96, 1242, 375), SMALL, [1, 2, 3]), ((128, 128, 1242, 375), SMALL, [2, 3]),
    ((96, 96, 1024, 436), SMALL, []), ((100, 75, 512, 224), SMALL, []),
    # as many patches as image 2 asks for
    ((1024, 436, 1024, 436), SMALL, []), ((1024, 436, 1024, 436), (16, 3), []), ((512, 224, 512, 224), SMALL, []),
    ((640, 480, 640, 480), SMALL, [1, 2, 3, 4]), ((1242, 375, 1242, 375), SMALL, [2, 3, 4, 5]),
    ((320, 240, 320, 240), SMALL, [1, 2, 3]), ((300, 124, 160, 96), SMALL, [1, 2]),
])
def test_routes(tiled, pair, tile, want):
    assert tiled(*pair, tile) == want
