"""Launch shapes that a caller names: an automatic z chunk is the one an untuned
lattice takes on that tile, and shapes that no launch takes are refused when they
are named (tile rows and z chunks are grid dimensions of at most 65535)."""
import pytest

PRECISIONS = ["f64", "f32", "bf16", "bf16_rest"]


@pytest.fixture(scope="module")
def lib():
    from paper_1112_5547_gb300 import build, lbm_sc
    build.build()
    return lbm_sc


def _handle(lib, lat, shape, prec, **kw):
    p = lib.make_params(lat, shape, 1.0, 1.0, 2.0, prec, **kw)
    return p, lib.lbm_sc_create(p, 256 * 1024, lib.lbm_sc_workspace_bytes(p), 0)


def test_automatic_chunk_is_the_untuned_one(lib):
    for shape in ((48, 48, 48), (128, 128, 128), (150, 130, 180), (512, 512, 512), (7, 9, 11), (1, 40, 40), (300, 8, 32)):
        for prec in PRECISIONS:
            for kw in ({}, {"forcing": "guo"}):
                p, h = _handle(lib, 1, shape, prec, **kw)
                try:
                    tile, zc = lib.lbm_sc_get_tuning(h)
                    lib.lbm_sc_set_tuning(h, tile, 0)
                    assert lib.lbm_sc_get_tuning(h) == (tile, zc)
                    for t in range(len(lib.TILES)):  # every tile the lattice takes gets a chunk within it
                        try:
                            lib.lbm_sc_set_tuning(h, t, 0)
                        except lib.LbmError:
                            continue
                        assert lib.lbm_sc_get_tuning(h)[0] == t and 1 <= lib.lbm_sc_get_tuning(h)[1] <= shape[0]
                finally:
                    lib.lbm_sc_destroy(h)


@pytest.mark.parametrize("lat,shape,tile,zchunk", [
    (0, (262141, 16), 3, 0), (0, (524281, 16), 0, 0), (1, (2, 262141, 8), 3, 0), (1, (65536, 8, 8), 3, 1),
    (1, (131071, 4, 4), 0, 1), (1, (2100000, 4, 4), 0, 32)])
def test_shapes_beyond_a_grid_are_refused(lib, lat, shape, tile, zchunk):
    p, h = _handle(lib, lat, shape, "f32")
    try:
        before = lib.lbm_sc_get_tuning(h)
        with pytest.raises(lib.LbmError):
            lib.lbm_sc_set_tuning(h, tile, zchunk)
        assert lib.lbm_sc_get_tuning(h) == before
        if lat == 1 and -(-shape[1] // lib.TILES[tile][1]) <= 65535:  # the automatic chunk and the next that fits
            lib.lbm_sc_set_tuning(h, tile, 0)
            assert -(-shape[0] // lib.lbm_sc_get_tuning(h)[1]) <= 65535
            least = -(-shape[0] // 65535)
            lib.lbm_sc_set_tuning(h, tile, least)
            assert lib.lbm_sc_get_tuning(h) == (tile, least)
    finally:
        lib.lbm_sc_destroy(h)
