"""Launch shapes of untuned lattices and the paths a step takes for them.

Every launch shape runs the same per-node arithmetic, so an untuned lattice
must give bit for bit what the 32x8 register kernel with one chunk gives.
"""
import numpy as np
import pytest

SIZES3 = [(1, 1, 1), (2, 5, 3), (7, 4, 15), (5, 3, 17), (9, 12, 32), (33, 11, 31), (20, 33, 47), (13, 64, 65),
          (40, 12, 96), (31, 70, 100)]
SIZES2 = [(1, 1), (3, 16), (4, 15), (5, 17), (64, 64), (37, 71), (130, 257)]
PRECISIONS = ["f64", "f32", "bf16", "bf16_rest"]


def _options(precision):
    yield {}
    yield {"forcing": "guo"}
    if precision in ("f64", "f32"):
        yield {"model": 1, "kappa": -1.0, "gamma": 0.5}


def test_untuned_shape_is_one_the_library_accepts():
    from paper_1112_5547_gb300 import build, lbm_sc as lib
    build.build()
    sizes = [(1, s) for s in SIZES3 + [(512, 512, 512), (3, 7, 1000), (1000, 8, 32), (100, 100, 20)]]
    sizes += [(0, s) for s in SIZES2 + [(4096, 4096)]]
    for lat, shape in sizes:
        for prec in PRECISIONS:
            for kw in _options(prec):
                p = lib.make_params(lat, shape, 1.0, 1.0, 2.0, prec, **kw)
                h = lib.lbm_sc_create(p, 256 * 1024, lib.lbm_sc_workspace_bytes(p), 0)
                try:
                    tile, zc = lib.lbm_sc_get_tuning(h)
                    assert lib.tile_supported(tile, lat, p.precision, p.forcing, p.model)
                    assert 1 <= zc <= p.nz
                    lib.lbm_sc_set_tuning(h, tile, zc)
                    assert lib.lbm_sc_get_tuning(h) == (tile, zc)
                finally:
                    lib.lbm_sc_destroy(h)


def test_untuned_shape_of_long_lattices_fits_a_grid():
    """Tiles along y and chunks along z are grid dimensions of at most 65535."""
    from paper_1112_5547_gb300 import build, lbm_sc as lib
    build.build()
    for lat, shape in ((0, (262140, 16)), (0, (262141, 16)), (0, (524280, 16)), (1, (1, 300000, 8)), (1, (2, 524280, 16)),
                       (1, (65536, 8, 8)), (1, (2100000, 4, 4)), (1, (2100000, 8, 32))):
        for prec in PRECISIONS:
            p = lib.make_params(lat, shape, 1.0, 1.0, 2.0, prec)
            h = lib.lbm_sc_create(p, 256 * 1024, lib.lbm_sc_workspace_bytes(p), 0)
            try:
                tile, zc = lib.lbm_sc_get_tuning(h)
                assert -(-p.ny // lib.TILES[tile][1]) <= 65535
                assert 1 <= zc <= p.nz and -(-p.nz // zc) <= 65535
            finally:
                lib.lbm_sc_destroy(h)


def _run(lib, lat, shape, prec, kw, tuning, fields, steps):
    import torch
    ref = dict(rho_ref_A=0.5, rho_ref_B=0.5) if prec == "bf16" else {}
    tau = (1.0, 0.9)
    G = 2.5 if kw.get("model") else 2.4 / 1.04
    lt = lib.Lattice(lat, shape, *tau, G, prec, **ref, **kw)
    if tuning:
        lt.set_tuning(*tuning)
    out = []
    for n in steps:  # a new init between the runs: the chained launches of one run end before the next
        lt.init(*fields).step(n)
        out.append([t.cpu().numpy() for t in lt.moments()])
    torch.cuda.synchronize()
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("lat,sizes", [(1, SIZES3), (0, SIZES2)])
def test_untuned_equals_one_register_kernel(lat, sizes, prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, inputs, lbm_sc as lib
    build.build()
    dt = np.float64 if prec == "f64" else np.float32
    for shape in sizes:
        for kw in _options(prec):
            hi, lo = (0.9, 0.14) if kw.get("model") else (1.0, 0.04)
            f = inputs.drop(shape, min(shape) / 3.0, rho_hi=hi, rho_lo=lo, seed=5, dtype=dt)
            a = _run(lib, lat, shape, prec, kw, None, f, (1, 6))
            b = _run(lib, lat, shape, prec, kw, (0, 1 if lat == 0 else shape[0]), f, (1, 6))
            for x, y in zip(a, b):
                for u, v in zip(x, y):
                    assert np.isfinite(v).all()
                    np.testing.assert_array_equal(u, v)


@pytest.mark.gpu
def test_many_steps_per_launch_equal_single_steps():
    """D2Q9 FP32: all steps in one cluster, two steps per launch, and both in a batch,
    for every remainder of the steps, against single steps of another tile."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, inputs, lbm_sc as lib
    build.build()
    G = 2.4 / 1.04
    # cluster kernel: one row band per CTA at least two rows high, ragged bands, wide and narrow rows, many steps
    # two-step tile: smallest frame, one more and one less than whole tiles
    shapes = [(4, 3), (5, 40), (33, 64), (8, 512), (100, 100), (22, 38), (22, 600), (161, 129), (192, 160), (127, 161)]
    for shape in shapes:
        for kw in ({}, {"forcing": "guo", "body_A": 1e-4}):
            f = inputs.drop(shape, min(shape) / 3.0, seed=6, dtype=np.float32)
            a = _run(lib, 0, shape, "f32", kw, None, f, (2, 3, 4, 5, 11))
            b = _run(lib, 0, shape, "f32", kw, (0, 1), f, (2, 3, 4, 5, 11))
            for x, y in zip(a, b):
                for u, v in zip(x, y):
                    np.testing.assert_array_equal(u, v)
    f = inputs.drop((8, 32), 2.0, seed=7, dtype=np.float32)  # more steps than one launch takes
    for u, v in zip(_run(lib, 0, (8, 32), "f32", {}, None, f, (4101,))[0],
                    _run(lib, 0, (8, 32), "f32", {}, (0, 1), f, (4101,))[0]):
        np.testing.assert_array_equal(u, v)
    stream = torch.cuda.Stream()
    shapes = [(64, 64), (22, 38), (100, 40), (257, 130)]
    fields = [inputs.drop(s, min(s) / 3.0, seed=8 + k, dtype=np.float32) for k, s in enumerate(shapes)]
    for tile, graph in ((0, 0), (1, 8), (7, 8)):
        for n in (4, 7, 18):
            with torch.cuda.stream(stream):
                solo = [lib.Lattice(0, s, 1.0, 0.9, G, "f32", stream=stream).set_tuning(0).init(*f).step(n)
                        for s, f in zip(shapes, fields)]
                lats = [lib.Lattice(0, s, 1.0, 0.9, G, "f32", stream=stream).init(*f) for s, f in zip(shapes, fields)]
                b = lib.Batch(lats, tile=tile, graph_steps=graph, stream=stream).step(n)
                for u, v in zip(solo, lats):
                    for x, y in zip(u.moments(), v.moments()):
                        assert torch.equal(x, y)
                b.close()
