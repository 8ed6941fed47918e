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
