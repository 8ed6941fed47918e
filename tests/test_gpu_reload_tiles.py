"""The tiles that pull a plane again for its collision, in every storage, against the
32x8 register tile, bit for bit: they differ in how and when they pull."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f32", "f64", "bf16", "f16", "bf16_rest", "f16_rest"])
@pytest.mark.parametrize("shape", [(37, 71), (1, 5), (11, 13, 40), (5, 33, 65), (1, 2, 3)])
def test_reload_tiles(shape, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, inputs, lbm_sc
    build.build()
    kw = dict(rho_ref_A=0.5, rho_ref_B=0.5) if precision in ("bf16", "f16") else {}
    f = inputs.drop(shape, 0.4 * min(shape), seed=6, dtype=np.float64 if precision == "f64" else np.float32)
    for forcing in ("shift", "guo"):
        lat = lbm_sc.Lattice(len(shape) - 2, shape, 1.0, 0.9, 2.4 / 1.04, precision, forcing=forcing, body_A=1e-4, **kw)
        want = lat.set_tuning(0, 3).init(*f).step(7).moments()
        for tile in (11, 12, 13, 14):
            for zchunk in (1, 4):
                # steps of both kinds in one stream: each waits for the one before
                got = lat.set_tuning(tile, zchunk).init(*f).step(3).set_tuning(0, 3).step(1).set_tuning(tile, zchunk).step(3)
                for x, y in zip(got.moments(), want):
                    assert torch.equal(x, y), (tile, zchunk)
