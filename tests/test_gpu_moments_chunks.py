"""Reported fields and diagnostics of thin, flat and tall lattices, whose z chunks the
launch shape chooses: fields equal to those of the populations summed in torch, in
FP64 and FP32, and whole numbers counted exactly."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C3 = [(0, 0, 0)] + [tuple(s * v for v in a) for a in ((1, 0, 0), (0, 1, 0), (0, 0, 1)) for s in (1, -1)] + [
    tuple(s * v for v in a) for a in ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)) for s in (1, -1)]


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(5, 93, 270), (2, 129, 136), (1, 40, 33), (48, 48, 48), (33, 8, 32), (152, 7, 31), (40, 100, 65)])
def test_fields_of_every_chunk(shape, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, lbm_sc
    build.build()
    rng = np.random.default_rng(2)
    rho = [rng.uniform(0.2, 1.0, shape) for _ in range(2)]
    lat = lbm_sc.Lattice(1, shape, 1.0, 0.9, 1.5, precision).init(*rho).step(2)
    gx, gy = lbm_sc.lbm_sc_layout(lat.handle)[4:6]
    nz, ny, nx = shape
    f = lat.populations()[:, :, :, gy:gy + ny, gx:gx + nx].double()
    want = [sum(torch.roll(f[s, i], c[::-1], (0, 1, 2)) for i, c in enumerate(C3)) for s in (0, 1)]
    rA, rB, u, p = lat.moments()
    eps = np.finfo(np.float64 if precision == "f64" else np.float32).eps
    for got, x in zip((rA, rB), want):  # 18 additions of positive values, half an ulp of the sum each
        assert float(((got.double() - x) / x).abs().max()) <= 9 * eps
    d = lat.diagnostics(check=False)
    assert d["droplet_nodes"] == int((rA >= rB).sum()) and d["nonfinite"] == 0
    assert d["min_rho_A"] == float(rA.double().min()) and d["min_rho_B"] == float(rB.double().min())
    for key, r in (("mass_A", rA), ("mass_B", rB)):
        assert abs(d[key] - float(r.double().sum())) <= 1e-12 * d[key]
    assert abs(d["max_speed"] - float(u.double().pow(2).sum(-1).sqrt().max())) <= 1e-12
