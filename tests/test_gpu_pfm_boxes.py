"""FP64 phase-field steps in the boxes that the fused kernels take, at the edges of
their range, against the numpy oracle: the smallest and largest plane boxes, the
longest lines, every radix of the row lengths and of the column lengths, short axes
in 3D, and boxes just outside (which go through cuFFT).  Tolerances as in
test_gpu_pfm.py: 1e-10 of the field's maximum on phi, 1e-9 on u (two FFT
algorithms)."""
import numpy as np
import pytest

from paper_1112_5547_gb300 import inputs

pytestmark = pytest.mark.gpu

RHO, TAU, G, DT = 1.4, 0.6, 0.3, 0.1


@pytest.mark.parametrize("shape", [
    (96, 1024), (128, 768), (384, 288), (320, 320), (240, 480), (160, 800), (128, 864), (400, 512), (432, 960), (1024, 320),
    (1024, 1024), (32, 64, 64), (16, 96, 96), (128, 16, 64), (48, 80, 160), (16, 16, 768), (1024, 16, 64), (32, 432, 64),
    (384, 256), (96, 960), (128, 1152), (128, 32, 32), (16, 128, 64)])
def test_boxes_match_the_oracle(oracle_mod, shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, phase_field
    build.build()
    rA, rB = inputs.drop(shape, min(shape) / 4.0, rho_hi=1.2, rho_lo=0.2, seed=9)
    phi0 = rA - rB
    ny, D = shape[-2], len(shape)
    u0 = np.zeros(shape + (D,))
    u0[..., 0] = 0.02 * np.sin(2 * np.pi * np.arange(ny) / ny)[:, None]
    s = phase_field.PFM(shape, RHO, TAU, G, DT, "f64", body_A=1e-4).init(phi0, u0)
    o = oracle_mod.OraclePFM(shape, RHO, TAU, G, DT, body_A=1e-4).init(phi0, u0)
    for n in (1, 2):  # the first step, and steps that continue one
        s.step(n)
        o.step(n)
        phi, u = (t.cpu().numpy() for t in s.fields())
        op, ou = o.fields()
        assert np.abs(phi - op).max() < 1e-10 * np.abs(op).max()
        assert np.abs(u - ou).max() < 1e-9 * np.abs(ou).max()
