"""FP64 phase-field steps with the transforms fused into the solver's kernels,
against the numpy oracle, at the sizes where they can go wrong: the shortest
lines, every middle radix, several of them, ragged column blocks, and sizes next to
those they take (which go through cuFFT).  Tolerances as in test_gpu_pfm.py: 1e-10
of the field's maximum on phi, 1e-9 on u (two FFT algorithms)."""
import numpy as np
import pytest

from paper_1112_5547_gb300 import inputs

pytestmark = pytest.mark.gpu

RHO, TAU, G, DT = 1.4, 0.6, 0.3, 0.1


@pytest.mark.parametrize("shape", [(16, 32), (32, 96), (48, 160), (80, 64), (128, 320), (240, 96), (512, 32), (16, 2048),
                                   (1024, 64), (16, 256, 32), (256, 16, 32), (32, 64, 96), (80, 48, 96), (64, 48, 160),
                                   (24, 32), (16, 34), (17, 64), (16, 20, 32), (30, 32, 32)])
def test_fused_steps_match_the_oracle(oracle_mod, shape):
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
    for n in (1, 4):  # the first step, and steps that continue one
        s.step(n)
        o.step(n)
        phi, u = (t.cpu().numpy() for t in s.fields())
        op, ou = o.fields()
        assert np.abs(phi - op).max() < 1e-10 * np.abs(op).max()
        assert np.abs(u - ou).max() < 1e-9 * np.abs(ou).max()
