"""The steps of a phase-field run may be divided over calls as one likes: the same
bits, whichever kernels begin and end a call."""
import numpy as np
import pytest

from paper_1112_5547_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(256, 512), (128, 960), (60, 100), (64, 48, 96), (32, 160, 64), (20, 24, 30)])
def test_calls_of_a_run_may_be_split(shape, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, phase_field
    build.build()
    a, b = inputs.drop(shape, min(shape) / 4.0, rho_hi=1.2, rho_lo=0.2, seed=9)
    ny = shape[-2]
    u = np.zeros(shape + (len(shape),))
    u[..., 0] = 0.02 * np.sin(2 * np.pi * np.arange(ny) / ny)[:, None]

    def run(*calls):
        s = phase_field.PFM(shape, 1.4, 0.6, 0.3, 0.1, precision, body_A=1e-4).init(a - b, u)
        for n in calls:
            s.step(n)
            out = s.fields()  # reading the fields in between changes nothing either
        return out

    whole = run(12)
    for calls in ((1,) * 12, (5, 1, 6), (0, 7, 5)):
        for x, y in zip(run(*calls), whole):
            assert torch.equal(x, y)
