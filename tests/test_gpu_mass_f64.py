"""Mass of the FP64 step over long runs, relaxation times away from 1.

The rest population relaxes by minus the sum of the increments that the moving
ones receive, so a step changes a node's mass by the roundings of the final
updates alone: at most about half an ulp of rho, of a sign that changes from node
to node.  Over N nodes they add up as sqrt(N), so a species' relative mass moves by
no more than eps / 2 / sqrt(N) a step even if every node repeated its rounding at
every step; a closure that rounds at the scale of rho repeats the same error in
all the nodes of a uniform region, and moves it by a good part of eps / 2 a step.
"""
import math

import numpy as np
import pytest

from paper_1112_5547_gb300 import inputs

pytestmark = pytest.mark.gpu

G0 = 2.4 / 1.04


@pytest.mark.parametrize("forcing", ["shift", "guo"])
@pytest.mark.parametrize("tau", [(0.7, 0.7), (0.9, 1.1), (3.0, 3.0), (3.0, 0.7)])
@pytest.mark.parametrize("shape,steps", [((48, 48), 4000), ((24, 24, 24), 2000)])
def test_fp64_mass_does_not_drift(shape, steps, tau, forcing):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, lbm_sc
    build.build()
    f = inputs.drop(shape, shape[0] / 4.0, seed=3, dtype=np.float64)
    lat = lbm_sc.Lattice(len(shape) - 2, shape, *tau, G0, "f64", forcing=forcing).init(*f)

    def masses():
        return [math.fsum(t.cpu().numpy().ravel()) for t in lat.moments()[:2]]

    before = masses()
    after = (lat.step(steps), masses())[1]
    bound = steps * np.finfo(np.float64).eps / 2 / math.sqrt(math.prod(shape))
    for a, b in zip(before, after):
        assert abs(b - a) / a < bound
