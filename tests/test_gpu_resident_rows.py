"""Tall, narrow and thin plane lattices in FP32: those whose steps run in one
cluster, at the edges of the rows a CTA takes (one, two and three passes), and
the next that do not, against single steps, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 9), (224, 5), (225, 31), (480, 24), (481, 20), (736, 16), (737, 16), (1000, 1), (1000, 12),
                                   (3000, 4), (16, 190), (17, 190), (32, 256), (33, 256)])
def test_tall_and_narrow_lattices(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, inputs, lbm_sc
    build.build()
    f = inputs.drop(shape, 0.4 * min(shape), seed=6, dtype=np.float32)
    for forcing in ("shift", "guo"):
        many = lbm_sc.Lattice(0, shape, 1.0, 0.9, 2.4 / 1.04, "f32", forcing=forcing, body_A=1e-4)
        one = lbm_sc.Lattice(0, shape, 1.0, 0.9, 2.4 / 1.04, "f32", forcing=forcing, body_A=1e-4)
        for n in (3, 6, 25):
            many.init(*f).step(n)
            one.init(*f)
            for _ in range(n):
                one.step(1)
            for x, y in zip(many.moments(), one.moments()):
                assert torch.equal(x, y), n
