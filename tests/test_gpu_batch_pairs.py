"""Two steps per launch in batches of plane FP32 lattices, for every collision that
such a lattice may have: each lattice equals its solo run, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["shift", "guo", "body", "guo_body", "fe"])
@pytest.mark.parametrize("tile,graph", [(0, 0), (1, 0), (7, 8)])
def test_pairs_equal_solo_steps(kind, tile, graph):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, inputs, lbm_sc
    build.build()
    stream = torch.cuda.Stream()
    shapes = [(64, 64), (22, 38), (100, 40), (33, 129)]
    hi, lo = (0.9, 0.14) if kind == "fe" else (1.0, 0.04)
    fields = [inputs.drop(s, min(s) / 3.0, rho_hi=hi, rho_lo=lo, seed=8 + k, dtype=np.float32) for k, s in enumerate(shapes)]

    def lattice(shape):
        if kind == "fe":
            return lbm_sc.FELattice(0, shape, 1.0, 0.9, 2.5, "f32", gamma=0.5, stream=stream)
        return lbm_sc.Lattice(0, shape, 1.0, 0.9, 2.4 / 1.04, "f32", stream=stream,
                              forcing="guo" if "guo" in kind else "shift", body_A=1e-4 if "body" in kind else 0.0)

    for n in (4, 10):
        with torch.cuda.stream(stream):
            solo = [lattice(s).set_tuning(0).init(*f).step(n) for s, f in zip(shapes, fields)]
            lats = [lattice(s).init(*f) for s, f in zip(shapes, fields)]
            b = lbm_sc.Batch(lats, tile=tile, graph_steps=graph, stream=stream).step(n)
            for u, v in zip(solo, lats):
                for x, y in zip(u.moments(), v.moments()):
                    assert torch.equal(x, y)
            b.close()
