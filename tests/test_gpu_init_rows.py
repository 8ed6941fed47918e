"""Initial populations at the edges of the row shapes the kernel chooses between
(narrow and wide rows of each storage width, few and many cells, resting and
moving fluids): every cell holds the equilibrium of the node that will pull it,
w_i rho (1 + 3 c.u + 9/2 (c.u)^2 - 3/2 u.u) at x + c_i, and the images of the
outermost nodes equal them bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C2 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
C3 = [(0, 0, 0)] + [tuple(s * v for v in a) for a in ((1, 0, 0), (0, 1, 0), (0, 0, 1)) for s in (1, -1)] + [
    tuple(s * v for v in a) for a in ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)) for s in (1, -1)]
# 12 sectors: 96 values of 32 bits, 48 of 64, 192 of 16
SHAPES = {"f32": [(3, 5, 1), (2, 3, 7), (4, 5, 95), (4, 5, 96), (40, 30, 97), (20, 30, 130)],
          "f64": [(3, 5, 1), (2, 3, 4), (4, 5, 47), (4, 5, 48), (50, 40, 49)],
          "bf16": [(3, 5, 1), (2, 3, 15), (4, 5, 191), (4, 5, 192), (20, 30, 193)],
          "bf16_rest": [(3, 5, 1), (2, 3, 7), (4, 5, 95), (4, 5, 96), (40, 30, 97)]}


@pytest.mark.parametrize("precision", list(SHAPES))
@pytest.mark.parametrize("moving", [False, True])
@pytest.mark.parametrize("D", [2, 3])
def test_initial_populations(precision, moving, D):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, lbm_sc
    build.build()
    c = C2 if D == 2 else C3
    w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if D == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    # one rounding of the stored value and a handful of the formula's; 16-bit values are of
    # f - w rho_ref (rho_ref 0.5) or of the deviation from w rho, at most w (1 + 3 |u|) each
    tol = {"f32": 8 * 2.0 ** -24, "f64": 8 * 2.0 ** -53, "bf16": 2.0 ** -8, "bf16_rest": 2.0 ** -8}[precision]
    kw = dict(rho_ref_A=0.5, rho_ref_B=0.5) if precision == "bf16" else {}
    rng = np.random.default_rng(6)
    for shape in SHAPES[precision]:
        shape = shape[1:] if D == 2 else shape
        rho = [rng.uniform(0.1, 1.0, shape).astype(np.float32) for _ in range(2)]
        u = rng.uniform(-0.05, 0.05, shape + (D,)).astype(np.float32) if moving else None
        lat = lbm_sc.Lattice(D - 2, shape, 1.0, 1.0, 2.0, precision, **kw).init(*rho, u)
        px, py, gx, gy = lbm_sc.lbm_sc_layout(lat.handle)[2:6]
        f = lat.populations().double().cpu().numpy()
        if precision == "bf16_rest":
            f = np.moveaxis(f, -1, 0)
        ny, nx = shape[-2:]
        xs = np.arange(-2, nx + 2)
        ys = np.arange(-2, ny + 2)
        cells = f[:, :, :, ys[:, None] + gy, xs[None, :] + gx]
        images = f[:, :, :, (ys % ny)[:, None] + gy, (xs % nx)[None, :] + gx]
        np.testing.assert_array_equal(cells, images)
        if precision == "bf16_rest":  # words hold the deviation from the storing node's own density
            continue
        for s in (0, 1):
            for i, ci in enumerate(c):
                ax = [-1 - d for d in range(D)]
                to = [-v for v in ci[:D]]
                r = np.roll(rho[s].astype(np.float64), to, ax)
                wi = w[sum(map(abs, ci))]
                want = wi * r
                if moving:
                    v = [np.roll(u[..., d].astype(np.float64), to, ax) for d in range(D)]
                    cu = sum(ci[d] * v[d] for d in range(D))
                    want = want * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * sum(x * x for x in v))
                got = f[s, i][:, gy:gy + ny, gx:gx + nx].reshape(shape)
                off = wi * 0.5 if precision == "bf16" else 0.0
                assert np.abs(got + off - want).max() <= tol * wi * 1.2, (shape, s, i)
