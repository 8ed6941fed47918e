"""FP32 steps with Guo forcing, bit for bit against a host evaluation that rounds
every operation by itself (fused multiply-adds once, everything else twice).

A product that a later addition takes up must be rounded before it: an assembler
that contracts the two would give other last digits, in every kernel alike, so
comparing kernels with each other does not show it.  A steep profile makes all
components of the force, and so c.F of the diagonal directions, non-zero from
the first step on.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

f32 = np.float32
AXES = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
C2 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0)]
C3 = [(0, 0, 0)] + [tuple(s * v for v in a) for a in AXES for s in (1, -1)] + [
    tuple(s * v for v in a) for a in ((1, 1, 0), (1, -1, 0), (1, 0, 1), (1, 0, -1), (0, 1, 1), (0, 1, -1)) for s in (1, -1)]


def fma(a, b, c):
    return (np.longdouble(a) * np.longdouble(b) + np.longdouble(c)).astype(f32)


def signed_sum(terms):
    """Sum of (sign, term) in order, the first one taken as it is."""
    out = None
    for s, t in terms:
        out = (t if s > 0 else -t) if out is None else (out + t if s > 0 else out - t)
    return np.zeros((), f32) if out is None else out


class HostGuo:
    def __init__(self, rA, rB, tau, G):
        self.D = rA.ndim
        self.c = C2 if self.D == 2 else C3
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if self.D == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.w = [f32(w[sum(map(abs, c))]) for c in self.c]
        self.G, self.om = f32(G), [f32(1.0 / t) for t in tau]
        self.f = [[w * r for w in self.w] for r in (rA, rB)]  # as pulled

    def at(self, a, c):
        """a(x + c) at every node; the arrays' axes are (z,) y, x."""
        return np.roll(a, [-v for v in c[:self.D]], [-1 - d for d in range(self.D)])

    def pairs(self):
        return range(1, len(self.c), 2)

    def density(self, f):
        r = f[1]
        for x in f[2:]:
            r = r + x
        return r + f[0]

    def along(self, i, v):
        """c_i . v"""
        return signed_sum([(self.c[i][d], v[d]) for d in range(self.D) if self.c[i][d]])

    def momentum(self, f):
        return [signed_sum([(self.c[i][d], f[i] - f[i + 1]) for i in self.pairs() if self.c[i][d]]) for d in range(self.D)]

    def accel(self, other):
        """F_s / rho_s from the other species' density."""
        g = [np.zeros(other.shape, f32) for _ in range(self.D)]
        for i in self.pairs():
            dr = self.at(other, self.c[i]) - self.at(other, self.c[i + 1])
            for d in range(self.D):
                if self.c[i][d]:
                    g[d] = fma(f32(self.c[i][d]) * self.w[i], dr, g[d])
        return [x * -self.G for x in g]

    def dot(self, a, b):
        s = a[self.D - 1] * b[self.D - 1]
        for d in range(self.D - 2, -1, -1):
            s = fma(a[d], b[d], s)
        return s

    def state(self):
        r = [self.density(f) for f in self.f]
        return r, [self.momentum(f) for f in self.f], [self.accel(r[1]), self.accel(r[0])]

    def step(self):
        r, j, g = self.state()
        oA, oB = self.om
        inv = f32(1) / fma(r[0], oA, r[1] * oB)
        F = [[r[s] * x for x in g[s]] for s in (0, 1)]
        m = [[fma(f32(0.5), F[s][d], j[s][d]) for d in range(self.D)] for s in (0, 1)]
        u = [fma(m[0][d], oA, m[1][d] * oB) * inv for d in range(self.D)]
        base = fma(f32(-1.5), self.dot(u, u), f32(1))
        for s in (0, 1):
            om, f, new = self.om[s], self.f[s], [None] * len(self.c)
            keep = fma(f32(-0.5), om, f32(1))
            m3uF = f32(-3) * self.dot(u, F[s])
            neq, src = [], []
            for i in self.pairs():
                cu, cF, w = self.along(i, u), self.along(i, F[s]), self.w[i]
                t1, t2 = fma(f32(9) * cu, cF, m3uF), f32(3) * cF
                for k, v, S in ((i, cu, w * (t1 + t2)), (i + 1, -cu, w * (t1 - t2))):
                    d = (w * r[s]) * fma(v, fma(f32(4.5), v, f32(3)), base) - f[k]
                    neq.append((1, d))
                    src.append((1, S))
                    new[k] = fma(keep, S, fma(om, d, f[k]))
            new[0] = fma(keep, -signed_sum(src), fma(om, -signed_sum(neq), f[0]))
            self.f[s] = [self.at(x, tuple(-v for v in c)) for x, c in zip(new, self.c)]

    def moments(self):
        r, j, g = self.state()
        inv = f32(1) / (r[0] + r[1])
        u = [(j[0][d] + j[1][d] + f32(0.5) * fma(r[0], g[0][d], r[1] * g[1][d])) * inv for d in range(self.D)]
        return r[0], r[1], np.stack(u, -1)


@pytest.mark.parametrize("shape", [(24, 70), (40, 16, 70)])
def test_fp32_guo_steps_round_every_operation(shape):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1112_5547_gb300 import build, lbm_sc
    build.build()
    rng = np.random.default_rng(4)
    rA, rB = (rng.uniform(0.1, 0.9, shape).astype(f32) for _ in range(2))
    tau, G = (0.8, 1.3), 1.7
    host, want = HostGuo(rA, rB, tau, G), []
    for _ in range(4):
        host.step()
        want.append(host.moments())
    assert all(np.abs(host.accel(rB)[d]).min() > 0 for d in range(len(shape)))
    lat = lbm_sc.Lattice(len(shape) - 2, shape, *tau, G, "f32", forcing="guo")
    shapes = [lat.tuning()] + [(t, 0) for t in range(len(lbm_sc.TILES)) if lat.tile_fits(t)]
    for tile, zc in shapes:
        lat.set_tuning(tile, zc)
        for n in (1, 2, 4):  # the untuned plane lattice takes four steps in one or two launches
            lat.init(rA, rB).step(n)
            for got, x in zip(lat.moments(), want[n - 1]):
                np.testing.assert_array_equal(got.cpu().numpy(), x, err_msg=str((tile, zc, n)))
