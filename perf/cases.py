"""The work that users of this framework have it do, as cases that can be timed.

A case is one job through the public entry points: initial densities in, a
number of time steps, fields (and, where a program monitors its run, the FP64
diagnostics) out.  The sizes are those of the README, the tests, the benchmark
and the serving stream; the numbers of steps are short stretches of runs that
take thousands of them.

``kind``:
  drop   two-component Shan-Chen drop on one lattice (``Lattice``), plain or with
         the Kolmogorov body force and / or Guo forcing;
  fe     the free-energy model on one lattice (``FELattice``);
  batch  independent drop lattices advanced together (``Batch``);
  pfm    the phase-field solver (``PFM``): a drop in a Kolmogorov flow kept up by its body force.
"""
import math

import numpy as np
import torch

from paper_1112_5547_gb300 import autotune, lbm_sc, phase_field, serving

G0 = 2.4 / 1.04          # coupling of the static-drop recipe (rho_hi + rho_lo = 1.04)
CS2 = 1.0 / 3.0
PFM_RHO, PFM_TAU, PFM_G, PFM_DT = 1.4, 0.6, 0.3, 0.1
PFM_U = 0.02             # amplitude of the Kolmogorov flow that the phase-field drops sit in
FE_G, FE_GAMMA = 2.5, 0.5
RAGGED = (32, 48, 64, 96, 128)  # edges of the benchmark's ragged batch
LAPLACE_RADII = (16, 24, 32, 40, 48, 56, 64, 72)


def listed():
    return [
        # the parity run and the smallest lattice of the serving stream: launches and latency count
        dict(name="drop2d_64", kind="drop", dim=2, nx=64, ny=64, nz=1, precision="f32", steps=500, monitor=100,
             forcing="shift", body_A=0.0, tuned=False),
        # Laplace's law: one drop per radius, all radii advanced as one batch under CUDA graphs
        dict(name="laplace2d_batch", kind="batch", dim=2, lattices=8, edge=256, steps=300, precision="f32", tile=7,
             zchunk=0, graph_steps=100),
        # a large plane lattice, fields read at the end
        dict(name="drop2d_4096", kind="drop", dim=2, nx=4096, ny=4096, nz=1, precision="f32", steps=60, monitor=0,
             forcing="shift", body_A=0.0, tuned=False),
        # a small box in FP64, as used to validate a set-up before the long FP32 run
        dict(name="drop3d_48_f64", kind="drop", dim=3, nx=48, ny=48, nz=48, precision="f64", steps=100, monitor=50,
             forcing="shift", body_A=0.0, tuned=False),
        # the README's drop, its peak speed and masses read every 50 steps
        dict(name="drop3d_128", kind="drop", dim=3, nx=128, ny=128, nz=128, precision="f32", steps=200, monitor=50,
             forcing="shift", body_A=0.0, tuned=False),
        # drop under Kolmogorov forcing with Guo's scheme in a box that no tile divides; leakage from the diagnostics
        dict(name="kolmogorov_guo_ragged", kind="drop", dim=3, nx=180, ny=130, nz=150, precision="f32", steps=100,
             monitor=50, forcing="guo", body_A=1e-6, tuned=False),
        # the free-energy model at the README's size
        dict(name="fe3d_128", kind="fe", dim=3, nx=128, ny=128, nz=128, precision="f32", steps=100, monitor=0),
        # a 256^3 drop in paired 16-bit storage
        dict(name="drop3d_256_bf16rest", kind="drop", dim=3, nx=256, ny=256, nz=256, precision="bf16_rest", steps=100,
             monitor=0, forcing="shift", body_A=0.0, tuned=False),
        # the benchmark's lattice with its launch shape of the tuning cache
        dict(name="drop3d_512", kind="drop", dim=3, nx=512, ny=512, nz=512, precision="f32", steps=40, monitor=0,
             forcing="shift", body_A=0.0, tuned=True),
        # 64 ragged lattices as the server batches them
        dict(name="ragged3d_batch", kind="batch", dim=3, lattices=64, edge=0, steps=60, precision="f32", tile=-1,
             zchunk=0, graph_steps=0),
        # the phase-field solver at the benchmark's size, and a plane one in FP64
        dict(name="pfm3d_256", kind="pfm", dim=3, nx=256, ny=256, nz=256, precision="f32", steps=20),
        dict(name="pfm2d_512_f64", kind="pfm", dim=2, nx=512, ny=512, nz=1, precision="f64", steps=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps(rng, nodes, budget, most=500):
    return max(10, min(int(most * rng.uniform(0.4, 1.0)), int(budget // nodes)))


def draw(rng):
    kind = rng.choice(["drop", "drop", "drop", "drop", "fe", "batch", "pfm"])
    if kind == "pfm":
        dim = rng.choice([2, 3])
        # powers of two and small multiples of them as users choose for transforms, and any odd edge
        edge = lambda lo, hi: rng.choice([1 << int(rng.uniform(math.log2(lo), math.log2(hi) + 1)),  # noqa: E731
                                          _log_int(rng, lo // 2, hi // 2) * 2, _log_int(rng, lo, hi)])
        n = [edge(48, 1024) for _ in range(2)] if dim == 2 else [edge(32, 256) for _ in range(3)]
        nodes = math.prod(n)
        return dict(kind="pfm", dim=dim, nx=n[0], ny=n[1], nz=n[2] if dim == 3 else 1,
                    precision=rng.choice(["f32", "f64"]), steps=_steps(rng, nodes, 1.5e8, 100))
    if kind == "batch":
        if rng.random() < 0.5:
            edge, count = _log_int(rng, 64, 512), rng.randint(2, 24)
            return dict(kind="batch", dim=2, lattices=count, edge=edge, steps=_steps(rng, edge * edge * count, 4e8, 300),
                        precision="f32", tile=7, zchunk=0, graph_steps=rng.choice([0, 20, 100]))
        return dict(kind="batch", dim=3, lattices=rng.randint(4, 64), edge=0, steps=rng.randint(20, 60),
                    precision=rng.choice(["f32", "f32", "bf16_rest"]), tile=-1, zchunk=0, graph_steps=0)
    dim = rng.choice([2, 3])
    if dim == 2:
        nx, ny, nz = _log_int(rng, 48, 4096), _log_int(rng, 48, 4096), 1
    else:
        e = _log_int(rng, 24, 320)
        nx, ny, nz = (max(16, int(e * rng.uniform(0.7, 1.4))) for _ in range(3))
    nodes = nx * ny * nz
    precision = rng.choice(["f32", "f32", "f32", "f64"] if kind == "fe" else
                           ["f32", "f32", "f32", "f64", "bf16_rest", "f16_rest"])
    case = dict(kind=kind, dim=dim, nx=nx, ny=ny, nz=nz, precision=precision,
                steps=_steps(rng, nodes, 2e8 if precision == "f64" else 1e9), monitor=rng.choice([0, 50]))
    if kind == "drop":
        case.update(forcing=rng.choice(["shift", "shift", "guo"]), body_A=rng.choice([0.0, 0.0, 1e-6]), tuned=False)
    return case


# ---- inputs -------------------------------------------------------------------
def _shape(c):
    return (c["ny"], c["nx"]) if c["dim"] == 2 else (c["nz"], c["ny"], c["nx"])


def _drop(shape, R, centre, hi, lo, seed, dtype):
    """The drop recipe (tanh profile of width 2 and seeded noise of 1e-3) made on the GPU."""
    r2 = 0.0
    for a, n in enumerate(shape):
        d = (torch.arange(n, device="cuda", dtype=torch.float64) - centre[a]).abs()
        d = torch.minimum(d, n - d) ** 2
        r2 = r2 + d.view([-1 if b == a else 1 for b in range(len(shape))])
    rA = lo + (hi - lo) * 0.5 * (1.0 - torch.tanh((r2.sqrt_() - R) / 2.0))
    del r2
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = lambda: torch.rand(shape, generator=g, device="cuda").mul_(2e-3).sub_(1e-3)  # noqa: E731
    rB = (hi + lo) - rA
    return rA.add_(noise()).to(dtype), rB.add_(noise()).to(dtype)


def _fields(shape, seed, dtype, hi=1.0, lo=0.04):
    g = torch.Generator().manual_seed(seed)
    v = torch.rand(4, generator=g, dtype=torch.float64).tolist()
    R = min(shape) * (0.2 + 0.1 * v[0])
    centre = [n * (0.3 + 0.4 * w) for n, w in zip(shape, v[1:])]
    return _drop(shape, R, centre, hi, lo, seed, dtype)


def _dtype(c):
    return torch.float64 if c["precision"] == "f64" else torch.float32


def _batch_specs(c, seed):
    """(shape, tau_A, tau_B, G, drop radius or None for the seeded one) of each lattice of a batch."""
    g = torch.Generator().manual_seed(seed)
    out = []
    for k in range(c["lattices"]):
        v = torch.rand(4, generator=g, dtype=torch.float64).tolist()
        if c["dim"] == 2:
            out.append(((c["edge"],) * 2, 1.0, 1.0, G0, LAPLACE_RADII[k % 8] * c["edge"] / 256.0))
        else:  # every edge of the recipe in turn, so that every seed is the same amount of work
            out.append(((RAGGED[k % len(RAGGED)],) * 3, 0.9 + 0.2 * v[0], 0.9 + 0.2 * v[1], (2.3 + 0.2 * v[2]) / 1.04,
                        None))
    return out


def _batch_fields(c, seed):
    out = []
    for k, (shape, tA, tB, G, R) in enumerate(_batch_specs(c, seed)):
        s = seed * 1009 + k
        out.append(_fields(shape, s, _dtype(c)) if R is None else
                   _drop(shape, R, [n / 2 for n in shape], 1.0, 0.04, s, _dtype(c)))
    return out


def _pfm_phi(c, seed):
    a, b = _fields(_shape(c), seed, torch.float64, 1.2, 0.2)
    return (a - b).to(_dtype(c))


def _pfm_flow(c):
    """(u, A): the steady flow u_x = U sin(2 pi y / ny) and the forcing amplitude that keeps it up."""
    k = 2 * math.pi / c["ny"]
    u = torch.zeros(_shape(c) + (c["dim"],), device="cuda", dtype=torch.float64)
    u[..., 0] = PFM_U * torch.sin(k * torch.arange(c["ny"], device="cuda", dtype=torch.float64)).view(-1, 1)
    return u.to(_dtype(c)), PFM_U * CS2 * (PFM_TAU - 0.5) * k * k


def prepare(case, seed):
    c = case
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(stream):
        st = {"case": c, "stream": stream}
        if c["kind"] == "pfm":
            st["phi"] = _pfm_phi(c, seed)
            st["u"], A = _pfm_flow(c)
            st["solver"] = phase_field.PFM(_shape(c), PFM_RHO, PFM_TAU, PFM_G, PFM_DT, c["precision"], stream=stream,
                                           body_A=A)
        elif c["kind"] == "batch":
            lat = lbm_sc.LBM_D2Q9 if c["dim"] == 2 else lbm_sc.LBM_D3Q19
            st["fields"] = _batch_fields(c, seed)
            lats = [lbm_sc.Lattice(lat, shape, tA, tB, G, c["precision"], stream=stream).init(*f)
                    for (shape, tA, tB, G, _), f in zip(_batch_specs(c, seed), st["fields"])]
            tile, zc = serving.Server.batch_shape(lats) if c["tile"] < 0 else (c["tile"], c["zchunk"])
            st["lattices"] = lats
            st["batch"] = lbm_sc.Batch(lats, tile=tile, zchunk=zc, graph_steps=c["graph_steps"], stream=stream)
        else:
            lat = lbm_sc.LBM_D2Q9 if c["dim"] == 2 else lbm_sc.LBM_D3Q19
            if c["kind"] == "fe":
                st["fields"] = _fields(_shape(c), seed, _dtype(c), 0.9, 0.14)
                st["lattice"] = lbm_sc.FELattice(lat, _shape(c), 1.0, 1.0, FE_G, c["precision"], gamma=FE_GAMMA,
                                                 stream=stream)
            else:
                st["fields"] = _fields(_shape(c), seed, _dtype(c))
                st["lattice"] = lbm_sc.Lattice(lat, _shape(c), 1.0, 1.0, G0, c["precision"], stream=stream,
                                               body_A=c["body_A"], forcing=c["forcing"])
            if c.get("tuned"):
                autotune.tuned(st["lattice"], store=False)  # the tuning cache holds this size
    torch.cuda.current_stream().wait_stream(stream)
    return st


def run(state):
    c = state["case"]
    with torch.cuda.stream(state["stream"]):
        if c["kind"] == "pfm":
            phi, u = state["solver"].init(state["phi"], state["u"]).step(c["steps"]).fields()
            return {"phi": phi, "u": u}
        if c["kind"] == "batch":
            b = state["batch"]
            # an even number of steps, so the lattices are where a new init() puts them
            for lat, f in zip(state["lattices"], state["fields"]):
                lat.init(*f)
            b.step(c["steps"] // 2 * 2)
            out = []
            for lat in state["lattices"]:
                out.append(lat.moments())
            # one array per field over the whole batch, as a program that stores the batch keeps them
            return {"rho_A": torch.cat([m[0].reshape(-1) for m in out]),
                    "rho_B": torch.cat([m[1].reshape(-1) for m in out]),
                    "u": torch.cat([m[2].reshape(-1) for m in out]),
                    "p": torch.cat([m[3].reshape(-1) for m in out])}
        lat = state["lattice"].init(*state["fields"])
        done, seen, counts = 0, [], []
        while done < c["steps"]:
            n = min(c["monitor"] or c["steps"], c["steps"] - done)
            lat.step(n)
            done += n
            if c["monitor"]:
                d = lat.diagnostics(check=False)
                # what a run is watched by: masses, energy, peak speed, extrema; leakage and instability counts
                seen.append([d[k] for k in ("mass_A", "mass_B", "kinetic_energy", "max_speed", "min_rho_A", "min_rho_B")])
                counts.append([d["droplet_nodes"], d["nonfinite"]])
        rA, rB, u, p = lat.moments()
        out = {"rho_A": rA, "rho_B": rB, "u": u, "p": p}
        if seen:
            out.update(watch=np.array(seen), counts=np.array(counts, dtype=np.int64))
        return out


# ---- the work of a pass ---------------------------------------------------------
def work(case):
    """Algorithmic bytes and operations of one pass.  A lattice step reads and
    writes every population once; initial densities are read, the reported
    fields and the initial populations written once.  A phase-field step reads
    and writes its spectral state (phi, u and the two previous right-hand sides)
    once and passes the fields once between spectral and physical space."""
    c = case
    D = c["dim"]
    if c["kind"] == "pfm":
        e = 8 if c["precision"] == "f64" else 4
        shape = _shape(c)
        N = math.prod(shape)
        M = 2 * N * (c["nx"] // 2 + 1) / c["nx"]  # reals of a half spectrum
        inv, fwd = 2 + 2 * D, 2 + D + D * (D + 1) // 2
        # phi, u and one derivative field inwards; two scalar, D force and D stress combinations outwards
        step = (4 * (1 + D) + 2 * (D + 3) + 2 * (2 + 2 * D)) * M * e
        fft = 2.5 * N * math.log2(N) * (inv + fwd) + 120 * N
        return {"bytes": c["steps"] * step + 2 * (1 + D) * N * e, "flops": c["steps"] * fft}
    Q = 9 if D == 2 else 19
    per = {"f64": 16 * Q, "f32": 8 * Q, "bf16_rest": 4 * Q + 8, "f16_rest": 4 * Q + 8}[c["precision"]]
    ce = 8 if c["precision"] == "f64" else 4
    ops = (230 if D == 2 else 480) * (1.6 if c["kind"] == "fe" or c.get("forcing") == "guo" else 1.0)
    if c["kind"] == "batch":
        N = sum(math.prod(s[0]) for s in _batch_specs(c, 0))
    else:
        N = math.prod(_shape(c))
    checks = (c["steps"] + c["monitor"] - 1) // c["monitor"] if c.get("monitor") else 0
    b = N * (c["steps"] * 2 * per + (2 * ce + per) + checks * per + (per + (3 + D) * ce))
    return {"bytes": b, "flops": N * (c["steps"] * ops + (1 + checks) * ops / 3)}


# ---- the same in plain torch, FP64 ----------------------------------------------
def _velocities(D):
    if D == 2:
        c = [(x, y) for y in (-1, 0, 1) for x in (-1, 0, 1)]
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}
    else:
        c = [(x, y, z) for z in (-1, 0, 1) for y in (-1, 0, 1) for x in (-1, 0, 1) if abs(x) + abs(y) + abs(z) < 3]
        w = {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
    return c, [w[sum(abs(a) for a in v)] for v in c]


def _shifted(a, c, sign):
    """a(x + sign c) for every node; the last axes of a are (z,) y, x."""
    axes = [-1 - k for k in range(len(c))]
    return torch.roll(a, [-sign * v for v in c], axes)


class _Exact:
    """Lattice Boltzmann step in FP64 on a stack of equally sized lattices (leading axis)."""

    def __init__(self, D, rA, rB, tA, tB, G, forcing="shift", body_A=0.0, fe=None):
        self.D, self.fe, self.forcing, self.G = D, fe, forcing, G
        self.c, self.w = _velocities(D)
        self.tau = (tA, tB)
        ny = rA.shape[-2]
        y = torch.arange(ny, device=rA.device, dtype=torch.float64)
        self.body = body_A * torch.sin(2 * math.pi * y / ny).view([ny, 1]) if body_A else None
        a, b = (rA + rB, rA - rB) if fe else (rA, rB)
        self.f = [[w * a for w in self.w], [w * b for w in self.w]]

    def cu(self, c, u):
        return sum(v * u[d] for d, v in enumerate(c) if v) if any(c) else torch.zeros_like(u[0])

    def sums(self):
        r = [sum(f) for f in self.f]
        j = [[sum(c[d] * f for c, f in zip(self.c, fs) if c[d]) for d in range(self.D)] for fs in self.f]
        return r, j

    def force(self, r):
        """F_s / rho_s of both species."""
        g = []
        for s in (0, 1):
            v = [0.0] * self.D
            for c, w in zip(self.c, self.w):
                if any(c):
                    o = _shifted(r[1 - s], c, 1)
                    for d in range(self.D):
                        if c[d]:
                            v[d] = v[d] + (w * c[d]) * o
            v = [-self.G * x for x in v]
            if self.body is not None:
                v[0] = v[0] + self.body
            g.append(v)
        return g

    def step(self):
        r, j = self.sums()
        if self.fe:
            self.collide_fe(r, j)
        else:
            g = self.force(r)
            den = r[0] / self.tau[0] + r[1] / self.tau[1]
            for_u = [[j[s][d] + (0.5 * r[s] * g[s][d] if self.forcing == "guo" else 0.0) for d in range(self.D)]
                     for s in (0, 1)]
            up = [(for_u[0][d] / self.tau[0] + for_u[1][d] / self.tau[1]) / den for d in range(self.D)]
            for s in (0, 1):
                t = self.tau[s]
                u = up if self.forcing == "guo" else [up[d] + t * g[s][d] for d in range(self.D)]
                uu = sum(x * x for x in u)
                F = [r[s] * x for x in g[s]]
                uF = sum(a * b for a, b in zip(u, F))
                for i, (c, w) in enumerate(zip(self.c, self.w)):
                    cu = self.cu(c, u)
                    feq = w * r[s] * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)
                    f = self.f[s][i] + (feq - self.f[s][i]) / t
                    if self.forcing == "guo":
                        cF = self.cu(c, F)
                        f = f + (1 - 0.5 / t) * w * (3 * (cF - uF) + 9 * cu * cF)
                    self.f[s][i] = f
        for s in (0, 1):
            self.f[s] = [_shifted(f, c, -1) if any(c) else f for f, c in zip(self.f[s], self.c)]

    def collide_fe(self, r, j):
        g, kappa, gamma = self.fe
        rho, phi = r
        D = self.D
        u = [x / rho for x in j[0]]
        gp, lap = [0.0] * D, 0.0
        for c, w in zip(self.c, self.w):
            if any(c):
                o = _shifted(phi, c, 1)
                lap = lap + 6 * w * (o - phi)
                for d in range(D):
                    if c[d]:
                        gp[d] = gp[d] + (3 * w * c[d]) * o
        uu, gg = sum(x * x for x in u), sum(x * x for x in gp)
        mu = 0.5 * CS2 * torch.log((rho + phi) / (rho - phi)) - 0.5 * g * CS2 * phi - kappa * lap
        s = 0.25 * g * CS2 * (rho * rho - phi * phi) - kappa * phi * lap - 0.5 * kappa * gg
        sg = gamma * mu - CS2 * phi
        for n, tau in ((0, self.tau[0]), (1, self.tau[1])):
            new, total = [None] * len(self.c), 0.0
            for i, (c, w) in enumerate(zip(self.c, self.w)):
                if not any(c):
                    rest = i
                    continue
                cu, cg = self.cu(c, u), self.cu(c, gp)
                iso = sum(v * v for v in c) - D / 3.0
                if n == 0:
                    h = s * iso + kappa * (cg * cg - CS2 * gg) + rho * (cu * cu - CS2 * uu)
                else:
                    h = sg * iso + phi * (cu * cu - CS2 * uu)
                base = r[n]
                feq = w * (base + 3 * base * cu + 4.5 * h)
                total = total + feq
                new[i] = self.f[n][i] + (feq - self.f[n][i]) / tau
            f0 = self.f[n][rest]
            new[rest] = f0 + (r[n] - total - f0) / tau
            self.f[n] = new

    def moments(self):
        r, j = self.sums()
        if self.fe:
            rho, phi = r
            rA, rB, u = 0.5 * (rho + phi), 0.5 * (rho - phi), [x / rho for x in j[0]]
            G = self.fe[0]
        else:
            rA, rB = r
            g = self.force(r)
            u = [(j[0][d] + j[1][d] + 0.5 * (rA * g[0][d] + rB * g[1][d])) / (rA + rB) for d in range(self.D)]
            G = self.G
        return rA, rB, torch.stack(u, -1), CS2 * (rA + rB) + CS2 * G * rA * rB


def _exact_pfm(c, seed):
    D, dt = c["dim"], PFM_DT
    phi0 = _pfm_phi(c, seed).double()
    shape = phi0.shape
    M = PFM_RHO * (PFM_TAU - 0.5)
    nu, g_tau = CS2 * (PFM_TAU - 0.5), PFM_TAU * PFM_G / (PFM_TAU - 0.5)
    Dc, xi2 = M * g_tau * CS2 / 2, CS2 / 2
    k2, kd = 0.0, []
    for d in range(D):  # component d along axis -1 - d; x is the half axis
        n = shape[-1 - d]
        f = (torch.fft.rfftfreq if d == 0 else torch.fft.fftfreq)(n, device="cuda", dtype=torch.float64)
        k = 2 * math.pi * f
        view = [1] * D
        view[-1 - d] = -1
        k2 = k2 + (k * k).view(view)
        k = k.clone()
        if n % 2 == 0:
            k[n // 2] = 0.0
        kd.append(k.view(view))
    kd2 = sum(k * k for k in kd)
    kd2 = torch.where(kd2 == 0, 1.0, kd2)
    F, B = (lambda a: torch.fft.rfftn(a)), (lambda a: torch.fft.irfftn(a, s=shape))
    u0, A = _pfm_flow(c)
    ph, uh = F(phi0), [F(u0[..., d].double()) for d in range(D)]
    y = torch.arange(c["ny"], device="cuda", dtype=torch.float64).view(-1, 1)
    body = F((A * torch.sin(2 * math.pi * y / c["ny"])).expand(shape))
    Sp = Np = None
    lam, vis = Dc * (2 * k2 + dt * Dc / 2 * k2 * k2), nu * k2
    for _ in range(c["steps"]):
        phi, lap, u = B(ph), B(-k2 * ph), [B(x) for x in uh]
        gp = [B(1j * k * ph) for k in kd]
        ln = torch.log((PFM_RHO + phi) / (PFM_RHO - phi))
        S = (-F(sum(a * b for a, b in zip(u, gp))) - Dc * k2 * F(ln / g_tau - 3 * phi)
             - Dc * (xi2 - dt * Dc / 2) * k2 * k2 * ph)
        mu = 0.5 * CS2 * ln - 0.5 * PFM_G * CS2 * phi - 0.25 * PFM_G * CS2 * CS2 * lap
        N = [F(mu * gp[a]) / PFM_RHO - sum(1j * kd[b] * F(u[a] * u[b]) for b in range(D)) for a in range(D)]
        N[0] = N[0] + body
        kN = sum(k * x for k, x in zip(kd, N)) / kd2
        N = [torch.where(k2 == 0, 0.0, x - k * kN) for k, x in zip(kd, N)]
        Sp, Np = Sp if Sp is not None else S, Np if Np is not None else N
        ph = (ph * (1 - dt * lam / 2) + dt * (3 * S - Sp) / 2) / (1 + dt * lam / 2)
        uh = [(x * (1 - dt * vis / 2) + dt * (3 * n - m) / 2) / (1 + dt * vis / 2) for x, n, m in zip(uh, N, Np)]
        Sp, Np = S, N
    return {"phi": B(ph), "u": torch.stack([B(x) for x in uh], -1)}


def exact(case, seed):
    c = case
    if c["kind"] == "pfm":
        return _exact_pfm(c, seed)
    if c["kind"] == "batch":
        specs, fields = _batch_specs(c, seed), _batch_fields(c, seed)
        got = [None] * len(specs)
        for shape in {s[0] for s in specs}:
            ks = [k for k, s in enumerate(specs) if s[0] == shape]
            one = [1] * len(shape)
            par = [torch.tensor([specs[k][m] for k in ks], dtype=torch.float64, device="cuda").view([-1] + one)
                   for m in (1, 2, 3)]
            e = _Exact(c["dim"], *(torch.stack([fields[k][s] for k in ks]).double() for s in (0, 1)), *par)
            for _ in range(c["steps"] // 2 * 2):
                e.step()
            m = e.moments()
            for i, k in enumerate(ks):
                got[k] = [x[i].reshape(-1) for x in m]
        return {k: torch.cat([m[i] for m in got]) for i, k in enumerate(("rho_A", "rho_B", "u", "p"))}
    nodes = math.prod(_shape(c))
    if nodes > 4e7 or nodes * c["steps"] > 2.5e9:
        return None  # over 20 s, and more memory than is free
    rA, rB = (x.double() for x in _fields(_shape(c), seed, _dtype(c), *((0.9, 0.14) if c["kind"] == "fe" else ())))
    fe = (FE_G, FE_G * CS2 * CS2 / 4, FE_GAMMA) if c["kind"] == "fe" else None
    e = _Exact(c["dim"], rA, rB, 1.0, 1.0, G0, c.get("forcing", "shift"), c.get("body_A", 0.0), fe)
    seen = []
    for t in range(1, c["steps"] + 1):
        e.step()
        if c["monitor"] and (t % c["monitor"] == 0 or t == c["steps"]):
            a, b, u, p = e.moments()
            uu = (u * u).sum(-1)
            seen.append([float(a.sum()), float(b.sum()), float((0.5 * (a + b) * uu).sum()), float(uu.max().sqrt()),
                         float(a.min()), float(b.min())])
    rA, rB, u, p = e.moments()
    out = {"rho_A": rA, "rho_B": rB, "u": u, "p": p}
    if seen:
        out.update(watch=np.array(seen), counts=None)
    return out
