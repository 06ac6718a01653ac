"""The work that users of this framework have it do, as cases that can be timed and compared.

A case is one of three jobs, each through the public Python entry points:

  "run"       initial fields -> n steps -> the final state (Solver.init, step, get_state); with
              "filtered", the steps are step_filtered's (turbulence as forcing, closure and step)
  "optimise"  one iteration of an optimisation of the force field: a rollout, a loss on its final
              velocity, and the gradient (rollout.velocity_after and backward)

The listed cases are the flows of the repository's benchmark, tests and README at their sizes, and
ragged sizes beside them; draw() spreads the same kinds of flow over the range of sizes, storage
types, boundaries, forces and collision options that the entry points take. exact() computes the
same results in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1202_6074_gb300 import cmlbm, rollout

DEVICE = "cuda"
BYTES = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}
EXACT_CELL_STEPS = 1.5e9        # exact() of a larger case would take too long


def _case(name=None, job="run", lattice="D3Q27", nx=32, ny=32, nz=32, storage="f32", steps=20, flow="vortices",
          bc="periodic", force="none", tau=0.51, omega_bulk=1.0, omega_3=1.0, omega_4=1.0, cs=0.0, van_driest=False,
          attractor="maxwell", reduced=False, segment=10):
    c = dict(job=job, lattice=lattice, nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, flow=flow, bc=bc, force=force,
             tau=tau, omega_bulk=omega_bulk, omega_3=omega_3, omega_4=omega_4, cs=cs, van_driest=van_driest,
             attractor=attractor, reduced=reduced, segment=segment)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's lattice at its smallest use: a force-driven channel, many steps of a few us
        # each (launches and latency)
        _case("channel2d_f64_64x32", lattice="D2Q9", nx=64, ny=32, nz=1, storage="f64", steps=500, flow="rest",
              bc="channel", force="uniform", tau=0.8, omega_bulk=0.0),
        # a 2D flow of an ordinary, ragged size between moving walls
        _case("couette2d_f32_1500x701", lattice="D2Q9", nx=1500, ny=701, nz=1, storage="f32", steps=100,
              bc="couette", tau=0.55, omega_bulk=0.0),
        # a small 3D box, the default grid of a new handle: a parameter study, a unit test, a first try
        _case("vortices_f32_32", nx=32, ny=32, nz=32, storage="f32", steps=100),
        # the benchmark's headline: decaying vortices, FP32
        _case("vortices_f32_256", nx=256, ny=256, nz=256, storage="f32", steps=20, tau=0.50382),
        # the same flow with 16-bit storage, which users take for twice the grid
        _case("vortices_bf16_256", nx=256, ny=256, nz=256, storage="bf16", steps=20, tau=0.50382),
        # forced isotropic turbulence, large-eddy simulation, a force per cell: the largest
        _case("forced_les_bf16_512", nx=512, ny=512, nz=512, storage="bf16", steps=10, force="field", tau=0.5005, cs=0.1),
        # a wall-bounded channel, large-eddy simulation with wall damping
        _case("channel_les_bf16_1024x256x256", nx=1024, ny=256, nz=256, storage="bf16", steps=20, flow="channel",
              bc="channel", force="uniform", tau=0.5107, cs=0.1, van_driest=True),
        # a lid-driven cavity: walls on every axis, one of them moving, a size that no tile divides
        _case("cavity_f32_130x111x90", nx=130, ny=111, nz=90, storage="f32", steps=50, flow="rest", bc="cavity",
              tau=0.53),
        # a ragged periodic box, FP16 storage, factorized attractor, a uniform force
        _case("factorized_f16_150x97x75", nx=150, ny=97, nz=75, storage="f16", steps=50, force="uniform", tau=0.52,
              attractor="factorized"),
        # the reference precision, for a run that others are checked against
        _case("forced_f64_128", nx=128, ny=128, nz=128, storage="f64", steps=5, force="uniform", tau=0.6),
        # the gradient of a loss on the final velocity with respect to the force field
        _case("optimise_f32_128", job="optimise", nx=128, ny=128, nz=128, storage="f32", steps=40, segment=20, force="field",
              tau=0.6, omega_bulk=0.0),
        # turbulence as forcing: the eddy stress of the resolved field enters as a force each step
        _case("filtered_f32_256", job="filtered", nx=256, ny=256, nz=256, storage="f32", steps=10, tau=0.50382, cs=0.1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, lo, hi):
    """A grid extent: spread over its logarithm, half of them the multiples of 16 or 32 that users like."""
    n = _log_int(rng, lo, hi)
    step = 32 if n >= 64 else 16
    return max(step, n // step * step) if rng.random() < 0.5 else n


def _steps(rng, cells, most=100):
    """A number of steps for which a pass stays below a hundred milliseconds or so."""
    return max(4, min(most, int(4e8 / cells), _log_int(rng, 4, most)))


def draw(rng):
    kind = rng.choice(["2d", "3d", "3d", "3d", "3d", "channel", "filtered", "optimise"])
    if kind == "2d":
        nx, ny = _size(rng, 16, 2500), _size(rng, 16, 1500)
        bc = rng.choice(["periodic", "channel", "couette"])
        return _case(lattice="D2Q9", nx=nx, ny=ny, nz=1, storage=rng.choice(["f64", "f32", "f32", "bf16", "f16"]),
                     steps=_steps(rng, nx * ny, 300), flow="rest" if bc == "channel" else "vortices", bc=bc,
                     force="uniform" if bc == "channel" else rng.choice(["none", "uniform"]),
                     tau=round(rng.uniform(0.52, 1.0), 4), omega_bulk=rng.choice([0.0, 1.0]))
    if kind == "filtered":
        nx, ny, nz = (_size(rng, 24, 256) for _ in range(3))
        return _case(job="filtered", nx=nx, ny=ny, nz=nz, storage=rng.choice(["f32", "f32", "bf16", "f16"]),
                     steps=min(10, _steps(rng, nx * ny * nz)), tau=round(rng.uniform(0.503, 0.55), 4), cs=0.1,
                     force=rng.choice(["none", "uniform"]))
    if kind == "optimise":
        storage = rng.choice(["f32", "f32", "f32", "f64"])
        nx, ny, nz = (_size(rng, 16, 64 if storage == "f64" else 128) for _ in range(3))
        return _case(job="optimise", nx=nx, ny=ny, nz=nz, storage=storage,
                     steps=rng.choice([10, 20, 30]), segment=rng.choice([5, 10, 20]), force="field",
                     bc=rng.choice(["periodic", "periodic", "cavity"]), tau=round(rng.uniform(0.55, 0.9), 4),
                     omega_bulk=rng.choice([0.0, 1.0]))
    if kind == "channel":
        nx, ny, nz = _size(rng, 32, 1024), _size(rng, 24, 256), _size(rng, 24, 256)
        storage = rng.choice(["f32", "bf16", "bf16", "f16"])
        return _case(nx=nx, ny=ny, nz=nz, storage=storage, steps=_steps(rng, nx * ny * nz, 20), flow="channel", bc="channel",
                     force="uniform", tau=round(rng.uniform(0.505, 0.53), 4), cs=0.1, van_driest=rng.random() < 0.7)
    storage = rng.choice(["f32", "f32", "bf16", "bf16", "f16", "f64"])
    nx, ny, nz = (_size(rng, 16, 128 if storage == "f64" else 320) for _ in range(3))
    bc = rng.choice(["periodic", "periodic", "periodic", "channel", "cavity"])
    steps = _steps(rng, nx * ny * nz * (10 if storage == "f64" else 1), 100 if storage in ("f32", "f64") else 20)
    les = rng.random() < 0.3
    general = rng.random() < 0.2
    return _case(nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, bc=bc,
                 flow="rest" if bc == "cavity" else "channel" if bc == "channel" else "vortices",
                 force="none" if bc == "cavity" else rng.choice(["none", "uniform", "field"]),
                 tau=round(rng.uniform(0.505, 0.7), 4), omega_3=1.3 if general else 1.0, omega_4=0.9 if general else 1.0,
                 cs=0.1 if les else 0.0, attractor=rng.choice(["maxwell"] * 4 + ["factorized"]),
                 reduced=rng.random() < 0.15)


# ---- inputs ------------------------------------------------------------------------------------
class _Fields:
    """Density, velocity and force of a case, made from the seed alone (FP64, on the GPU)."""

    def __init__(self, case, seed):
        self.rng = np.random.default_rng(seed)
        self.dev = torch.device(DEVICE)
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        self.shape = (nz, ny, nx)
        flat = case["lattice"] == "D2Q9"
        self.rho = torch.ones(self.shape, dtype=torch.float64, device=self.dev)
        self.u = torch.zeros((3,) + self.shape, dtype=torch.float64, device=self.dev)
        self.rho += 1e-3 * self._wave(0, 1, flat)
        if case["flow"] == "vortices":
            self._solenoidal(self.u, 0.04, flat)
        elif case["flow"] == "channel":
            eta = (torch.arange(ny, device=self.dev, dtype=torch.float64) + 0.5) / ny
            shape = (6.0 * eta * (1.0 - eta)).reshape(1, ny, 1)
            self.u[0] = 0.05 * shape
            g = torch.Generator(device=self.dev).manual_seed(int(seed) + 1)
            for d in range(3):
                self.u[d] += 0.003 * shape * torch.randn(self.shape, generator=g, device=self.dev)
        if flat:
            self.u[2] = 0.0
        # the force: none, a constant along x, or a solenoidal field
        self.uniform = (float(self.rng.uniform(0.5, 1.5) * 1e-5), 0.0, 0.0) if case["force"] == "uniform" else (0.0, 0.0, 0.0)
        self.field = None
        if case["force"] == "field":
            self.field = torch.zeros((3,) + self.shape, dtype=torch.float64, device=self.dev)
            self._solenoidal(self.field, 1e-5, flat)
        # wall velocities [axis][side][component] and the kinds of the boundaries
        self.wall = np.zeros((3, 2, 3))
        self.kinds = ["periodic"] * 3
        if case["bc"] in ("channel", "couette"):
            self.kinds[1] = "bounceback"
        if case["bc"] == "couette":
            self.wall[1, 1, 0] = self.rng.uniform(0.02, 0.05)
        if case["bc"] == "cavity":
            self.kinds = ["bounceback"] * 3
            self.wall[1, 1, 0] = self.rng.uniform(0.02, 0.05)

    def _wave(self, a, b, flat):
        """sin along one axis (0 = x) times cos along another, with random phases and wave numbers 1 or 2"""
        out = torch.ones((1, 1, 1), dtype=torch.float64, device=self.dev)
        for axis, shift in ((a, 0.0), (b, math.pi / 2)):
            n = self.shape[2 - axis]
            k = 2 * math.pi * int(self.rng.integers(1, 3))
            phase = shift + self.rng.uniform(0.0, 2 * math.pi)
            view = [1, 1, 1]
            view[2 - axis] = n
            line = torch.sin(k / n * torch.arange(n, dtype=torch.float64, device=self.dev) + phase)
            if not (flat and axis == 2):
                out = out * line.reshape(view)
        return out

    def _solenoidal(self, out, amplitude, flat):
        """Component d depends on the other two coordinates only, so that the divergence is zero."""
        for d in range(2 if flat else 3):
            out[d] += amplitude * self.rng.uniform(0.7, 1.3) * self._wave((d + 1) % (2 if flat else 3), (d + 2) % 3, flat)


def _solver(case, f):
    return cmlbm.Solver(lattice=case["lattice"], nx=case["nx"], ny=case["ny"], nz=case["nz"], storage=case["storage"],
                     bc=tuple(f.kinds), wall_velocity=f.wall, tau=case["tau"], omega_bulk=case["omega_bulk"],
                     omega_3=case["omega_3"], omega_4=case["omega_4"],
                     smagorinsky_cs=case["cs"] if case["job"] == "run" else 0.0,
                     van_driest=(26.0, 0.28) if case["van_driest"] else None, attractor=case["attractor"],
                     reduced_compressibility=case["reduced"])


def prepare(case, seed):
    f = _Fields(case, seed)
    s = _solver(case, f)
    if case["job"] == "optimise":
        s.init(f.rho, f.u)
        return {"case": case, "solver": s, "s0": s.get_state(), "force": f.field.float().requires_grad_(True),
                "target": 0.9 * f.u}
    s.set_force(f.uniform, f.field)
    return {"case": case, "solver": s, "rho": f.rho, "u": f.u, "uniform": f.uniform, "out": s.new_state()}


# ---- one pass ----------------------------------------------------------------------------------
def run(state):
    case, s = state["case"], state["solver"]
    if case["job"] == "optimise":
        force = state["force"]
        force.grad = None
        u = rollout.velocity_after(s, force.double(), state["s0"], case["steps"], case["segment"])
        loss = ((u - state["target"]) ** 2).sum(0).mean()
        loss.backward()
        return {"u": u.detach().float() if case["storage"] == "f32" else u.detach(), "gradient": force.grad}
    if case["job"] == "filtered":
        s.set_force(state["uniform"])       # the last run's turbulence force goes
        s.init(state["rho"], state["u"])
        s.step_filtered(case["steps"], case["cs"])
    else:
        s.init(state["rho"], state["u"])
        s.step(case["steps"])
    return s.get_state(out=state["out"])


# ---- bytes and operations ----------------------------------------------------------------------
def work(case):
    """Per step: every population read and written once, the force field read once; around the steps
    the initial fields read once and the final state written once. A filtered step also needs the
    velocity field of the whole neighbourhood before any cell can be updated: the populations once
    more, and rho and u written and read. An optimisation iteration: a forward step and an adjoint
    step (the state, the adjoint in and out, the force, the gradient sum in and out) for each step;
    the recomputation between the checkpoints is the caller's choice of segment."""
    q, flops = (9, 160) if case["lattice"] == "D2Q9" else (27, 600)
    e = BYTES[case["storage"]]
    r = 8 if case["storage"] == "f64" else 4
    n, steps = case["nx"] * case["ny"] * case["nz"], case["steps"]
    step = 2 * q * e + (3 * r if case["force"] == "field" else 0)
    if case["force"] != "none":
        flops += flops // 4
    if case["job"] == "optimise":
        adjoint = 3 * q * e + 3 * r + 6 * r
        return {"bytes": float(n * steps * (step + adjoint) + n * 24 * 3), "flops": float(n * steps * (flops + 2 * flops + flops))}
    if case["job"] == "filtered":
        step += q * e + 2 * 4 * r
        flops += 120
    return {"bytes": float(n * (steps * step + 32 + q * e)), "flops": float(n * steps * flops)}


# ---- the same in 64 bits, in plain torch -------------------------------------------------------
class _Exact:
    """The step on populations f[ez + 1, ey + 1, ex + 1, z, y, x] (D2Q9: one ez, one z)."""

    def __init__(self, case, f):
        self.c, self.f, self.flat = case, f, case["lattice"] == "D2Q9"
        self.ez = [0] if self.flat else [-1, 0, 1]
        self.dims = 2 if self.flat else 3

    def weight(self, e):
        w = 1.0
        for v in e[: self.dims]:
            w *= 2 / 3 if v == 0 else 1 / 6
        return w

    @staticmethod
    def _lines(m, dim):
        return m.select(dim, 0), m.select(dim, 1), m.select(dim, 2)

    def to_central(self, m, u):
        """Populations -> central moments, exponents [c, b, a] in the places of [ez, ey, ex]."""
        for axis in range(self.dims):
            v = u[axis]
            lo, mid, hi = self._lines(m, 2 - axis)
            m0, s1, s2 = lo + mid + hi, hi - lo, hi + lo
            m = torch.stack((m0, s1 - v * m0, s2 - 2 * v * s1 + v * v * m0), 2 - axis)
        return m

    def from_central(self, m, u):
        for axis in range(self.dims):
            v = u[axis]
            m0, m1, m2 = self._lines(m, 2 - axis)
            r1, r2 = m1 + v * m0, m2 + 2 * v * m1 + v * v * m0
            m = torch.stack(((r2 - r1) / 2, m0 - r2, (r2 + r1) / 2), 2 - axis)
        return m

    def exponents(self):
        return [(a, b, c) for c in (range(1) if self.flat else range(3)) for b in range(3) for a in range(3)]

    def hydro(self, g, F):
        """rho and u = (sum f e + F / 2) / rho (rho0 = 1 in the place of rho with reduced compressibility)."""
        rho = g.sum((0, 1, 2))
        j = [(g[:, :, 2] - g[:, :, 0]).sum((0, 1)), (g[:, 2] - g[:, 0]).sum((0, 1)),
             torch.zeros_like(rho) if self.flat else (g[2] - g[0]).sum((0, 1))]
        den = 1.0 if self.c["reduced"] else rho
        return rho, [(j[d] + 0.5 * F[d]) / den if d < self.dims else j[d] for d in range(3)]

    def collide(self, g, F, y0=0):
        c = self.c
        rho, u = self.hydro(g, F)
        m = self.to_central(g, u)
        K = {(a, b, d): m[d, b, a] for (a, b, d) in self.exponents()}
        kap, post = dict(K), {}
        unit = [(1, 0, 0), (0, 1, 0), (0, 0, 1)][: self.dims]
        post[(0, 0, 0)] = K[(0, 0, 0)]
        for d, e in enumerate(unit):
            post[e] = K[e] + F[d]
        # second order
        diag = [tuple(2 * v for v in e) for e in unit]
        off = [e for e in K if sum(e) == 2 and e not in diag]
        P = {e: K[e] - rho / 3 for e in diag}
        omega = 1.0 / c["tau"]
        if c["cs"] > 0 and c["job"] == "run":
            cs = c["cs"]
            if c["van_driest"]:
                y = torch.arange(c["ny"], dtype=torch.float64, device=g.device)
                wall = torch.minimum(y + 0.5, c["ny"] - 0.5 - y)
                cs = (cs * (1.0 - torch.exp(-wall * 0.28 / 26.0))).reshape(1, -1, 1)
            norm = torch.sqrt(sum(P[e] ** 2 for e in diag) + 2.0 * sum(K[e] ** 2 for e in off))
            omega = 2.0 / (c["tau"] + torch.sqrt(c["tau"] ** 2 + 18.0 * math.sqrt(2.0) * cs * cs * norm / rho))
        bulk = c["omega_bulk"] if c["omega_bulk"] > 0 else omega
        trace = sum(P[e] for e in diag)
        for e in diag:
            post[e] = rho / 3 + (1.0 - omega) * P[e] + (omega - bulk) * trace / self.dims
        for e in off:
            post[e] = (1.0 - omega) * K[e]
        # higher orders: source by the recursion, attractor, relaxation
        for e in sorted((e for e in K if sum(e) >= 3), key=sum):
            sigma = 0.0
            for d in range(self.dims):
                if e[d] > 0:
                    below = tuple(v - (k == d) for k, v in enumerate(e))
                    sigma = sigma + e[d] * F[d] / rho * kap[below]
            kap[e] = K[e] + 0.5 * sigma
            ones, twos = [d for d in range(3) if e[d] == 1], [d for d in range(3) if e[d] == 2]
            attract = rho / 3.0 ** len(twos) if not ones else 0.0
            if c["attractor"] == "factorized":
                if not ones:
                    attract = 1.0
                    for d in twos:
                        attract = attract * post[diag[d]]
                    attract = attract / rho ** (len(twos) - 1)
                elif len(ones) == 2 and len(twos) == 1:
                    attract = post[diag[twos[0]]] * post[tuple(1 if d in ones else 0 for d in range(3))] / rho
            w = c["omega_3"] if sum(e) == 3 else c["omega_4"]
            post[e] = (1.0 - w) * K[e] + w * attract + (1.0 - 0.5 * w) * sigma
        rows = [torch.stack([torch.stack([post[(a, b, d)] for a in range(3)]) for b in range(3)])
                for d in (range(1) if self.flat else range(3))]
        return self.from_central(torch.stack(rows), u)

    def initial(self, rho, u, F):
        """fbar = f^M - S / 2: the Maxwellian's central moments less half the source's"""
        c = self.c
        rows = []
        for d in (range(1) if self.flat else range(3)):
            for b in range(3):
                for a in range(3):
                    e = (a, b, d)
                    ones, scale = [k for k in range(3) if e[k] == 1], 3.0 ** -sum(v == 2 for v in e)
                    rows.append(rho * scale if not ones else -0.5 * F[ones[0]] * scale + 0.0 * rho if len(ones) == 1
                                else torch.zeros_like(rho))
        m = torch.stack(rows).reshape(len(self.ez), 3, 3, *rho.shape)
        v = [u[d] / rho if c["reduced"] else u[d] for d in range(3)]
        return self.from_central(m, v)

    def pull(self, f, z0, z1):
        """The populations that arrive in the planes z0 .. z1 - 1."""
        nz, ny, nx = self.f.shape
        planes = torch.arange(z0, z1, device=f.device)
        out = []
        for c in range(len(self.ez)):
            for b in range(3):
                for a in range(3):
                    e = (a - 1, b - 1, self.ez[c])
                    g = f[c, b, a].index_select(0, (planes - e[2]) % nz)
                    g = torch.roll(g, (e[1], e[0]), (1, 2))
                    count, eu = 0, 0.0
                    for axis, place in enumerate((torch.arange(nx, device=f.device).reshape(1, 1, -1),
                                                  torch.arange(ny, device=f.device).reshape(1, -1, 1),
                                                  planes.reshape(-1, 1, 1))):
                        if self.f.kinds[axis] == "bounceback" and e[axis] != 0:
                            side = 0 if e[axis] > 0 else 1
                            hit = place == (0 if side == 0 else (nx, ny, nz)[axis] - 1)
                            count = count + hit.double()
                            eu = eu + hit.double() * float(sum(e[k] * self.f.wall[axis, side, k] for k in range(3)))
                    if torch.is_tensor(count):
                        back = f[len(self.ez) - 1 - c, 2 - b, 2 - a][z0:z1] + 6.0 * self.weight(e) * eu / count.clamp(min=1.0)
                        g = torch.where(count > 0, back, g)
                    out.append(g)
        return torch.stack(out).reshape(len(self.ez), 3, 3, z1 - z0, ny, nx)

    def chunks(self):
        nz, ny, nx = self.f.shape
        k = max(1, int(2e6) // (ny * nx))
        return [(z, min(nz, z + k)) for z in range(0, nz, k)]

    def force(self, z0, z1, field):
        return [field[d][z0:z1] if field is not None else self.f.uniform[d] for d in range(3)]

    def eddy_force(self, rho, u):
        """rho d_j (2 nu_t S_ij), nu_t = C^2 |S|, central differences on the periodic box, plus the uniform force"""
        def diff(v, axis):
            return 0.5 * (torch.roll(v, -1, 2 - axis) - torch.roll(v, 1, 2 - axis)) if axis < self.dims else torch.zeros_like(v)

        S = [[0.5 * (diff(u[j], i) + diff(u[i], j)) for j in range(3)] for i in range(3)]
        size = torch.sqrt(2.0 * sum(S[i][j] ** 2 for i in range(3) for j in range(3)))
        k = 2.0 * self.c["cs"] ** 2 * size
        return [rho * sum(diff(k * S[i][j], j) for j in range(3)) + self.f.uniform[i] for i in range(3)]

    def states(self):
        """The populations after the case's steps."""
        field = self.f.field
        f, g = None, None
        filtered = self.c["job"] == "filtered"
        for t in range(self.c["steps"]):
            new = torch.empty((len(self.ez), 3, 3) + self.f.shape, dtype=torch.float64, device=self.f.dev)

            def arriving(z0, z1):
                if t > 0:
                    return self.pull(f, z0, z1)
                part = self.force(z0, z1, field)
                return self.initial(self.f.rho[z0:z1], self.f.u[:, z0:z1], part)

            if filtered:
                rho, u = torch.empty_like(self.f.rho), torch.empty_like(self.f.u)
                for z0, z1 in self.chunks():
                    r, v = self.hydro(arriving(z0, z1), self.force(z0, z1, field))
                    rho[z0:z1] = r
                    for d in range(3):
                        u[d, z0:z1] = v[d]
                started, field = field, torch.stack(self.eddy_force(rho, u))
            for z0, z1 in self.chunks():
                if filtered and t == 0:
                    g = self.initial(self.f.rho[z0:z1], self.f.u[:, z0:z1], self.force(z0, z1, started))
                else:
                    g = arriving(z0, z1)
                new[:, :, :, z0:z1] = self.collide(g, self.force(z0, z1, field))
            f = new
        return f

    def stored(self, f):
        """d = f / w - 1 in the order in which a state holds the directions"""
        if self.flat:
            order = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
            return torch.stack([f[0, ey + 1, ex + 1] / self.weight((ex, ey, 0)) - 1.0 for ex, ey in order])
        for c in range(3):
            for b in range(3):
                for a in range(3):
                    f[c, b, a] = f[c, b, a] / self.weight((a - 1, b - 1, c - 1)) - 1.0
        return f.reshape((27,) + self.f.shape)


def exact(case, seed):
    n = case["nx"] * case["ny"] * case["nz"]
    if n * case["steps"] > EXACT_CELL_STEPS:
        return None
    f = _Fields(case, seed)
    sim = _Exact(case, f)
    if case["job"] != "optimise":
        with torch.no_grad():
            return sim.stored(sim.states())
    nz = f.shape[0]
    force = f.field.float().requires_grad_(True)
    F = force.double()
    zero = [0.0, 0.0, 0.0]
    with torch.no_grad():
        g = sim.initial(f.rho, f.u, zero)
    for t in range(case["steps"]):
        def step(g, F):
            return sim.pull(sim.collide(g, F), 0, nz)
        g = checkpoint(step, g, F, use_reentrant=False)
    _, u = sim.hydro(g, F)
    u = torch.stack(u)
    loss = ((u - 0.9 * f.u) ** 2).sum(0).mean()
    loss.backward()
    return {"u": u.detach(), "gradient": force.grad.double()}
