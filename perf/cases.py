"""The measured cases: what a user's program asks of the framework, through
its public entry points (Simulation and Batch of the Python binding).

Three kinds of pass:
  "job"    a whole design-sweep job, as the job server runs it: a simulation
           made from the bunch's host arrays, its steps, its results copied
           out, the simulation closed;
  "run"    the next stretch of a run whose simulation is kept: some steps,
           then the outputs a program saves;
  "batch"  the next stretch of several simulations stepped together, then
           every member's outputs.

The workloads are the package's own (inputs.WORKLOADS) or generic FEL cases
of the same recipe: a lab beam of gamma and K boosted to the rest frame, 50
steps per rest-frame undulator period, c dt = 0.95 dz, dx = dy = 3 dz, a
transverse Gaussian bunch (sigma nx dx / 12, cut at 3 sigma) over the central
half of the grid, the undulator entrance one period ahead of it.  The generic
bunches are dilute, so that a run keeps its shape through however many
stretches it is stepped.
"""
import math

import numpy as np
import torch

from paper_1612_03310_gb300 import inputs, mithra

PRECISION = {"p64": mithra.P64, "p32": mithra.P32, "p32_u64": mithra.P32_U64, "p32_c": mithra.P32_C}

C = 299792458.0
QE = 1.602176634e-19
ME = 9.1093837015e-31
EPS0 = 8.8541878128e-12
MU0 = 1.0 / (EPS0 * C * C)


def _case(name, kind, nx, ny, nz, particles, prec, steps, **more):
    case = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, particles=particles, prec=prec, steps=steps,
                workload="", boundary=1, n_sub=1, undulator="static", seed_wave="", spectrum=0,
                power=False, copy_particles=True, fields="Ex,rho", members=1, uneven=False)
    case.update(more)
    return case


def listed():
    return [
        # the smallest calls: one small design job (the package's c1), where launches and latency
        # count, in the fast form and in the plain FP64 form that serves as its reference
        _case("job_c1_p32", "job", 32, 32, 64, 4096, "p32", 200, workload="c1", fields="Ex,By,phi,rho"),
        _case("job_c1_p64", "job", 32, 32, 64, 4096, "p64", 200, workload="c1", fields="Ex,By,phi,rho"),
        # an ordinary sweep point
        _case("run_sweep_p32", "run", 64, 64, 256, 262144, "p32", 200, fields="Ex,By,phi,rho"),
        # odd sizes, second-order boundary, sub-cycled particles, compensated potentials
        _case("run_ragged_p32c", "run", 101, 75, 413, 600011, "p32_c", 100, boundary=2, n_sub=2),
        # the plain FP64 form at an ordinary size
        _case("run_p64", "run", 96, 80, 384, 400000, "p64", 20),
        # the package's paper-sized run (c2) in its headline form, recording power, and in FP32
        _case("run_c2_p32u64", "run", 128, 128, 1024, 2097152, "p32_u64", 200, workload="c2", power=True,
              fields="Ex"),
        _case("run_c2_p32", "run", 128, 128, 1024, 2097152, "p32", 200, workload="c2", copy_particles=False),
        # the largest: the precision study's grid (c3)
        _case("run_c3_p32u64", "run", 256, 256, 2048, 16777216, "p32_u64", 60, workload="c3", power=True,
              copy_particles=False, fields="Ex"),
        # a seeded run without particles: the wave injected and its spectrum taken
        _case("run_seeded_p32", "run", 128, 128, 768, 0, "p32", 100, seed_wave="gaussian-beam", spectrum=16,
              power=True, copy_particles=False, fields="Ax"),
        # few particles in a large grid and a laser as the undulator (inverse Compton scattering)
        _case("run_optical_p32u64", "run", 192, 192, 768, 2800, "p32_u64", 100, undulator="optical"),
        # design sweeps stepped together: many small members, and uneven ones (the package's c4 sizes)
        _case("batch_small_p32", "batch", 32, 32, 128, 2000, "p32", 100, members=64, fields="Ex"),
        _case("batch_uneven_p32u64", "batch", 128, 128, 512, 256 * 128 * 128, "p32_u64", 40, members=8,
              uneven=True, fields="Ex", copy_particles=False),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["job", "run", "run", "run", "batch"])
    prec = rng.choice(["p32", "p32_u64", "p32_u64", "p32_c", "p64"])
    top = 48 if kind == "batch" else 160
    nx = log_int(32, top)
    ny = nx if rng.random() < 0.5 else log_int(32, top)
    nz = log_int(64, 256 if kind == "batch" else 1200)
    members = log_int(4, 64) if kind == "batch" else 1
    per_column = math.exp(rng.uniform(math.log(2.0), math.log(256.0)))
    particles = int(min(4.0e6 / members, per_column * nx * ny)) if kind == "batch" or rng.random() < 0.9 else 0
    undulator = rng.choice(["static", "static", "static", "optical"])
    n_sub = rng.choice([1, 1, 1, 2, 3])
    # work of a step in cell updates; a pass of some 2e9 of them (FP64: a tenth)
    work = members * (nx * ny * nz + 4.0 * n_sub * particles) + 2.0e5
    steps = int(max(8, min(200, (2.0e8 if prec == "p64" else 2.0e9) / work)))
    seeded = kind != "batch" and (not particles or rng.random() < 0.2)
    return _case("", kind, nx, ny, nz, particles, prec, steps, boundary=rng.choice([1, 1, 2]), n_sub=n_sub,
                 undulator=undulator, seed_wave=rng.choice(["plane-wave", "gaussian-beam"]) if seeded else "",
                 spectrum=rng.choice([0, 8]) if kind == "run" else 0, power=rng.random() < 0.5, members=members,
                 fields="Ex,rho" if particles else "Ax")


# --- inputs ------------------------------------------------------------------

def _shape(case, k):
    """Sizes of member k: all alike, or the package's c4 sizes in turn."""
    if not case["uneven"]:
        return case["nx"], case["ny"], case["nz"], case["particles"]
    nx = max(32, case["nx"] - 16 * (k % 6))
    per_column = case["particles"] / (case["nx"] * case["ny"]) * 0.5 ** (k % 3)
    return nx, nx, 4 * nx, int(per_column * nx * nx)


def _setup(case, seed, k=0):
    """Grid, undulator and bunch description of member k, host numbers only."""
    rng = np.random.Generator(np.random.PCG64([int(seed), k]))
    if case["workload"]:
        w = inputs.workload(case["workload"])
        grid = dict(w["grid"], boundary=case["boundary"])
        spec = dict(w["bunch_spec"])
        return grid, w["undulator"], dict(spec, q_macro=-spec["charge"] / spec["n"])
    nx, ny, nz, n = _shape(case, k)
    # one sweep point each: beam energy and undulator strength
    gamma, K, lam = float(rng.uniform(50.0, 150.0)), float(rng.uniform(0.7, 1.8)), 0.03
    f = mithra.boost_from_lab(gamma, lam, K, 50, 0.95, sigma_gamma_rel=1e-4)
    dz = f["dz"]
    dx = 3.0 * dz
    grid = inputs.centred_grid(dict(nx=nx, ny=ny, nz=nz, dx=dx, dy=dx, dz=dz, dt=f["dt"], n_sub=case["n_sub"],
                                    stencil=0, space_charge=1))
    grid["boundary"] = case["boundary"]
    z_lo, z_hi = 0.25 * nz * dz, 0.75 * nz * dz
    g0 = f["gamma0"]
    if case["undulator"] == "optical":
        lam_l = 2.0 * lam  # a laser of the wavelength that shakes the beam as the static undulator does
        a0 = 0.3 * K
        und = dict(type="optical", gamma0=g0, a0=a0, lambda_l=lam_l, polarization=(1.0, 0.0), direction=-1,
                   z0_lab=g0 * z_hi, offset=6.0 * lam_l, variance=3.0 * lam_l, cep=float(rng.uniform(0.0, 6.0)),
                   signal="flat-top")
        uz = 0.25 * a0 * a0 / math.sqrt(1.0 + 0.5 * a0 * a0)  # at rest, on average, once inside the wave
    else:
        und = dict(gamma0=g0, lambda_u=lam, K=K, z_ent_lab=g0 * z_hi + lam, length_lab=0.0, fringe=1)
        uz = f["uz_mean"]
    sigma = min(nx, ny) * dx / 12.0
    # the bunch's own field moves an electron by about two cells in 20000 steps
    t = 2.0e4 * f["dt"]
    charge = 4.0 * dx / (t * t) * 2.0 * math.pi * EPS0 * sigma * (z_hi - z_lo) * ME / QE
    spec = dict(n=n, charge=charge, sigma_r=sigma, trunc=3.0, z_lo=z_lo, z_hi=z_hi, uz_mean=uz,
                uz_sigma=f["uz_sigma"], ut_sigma=0.0, bf=1.0e-3, kb=f["k_b"], q_macro=-charge / max(n, 1))
    return grid, und, spec


def _bunch(spec, seed, k=0):
    """The bunch's arrays in 64 bits, drawn on the GPU: a transverse Gaussian cut at trunc sigma, uniform along z
    with the density modulation of the shot-noise recipe, Gaussian momenta."""
    n = int(spec["n"])
    g = torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + k)

    def uniform():
        return torch.rand(n, generator=g, device="cuda", dtype=torch.float64)

    def normal():
        return torch.randn(n, generator=g, device="cuda", dtype=torch.float64)

    cut = math.erf(spec["trunc"] / math.sqrt(2.0))

    def transverse():
        return spec["sigma_r"] * math.sqrt(2.0) * torch.erfinv(cut * (2.0 * uniform() - 1.0))

    x, y = transverse(), transverse()
    z = spec["z_lo"] + (spec["z_hi"] - spec["z_lo"]) * uniform()
    z = z - (2.0 * spec["bf"] / spec["kb"]) * torch.sin(spec["kb"] * z)
    u = [spec["ut_sigma"] * normal(), spec["ut_sigma"] * normal(), spec["uz_mean"] + spec["uz_sigma"] * normal()]
    return dict(x=x, y=y, z=z, ux=u[0], uy=u[1], uz=u[2])


def _host_bunch(spec, seed, k=0):
    if not spec["n"]:
        return None
    return dict({a: v.cpu().numpy() for a, v in _bunch(spec, seed, k).items()}, q_macro=spec["q_macro"])


def _seed_wave(case, grid, und, seed):
    """A seed that enters through the planes next to z_min, its wavelength 20 cells along z in the rest frame."""
    rng = np.random.Generator(np.random.PCG64([int(seed), 77]))
    g0 = und["gamma0"]
    b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
    lam = 20.0 * grid["dz"] / (g0 * (1.0 + b0))
    w = grid["nx"] * grid["dx"] / float(rng.uniform(5.0, 7.0))
    return dict(beam=case["seed_wave"], a0=1.0e-6, lambda_l=lam, polarization=(1.0, 0.3), direction=1, z0_lab=0.0,
                rayleigh_radius=(w, 1.2 * w), signal="gaussian", offset=30.0 * lam, variance=20.0 * lam,
                cep=float(rng.uniform(0.0, 6.0)))


def _power_plane(grid):
    return grid["nz"] - max(8, grid["nz"] // 16)


def _wavelengths(case, grid, und):
    g0 = und["gamma0"]
    b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
    return 20.0 * grid["dz"] / (g0 * (1.0 + b0)) * np.linspace(0.8, 1.25, case["spectrum"])


def _simulation(case, grid, und, bunch, seed):
    sim = mithra.Simulation(grid, und, bunch, precision=PRECISION[case["prec"]])
    if case["seed_wave"]:
        sim.set_seed(_seed_wave(case, grid, und, seed))
    if case["power"]:
        sim.set_power_sampling(_power_plane(grid), 5000)
    if case["spectrum"]:
        sim.set_spectrum(grid["nz"] // 3, _wavelengths(case, grid, und))
    return sim


def prepare(case, seed):
    members = []
    for k in range(case["members"]):
        grid, und, spec = _setup(case, seed, k)
        members.append((grid, und, _host_bunch(spec, seed, k)))
    state = dict(case=case, seed=seed)
    if case["kind"] == "job":  # the job's request: plain host data
        state["request"] = members[0]
        return state
    state["sims"] = [_simulation(case, g, u, b, seed) for g, u, b in members]
    if case["kind"] == "batch":
        state["batch"] = mithra.Batch()
        for sim in state["sims"]:
            state["batch"].add(sim)
    return state


# --- one pass ----------------------------------------------------------------

def _outputs(case, sim):
    out = {name: sim.copy_field(name) for name in case["fields"].split(",")}
    out["power"] = sim.read_power() if case["power"] else np.array(sim.radiated_power(_power_plane(sim.grid)))
    if case["spectrum"]:
        out["spectrum"] = sim.read_spectrum()[0]
    if case["copy_particles"] and sim.n_particles:
        p = sim.copy_particles()
        out.update({"particle_" + a: p[a] for a in ("x", "y", "z", "ux", "uy", "uz", "lost")})
    return out


def _joined(outs):
    """The members' outputs: each by itself, or (many members) end to end in one array for each name."""
    return outs if len(outs) <= 8 else {a: np.concatenate([np.ravel(o[a]) for o in outs]) for a in outs[0]}


def run(state):
    case = state["case"]
    if case["kind"] == "job":
        grid, und, bunch = state["request"]
        with _simulation(case, grid, und, bunch, state["seed"]) as sim:
            sim.step(case["steps"])
            return _outputs(case, sim)
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
        state["batch"].sync()
        return _joined([_outputs(case, sim) for sim in state["sims"]])
    sim = state["sims"][0]
    sim.step(case["steps"])
    return _outputs(case, sim)


# --- what a pass cannot do without ------------------------------------------

def work(case):
    """Per step and vertex: the newest level and the increment, four components each, read and written (the
    compensated forms' 16-bit rest too).  Per step and particle: cell, fractions and momenta, read and written.  Each
    output written once.  Operations: 17 a vertex and component, and about 500 a particle and sub-step."""
    real = 8 if case["prec"] == "p64" else 4
    mom = 8 if case["prec"] in ("p64", "p32_u64") else 4
    vertex = 4 * 4 * real + (16 if case["prec"] in ("p32_u64", "p32_c") else 0)
    particle = 2 * (4 + 3 * real + 3 * mom)
    total, flops = 0, 0
    for k in range(case["members"]):
        nx, ny, nz, n = _shape(case, k)
        cells = nx * ny * nz
        total += case["steps"] * (vertex * cells + particle * n)
        flops += case["steps"] * (4 * 17 * cells + 500 * n * case["n_sub"])
        total += 8 * cells * len(case["fields"].split(",")) + (52 * n if case["copy_particles"] else 0)
    return {"bytes": total, "flops": flops}


def tolerance(case):
    # Measured against exact() over the ranges of draw(): FP64 up to 2e-10 (E of a dilute bunch, a difference of
    # potentials); single FP32 levels and momenta up to 8e-5 after 200 steps (rho and J, through the particles); the
    # compensated levels up to 3e-5 (rho).  About four times that; "max" is the largest of a few million vertices.
    if case["prec"] == "p64":
        return {"rel": 1e-9, "max": 1e-6}
    return {"rel": 4e-4, "max": 0.05} if case["prec"] == "p32" else {"rel": 1e-4, "max": 0.01}


# --- the same in 64 bits, in plain torch ------------------------------------

def _signal(w, x, phase):
    """Signal "gaussian" or "flat-top" and its derivative at retarded time x with carrier phase offset `phase`."""
    w0 = 2.0 * math.pi * C / w["lambda_l"]
    tv = w["variance"] / C
    a = 2.0 * math.log(2.0) / (tv * tv)
    arg = w0 * x + w["cep"] + phase
    env, denv = torch.exp(-a * x * x), -2.0 * a * x * torch.exp(-a * x * x)
    if w["signal"] == "flat-top":
        env, denv = torch.where(x > 0, torch.ones_like(x), env), torch.where(x > 0, torch.zeros_like(x), denv)
    return env * torch.cos(arg), denv * torch.cos(arg) - w0 * env * torch.sin(arg)


class _Exact:
    """One simulation in 64 bits: potentials and increment as (4, nz, ny, nx) arrays."""

    def __init__(self, case, grid, und, spec, seed, k):
        self.case, self.g, self.u = case, grid, und
        self.dev = torch.device("cuda")
        nx, ny, nz = grid["nx"], grid["ny"], grid["nz"]
        self.n = nx * ny * nz
        z4 = lambda: torch.zeros((4, nz, ny, nx), dtype=torch.float64, device=self.dev)  # noqa: E731
        self.cur, self.D = z4(), z4()
        self.steps = 0
        cdt = C * grid["dt"]
        self.cdt = cdt
        self.r2 = [(cdt / grid[d]) ** 2 for d in ("dx", "dy", "dz")]
        qx, qy = grid["dz"] / grid["dx"], grid["dz"] / grid["dy"]
        self.A = 0.25 * (1.0 + 0.02 / (qx * qx + qy * qy))
        self._boundary()
        self.np = int(spec["n"])
        self.q = spec["q_macro"]
        self.src = torch.zeros((self.n, 4), dtype=torch.float64, device=self.dev)
        if self.np:
            b = _bunch(spec, seed, k)
            self.r = [b["x"], b["y"], b["z"]]
            self.uu = [b["ux"], b["uy"], b["uz"]]
            self.alive = self._valid(self.r)
            self._deposit(self.r, self.alive, [3], [self.q / (grid["dx"] * grid["dy"] * grid["dz"])])
        self.wave = _seed_wave(case, grid, und, seed) if case["seed_wave"] else None
        self.power = []
        if case["spectrum"]:
            b0 = math.sqrt(1.0 - 1.0 / und["gamma0"] ** 2)
            lam = torch.tensor(_wavelengths(case, grid, und), dtype=torch.float64, device=self.dev)
            self.omega = 2.0 * math.pi * C * (1.0 - b0) / lam
            self.acc = torch.zeros((case["spectrum"], 4, ny - 2, nx - 2), dtype=torch.complex128, device=self.dev)

    # potentials
    def _boundary(self):
        g = self.g
        nx, ny, nz = g["nx"], g["ny"], g["nz"]
        i = torch.arange(self.n, device=self.dev)
        ix, iy, iz = i % nx, (i // nx) % ny, i // (nx * ny)
        q = [ix.clamp(1, nx - 2), iy.clamp(1, ny - 2), iz.clamp(1, nz - 2)]
        off = [q[0] != ix, q[1] != iy, q[2] != iz]
        at = torch.nonzero(off[0] | off[1] | off[2]).squeeze(1)
        self.b = at
        self.bq = ((q[2] * ny + q[1]) * nx + q[0])[at]
        d2 = sum(o[at].double() * g[d] ** 2 for o, d in zip(off, ("dx", "dy", "dz")))
        d = torch.sqrt(d2)
        self.beta = (self.cdt - d) / (self.cdt + d)
        self.faces = []
        if g["boundary"] == 2:
            stride = [1, nx, nx * ny]
            one = off[0].int() + off[1].int() + off[2].int() == 1
            for a in range(3):
                sel = torch.nonzero((one & off[a])[at]).squeeze(1)
                d_a = g[("dx", "dy", "dz")[a]]
                terms = [(stride[t], self.r2[t] * d_a / (2.0 * (self.cdt + d_a))) for t in range(3) if t != a]
                self.faces.append((sel, terms))

    def _update(self):
        c, A = self.cur, self.A
        rx, ry, rz = self.r2
        mid = c[:, :, 1:-1, 1:-1]
        T = rx * (c[:, :, 1:-1, 2:] + c[:, :, 1:-1, :-2] - 2.0 * mid)
        T += ry * (c[:, :, 2:, 1:-1] + c[:, :, :-2, 1:-1] - 2.0 * mid)
        L = A * (T[:, 2:] + T[:, :-2])
        L += (1.0 - 2.0 * A) * T[:, 1:-1]
        L += rz * (mid[:, 2:] + mid[:, :-2] - 2.0 * mid[:, 1:-1])
        g = self.g
        s = self.src.view(g["nz"], g["ny"], g["nx"], 4)[1:-1, 1:-1, 1:-1]
        for m in range(3):
            L[m] += (self.cdt ** 2 * MU0) * s[..., m]
        L[3] += (self.cdt ** 2 / EPS0) * s[..., 3]
        Df, cf = self.D.view(4, -1), c.reshape(4, -1)
        old_b, old_q = Df[:, self.b], Df[:, self.bq]
        self.D[:, 1:-1, 1:-1, 1:-1] += L
        new_b = self.beta * (Df[:, self.bq] - old_b) + old_q
        for sel, terms in self.faces:
            b, q = self.b[sel], self.bq[sel]
            for o, w in terms:
                for v in (b, q):
                    new_b[:, sel] += w * (cf[:, v + o] + cf[:, v - o] - 2.0 * cf[:, v])
        Df[:, self.b] = new_b
        self.cur = c + self.D
        if self.wave:
            self._inject()

    def _inject(self):
        g, w = self.g, self.wave
        g0 = self.u["gamma0"]
        b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
        t = self.steps * g["dt"]
        x = g["x0"] + g["dx"] * torch.arange(g["nx"], device=self.dev, dtype=torch.float64)
        y = g["y0"] + g["dy"] * torch.arange(g["ny"], device=self.dev, dtype=torch.float64)
        p = np.array(w["polarization"]) / math.hypot(*w["polarization"])
        A0 = w["a0"] * ME * C / QE
        s = {}
        for k in (2, 3):
            zl = g0 * (g["z0"] + k * g["dz"] + b0 * C * t)
            tl = g0 * (t + b0 * (g["z0"] + k * g["dz"]) / C)
            tau = tl - (zl - w["z0_lab"]) / C - w["offset"] / C
            X, Y = x[None, :], y[:, None]
            if w["beam"] == "plane-wave":
                s[k] = _signal(w, torch.full((g["ny"], g["nx"]), tau, dtype=torch.float64, device=self.dev), 0.0)[0]
                continue
            zeta = zl - w["z0_lab"]
            amp, phase, expo, delay = 1.0, 0.0, 0.0, 0.0
            for a, wa in ((p[0] * X + p[1] * Y, w["rayleigh_radius"][0]), (p[0] * Y - p[1] * X, w["rayleigh_radius"][1])):
                zr = math.pi * wa * wa / w["lambda_l"]
                amp *= (zr * zr / (zeta * zeta + zr * zr)) ** 0.25
                phase += 0.5 * math.atan2(zeta, zr)
                expo = expo - a * a / (wa * wa * (1.0 + (zeta / zr) ** 2))
                delay = delay + a * a * zeta / (2.0 * C * (zeta * zeta + zr * zr))
            s[k] = amp * torch.exp(expo) * _signal(w, tau - delay, phase)[0]
        rx, ry, rz = self.r2
        for k, other, sign in ((2, 3, -1.0), (3, 2, 1.0)):
            f = s[other]
            m = f[1:-1, 1:-1]
            cpl = m * rz + self.A * (rx * (f[1:-1, 2:] + f[1:-1, :-2] - 2 * m) + ry * (f[2:, 1:-1] + f[:-2, 1:-1] - 2 * m))
            for a in range(2):
                self.D[a, k, 1:-1, 1:-1] += sign * A0 * p[a] * cpl
                self.cur[a, k, 1:-1, 1:-1] += sign * A0 * p[a] * cpl

    def _fields(self):
        """E and B at the half step, (n, 6) rows, zero on boundary vertices."""
        g = self.g
        out = torch.zeros((g["nz"], g["ny"], g["nx"], 6), dtype=torch.float64, device=self.dev)
        v = out[1:-1, 1:-1, 1:-1]
        i = slice(1, -1)
        lo, hi = slice(None, -2), slice(2, None)

        def diff(a, axis):
            at = [[i, i, i], [i, i, i]]
            at[0][2 - axis], at[1][2 - axis] = hi, lo
            return (a[tuple(at[0])] - a[tuple(at[1])]) / (2.0 * g[("dx", "dy", "dz")[axis]])

        mid = [self.cur[m] - 0.5 * self.D[m] for m in range(3)]
        phi = self.cur[3] - self.D[3]
        for a in range(3):
            v[..., a] = -self.D[a][i, i, i] / g["dt"] - diff(phi, a)
        v[..., 3] = diff(mid[2], 1) - diff(mid[1], 2)
        v[..., 4] = diff(mid[0], 2) - diff(mid[2], 0)
        v[..., 5] = diff(mid[1], 0) - diff(mid[0], 1)
        return out.view(-1, 6)

    # particles
    def _split(self, r):
        g = self.g
        cell, frac = [], []
        for a in range(3):
            s = (r[a] - g[("x0", "y0", "z0")[a]]) / g[("dx", "dy", "dz")[a]]
            f = torch.floor(s)
            cell.append(f.long())
            frac.append(s - f)
        return cell, frac

    def _valid(self, r):
        cell, _ = self._split(r)
        ok = torch.ones_like(cell[0], dtype=torch.bool)
        for c, n in zip(cell, (self.g["nx"], self.g["ny"], self.g["nz"])):
            ok &= (c >= 1) & (c <= n - 3)
        return ok

    def _corners(self, r):
        cell, f = self._split(r)
        nx, ny = self.g["nx"], self.g["ny"]
        base = (cell[2] * ny + cell[1]) * nx + cell[0]
        for k in range(2):
            for j in range(2):
                for i in range(2):
                    w = (f[0] if i else 1 - f[0]) * (f[1] if j else 1 - f[1]) * (f[2] if k else 1 - f[2])
                    yield base + (k * ny + j) * nx + i, w

    def _deposit(self, r, alive, comps, values):
        r = [torch.where(alive, a, torch.full_like(a, o + 2.5 * d)) for a, o, d in
             zip(r, (self.g["x0"], self.g["y0"], self.g["z0"]), (self.g["dx"], self.g["dy"], self.g["dz"]))]
        for at, w in self._corners(r):
            w = torch.where(alive, w, torch.zeros_like(w))
            for m, v in zip(comps, values):
                self.src.view(-1).index_add_(0, 4 * at + m, w * v)

    def _undulator(self, r, t):
        u, g0 = self.u, self.u["gamma0"]
        b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
        zl = g0 * (r[2] + b0 * C * t)
        zero = torch.zeros_like(zl)
        if u.get("type") == "optical":
            d = u["direction"]
            tau = g0 * (t + b0 * r[2] / C) - d * (zl - u["z0_lab"]) / C - u["offset"] / C
            ds = _signal(u, tau, 0.0)[1]
            A0 = u["a0"] * ME * C / QE
            px, py = u["polarization"]
            e, b = -g0 * (1.0 - d * b0) * A0 * ds, g0 * (d - b0) * A0 / C * ds
            return [px * e, py * e, zero], [py * b, -px * b, zero]
        ku = 2.0 * math.pi / u["lambda_u"]
        B0 = 2.0 * math.pi * ME * C * u["K"] / (QE * u["lambda_u"])
        zeta = zl - u["z_ent_lab"]
        a = ku * zeta
        inside_y, inside_z = torch.sin(a), torch.cos(a)
        before = zeta < 0
        L = u["length_lab"]
        after = zeta > L if L > 0 else torch.zeros_like(before)
        out = torch.where(after, ku * (zeta - L), a)
        e = torch.exp(-0.5 * out * out)
        by = B0 * torch.cosh(ku * r[1]) * torch.where(before | after, out * e, inside_y)
        bz = B0 * torch.sinh(ku * r[1]) * torch.where(before | after, e, inside_z)
        return [-g0 * b0 * C * by, zero, zero], [zero, g0 * by, bz]

    def _push(self, EB):
        g = self.g
        qm, dtb = -QE / ME, g["dt"] / g["n_sub"]
        h = qm * dtb / (2.0 * C)
        start = [a.clone() for a in self.r]
        r, u, alive = list(self.r), list(self.uu), self.alive
        for m in range(g["n_sub"]):
            safe = [torch.where(alive, a, torch.full_like(a, o + 2.5 * d)) for a, o, d in
                    zip(r, (g["x0"], g["y0"], g["z0"]), (g["dx"], g["dy"], g["dz"]))]
            F = torch.zeros((self.np, 6), dtype=torch.float64, device=self.dev)
            for at, w in self._corners(safe):
                F += w[:, None] * EB[at]
            Eu, Bu = self._undulator(safe, (self.steps + 0.5) * g["dt"] + m * dtb)
            E = [F[:, a] + Eu[a] for a in range(3)]
            B = [F[:, 3 + a] + Bu[a] for a in range(3)]
            t1 = [u[a] + h * E[a] for a in range(3)]
            al = qm * dtb / 2.0 / torch.sqrt(1.0 + t1[0] ** 2 + t1[1] ** 2 + t1[2] ** 2)
            cross = lambda p, q: [p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]]  # noqa: E731
            t = [al * b for b in B]
            c = cross(t1, t)
            t2 = [t1[a] + c[a] for a in range(3)]
            f = 2.0 / (1.0 + t[0] ** 2 + t[1] ** 2 + t[2] ** 2)
            c = cross(t2, [f * a for a in t])
            un = [t1[a] + c[a] + h * E[a] for a in range(3)]
            ig = 1.0 / torch.sqrt(1.0 + un[0] ** 2 + un[1] ** 2 + un[2] ** 2)
            rn = [r[a] + C * dtb * ig * un[a] for a in range(3)]
            u = [torch.where(alive, un[a], u[a]) for a in range(3)]
            r = [torch.where(alive, rn[a], r[a]) for a in range(3)]
            alive = alive & self._valid(r)
        V = g["dx"] * g["dy"] * g["dz"]
        self._deposit(r, alive, [3], [self.q / V])
        self._deposit([0.5 * (a + b) for a, b in zip(r, start)], alive, [0, 1, 2],
                      [self.q / V / g["dt"] * (a - b) for a, b in zip(r, start)])
        self.r, self.uu, self.alive = r, u, alive

    # diagnostics
    def _lab(self, EB, k):
        g, g0 = self.g, self.u["gamma0"]
        b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
        p = EB.view(g["nz"], g["ny"], g["nx"], 6)[k, 1:-1, 1:-1]
        Ex, Ey, Bx, By = p[..., 0], p[..., 1], p[..., 3], p[..., 4]
        return [g0 * (Ex + b0 * C * By), g0 * (Ey - b0 * C * Bx), g0 * (Bx - b0 / C * Ey), g0 * (By + b0 / C * Ex)]

    def _record(self, EB):
        g, g0 = self.g, self.u["gamma0"]
        b0 = math.sqrt(1.0 - 1.0 / (g0 * g0))
        t = (self.steps + 0.5) * g["dt"]
        k = _power_plane(g)
        e = self._lab(EB, k)
        z = g["z0"] + k * g["dz"]
        P = (e[0] * e[3] - e[1] * e[2]).sum() * (g["dx"] * g["dy"] / MU0)
        self.power.append((P, g0 * (t + b0 * z / C), g0 * (z + b0 * C * t)))
        if self.case["spectrum"]:
            k = g["nz"] // 3
            tl = g0 * (t + b0 * (g["z0"] + k * g["dz"]) / C)
            w = torch.exp(-1j * self.omega * tl) * (g0 * g["dt"])
            self.acc += w[:, None, None, None] * torch.stack(self._lab(EB, k))

    def run(self, steps):
        for s in range(steps):
            self._update()
            last = s + 1 == steps
            if self.np or last or self.case["power"] or self.case["spectrum"]:
                EB = self._fields()
                if last or self.case["power"] or self.case["spectrum"]:
                    self._record(EB)
            self.src.zero_()
            if self.np:
                self._push(EB)
            self.steps += 1
        self.EB = EB

    def outputs(self):
        case, g = self.case, self.g
        shape = (g["nz"], g["ny"], g["nx"])
        out = {}
        for name in case["fields"].split(","):
            if name in ("Ax", "Ay", "Az", "phi"):
                v = self.cur[("Ax", "Ay", "Az", "phi").index(name)]
            elif name in ("Jx", "Jy", "Jz", "rho"):
                v = self.src[:, ("Jx", "Jy", "Jz", "rho").index(name)].reshape(shape)
            else:
                v = self.EB[:, ("Ex", "Ey", "Ez", "Bx", "By", "Bz").index(name)].reshape(shape)
            out[name] = v.cpu().numpy()
        rec = np.array([[float(a) for a in row] for row in self.power])
        out["power"] = rec if case["power"] else rec[-1]
        if case["spectrum"]:
            a = self.acc
            s = (a[:, 0] * a[:, 3].conj() - a[:, 1] * a[:, 2].conj()).real.sum((1, 2))
            out["spectrum"] = (s * (g["dx"] * g["dy"] / (math.pi * MU0))).cpu().numpy()
        if case["copy_particles"] and self.np:
            for a, v in zip("xyz", self.r):
                out["particle_" + a] = torch.where(self.alive, v, torch.zeros_like(v)).cpu().numpy()
            for a, v in zip("xyz", self.uu):
                out["particle_u" + a] = v.cpu().numpy()
            out["particle_lost"] = (~self.alive).to(torch.int32).cpu().numpy()
        return out


def exact(case, seed):
    outs = []
    for k in range(case["members"]):
        grid, und, spec = _setup(case, seed, k)
        e = _Exact(case, grid, und, spec, seed, k)
        e.run(case["steps"])
        outs.append(e.outputs())
        del e
    return _joined(outs) if case["kind"] == "batch" else outs[0]
