"""What a user of this package has it do, as a set of timed cases.

A case is one pass through the public entry points (fs.FauxShock, fs.FsBatch,
window.FauxShockWindow): a few steps of a box and its fields read back, a
batched ensemble, a differentiable window with its gradient, the diagnostics
of one output time, or a checkpoint and restart. listed() holds the named
cases, draw() gives more of the same ranges, and exact() evaluates the same
inputs in 64 bits with plain torch operations (its own Philox draws, particle
step and field solver, below), for comparison.
"""
import math

import numpy as np
import torch

from paper_2507_14282_gb300 import fs
from paper_2507_14282_gb300.window import FauxShockWindow

DEVICE = "cuda:0"


# --------------------------------------------------------------------- cases
def _box(kind, dim, nx, ny, ppc, fp64, steps, **kw):
    """A box case: the physics the runs of this repository vary, as plain
    values. thermal_open: the paper's thermal plasma, which always leaves
    through the faux shock; otherwise it is returned with Eq. 1's probability.
    cr: the cosmic-ray source at the faux shock. c_light: relativistic ions."""
    c = dict(kind=kind, dim=dim, nx=nx, ny=ny, ppc=ppc, fp64=fp64, steps=steps, mach=20.0,
             theta=0.0, beta=1.0, dx=0.5, dt=0.0025, thermal_open=False, cr=False, p_iso=100.0,
             c_light=0.0, n_sub=2, periodic=False)
    unknown = set(kw) - set(c)
    assert not unknown, unknown
    c.update(kw)
    return c


def listed():
    cases = {
        # one short 1D run of the paper's kind (thermal plasma open, cosmic rays
        # from the faux shock): 16 K particles, all launch latency
        "box1d_fp64": _box("box", 1, 512, 1, 32, True, 20, mach=10.0, dt=0.005,
                           thermal_open=True, cr=True),
        # a long 1D precursor run in single precision, no power of two in its sizes
        "box1d_fp32": _box("box", 1, 8100, 1, 100, False, 10, mach=40.0, theta=20.0, dt=0.00125,
                           thermal_open=True, cr=True),
        # the 2D production-shaped box in double precision (the benchmark's)
        "box2d_fp64": _box("box", 2, 4096, 256, 16, True, 2),
        # the 2D precision form in single precision, 268 M particles (the benchmark's)
        "box2d_fp32": _box("box", 2, 8192, 512, 64, False, 2, mach=30.0, theta=30.0, dt=0.002),
        # a 2D box whose sides are no whole number of field tiles, with cosmic rays
        "box2d_fp32_ragged": _box("box", 2, 3000, 250, 20, False, 4, mach=30.0, theta=45.0,
                                  dt=0.002, thermal_open=True, cr=True),
        # relativistic ions in double precision, ragged sizes
        "box2d_fp64_rel": _box("box", 2, 1002, 150, 24, True, 4, theta=60.0, cr=True,
                               thermal_open=True, p_iso=1000.0, c_light=300.0),
        # 64 uneven 1D runs stepped together (a parameter study), fields read every 24 steps
        "ensemble_fp32": dict(kind="ensemble", runs=64, first=100, fp64=False, steps=24),
        # loss and gradient of a 200-step window, single precision
        "window_fp32": dict(kind="window", nx=2048, ppc=128, fp64=False, steps=200, ckpt=20,
                            modes=16),
        # the same in double precision on a smaller, odd-sized window
        "window_fp64": dict(kind="window", nx=777, ppc=50, fp64=True, steps=60, ckpt=15, modes=16),
        # what a run writes out at an output time: profiles, spectra, phase
        # space, energies (rows of a power of two)
        "analysis_fp64": _box("analysis", 2, 4096, 256, 16, True, 0, cr=True),
        # the same on a ragged single-precision box
        "analysis_fp32": _box("analysis", 2, 3000, 250, 20, False, 0, cr=True, theta=45.0,
                              mach=30.0),
        # a run saved to host arrays and restored into a new handle
        "checkpoint": _box("checkpoint", 2, 512, 96, 20, True, 2, cr=True, theta=30.0),
    }
    return [dict(c, name=name) for name, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _side(rng, lo, hi):
    """A side length with a small factor (boxes are cut into tiles), often odd."""
    f = rng.choice([2, 3, 4, 5, 6, 7, 8, 16])
    return f * max(2, round(_log_uniform(rng, lo, hi) / f))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "box", "ensemble", "window", "analysis", "checkpoint"])
    fp64 = rng.random() < 0.5
    if kind == "ensemble":
        return dict(kind=kind, runs=rng.randint(24, 64), first=rng.randint(100, 10000), fp64=fp64,
                    steps=4 if fp64 else rng.choice([8, 16, 24]))
    if kind == "window":
        return dict(kind=kind, nx=round(_log_uniform(rng, 64, 2048)), ppc=rng.randint(8, 128),
                    fp64=fp64, steps=rng.randint(20, 100), ckpt=rng.choice([7, 10, 20]),
                    modes=rng.randint(2, 16))
    mach = rng.uniform(10.0, 50.0)
    kw = dict(mach=mach, theta=rng.choice([0.0, rng.uniform(0.0, 60.0)]),
              beta=rng.choice([0.5, 1.0, 2.0]), dt=min(0.005, 0.05 / mach),
              cr=rng.random() < 0.5, thermal_open=rng.random() < 0.5)
    dim = 2 if kind != "box" else rng.choice([1, 2, 2])
    if dim == 1:
        nx, ny, ppc = _side(rng, 256, 16384), 1, round(_log_uniform(rng, 8, 256))
    else:
        cells = _log_uniform(rng, 4096, (1 << 20) if kind != "checkpoint" else (1 << 14))
        ny = _side(rng, 16, max(17, min(512, cells / 32)))
        nx, ppc = _side(rng, 32, 64), round(_log_uniform(rng, 8, 64))
        nx = max(32, min(8192, nx * round(cells / (nx * ny)) or nx))
    if nx * ny * ppc < 1 << 22:  # a small box's run is short: no pile-up at the wall
        kw["thermal_open"] = True
    if kind == "box":
        kw["n_sub"] = rng.choice([1, 2, 2, 2, 3])
        if rng.random() < 0.2:
            kw["c_light"] = 300.0
        if rng.random() < 0.2:
            kw.update(periodic=True, cr=False)
    steps = 0 if kind == "analysis" else rng.choice([2, 4]) if dim == 2 else 10
    return _box(kind, dim, nx, ny, ppc, fp64, steps, **kw)


# ----------------------------------------------------------- the package's run
def _params(c, seed):
    p = dict(dim=c["dim"], nx=c["nx"], ny=c["ny"], dx=c["dx"], dy=c["dx"], dt=c["dt"],
             precision=fs.FS_FP64 if c["fp64"] else fs.FS_FP32, mach_a=c["mach"],
             theta_bn_deg=c["theta"], beta_i=c["beta"], beta_e=c["beta"], ppc=c["ppc"],
             bc_x=fs.FS_BC_PERIODIC if c["periodic"] else fs.FS_BC_FAUXSHOCK,
             fs_mode_thermal=fs.FS_OPEN if c["thermal_open"] else fs.FS_SHOCK,
             cr_enable=int(c["cr"]), p_iso=c["p_iso"], c_light=c["c_light"], n_sub=c["n_sub"],
             seed=seed + 1)
    if c["kind"] == "analysis":
        p.update(hist_nx=256, hist_np=128, hist_pmin=-120.0, hist_pmax=120.0, spec_np=128,
                 spec_pmin=1.0, spec_pmax=1000.0)
    return p


def _ensemble_params(c, seed):
    """Uneven 1D runs as the batched-ensemble configuration draws them (Philox,
    key first + r), with the tile widths the autotuner picks for each ppc."""
    runs = []
    for r in range(c["runs"]):
        g = np.random.Generator(np.random.Philox(key=c["first"] + r))
        nx = int(round(float(np.exp(g.uniform(np.log(512.0), np.log(8192.0)))) / 32.0)) * 32
        ppc = int(g.choice([32, 64, 128, 256]))
        mach = float(g.uniform(5.0, 100.0))
        theta = float(g.uniform(0.0, 60.0))
        beta = float(g.choice([0.5, 1.0, 2.0]))
        runs.append(dict(dim=1, nx=nx, ny=1, dx=0.5, dy=0.5, dt=min(0.005, 0.1 * 0.5 / mach),
                         mach_a=mach, theta_bn_deg=theta, beta_i=beta, beta_e=beta, ppc=ppc,
                         seed=1000 * (seed + 1) + r, precision=int(not c["fp64"]),
                         capacity_factor=4.0,
                         tile_x={32: 16, 64: 16, 128: 8, 256: 4}[ppc], tile_y=1))
    return runs


FIELDS = ((fs.FS_B, "B"), (fs.FS_E, "E"), (fs.FS_N, "n"), (fs.FS_U, "u"))


def _buffers(sim):
    """Device tensors for the fields a program reads after its steps (FP64, as
    the interface delivers them)."""
    nn, out = (sim.ny, sim.nxn), {}
    for what, name in FIELDS:
        shape = {"B": (sim.ny, sim.nx, 3), "n": nn}.get(name, nn + (3,))
        out[name] = torch.empty(shape, dtype=torch.float64, device=DEVICE)
    return out


def _read(sim, out):
    for what, name in FIELDS:
        sim.grid_device(what, out[name])


def _own_type(values, fp64):
    """Results in the type the run computes in: a single-precision run's
    numbers are kept in 32 bits."""
    return values if fp64 else {k: v.float() if torch.is_tensor(v) else v.astype(np.float32)
                                for k, v in values.items()}


def _seeded_B(c, seed):
    """B0 plus 24 seeded transverse modes along x with a weak y dependence."""
    g = np.random.default_rng(seed)
    x = (np.arange(c["nx"]) + 0.5) / c["nx"]
    y = (np.arange(c["ny"]) + 0.5) / c["ny"]
    th = math.radians(c["theta"])
    B = np.empty((c["ny"], c["nx"], 3))
    B[...] = (math.cos(th), math.sin(th), 0.0)
    for _ in range(24):
        m, l = int(g.integers(1, max(2, c["nx"] // 8))), int(g.integers(0, 4))
        ph = 2 * np.pi * (m * x[None, :] + l * y[:, None] + g.uniform())
        a = g.uniform(0.005, 0.05)
        B[..., 1] += a * np.cos(ph)
        B[..., 2] += a * np.sin(ph)
    return B


def _seeded_cr(c, seed):
    """A population of cosmic rays streaming away from the wall (ids flagged)."""
    g = np.random.default_rng(seed + 7)
    n = c["nx"] * c["ny"] * c["ppc"] // 16
    p = c["p_iso"] * np.exp(g.normal(0.0, 0.3, n))
    mu, ph = g.uniform(-0.2, 1.0, n), g.uniform(0.0, 2 * np.pi, n)
    s = np.sqrt(1 - mu * mu)
    first = c["nx"] * c["ny"] * c["ppc"]
    return dict(ci=g.integers(0, c["nx"], n).astype(np.int32),
                cj=g.integers(0, c["ny"], n).astype(np.int32), fx=g.uniform(0, 1, n),
                fy=g.uniform(0, 1, n), vx=p * mu, vy=p * s * np.cos(ph), vz=p * s * np.sin(ph),
                ids=((first + np.arange(n)) | fs.ID_CR).astype(np.uint32))


def _window_inputs(c, seed):
    g = np.random.default_rng(seed)
    nx, ppc = c["nx"], c["ppc"]
    x = np.repeat(np.arange(nx), ppc) + g.uniform(0.0, 1.0, nx * ppc)
    v = g.normal(0.0, math.sqrt(0.5), (nx * ppc, 3))
    v[:, 0] -= 20.0
    amps = g.uniform(-0.01, 0.01, c["modes"])
    phases = g.uniform(0.0, 2 * np.pi, c["modes"])
    params = dict(nx=nx, ppc=ppc, dx=0.5, dt=0.0025, mach_a=20.0, theta_bn_deg=0.0, beta_i=1.0,
                  beta_e=1.0, seed=seed + 1, precision=int(not c["fp64"]), cr_enable=1,
                  p_iso=100.0, n_cr_ratio=0.01)
    return x, v, phases, np.concatenate([amps, [5.0, 5.0]]), params


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "ensemble":
        sims = [fs.FauxShock(device=DEVICE, **p) for p in _ensemble_params(c, seed)]
        return dict(case=c, sims=sims, batch=fs.FsBatch(sims), out=[_buffers(s) for s in sims])
    if kind == "window":
        x, v, phases, theta, params = _window_inputs(c, seed)
        win = FauxShockWindow(x, v, phases, steps=c["steps"], ckpt=c["ckpt"], device=DEVICE,
                              **params)
        return dict(case=c, win=win, theta=theta)
    params = _params(c, seed)
    sim = fs.FauxShock(device=DEVICE, **params)
    state = dict(case=c, sim=sim, params=params)
    if kind == "analysis":
        sim.load_fields(_seeded_B(c, seed))
        sim.inject(**_seeded_cr(c, seed))
    elif kind == "checkpoint":
        sim.step(c["steps"])
    else:
        state.update(out=_buffers(sim), left=_run_steps(c))
    return state


def _run_steps(c):
    """Steps of one whole run: 5 / Omega_ci in 1D (the 1000 steps of the 1D
    configuration), 1 / Omega_ci in 2D."""
    return round((5.0 if c["dim"] == 1 else 1.0) / c["dt"])


def run(state):
    c, kind = state["case"], state["case"]["kind"]
    if kind == "box":  # some steps, then the fields at the output time
        if state["left"] < c["steps"]:  # the run has reached its end: the next one starts
            state["sim"].close()
            state.update(sim=fs.FauxShock(device=DEVICE, **state["params"]), left=_run_steps(c))
        state["left"] -= c["steps"]
        state["sim"].step(c["steps"])
        _read(state["sim"], state["out"])
        return _own_type(state["out"], c["fp64"])
    if kind == "ensemble":
        state["batch"].step(c["steps"])
        for sim, out in zip(state["sims"], state["out"]):
            _read(sim, out)
        whole = {name: torch.cat([o[name].reshape(-1) for o in state["out"]])
                 for _, name in FIELDS}
        return _own_type(whole, c["fp64"])
    if kind == "window":
        loss, grad = state["win"].loss_and_grad(state["theta"])
        m = c["modes"]
        out = {"loss": np.array([loss]), "modes": grad[:m], "u_cr": grad[m:m + 1],
               "u2": grad[m + 1:]}
        return _own_type(out, c["fp64"])
    sim = state["sim"]
    if kind == "analysis":
        d = sim.diag()
        moments = {"n": sim.grid(fs.FS_PROFILE_N), "max_z": np.array([d["max_z"]])}
        return dict(_own_type(moments, c["fp64"]), db2=sim.grid(fs.FS_PROFILE_DB2),
                    B=sim.grid(fs.FS_PROFILE_B), spectrum=sim.grid(fs.FS_SPECTRUM_BPERP),
                    hist=sim.histogram(), hist_cr=sim.histogram(cr_only=True),
                    p_all=sim.spectrum_p(cr_only=False), p_cr=sim.spectrum_p(),
                    energy=np.array([d["kinetic"], d["magnetic"]]),
                    momentum=np.array([d["px"], d["py"], d["pz"]]),
                    particles=d["n_particles"])
    ck = sim.checkpoint()
    new = fs.FauxShock.restart(ck, device=DEVICE, **state["params"])
    out = {name: new.grid(what) for what, name in FIELDS}
    n = new.num_particles()
    new.close()
    return dict(_own_type(out, c["fp64"]), particles=n)


def work(case):
    c, kind = case, case["kind"]
    T = 8 if c["fp64"] else 4
    if kind == "window":
        # the forward and the reverse sweep each read and write the particles
        # once per step; the fields are small
        n = c["nx"] * c["ppc"] * c["steps"]
        return {"bytes": 2.0 * n * 2 * (4 * T + 4), "flops": 600.0 * n}
    if kind == "ensemble":
        boxes = [(1, p["nx"], 1, p["ppc"]) for p in _ensemble_params(c, 0)]
    else:
        boxes = [(c["dim"], c["nx"], c["ny"], c["ppc"])]
    b = f = 0.0
    for dim, nx, ny, ppc in boxes:
        n, cells = nx * ny * ppc, nx * ny
        state = 8 + (dim + 3) * T  # cell, offsets, velocity, id
        if kind == "analysis":  # every particle and the grid once
            b += 17 / 16 * n * state + 10 * cells * T
            f += 30.0 * n + 60.0 * cells
        elif kind == "checkpoint":  # out to the host, back, and in place
            b += n * (4 * state + 56)
            f += 60.0 * n
        else:
            b += c["steps"] * (2.0 * n * state + 23 * T * cells) + 10 * cells * (T + 8)
            f += c["steps"] * ((250.0 if dim == 2 else 160.0) * n + 900.0 * cells)
    return {"bytes": b, "flops": f}


# ------------------------------------------- the same inputs in 64 bits (torch)
M32 = 0xFFFFFFFF


def _philox(seed, pid, step, purpose):
    """Philox4x32-10 (Salmon et al., SC'11), counter (pid, step, purpose, 0)."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    c = [pid, torch.full_like(pid, step & M32), torch.full_like(pid, purpose),
         torch.zeros_like(pid)]
    for r in range(10):
        p0, p1 = c[0] * 0xD2511F53, c[2] * 0xCD9E8D57  # wraps mod 2^64: bits kept
        c = [((p1 >> 32) & M32) ^ c[1] ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c[3] ^ k1, p0 & M32]
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return [(x.double() + 0.5) * 2.0 ** -32 for x in c]


def _gauss(a, b):
    r = torch.sqrt(-2.0 * torch.log(a))
    return r * torch.cos(2 * math.pi * b), r * torch.sin(2 * math.pi * b)


class _Box64:
    """One box in double precision: the scheme with whole-array operations.
    A 1D box is the 2D scheme with one row and no y differences."""

    def __init__(self, p, u_cr=None, u2=None):
        d = fs.params_default(p.get("dim", 1))
        d.update(p)
        self.p = d
        self.nx, self.ny = d["nx"], d["ny"]
        self.per = d["bc_x"] == fs.FS_BC_PERIODIC
        self.nxn = self.nx + (0 if self.per else 1)
        self.dim2 = d["dim"] == 2
        self.c2 = 1.0 / d["c_light"] ** 2 if d["c_light"] > 0 else 0.0
        self.u2 = u2 if u2 is not None else d["mach_a"] / d["r_comp"]
        self.u_cr = u_cr if u_cr is not None else self.u2
        self.piso = d["p_iso"] / math.sqrt(1 + d["p_iso"] ** 2 * self.c2)
        self.w = (1.0 / d["ppc"], d["n_cr_ratio"] / d["ppc"])
        self.vth, self.te = math.sqrt(0.5 * d["beta_i"]), 0.5 * d["beta_e"]
        th = math.radians(d["theta_bn_deg"])
        self.B0 = (math.cos(th), math.sin(th), 0.0)
        self.acc, self.step_no, self.next_id = np.zeros(self.ny), 0, 0
        i, j = torch.arange(self.nxn, device=DEVICE), torch.arange(self.ny, device=DEVICE)
        if self.per:
            self.im, self.ip = (i - 1) % self.nx, i
            self.nl, self.nr = (i - 1) % self.nx, (i + 1) % self.nx
        else:
            self.im, self.ip = (i - 1).clamp(min=0), i.clamp(max=self.nx - 1)
            self.nl, self.nr = (i - 1).abs(), self.nx - (self.nx - (i + 1)).abs()
        self.jm, self.jp = (j - 1) % self.ny, (j + 1) % self.ny

    def store(self, x):
        """A value as the run holds it (single-precision runs round the state
        they start from)."""
        return x if self.p["precision"] == fs.FS_FP64 else x.float().double()

    # ---- fields
    def ohm(self, B, n, u):
        d = self.p
        a, b = B[:, self.jm], B  # rows below and above the node
        mm, pm, mp, pp = a[:, :, self.im], a[:, :, self.ip], b[:, :, self.im], b[:, :, self.ip]
        bb = 0.25 * (mm + pm + mp + pp)
        dx = (pp + pm - mp - mm) * (0.5 / d["dx"])
        dy = (pp + mp - pm - mm) * (0.5 / d["dy"]) if self.dim2 else torch.zeros_like(dx)
        curl = torch.stack([dy[2], -dx[2], dx[1] - dy[0]])
        j = torch.stack([curl[0] - d["j_cr_ext"], curl[1], curl[2]])
        gx = (n[:, self.nr] - n[:, self.nl]) * (0.5 / d["dx"])
        gy = (n[self.jp] - n[self.jm]) * (0.5 / d["dy"]) if self.dim2 else torch.zeros_like(gx)
        grad = torch.stack([gx, gy, torch.zeros_like(gx)])
        hall, motional = torch.linalg.cross(j, bb, dim=0), torch.linalg.cross(u, bb, dim=0)
        E = (hall - self.te * grad) / n - motional
        return E + d["eta"] * curl, bb

    def curl_e(self, E):
        d = self.p
        right = torch.roll(E, -1, 2)[:, :, :self.nx]  # (a box with walls has node nx)
        left = E[:, :, :self.nx]
        up_r, up_l = right[:, self.jp], left[:, self.jp]
        dx = (right + up_r - left - up_l) * (0.5 / d["dx"])
        dy = (up_l + up_r - left - right) * (0.5 / d["dy"]) if self.dim2 else torch.zeros_like(dx)
        return torch.stack([dy[2], -dx[2], dx[1] - dy[0]])

    def advance(self, B, n, u):
        h = self.p["dt"] / self.p["n_sub"]
        for _ in range(self.p["n_sub"]):
            k1 = -self.curl_e(self.ohm(B, n, u)[0])
            k2 = -self.curl_e(self.ohm(B + 0.5 * h * k1, n, u)[0])
            k3 = -self.curl_e(self.ohm(B + 0.5 * h * k2, n, u)[0])
            k4 = -self.curl_e(self.ohm(B + h * k3, n, u)[0])
            B = B + (h / 6.0) * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        return B

    # ---- particles: (i, j, fx, fy, v[N, 3], id); v holds u = gamma v with c
    def corners(self, i, j, fx, fy):
        i1, j1 = i + 1, (j + 1) % self.ny
        i1 = i1 % self.nx if self.per else i1
        gx, gy = 1.0 - fx, 1.0 - fy
        out = [(j * self.nxn + i, gx * gy), (j * self.nxn + i1, fx * gy)]
        if self.dim2:
            out += [(j1 * self.nxn + i, gx * fy), (j1 * self.nxn + i1, fx * fy)]
        return out

    def weight(self, pid):
        w = torch.tensor(self.w, dtype=torch.float64, device=DEVICE)
        return w[((pid & fs.ID_CR) != 0).long()]

    def inv_gamma(self, v):
        return 1.0 / torch.sqrt(1.0 + (v * v).sum(1) * self.c2) if self.c2 else None

    def moments(self, parts):
        nn = self.nxn * self.ny
        total = torch.zeros(nn, 4, dtype=torch.float64, device=DEVICE)
        for s in range(0, len(parts[0]), 1 << 24):
            i, j, fx, fy, v, pid = (x[s:s + (1 << 24)] for x in parts)
            w = self.weight(pid)
            ig = self.inv_gamma(v)
            q = torch.cat([torch.ones_like(v[:, :1]), v if ig is None else v * ig[:, None]], 1)
            for node, cw in self.corners(i, j, fx, fy):
                total = total.index_add(0, node, (w * cw)[:, None] * q)
        total = total.reshape(self.ny, self.nxn, 4)
        if not self.per:
            wall = torch.ones(self.nxn, dtype=torch.float64, device=DEVICE)
            wall[0] = wall[-1] = 2.0
            total = total * wall[None, :, None]
        n = total[..., 0].clamp(min=self.p["n_floor"])
        return n, (total[..., 1:] / n[..., None]).permute(2, 0, 1)

    def push(self, parts, F):
        i, j, fx, fy, v, pid = parts
        d = self.p
        eb = sum(cw[:, None] * F[node] for node, cw in self.corners(i, j, fx, fy))
        half = 0.5 * d["dt"] * eb[:, :3]
        v = v + half
        ig = self.inv_gamma(v)
        t = 0.5 * d["dt"] * eb[:, 3:] * (1.0 if ig is None else ig[:, None])
        s = 2.0 * t / (1.0 + (t * t).sum(1, keepdim=True))
        v = v + torch.linalg.cross(v + torch.linalg.cross(v, t, dim=1), s, dim=1) + half
        ig = self.inv_gamma(v)
        vel = v if ig is None else v * ig[:, None]
        fxr = fx + vel[:, 0] * (d["dt"] / d["dx"])
        shift = torch.floor(fxr.detach())
        Xo, Xn = i + fx, i + fxr
        inew, fxn = i + shift.long(), fxr - shift
        if self.dim2:
            fyr = fy + vel[:, 1] * (d["dt"] / d["dy"])
            up = torch.floor(fyr.detach())
            j, fy = (j + up.long()) % self.ny, fyr - up
        if self.per:
            return inew % self.nx, j, fxn, fy, v, pid
        keep = (inew >= 0) & (inew < self.nx)
        hit = torch.nonzero(inew < 0).squeeze(1)
        if len(hit):
            vn, back = self.returned(vel[hit], pid[hit])
            hit = hit[back]
        if len(hit):
            vn = vn[back]
            g = Xn[hit] / (Xn[hit] - Xo[hit])
            f = (g * vn[:, 0] * (d["dt"] / d["dx"])).clamp(0.0, 1.0 - 2.0 ** -53)
            if self.c2:
                vn = vn / torch.sqrt(1.0 - (vn * vn).sum(1, keepdim=True) * self.c2)
            fxn, v = fxn.index_put((hit,), f), v.index_put((hit,), vn)
            inew, keep = inew.index_fill(0, hit, 0), keep.index_fill(0, hit, True)
        return inew[keep], j[keep], fxn[keep], fy[keep], v[keep], pid[keep]

    def returned(self, v, pid):
        """Eq. 1 and the return map for particles beyond the faux shock."""
        u2, num = self.u2, pid & fs.ID_MASK
        shift = torch.stack([torch.ones_like(v[:, 0]), torch.zeros_like(v[:, 0]),
                             torch.zeros_like(v[:, 0])], 1) * u2
        w = torch.sqrt(((v + shift) ** 2).sum(1))
        a = u2 / torch.sqrt((v * v).sum(1))
        prob = torch.where(a < 1.0, ((1.0 - a) / (1.0 + a)) ** 2, torch.zeros_like(a))
        r = _philox(self.p["seed"], num, self.step_no, 3)
        back = (r[0] < prob.detach()) & (w.detach() > u2)
        if self.p["fs_mode_thermal"] == fs.FS_OPEN:
            back = back & ((pid & fs.ID_CR) != 0)
        a = u2 / w
        mu = a + (1.0 - a) * torch.sqrt(r[1])
        sn = torch.sqrt((1.0 - mu * mu).clamp(min=1e-300))
        ph = 2 * math.pi * r[2]
        return torch.stack([w * mu - u2, w * sn * torch.cos(ph), w * sn * torch.sin(ph)], 1), back

    def inflow(self):
        """The step's new particles, ids in (row, thermal then cosmic ray) order."""
        d = self.p
        if self.per or not (d["inject_thermal"] or d["cr_enable"]):
            return []
        self.acc = self.acc + ((float(d["ppc"]) * d["mach_a"]) * d["dt"]) / d["dx"]
        k = np.floor(self.acc).astype(np.int64)
        self.acc = self.acc - k
        mult = int(bool(d["inject_thermal"])) + int(bool(d["cr_enable"]))
        off = np.concatenate([[0], np.cumsum(k * mult)])
        rows = np.repeat(np.arange(self.ny), k)
        slot = np.arange(len(rows)) - np.repeat(np.cumsum(k) - k, k)
        first = self.next_id + off[rows] + slot
        self.next_id += int(off[-1])
        new, seed, dtdx = [], d["seed"], d["dt"] / d["dx"]
        row = torch.as_tensor(rows, device=DEVICE)
        if d["inject_thermal"] and len(rows):
            pid = torch.as_tensor(first, device=DEVICE)
            a, b = _philox(seed, pid, self.step_no, 4), _philox(seed, pid, self.step_no, 5)
            g0, g1 = _gauss(a[0], a[1])
            g2, _ = _gauss(a[2], a[3])
            v = torch.stack([self.vth * g0 - d["mach_a"], self.vth * g1, self.vth * g2], 1)
            new.append((self.nx - b[0] * v[:, 0].abs() * dtdx, row, b[1], v, pid))
        if d["cr_enable"] and len(rows):
            pid = torch.as_tensor(first + (k[rows] if d["inject_thermal"] else 0), device=DEVICE)
            r = _philox(seed, pid, self.step_no, 6)
            a = self.u_cr / self.piso
            mu = a + (1.0 - a) * torch.sqrt(r[0])
            sn, ph = torch.sqrt(1.0 - mu * mu), 2 * math.pi * r[1]
            v = torch.stack([self.piso * mu - self.u_cr, self.piso * sn * torch.cos(ph),
                             self.piso * sn * torch.sin(ph)], 1)
            new.append((r[2] * v[:, 0] * dtdx, row, r[3], v, pid | fs.ID_CR))
        out = []
        for X, j, fy, v, pid in new:
            i = torch.floor(X.detach()).clamp(0, self.nx - 1)
            f = (X - i).clamp(0.0, 1.0 - 2.0 ** -53)
            if self.c2:
                v = v / torch.sqrt(1.0 - (v * v).sum(1, keepdim=True) * self.c2)
            out.append((i.long(), j, f, fy if self.dim2 else torch.zeros_like(f), v, pid))
        return out

    def load(self):
        """The uniform drifting plasma at t = 0."""
        d, out = self.p, []
        total = self.nx * self.ny * d["ppc"]
        for s in range(0, total, 1 << 24):
            pid = torch.arange(s, min(total, s + (1 << 24)), device=DEVICE)
            cell = pid // d["ppc"]
            a, b = _philox(d["seed"], pid, 0, 1), _philox(d["seed"], pid, 0, 2)
            g0, g1 = _gauss(a[2], a[3])
            g2, _ = _gauss(b[0], b[1])
            v = torch.stack([self.vth * g0 - d["mach_a"], self.vth * g1, self.vth * g2], 1)
            if self.c2:
                v = v / torch.sqrt(1.0 - (v * v).sum(1, keepdim=True) * self.c2)
            top = 1.0 - 2.0 ** (-53 if d["precision"] == fs.FS_FP64 else -24)
            out.append((cell % self.nx, cell // self.nx, self.store(a[0]).clamp(max=top),
                        self.store(a[1]).clamp(max=top) if self.dim2 else torch.zeros_like(a[0]),
                        self.store(v), pid))
        self.next_id = total
        return tuple(torch.cat(x) for x in zip(*out))

    def uniform_B(self):
        b = torch.tensor(self.B0, dtype=torch.float64, device=DEVICE)
        return self.store(b)[:, None, None].expand(3, self.ny, self.nx).clone()

    def steps(self, parts, B, count):
        n, u = self.moments(parts)
        E, bb = self.ohm(B, n, u)
        block = (1 << 24) if not B.requires_grad else len(parts[0]) + (1 << 24)
        for _ in range(count):
            F = torch.cat([E, bb]).reshape(6, -1).t().contiguous()
            moved = [self.push(tuple(x[s:s + block] for x in parts), F)
                     for s in range(0, len(parts[0]), block)]
            parts = tuple(torch.cat(x) for x in zip(*(moved + self.inflow())))
            del moved
            n, u = self.moments(parts)
            B = self.advance(B, n, u)
            E, bb = self.ohm(B, n, u)
            self.step_no += 1
        return parts, dict(B=B.permute(1, 2, 0), E=E.permute(1, 2, 0), n=n, u=u.permute(1, 2, 0))


def _exact_window(c, seed):
    x, v, phases, theta, params = _window_inputs(c, seed)
    th = torch.tensor(theta, dtype=torch.float64, device=DEVICE, requires_grad=True)
    m = c["modes"]
    box = _Box64(dict(params, dim=1, ny=1), u_cr=th[m], u2=th[m + 1])
    X = torch.as_tensor(x, device=DEVICE)
    i = torch.floor(X)
    parts = (i.long(), torch.zeros_like(i).long(), box.store(X - i), torch.zeros_like(X),
             box.store(torch.as_tensor(v, device=DEVICE)), torch.arange(len(x), device=DEVICE))
    box.next_id = len(x)
    xc = (torch.arange(c["nx"], dtype=torch.float64, device=DEVICE) + 0.5) / c["nx"]
    k = torch.arange(1, m + 1, dtype=torch.float64, device=DEVICE)
    ph = 2 * math.pi * k[:, None] * xc[None, :] + torch.as_tensor(phases, device=DEVICE)[:, None]
    B = torch.stack([torch.full_like(xc, box.B0[0]),
                     box.B0[1] + (th[:m, None] * torch.cos(ph)).sum(0),
                     box.B0[2] + (th[:m, None] * torch.sin(ph)).sum(0)])[:, None, :]
    _, out = box.steps(parts, B, c["steps"])
    dB = out["B"][0, :, 1:] - torch.tensor(box.B0[1:], dtype=torch.float64, device=DEVICE)
    loss = (dB * dB).sum() * params["dx"]
    loss.backward()
    g = th.grad
    # (over a long window a single-precision forward returns a few other ions than
    # the 64-bit one; the small derivative by u_cr then belongs to another trajectory)
    return {"loss": loss.detach().reshape(1), "modes": g[:m], "u2": g[m + 1:],
            "u_cr": g[m:m + 1] if c["fp64"] else None}


def _exact_analysis(c, seed):
    box = _Box64(_params(c, seed))
    B = box.store(torch.as_tensor(_seeded_B(c, seed), device=DEVICE))
    cr = {k: torch.as_tensor(v.astype(np.int64) if v.dtype.kind in "iu" else v, device=DEVICE)
          for k, v in _seeded_cr(c, seed).items()}
    top = 1.0 - 2.0 ** (-53 if c["fp64"] else -24)
    v = torch.stack([cr["vx"], cr["vy"], cr["vz"]], 1)
    more = (cr["ci"], cr["cj"], box.store(cr["fx"]).clamp(max=top),
            box.store(cr["fy"]).clamp(max=top), box.store(v), cr["ids"])
    parts = tuple(torch.cat(x) for x in zip(box.load(), more))
    n, u = box.moments(parts)
    _, bb = box.ohm(B.permute(2, 0, 1), n, u)
    w = box.weight(parts[5]) * c["dx"] ** 2
    v = parts[4]
    B0 = torch.tensor(box.B0, dtype=torch.float64, device=DEVICE)
    F = torch.fft.fft(torch.complex(B[..., 1], torch.zeros_like(B[..., 1])), dim=1) / c["nx"]
    G = torch.fft.fft(torch.complex(B[..., 2], torch.zeros_like(B[..., 2])), dim=1) / c["nx"]
    h = c["dt"] / c["n_sub"]
    z = h * (8.0 / c["dx"] ** 2 * torch.sqrt((bb * bb).sum(0)) / n +
             4.0 / c["dx"] * torch.sqrt((u * u).sum(0)))
    return dict(n=n.mean(0), max_z=z.max().reshape(1), db2=((B - B0) ** 2).sum(2).mean(0),
                B=B.mean(0), spectrum=(F.abs() ** 2 + G.abs() ** 2).mean(0)[:c["nx"] // 2 + 1],
                energy=torch.stack([0.5 * (w * (v * v).sum(1)).sum(),
                                    0.5 * (B * B).sum() * c["dx"] ** 2]),
                momentum=(w[:, None] * v).sum(0))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "window":
        return _exact_window(c, seed)
    if kind == "analysis":
        return _exact_analysis(c, seed)
    with torch.no_grad():
        if kind == "ensemble":
            runs = []
            for p in _ensemble_params(c, seed):
                box = _Box64(p)
                runs.append(box.steps(box.load(), box.uniform_B(), c["steps"])[1])
            return {name: torch.cat([r[name].reshape(-1) for r in runs]) for _, name in FIELDS}
        box = _Box64(_params(c, seed))
        return box.steps(box.load(), box.uniform_B(), c["steps"])[1]
