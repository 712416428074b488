"""What a user of this library has it do, as cases that can be timed and checked.

A case is one call pattern of a particle-in-cell program: `pic_step` on a
simulation that is set up and kept (`kind` restart, run, vacuum), a batched
step (`batch`), or a round of diagnostics (`diag`).  `exact` is the same
physics as plain torch arithmetic in 64 bits, written from the method (cubic
B-spline shapes, Boris push, Esirkepov current, smoothed-curl field update,
moving window, absorbing layers); it shares no code with the package.

The fields that a pass returns are the library's own: one block of nine
component arrays [slab][j][k] (E, B, J), x slabs in ring order (window slab i
at storage slab (i + shifts) mod nx), read in place in the memory that the
program hands the library through the `pic_alloc` hooks.
"""
import math

import numpy as np
import torch

from paper_1204_0838_gb300 import pic

LAM = 0.8e-6
C0 = 299792458.0
QE, ME, EPS0 = 1.602176634e-19, 9.1093837015e-31, 8.8541878128e-12
K0 = 2.0 * math.pi / LAM
OMEGA0 = K0 * C0
BINS, P_BINS, E_MAX = 200, 64, 50.0   # spectrum bins, p_x bins, MeV
P_MIN, P_MAX, GAMMA_MIN = -4.0, 40.0, 5.0


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _case(kind, prec, nx, ny, nz, **more):
    c = dict(kind=kind, prec=prec, nx=nx, ny=ny, nz=nz, ppc=2.0, steps=2, dx=1 / 24, dt_=1 / 3, solver="perfect",
             open_x=True, pml=0, dens=0.01, lattice=True, start=0, a0=4.0, waist=16e-6, fwhm=30e-15, ramp=50e-6,
             members=0, gauss=False)
    c.update(more)
    return c


def listed():
    out = []

    def add(name, *a, **k):
        out.append(dict(_case(*a, **k), name=name))

    # One step of a few thousand particles: what a first script or a unit test
    # of a user's does; launches and latency.
    add("smoke_fp64", "restart", "fp64", 32, 8, 8, ppc=1.5, steps=1, dx=1 / 8, open_x=True)
    # A small periodic box with the standard Yee curl, odd sizes: a solver comparison.
    add("yee_fp32", "restart", "fp32", 49, 21, 27, ppc=3.0, dx=1 / 8, solver="yee", open_x=False)
    # The small full workload: boundary laser source, no window, random loading,
    # ten steps a call.
    add("source_fp64", "run", "fp64", 128, 32, 32, ppc=1.0, steps=10, dx=1 / 8, dt_=1 / 2, lattice=False, a0=2.0,
        waist=4 * LAM, fwhm=4 * LAM / C0, dens=0.02, ramp=0.0)
    # A mid-run state (wake-like density, thermal and relativistic electrons)
    # taken up again: uneven tiles, ragged sizes, every particle at a random place.
    add("restart_fp64", "restart", "fp64", 131, 45, 37, ppc=2.0, open_x=False)
    add("restart_fp32", "restart", "fp32", 251, 67, 93, ppc=2.0, open_x=True)
    # The trapping run: dense plasma, short pulse, moving window, FP64.
    add("trapping_fp64", "run", "fp64", 384, 96, 96, ppc=2.0, dens=0.03, start=900, a0=5.0, waist=4e-6, fwhm=15e-15,
        ramp=10e-6)
    # Window run with 16 absorbing layers and 4 particles a cell, FP32: the
    # paper's boundary and particle count.
    add("layers_fp32", "run", "fp32", 384, 128, 128, ppc=4.0, pml=16, dens=0.01, start=900, waist=4e-6, fwhm=15e-15,
        ramp=10e-6)
    # A parameter scan: instances of several sizes stepped together, FP32.
    add("scan_fp32", "batch", "fp32", 256, 64, 64, dx=1 / 16, members=4, fwhm=15e-15, ramp=20e-6)
    # Laser in vacuum: the field solver and the window alone, FP64.
    add("vacuum_fp64", "vacuum", "fp64", 512, 128, 128, fwhm=15e-15, waist=8e-6)
    # The diagnostics between steps of a large run, FP32.
    add("figures_fp32", "diag", "fp32", 320, 96, 96, ppc=2.0)
    # The full laser-wakefield runs, one step a call, FP32 and FP64.
    add("wakefield_fp32", "run", "fp32", 1536, 256, 256, steps=1, dens=0.004, start=900)
    add("wakefield_fp64", "run", "fp64", 1536, 256, 256, steps=1, dens=0.004, start=900)
    return out


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["restart", "restart", "run", "run", "vacuum", "batch", "diag"])
    prec = rng.choice(["fp64", "fp32"])
    dx = rng.choice([1 / 8, 1 / 16, 1 / 24, 1 / 32])
    if kind == "restart":
        pml = rng.choice([0, 0, 0, 8])
        return _case(kind, prec, size(24, 300), size(24, 110), size(24, 110), ppc=round(rng.uniform(0.5, 5.0), 2), dx=dx,
                     solver=rng.choice(["perfect", "perfect", "yee"]), open_x=rng.random() < 0.5 or pml > 0, pml=pml)
    if kind == "run":
        pml = rng.choice([0, 0, 16])
        return _case(kind, prec, size(256, 700), size(40, 160), size(40, 160), ppc=float(rng.choice([1, 2, 4, 8])),
                     dx=dx, pml=pml, dens=round(rng.uniform(0.003, 0.03), 4), lattice=rng.random() < 0.7,
                     start=rng.randint(800, 1200), a0=round(rng.uniform(2, 5), 2), waist=4e-6, fwhm=15e-15, ramp=10e-6)
    if kind == "vacuum":
        return _case(kind, prec, size(64, 600), size(24, 220), size(24, 220), dx=dx, fwhm=15e-15, waist=8e-6)
    if kind == "batch":
        return _case(kind, "fp32", size(160, 320), size(48, 80), size(48, 80), dx=1 / 16, members=rng.randint(2, 6),
                     fwhm=15e-15, ramp=20e-6)
    return _case(kind, prec, size(64, 320), size(40, 120), size(40, 120), ppc=round(rng.uniform(1.0, 4.0), 2), dx=dx,
                 gauss=rng.random() < 0.3)


def _members(case):
    """The simulations of a case: itself, or the instances of a scan."""
    if case["kind"] != "batch":
        return [case]
    out = []
    for i in range(case["members"]):
        nt = (1.0, 1.5, 2.0)[i % 3]
        out.append(dict(case, kind="run", nx=int(case["nx"] * (1 + 0.5 * (i % 2))), ny=int(case["ny"] * nt),
                        nz=int(case["nz"] * nt), ppc=float(1 + i % 2), start=700 + 20 * i))
    return out


def _x_range(case):
    """Cells along x that may hold particles."""
    return (2, case["nx"] - 4) if case["open_x"] else (0, case["nx"] - 1)


def _count(case):
    if case["kind"] == "vacuum":
        return 0
    lo, hi = _x_range(case)
    if case["kind"] == "run" and case["start"]:  # the window has entered the plasma by `start` cells
        lo = max(lo, case["nx"] - case["start"])
    m = case["pml"]
    return int(case["ppc"] * (hi - lo + 1) * (case["ny"] - 2 * m) * (case["nz"] - 2 * m))


def work(case):
    """Per step: every particle record read and written, E and B read and
    written, J written; 1613 flops a particle (shapes, gather, Boris, deposit),
    about 120 a cell (field update).  A round of diagnostics reads the momenta
    and weights once, the fields once and writes its results."""
    size = 8 if case["prec"] == "fp64" else 4
    b = f = 0.0
    for m in _members(case):
        n, cells = _count(m), m["nx"] * m["ny"] * m["nz"]
        if case["kind"] == "diag":
            return {"bytes": n * (4 + 7 * size) + 6.0 * cells * size, "flops": n * 40.0 + 12.0 * cells}
        b += m["steps"] * (n * 2 * (4 + 7 * size) + 15.0 * cells * size)
        f += m["steps"] * (n * 1613.0 + cells * 120.0)
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _state(case, seed):
    """A mid-run state from the seed, as float64 tensors on the GPU: fields
    (6, nx, ny, nz), cells (3, n), offsets and momenta (3, n), weights (n).
    Density crests and a drift of a plasma wave along x, a thermal spread and
    one electron in a hundred fast; fields of the wave and of a pulse in the
    front third, with noise.  Values are float32 numbers."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n, f32 = _count(case), torch.float32

    def uniform(k):
        return torch.rand(k, generator=g, device="cuda", dtype=torch.float64)

    def normal(*k):
        return torch.randn(*k, generator=g, device="cuda", dtype=torch.float64)

    lo, hi = _x_range(case)
    m = case["pml"]
    s = uniform(n)
    ph = 2 * math.pi * 3 * s
    x = lo + (hi + 1 - lo) * (s + 0.6 / (2 * math.pi * 3) * torch.sin(ph)).clamp(0.0, 1.0)
    y, z = m + (ny - 2 * m) * uniform(n), m + (nz - 2 * m) * uniform(n)
    cell, off = [], []
    for p, a, b in ((x, lo, hi), (y, m, ny - m - 1), (z, m, nz - m - 1)):
        c = p.floor().clamp(a, b)
        cell.append(c.to(torch.int64))
        off.append((p - c).clamp(0.0, 0.9999).to(f32).double())
    u = 0.05 * normal(3, n)
    u[0] += 0.4 * torch.sin(ph)
    u[1:] *= 2.0
    fast = uniform(n) < 0.01
    u[0] += 20.0 * fast
    w = case["dens"] / max(case["ppc"], 1e-3) * _cell_volume(case) * (0.5 + uniform(n))
    F = 1e-3 * normal(6, nx, ny, nz)
    i = torch.arange(nx, device="cuda", dtype=torch.float64)
    wave = torch.sin(2 * math.pi * 3 * (i + 0.5) / nx)
    pulse = 1.5 * torch.exp(-((i - 0.8 * nx) / (0.08 * nx)) ** 2) * torch.sin(2 * math.pi * case["dx"] * i)
    F[0] += 0.1 * wave[:, None, None]
    F[1] += pulse[:, None, None]
    F[5] += pulse[:, None, None]
    return F.to(f32).double(), torch.stack(cell), torch.stack(off), u.to(f32).double(), w.to(f32).double()


def _cell_volume(case):
    return (2 * math.pi) ** 3 * case["dx"] * case["dt_"] ** 2


def _laser(case, seed):
    """(a0, waist, fwhm, focus, peak time) of a case and seed."""
    r = np.random.RandomState(seed % (1 << 31))
    a0 = case["a0"] * float(r.uniform(0.95, 1.05))
    return a0, case["waist"], case["fwhm"], 0.0, 2 * case["fwhm"] - case["start"] * case["dx"] * LAM / C0


def _profile(case):
    if case["ramp"] > 0:
        return [0.0, case["ramp"], 1.0], [0.0, case["dens"], case["dens"]]
    return [-1.0, 1.0], [case["dens"], case["dens"]]


def _x0(case):
    """Lab x of the window's back at t = 0 (m): a window enters the plasma by `start` cells."""
    return (case["start"] - case["nx"]) * case["dx"] * LAM if _windowed(case) else 0.0


def _windowed(case):
    return case["kind"] == "vacuum" or (case["kind"] == "run" and case["start"] > 0)


class Memory:
    """The program's own device memory, handed out through the pic_alloc hooks."""

    def __init__(self):
        kinds = dict(pic.pic_alloc._fields_)
        self.blocks = {}
        self._hooks = kinds["alloc"](self._give), kinds["free"](self._take)
        self.struct = pic.pic_alloc(self._hooks[0], self._hooks[1], None)

    def _give(self, size, ctx):
        try:
            t = torch.empty(int(size), dtype=torch.uint8, device="cuda")
        except RuntimeError:
            return None
        self.blocks[t.data_ptr()] = t
        return t.data_ptr()

    def _take(self, ptr, ctx):
        self.blocks.pop(ptr, None)


def _simulation(case, seed):
    """(simulation, E, B, J): set up as the case says, its fields read in place."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    mem = Memory()
    s = pic.Sim(nx, ny, nz, case["dx"] * LAM, case["dt_"] * LAM, case["dt_"] * LAM, LAM, x0=_x0(case),
                periodic_x=not case["open_x"], precision=case["prec"], seed=seed, solver=case["solver"],
                window=(1.0, 0.0) if _windowed(case) else None, pml=case["pml"], memory=mem)
    kind = torch.float64 if case["prec"] == "fp64" else torch.float32
    want = 9 * nx * ny * nz
    size = (want * kind.itemsize + 255) // 256 * 256
    block = next(t for t in mem.blocks.values() if t.numel() == size)
    F = block[: want * kind.itemsize].view(kind).view(9, nx, ny, nz)
    if case["kind"] in ("restart", "diag"):
        fields, cell, off, u, w = _state(case, seed)
        for c in range(6):
            s.set_field(c, fields[c].cpu().numpy())
        s.set_particles((cell + off).cpu().numpy(), u.cpu().numpy(), w.cpu().numpy())
    else:
        if case["kind"] != "vacuum":
            s.add_species(*_profile(case), int(case["ppc"]), loading="lattice" if case["lattice"] else "random")
        a0, waist, fwhm, focus, peak = _laser(case, seed)
        s.add_laser(a0, waist, fwhm, LAM, x_focus=focus, t_peak=peak)
    return s, {"E": F[0:3], "B": F[3:6], "J": F[6:9]}


class _Scan:
    """Simulations stepped together, ended in the order that the library asks for."""

    def __init__(self, sims):
        self.sims = sims
        self.handle = pic.pic_batch_create([s.h for s in sims])

    def __del__(self):
        pic.pic_batch_destroy(self.handle)


def prepare(case, seed):
    made = [_simulation(m, seed + i) for i, m in enumerate(_members(case))]
    state = {"case": case, "sims": [s for s, _ in made], "fields": [f for _, f in made]}
    if case["kind"] == "batch":
        state["scan"] = _Scan(state["sims"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        pic.pic_batch_step(state["scan"].handle, case["steps"])
        return state["fields"]
    s = state["sims"][0]
    if case["kind"] != "diag":
        s.step(case["steps"])
        return state["fields"][0]
    out = {"lineout": s.diag("ex_lineout"), "energy": s.diag("field_energy"), "charge": s.diag("charge", 1, GAMMA_MIN),
           "spectrum": s.diag("spectrum", BINS, 0.0, E_MAX), "emittance": s.diag("emittance", 2, GAMMA_MIN),
           "phase": s.diag("phase_x_px", case["nx"] * P_BINS, P_MIN, P_MAX), "density": s.diag("density_xy")}
    if case["gauss"]:
        out["gauss"] = s.diag("dive_residual", 3)
    return out


# ---------------------------------------------------------------------------
# The same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _at(a, axis, by, wrap):
    """a at index + by along an axis: periodic, or zero beyond the ends."""
    r = torch.roll(a, -by, axis)
    if not wrap:
        n = a.shape[axis]
        r.narrow(axis, n - by if by > 0 else 0, abs(by)).zero_()
    return r


def _m4(d):
    """The centred cubic B-spline."""
    a = d.abs()
    return torch.where(a < 1, (4 - 6 * a * a + 3 * a ** 3) / 6, (2 - a).clamp(min=0) ** 3 / 6)


def _mix64(seed, n):
    """(n + 1)-th SplitMix64 output of the stream `seed`, as a uniform in [0, 1)."""
    def signed(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >> 63 else v

    def down(v, k):
        return (v >> k) & ((1 << (64 - k)) - 1)

    z = signed(seed) + (n + 1) * signed(0x9E3779B97F4A7C15)
    z = (z ^ down(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ down(z, 27)) * signed(0x94D049BB133111EB)
    return down(z ^ down(z, 31), 11).double() / 9007199254740992.0


class Exact:
    """One simulation in 64 bits; arrays in window order."""

    def __init__(self, case, seed):
        self.case, self.seed = case, seed
        self.n = case["nx"], case["ny"], case["nz"]
        self.d = [2 * math.pi * case["dx"], 2 * math.pi * case["dt_"], 2 * math.pi * case["dt_"]]
        self.yee = case["solver"] == "yee"
        self.dt = 0.999 / math.sqrt(sum(1 / v ** 2 for v in self.d)) if self.yee else self.d[0]
        self.wrap = [not case["open_x"], case["pml"] == 0, case["pml"] == 0]
        self.window, self.x0 = _windowed(case), _x0(case) * K0
        self.t_step = self.shifts = 0
        self.E, self.B, self.J = (torch.zeros(3, *self.n, device="cuda", dtype=torch.float64) for _ in range(3))
        r = [1.0, (self.d[0] / self.d[1]) ** 2, (self.d[0] / self.d[2]) ** 2]
        self.smooth = []
        for a, b in ((1, 2), (0, 2), (0, 1)):
            g = 0.0 if self.yee else r[a] * r[b] / 48
            e = [0.0 if self.yee else r[k] / 8 - 2 * g for k in (a, b)]
            self.smooth.append((a, b, 1 - 2 * e[0] - 2 * e[1] - 4 * g, e[0], e[1], g))
        self._layers()
        self.cell = torch.zeros(3, 0, device="cuda", dtype=torch.int64)
        self.o = self.u = torch.zeros(3, 0, device="cuda", dtype=torch.float64)
        self.w = torch.zeros(0, device="cuda", dtype=torch.float64)
        self.source = None
        if case["kind"] in ("restart", "diag"):
            F, self.cell, self.o, self.u, self.w = _state(case, seed)
            self.E, self.B = F[:3].clone(), F[3:].clone()
        else:
            if case["kind"] != "vacuum":
                self._load(*_x_range(case))
            self._add_laser()
        self.C = self._curl_e(False)

    # absorbing layers: coefficients per position, memory variables per derivative
    def _layers(self):
        self.psi, self.ab = {}, {}
        L = self.case["pml"]
        for ax in (1, 2):
            for half in (0, 1):
                pos = torch.arange(self.n[ax], device="cuda", dtype=torch.float64) + 0.5 * half
                depth = torch.maximum(L - pos, pos - (self.n[ax] - 1 - L)).clamp(min=0) / max(L, 1)
                sigma = 2 * math.log(1e6) / (max(L, 1) * self.d[ax]) * depth ** 3
                b = torch.exp(-sigma * self.dt)
                self.ab[ax, half] = [v.view([-1 if k == ax else 1 for k in range(3)]) for v in (b - 1, b)]

    def _stretch(self, key, ax, half, v, advance):
        if not self.case["pml"]:
            return v
        p = self.psi.setdefault(key, torch.zeros_like(v))
        if advance:
            a, b = self.ab[ax, half]
            p = self.psi[key] = b * p + a * v
        return v + p

    def _s(self, a, F):
        t1, t2, c, e1, e2, g = self.smooth[a]
        if self.yee:
            return F
        pair = [_at(F, t, 1, self.wrap[t]) + _at(F, t, -1, self.wrap[t]) for t in (t1, t2)]
        corner = _at(pair[0], t2, 1, self.wrap[t2]) + _at(pair[0], t2, -1, self.wrap[t2])
        return c * F + e1 * pair[0] + e2 * pair[1] + g * corner

    def _up(self, a, F):  # forward difference along a of the field smoothed across it
        S = self._s(a, F)
        return (_at(S, a, 1, self.wrap[a]) - S) / self.d[a]

    def _curl_e(self, advance):
        E = self.E
        dyEz, dyEx = (self._stretch(k, 1, 1, self._up(1, E[c]), advance) for k, c in (("cxy", 2), ("czy", 0)))
        dzEy, dzEx = (self._stretch(k, 2, 1, self._up(2, E[c]), advance) for k, c in (("cxz", 1), ("cyz", 0)))
        return torch.stack([dyEz - dzEy, dzEx - self._up(0, E[2]), self._up(0, E[1]) - dyEx])

    def _down(self, a, F):
        return (F - _at(F, a, -1, self.wrap[a])) / self.d[a]

    def _fields(self):
        Bh = self.B - 0.5 * self.dt * self.C
        dyBz, dyBx = (self._stretch(k, 1, 0, self._down(1, Bh[c]), True) for k, c in (("exy", 2), ("ezy", 0)))
        dzBy, dzBx = (self._stretch(k, 2, 0, self._down(2, Bh[c]), True) for k, c in (("exz", 1), ("eyz", 0)))
        curl = torch.stack([dyBz - dzBy, dzBx - self._down(0, Bh[2]), self._down(0, Bh[1]) - dyBx])
        self.E = self.E + self.dt * (curl - self.J)
        if self.source:
            self.E[1][0] = self._laser_at(self.x0, self.t_step * self.dt)
        self.C = self._curl_e(True)
        self.B = Bh - 0.5 * self.dt * self.C

    def _laser_at(self, x, t):
        """E_y at lab x (number or (nx, 1, 1)) over the transverse nodes (j + 1/2, k)."""
        a0, w0, zr, tau, xf, tpk = self.source or self.pulse
        y = (torch.arange(self.n[1], device="cuda", dtype=torch.float64) + 0.5)[:, None] * self.d[1] - 0.5 * self.n[1] * self.d[1]
        z = torch.arange(self.n[2], device="cuda", dtype=torch.float64)[None, :] * self.d[2] - 0.5 * self.n[2] * self.d[2]
        r2 = y * y + z * z
        xi = torch.as_tensor(x - xf, device="cuda", dtype=torch.float64)
        w = w0 * torch.sqrt(1 + (xi / zr) ** 2)
        lag = xi - (t - tpk)
        phase = torch.atan2(xi, torch.full_like(xi, zr)) - lag - 0.5 * r2 * xi / (xi * xi + zr * zr)
        return a0 * (w0 / w) * torch.exp(-r2 / (w * w)) * torch.exp(-2 * math.log(2) * (lag / tau) ** 2) * torch.sin(phase)

    def _add_laser(self):
        a0, waist, fwhm, focus, peak = _laser(self.case, self.seed)
        self.pulse = a0, waist * K0, 0.5 * (waist * K0) ** 2, fwhm * OMEGA0, focus * K0, peak * OMEGA0
        if not self.window:
            self.source = self.pulse
            self.E[1][0] = self._laser_at(self.x0, 0.0)
            return
        x = (torch.arange(self.n[0], device="cuda", dtype=torch.float64) * self.d[0] + self.x0)[:, None, None]
        Ey, Bz = self._laser_at(x, 0.0), self._laser_at(x + 0.5 * self.d[0], 0.5 * self.dt)
        Ex = torch.cumsum(-self.d[0] * self._down(1, Ey), 0)
        slope = -self.d[0] * (_at(Bz, 2, 1, self.wrap[2]) - Bz) / self.d[2]
        self.E = torch.stack([Ex, Ey, torch.zeros_like(Ex)])
        B = torch.stack([torch.cumsum(slope, 0) - slope, torch.zeros_like(Ex), Bz])
        pml, self.case = self.case["pml"], dict(self.case, pml=0)  # the set-up curl has no memory variables
        self.B = B + 0.5 * self.dt * self._curl_e(False)
        self.case = dict(self.case, pml=pml)

    def _load(self, lo, hi):
        c, (nx, ny, nz) = self.case, self.n
        ppc, lat = int(c["ppc"]), (1, 1, 1)
        if c["lattice"]:
            lat = {1: (1, 1, 1), 2: (1, 2, 1), 4: (1, 2, 2), 8: (2, 2, 2)}[ppc]
        m = c["pml"]
        ranges = ((lo, hi + 1), (m, ny - m), (m, nz - m), (0, ppc))
        i, j, k, s = (v.reshape(-1) for v in torch.meshgrid(*(torch.arange(*r, device="cuda") for r in ranges), indexing="ij"))
        key = ((((self.shifts + i) * ny + j) * nz + k) * ppc + s) * 3
        o = torch.stack([_mix64(self.seed, key + a) for a in range(3)])
        if c["lattice"]:
            part = [s // (lat[1] * lat[2]), (s // lat[2]) % lat[1], s % lat[2]]
            o = torch.stack([(part[a] + o[a]) / lat[a] for a in range(3)])
        x = self.x0 + (self.shifts + i + o[0]) * self.d[0]
        px, pn = _profile(c)
        dens = torch.zeros_like(x)
        for a in range(len(px) - 1):
            a0, a1 = px[a] * K0, px[a + 1] * K0
            dens = torch.where((x >= a0) & (x <= a1), pn[a] + (x - a0) / (a1 - a0) * (pn[a + 1] - pn[a]), dens)
        keep = dens > 0
        if c["prec"] == "fp32":
            o = o.float().clamp(max=0.99999994).double()
        w = dens * (self.d[0] * self.d[1] * self.d[2] / ppc)
        w = w.float().double() if c["prec"] == "fp32" else w
        self.cell = torch.cat([self.cell, torch.stack([i, j, k])[:, keep]], 1)
        self.o = torch.cat([self.o, o[:, keep]], 1)
        self.u = torch.cat([self.u, torch.zeros_like(o[:, keep])], 1)
        self.w = torch.cat([self.w, w[keep]])

    def _flat(self, idx):
        return ((idx[0] % self.n[0]) * self.n[1] + idx[1] % self.n[1]) * self.n[2] + idx[2] % self.n[2]

    def _gather(self, F, stag, cell, o):
        base, wt = [], []
        for a in range(3):
            low = (o[a] < 0.5).long() if stag[a] else 0
            base.append(cell[a] - 1 - low)
            t = o[a] - 0.5 * stag[a]
            wt.append([_m4(t + 1 + low - m) for m in range(4)])
        out = torch.zeros_like(o[0])
        F = F.reshape(-1)
        for a in range(4):
            for b in range(4):
                for c in range(4):
                    out += F[self._flat((base[0] + a, base[1] + b, base[2] + c))] * (wt[0][a] * wt[1][b] * wt[2][c])
        return out

    def _deposit(self, cell, o0, o1, qw, lo, hi):
        """Esirkepov current over nodes cell + lo .. cell + hi; o1 relative to the old cell."""
        S0 = [[_m4(o0[a] - m) for m in range(lo, hi + 1)] for a in range(3)]
        D = [[_m4(o1[a] - m) - S0[a][m - lo] for m in range(lo, hi + 1)] for a in range(3)]
        n = hi - lo + 1
        for comp in range(3):
            b_, c_ = [a for a in range(3) if a != comp]
            f = -qw / (self.dt * self.d[b_] * self.d[c_])
            J = self.J[comp].reshape(-1)
            for b in range(n):
                for c in range(n):
                    A = f * (S0[b_][b] * (S0[c_][c] + D[c_][c] / 2) + D[b_][b] * (S0[c_][c] / 2 + D[c_][c] / 3))
                    run = torch.zeros_like(qw)
                    for m in range(n - 1):
                        run = run + D[comp][m]
                        at = [None] * 3
                        at[comp], at[b_], at[c_] = cell[comp] + lo + m, cell[b_] + lo + b, cell[c_] + lo + c
                        J.index_add_(0, self._flat(at), run * A)

    def _push(self):
        self.J.zero_()
        h, parts = -0.5 * self.dt, []
        for i in range(0, self.w.numel(), 1 << 21):
            s = slice(i, i + (1 << 21))
            cell, o, u, w = self.cell[:, s], self.o[:, s], self.u[:, s], self.w[s]
            e = [self._gather(self.E[a], [int(a == k) for k in range(3)], cell, o) for a in range(3)]
            b = [self._gather(self.B[a], [int(a != k) for k in range(3)], cell, o) for a in range(3)]
            e, b = torch.stack(e), torch.stack(b)
            um = u + h * e
            t = h * b / torch.sqrt(1 + (um * um).sum(0))
            sv = 2 * t / (1 + (t * t).sum(0))
            u = um + torch.cross(um + torch.cross(um, t, dim=0), sv, dim=0) + h * e
            move = torch.stack([self.dt / self.d[a] * u[a] for a in range(3)]) / torch.sqrt(1 + (u * u).sum(0))
            end = o + move
            step = end.floor().long()
            still = (step == 0).all(0)
            for pick, lo, hi in ((still, -1, 2), (~still, -2, 3)):
                self._deposit(cell[:, pick], o[:, pick], end[:, pick], -w[pick], lo, hi)
            parts.append((cell + step, end - step, u, w))
        if parts:
            self.cell, self.o, self.u = (torch.cat([p[k] for p in parts], 1) for k in range(3))
            self.w = torch.cat([p[3] for p in parts])

    def step(self):
        self._push()
        self.t_step += 1
        self._fields()
        if self.window:  # v = c and c dt = dx: one cell every step
            self.shifts += 1
            self.E, self.B, self.J = (_at(v, 1, 1, False) for v in (self.E, self.B, self.J))
            self.psi = {k: _at(v, 0, 1, False) for k, v in self.psi.items()}
            self.C = self._curl_e(False)
            self.cell[0] -= 1
        lo, hi = _x_range(self.case)
        m = self.case["pml"]
        keep = torch.ones_like(self.w, dtype=torch.bool)
        if not self.wrap[0]:
            keep &= (self.cell[0] >= lo) & (self.cell[0] <= hi)
        for a in (1, 2):
            if m:
                keep &= (self.cell[a] >= m) & (self.cell[a] < self.n[a] - m)
        self.cell = torch.stack([self.cell[a] % self.n[a] if self.wrap[a] else self.cell[a] for a in range(3)])
        self.cell, self.o, self.u, self.w = self.cell[:, keep], self.o[:, keep], self.u[:, keep], self.w[keep]
        if self.window and self.case["kind"] == "run":
            self._load(hi, hi)

    def fields(self):
        return {k: torch.roll(v, self.shifts % self.n[0], 1) for k, v in (("E", self.E), ("B", self.B), ("J", self.J))}

    def figures(self):
        nx, ny, nz = self.n
        e0, length = ME * C0 * OMEGA0 / QE, C0 / OMEGA0
        nc = EPS0 * ME * OMEGA0 ** 2 / QE ** 2
        q = QE * nc * length ** 3
        dv = self.d[0] * self.d[1] * self.d[2]
        gam = torch.sqrt(1 + (self.u * self.u).sum(0))
        mev = (gam - 1) * ME * C0 * C0 / (QE * 1e6)

        def hist(idx, w, n):
            return torch.zeros(n, device="cuda", dtype=torch.float64).index_add_(0, idx, w)

        fast = gam > GAMMA_MIN
        w = self.w[fast]
        emit = []
        for a in (1, 2):
            r = (self.cell[a][fast] + self.o[a][fast] - 0.5 * self.n[a]) * self.d[a]
            u = self.u[a][fast]
            mean = [(w * v).sum() / w.sum() for v in (u, r, u * u, r * r, u * r)]
            det = (mean[2] - mean[0] ** 2) * (mean[3] - mean[1] ** 2) - (mean[4] - mean[0] * mean[1]) ** 2
            emit.append(math.sqrt(max(float(det), 0.0)) * length)
        at = (mev >= 0) & (mev < E_MAX)
        spectrum = hist((mev[at] / E_MAX * BINS).long().clamp(max=BINS - 1), self.w[at], BINS)
        ux = self.u[0]
        pin = (ux >= P_MIN) & (ux < P_MAX)
        pb = ((ux[pin] - P_MIN) / (P_MAX - P_MIN) * P_BINS).long().clamp(max=P_BINS - 1)
        mid = self.cell[2] == nz // 2
        out = {"lineout": (self.E[0][:, ny // 2, nz // 2] * e0).cpu().numpy(),
               "energy": np.array([0.5 * dv * EPS0 * e0 ** 2 * length ** 3 * float((self.E ** 2).sum() + (self.B ** 2).sum())]),
               "charge": np.array([float(w.sum()) * q]), "spectrum": (spectrum * q).cpu().numpy(), "emittance": np.array(emit),
               "phase": (hist(self.cell[0][pin] * P_BINS + pb, self.w[pin], nx * P_BINS) * q).cpu().numpy(),
               "density": (hist(self.cell[0][mid] * ny + self.cell[1][mid], self.w[mid], nx * ny) / dv).cpu().numpy()}
        if self.case["gauss"]:
            rho = torch.zeros(nx * ny * nz, device="cuda", dtype=torch.float64)
            wt = [[_m4(self.o[a] - m) for m in range(-1, 3)] for a in range(3)]
            for i in range(4):
                for j in range(4):
                    for k in range(4):
                        rho.index_add_(0, self._flat((self.cell[0] + i - 1, self.cell[1] + j - 1, self.cell[2] + k - 1)),
                                       -self.w / dv * wt[0][i] * wt[1][j] * wt[2][k])
            rho = rho.view(nx, ny, nz)
            div = sum(self._down(a, self.E[a]) for a in range(3))
            r, e = float((div - rho).abs().max()), float(rho.abs().max())
            out["gauss"] = np.array([r / e, r * QE * nc, e * QE * nc])
        return out


def exact(case, seed):
    members = _members(case)
    if sum(_count(m) * m["steps"] for m in members) > 150e6:
        return None  # half a minute and more
    got = []
    for i, m in enumerate(members):
        sim = Exact(m, seed + i)
        if case["kind"] == "diag":
            return sim.figures()
        for _ in range(m["steps"]):
            sim.step()
        got.append(sim.fields())
    return got if case["kind"] == "batch" else got[0]
