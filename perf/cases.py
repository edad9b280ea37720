"""Benchmark cases of the split-step Crank-Nicolson solver: what users have it compute.

Each case is one pass of a simulation program through the public entry points (the
``Solver`` and ``Pool`` classes and the C-named calls of ``paper_1605_03958_gb300.gp``):
some time steps of the resident field, then the outputs that such a program keeps (the
field itself, and where ``sample`` is set the observables and the integrated densities
that the paper's programs write).  The field stays on the GPU from pass to pass, as in
a run that reads its state every so many steps; with ``upload`` the pass begins with
the host's field.

Kinds of cases
  solve  one ``Solver``: imaginary time (ground states) or real time (quench dynamics),
         FP64 (the paper's precision) or FP32 fields, Lie or Strang splitting, 3D grids
         or planes (nz = 1)
  pool   uneven FP32 solves resident in one ``Pool``, ground states and quenches mixed,
         as the server steps and retires them
"""
import math

import numpy as np
import torch

from paper_1605_03958_gb300 import gp

OBS = ("norm", "mu", "energy", "ekin", "epot", "eint", "rms_x", "rms_y", "rms_z", "rms_r")
TRAP = (1.0, 1.41, 2.0)   # trap ratios of the benchmark's configurations


def _solve(name, shape, prec, mode, steps, h, dtf, g, scheme="lie", sample=False, upload=False):
    return dict(name=name, kind="solve", nx=shape[0], ny=shape[1], nz=shape[2], prec=prec,
                mode=mode, steps=steps, h=h, dtf=dtf, g=float(g), scheme=scheme, sample=sample,
                upload=upload)


def listed():
    return [
        # a controller that hands a small FP32 field over, advances one step and reads it
        # back: copies, launches and latency
        _solve("step_f32_small", (64, 48, 32), "f32", "imag", 1, 0.2, 0.1, 20, upload=True),
        # the small ground state in the paper's precision (64x48x32, h = 0.2), run between
        # two looks at the energy
        _solve("ground_f64_small", (64, 48, 32), "f64", "imag", 100, 0.2, 0.1, 20, sample=True),
        # imag2d: a ground state in the plane
        _solve("ground_plane_f32", (300, 256, 1), "f32", "imag", 100, 0.08, 0.1, 200),
        # an odd grid whose rows do not fill the 16-byte vectors, FP32 ground state
        _solve("ground_f32_ragged", (131, 97, 61), "f32", "imag", 50, 0.15, 0.1, 300),
        # an odd grid in the time-reversible splitting, complex128 dynamics
        _solve("strang_c128_ragged", (101, 77, 53), "f64", "real", 20, 0.2, 0.05, 60, scheme="strang"),
        # the benchmark's workload: imag3d 240x200x160, FP32 field
        _solve("ground_f32_240x200x160", (240, 200, 160), "f32", "imag", 50, 0.1, 0.1, 100),
        # the same in the paper's precision
        _solve("ground_f64_240x200x160", (240, 200, 160), "f64", "imag", 20, 0.1, 0.1, 100),
        # real3d quench, complex64
        _solve("quench_c64_240x200x160", (240, 200, 160), "f32", "real", 50, 0.1, 0.02, 200),
        # real3d quench, complex128
        _solve("quench_c128_240x200x160", (240, 200, 160), "f64", "real", 10, 0.1, 0.02, 200),
        # what the paper's programs write at each output time of a quench: observables,
        # 1D and 2D densities
        _solve("sample_c64_240x200x160", (240, 200, 160), "f32", "real", 1, 0.1, 0.02, 200, sample=True),
        # the largest single solve: every sweep streams through HBM
        _solve("ground_f32_512x400x320", (512, 400, 320), "f32", "imag", 20, 0.1, 0.1, 100),
        # a quantum of the server: uneven ground states and quenches together, then their
        # observables and fields
        dict(name="pool_mixed_24", kind="pool", slots=24, sizes=3958, steps=200, real=0.3),
    ]


# Work units of one step and point, relative to the FP32 real field, that keep drawn
# cases below the largest listed one.
_UNIT = {("f32", "imag"): 1.0, ("f32", "real"): 2.0, ("f64", "imag"): 13.0, ("f64", "real"): 42.0}
_MOST = 1.3e9


def draw(rng):
    if rng.random() < 0.15:
        return dict(kind="pool", slots=rng.randint(3, 32), sizes=rng.randrange(1 << 20),
                    steps=rng.randint(20, 200), real=round(rng.random(), 2))
    prec = rng.choice(("f32", "f64"))
    mode = rng.choice(("imag", "real"))
    plane = rng.random() < 0.15

    def extent(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n if rng.random() < 0.5 else max(lo, n // 8 * 8)

    if plane:
        shape = (extent(64, 1024), extent(64, 1024), 1)
    else:
        shape = (extent(32, 512), extent(24, 400), extent(24, 320))
        while math.prod(shape) > (40e6 if prec == "f32" else 12e6):
            shape = tuple(max(24, int(n / 1.2)) for n in shape)
    steps = int(round(math.exp(rng.uniform(math.log(1), math.log(100)))))
    steps = max(1, min(steps, int(_MOST / (math.prod(shape) * _UNIT[prec, mode]))))
    h = round(rng.uniform(0.08, 0.25), 3)
    dtf = round(rng.uniform(0.05, 0.1) if mode == "imag" else rng.uniform(0.02, 0.1), 3)
    # a step's nonlinear phase or decay, dt g |psi|^2, stays below about 0.1 (the method's
    # regime: at phases of order 1 the dynamics of a step is chaotic)
    most = min(2000.0, 0.3 / (dtf * h * h))
    c = _solve("", shape, prec, mode, steps, h, dtf,
               round(math.exp(rng.uniform(0.0, math.log(most))), 1),
               scheme="strang" if rng.random() < 0.2 else "lie", sample=rng.random() < 0.2,
               upload=rng.random() < 0.2)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _axes(shape, h, dtype=torch.float64, device="cuda"):
    return [(torch.arange(n, dtype=dtype, device=device) - 0.5 * (n - 1)) * h for n in shape]


def _dims(c):
    return (c["nx"], c["ny"], c["nz"])


def _initial(c, seed):
    """A condensate on its way: a normalised anisotropic Gaussian, wider than the trap's
    by a seeded factor (the interaction's swelling), with long waves on it and in real
    time a smooth flow (phase); [nz, ny, nx] float64 or complex128 on the GPU."""
    rng = np.random.default_rng(seed)
    x, y, z = _axes(_dims(c), c["h"])
    wide = rng.uniform(0.4, 1.0, 3) * np.array(TRAP)
    psi = torch.exp(-0.5 * wide[2] * z * z)[:, None, None] * torch.exp(-0.5 * wide[1] * y * y)[None, :, None] \
        * torch.exp(-0.5 * wide[0] * x * x)[None, None, :]

    def wave():
        k = rng.uniform(0.1, 1.0, 3)
        p = rng.uniform(0.0, 2 * math.pi)
        return torch.cos(k[2] * z[:, None, None] + k[1] * y[None, :, None] + k[0] * x[None, None, :] + p)

    for _ in range(3):
        psi = psi * (1.0 + 0.1 * wave())
    vol = c["h"] ** (2 if c["nz"] == 1 else 3)
    psi = psi / torch.sqrt((psi * psi).sum() * vol)
    if c["mode"] == "real":
        psi = torch.polar(psi, 0.5 * wave())
    return psi


def _host_field(c, seed):
    psi = _initial(c, seed)
    if psi.is_complex():
        psi = torch.view_as_real(psi)
    return psi.to(torch.float32 if c["prec"] == "f32" else torch.float64).contiguous()


def _pool_members(c, seed):
    """The pool's members: extents by the case, trap ratios and nonlinearities by the seed
    (the server's request distributions, g up to where a step's nonlinear phase or decay
    stays well below 1: beyond that a quench is chaotic and no two roundings agree)."""
    sizes = np.random.default_rng(c["sizes"])
    rng = np.random.default_rng(seed)
    out = []
    for i in range(c["slots"]):
        nx = int(sizes.choice(np.arange(32, 129, 16)))
        ny = int(sizes.choice(np.arange(32, 97, 16)))
        nz = int(sizes.choice(np.arange(32, 65, 16)))
        real = bool(sizes.uniform() < c["real"])
        gamma, nu, lam = (float(rng.uniform(0.5, 3.0)) for _ in range(3))
        g = float(np.exp(rng.uniform(0.0, np.log(20.0 if real else 300.0))))
        out.append((real, dict(nx=nx, ny=ny, nz=nz, dx=0.2, dt=0.1 * 0.2 * 0.2, gamma=gamma, nu=nu,
                               lam=lam, g=g)))
    return out


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = c = case
    if c["kind"] == "pool":
        members = _pool_members(c, seed)
        need = sum(gp.Pool.slot_bytes(**p) for _, p in members)
        s.pool = gp.Pool(need + (1 << 20), max_slots=max(64, c["slots"]))
        s.slots = []
        for real, p in members:
            slot = s.pool.add(**p)
            if real:
                s.pool.set_real_time(slot)
            s.slots.append((slot, real))
        return s
    s.solver = gp.Solver(c["nx"], c["ny"], c["nz"], c["h"], dt=c["dtf"] * c["h"] ** 2,
                         gamma=TRAP[0], nu=TRAP[1], lam=TRAP[2], g=c["g"], prec=c["prec"])
    s.solver.set_splitting(c["scheme"])
    dev = _host_field(c, seed)
    s.psi0 = torch.empty(dev.shape, dtype=dev.dtype, pin_memory=True)
    s.psi0.copy_(dev)
    s.psi = torch.empty(dev.shape, dtype=dev.dtype, pin_memory=True)
    _upload(s)
    s.solver.sync()
    return s


def _upload(s):
    put = gp.gp_set_psi_f32_ptr if s.case["prec"] == "f32" else gp.gp_set_psi_ptr
    put(s.solver.handle, s.psi0.data_ptr(), s.case["mode"] == "real")


def run(state):
    s, c = state, state.case
    if c["kind"] == "pool":
        s.pool.step(c["steps"])
        obs = np.array([[o[k] for k in OBS] for o in (s.pool.observables(i) for i, _ in s.slots)])
        return {"obs": obs, "psi": [s.pool.get_psi(i, as_complex=real) for i, real in s.slots]}
    sv = s.solver
    real = c["mode"] == "real"
    if c["upload"]:
        _upload(s)
    (sv.step_real if real else sv.step_imag)(c["steps"])
    out = {}
    if c["sample"]:
        o = sv.observables()
        out["obs"] = np.array([o[k] for k in OBS])
        out["n1"] = [sv.density1d(a) for a in range(3)]
        out["n2"] = [sv.density2d(p) for p in range(3)]
    get = gp.gp_get_psi_f32_ptr if c["prec"] == "f32" else gp.gp_get_psi_ptr
    get(sv.handle, s.psi.data_ptr(), real)
    out["psi"] = s.psi
    return out


# -------------------------------------------------------------------- work

# Operations of one step and point: the pointwise substep (|psi|^2, the exponential's or
# phase's short polynomial, the products) and one Thomas solve per axis.
def _ops(mode, axes):
    return (39 if mode == "real" else 13) + (axes - 1) * (18 if mode == "real" else 5) + (mode == "imag")


def work(case):
    c = case
    if c["kind"] == "pool":
        b = f = 0.0
        for real, p in _pool_members(c, 0):
            n = p["nx"] * p["ny"] * p["nz"]
            e = 8 if real else 4
            # every sweep of a step reads and writes the field once; the field is read
            # once for the observables and once for the host's copy
            b += n * e * (6 * c["steps"] + 2) + n * 2 * e
            f += n * _ops("real" if real else "imag", 3) * c["steps"]
        return {"bytes": b, "flops": f}
    n = c["nx"] * c["ny"] * c["nz"]
    e = (4 if c["prec"] == "f32" else 8) * (2 if c["mode"] == "real" else 1)
    axes = 2 if c["nz"] == 1 else 3
    # a step reads and writes the field once per axis; the read-out and the samples
    # read it once, the host's copies cross once
    b = n * e * (2 * axes * c["steps"] + 2 + (1 if c["upload"] else 0) + (1 if c["sample"] else 0))
    return {"bytes": float(b), "flops": float(n * c["steps"] * _ops(c["mode"], axes))}


# ------------------------------------------------------- 64-bit reference

def _cn(n, a, dtype):
    """(I + aK)^-1 (I - aK), K the second difference with zero ghosts."""
    eye = torch.eye(n, dtype=dtype, device="cuda")
    off = torch.diag(torch.ones(n - 1, dtype=torch.float64), 1).to("cuda").to(dtype)
    k = 2 * eye - off - off.T
    return torch.linalg.solve(eye + a * k, eye - a * k)


class _Exact:
    """Plain dense 64-bit evaluation of the method on one field [nz, ny, nx]."""

    def __init__(self, shape, h, dt, trap, g, real):
        self.shape, self.h, self.dt, self.g, self.real = shape, h, dt, g, real
        self.dtype = torch.complex128 if real else torch.float64
        self.axes = 2 if shape[2] == 1 else 3
        self.x = _axes(shape, h)
        a = dt / (4 * h * h) * (1j if real else 1.0)
        self.T = [_cn(n, a, self.dtype) if i < self.axes else None for i, n in enumerate(shape)]
        vx, vy, vz = (0.5 * w * w * q * q for w, q in zip(trap, self.x))
        self.V = vz[:, None, None] + vy[None, :, None] + vx[None, None, :]
        self.dV = h ** self.axes

    def _point(self, u, dt):
        if self.real:
            # |u|^2 = re^2 + im^2: abs() takes a square root that squaring does not undo
            n = u.real * u.real + u.imag * u.imag
            return u * torch.polar(torch.ones_like(n), -dt * (self.V + self.g * n))
        return u * torch.exp(-dt * (self.V + self.g * u * u))

    def _kinetic(self, u):
        u = torch.matmul(u, self.T[0])
        u = torch.matmul(self.T[1], u)
        if self.axes == 3:
            nz = u.shape[0]
            u = torch.matmul(self.T[2], u.reshape(nz, -1)).reshape(u.shape)
        return u

    def dens(self, u):
        return u.real * u.real + u.imag * u.imag if self.real else u * u

    def step(self, u, scheme):
        if scheme == "strang":
            u = self._point(self._kinetic(self._point(u, 0.5 * self.dt)), 0.5 * self.dt)
        else:
            u = self._kinetic(self._point(u, self.dt))
        return u if self.real else u / torch.sqrt((u * u).sum() * self.dV)

    def observables(self, u):
        d = self.dens(u)
        norm = d.sum() * self.dV
        kin = 0.0
        for dim in range(3):
            if u.shape[dim] == 1:
                continue
            first, last = u.narrow(dim, 0, 1), u.narrow(dim, u.shape[dim] - 1, 1)
            diff = torch.diff(u, dim=dim)
            kin = kin + (self.dens(diff).sum() + self.dens(first).sum() + self.dens(last).sum())
        kin = 0.5 * kin / self.h ** 2 * self.dV
        pot = (self.V * d).sum() * self.dV
        inter = 0.5 * self.g * (d * d).sum() * self.dV
        x, y, z = self.x
        r2 = [(q * q * d.sum(dim=dims)).sum() * self.dV / norm
              for q, dims in ((x, (0, 1)), (y, (0, 2)), (z, (1, 2)))]
        r2[2] = r2[2] * (1.0 if self.axes == 3 else 0.0)
        v = [norm, kin + pot + 2 * inter, kin + pot + inter, kin, pot, inter, *(torch.sqrt(q) for q in r2),
             torch.sqrt(sum(r2))]
        return np.array([float(q) for q in v])

    def densities(self, u):
        d = self.dens(u)
        h = self.h
        hz = h if self.axes == 3 else 1.0
        n1 = [d.sum(dim=(0, 1)) * h * hz, d.sum(dim=(0, 2)) * h * hz, d.sum(dim=(1, 2)) * h * h]
        n2 = [d.sum(dim=0) * hz, d.sum(dim=1) * h, d.sum(dim=2) * h]
        return [t.cpu().numpy() for t in n1], [t.cpu().numpy() for t in n2]


def exact(case, seed):
    c = case
    if c["kind"] == "pool":
        if c["steps"] * c["slots"] > 8000:
            return None
        obs, psi = [], []
        for real, p in _pool_members(c, seed):
            shape = (p["nx"], p["ny"], p["nz"])
            e = _Exact(shape, p["dx"], p["dt"], (p["gamma"], p["nu"], p["lam"]), p["g"], real)
            x, y, z = e.x
            u = torch.exp(-0.5 * p["lam"] * z * z)[:, None, None] * torch.exp(-0.5 * p["nu"] * y * y)[None, :, None] \
                * torch.exp(-0.5 * p["gamma"] * x * x)[None, None, :]
            u = (u / torch.sqrt((u * u).sum() * e.dV)).to(e.dtype)
            for _ in range(c["steps"]):
                u = e.step(u, "lie")
            obs.append(e.observables(u))
            psi.append(u.cpu().numpy())
        return {"obs": np.array(obs), "psi": psi}
    real = c["mode"] == "real"
    e = _Exact(_dims(c), c["h"], c["dtf"] * c["h"] ** 2, TRAP, c["g"], real)
    u = _host_field(c, seed).double()   # the field as the solver is given it
    if real:
        u = torch.view_as_complex(u)
    for _ in range(c["steps"]):
        u = e.step(u, c["scheme"])
    out = {}
    if c["sample"]:
        out["obs"] = e.observables(u)
        out["n1"], out["n2"] = e.densities(u)
    out["psi"] = torch.view_as_real(u) if real else u
    return out
