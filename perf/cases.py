"""Workloads of the Maxwell–Bloch FDTD framework as a user's program runs them.

``listed()`` names the workloads, ``draw`` makes more of the same ranges,
``prepare`` builds what a program holds before the timed call (contexts with
their materials, probes and tuned launches), ``run`` is one pass through the
public entry points and ``exact`` the same results in plain 64-bit torch and
numpy.

Kinds:

* ``step``     one realization advanced and its state read (``MBSimulation``);
* ``ensemble`` several realizations advanced together (``MBBatch``);
* ``adjoint``  a gradient of the energy through the +z face on a context;
* ``design``   the same gradient through ``torch.autograd`` with a graded map;
* ``readout``  what a long run reads at its recorded times;
* ``theory``   the spectral features of the envelope equation versus pump.

The samples are packings of spheres (d = 300 nm, 10 % spread, about 45 % fill,
dx = 20 nm) with the gain medium in the voids and the background in the CPML,
as in ``inputs.py``, made from a periodic 64-cell tile so that they are quick
to make at every size.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_0809_1547_gb300 import gp
from paper_0809_1547_gb300.autograd import Realization, emitted_energy
from paper_0809_1547_gb300.binding import MBBatch, MBSimulation, mb_default_params

C0 = 299_792_458.0
EPS0 = 8.8541878128e-12
HBAR = 1.054571817e-34
QE = 1.602176634e-19
DX = 20e-9
DT = 0.99 * DX / (C0 * math.sqrt(3.0))
PUMP = 1e13
EPS_SPHERE = 8.41
LAM_MIN, LAM_MAX, N_FREQ = 475e-9, 705e-9, 128
FACE_STRIDE, FACE_EVERY = 8, 4
CW_LAM, PULSE_LAM = 586.5e-9, 532e-9
TILE = 64

EH = ("Ex", "Ey", "Ez", "Hx", "Hy", "Hz")
STATE = EH + ("Px", "Py", "Pz", "Jx", "Jy", "Jz", "N1", "N2", "N3")
MEMBER = ("Ez", "Hz", "Jz", "N2")   # read of every ensemble member beside its spectrum


# ------------------------------------------------------------------ the cases

def _step(name, nx, ny, nz, steps, npml=8, eps="packed", gain=True, source="none", point=True,
          faces=False, plane=False, state=True):
    c = {"kind": "step", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "npml": npml, "eps": eps,
         "gain": gain, "source": source, "point": point, "faces": faces, "plane": plane,
         "state": state}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a program that looks at the fields after every
        # step of a test-sized ragged grid
        _step("monitor_24", 24, 22, 20, 1, npml=4, point=False, state=False),
        # the 48^3 parity configuration, a stretch of its 500 steps
        _step("burst_48", 48, 48, 48, 100),
        # one member of the pump-sweep ensemble on its own: an odd cube
        _step("member_139", 139, 139, 139, 64),
        # a ragged box with a graded map (more than 128 eps_r values) and the
        # single-cycle pulse
        _step("graded_157", 157, 131, 110, 48, eps="graded", source="pulse"),
        # the benchmark: the paper-scale sample with the centre and the six
        # face probes
        _step("paper_320", 320, 320, 320, 64, faces=True),
        # the same geometry without gain under CW excitation: the mode map of
        # the middle section
        _step("passive_cw_320", 320, 320, 320, 48, gain=False, source="cw", point=False, plane=True),
        # the largest sample
        _step("large_448", 448, 448, 448, 16, faces=True),
        # the pump sweep: uneven cubes (sides of the 80-member ensemble) at
        # several atomic densities
        {"name": "ensemble_12", "kind": "ensemble", "sides": "97,126,148", "levels": 4, "steps": 40},
        # the adjoint configuration, three of its checkpoint segments
        {"name": "adjoint_96", "kind": "adjoint", "nx": 96, "ny": 96, "nz": 96, "steps": 600,
         "ckpt": 200, "npml": 8, "eps": "packed"},
        # one iteration of a small inverse-design loop through autograd
        {"name": "design_40", "kind": "design", "nx": 40, "ny": 37, "nz": 24, "steps": 120, "ckpt": 30,
         "npml": 4, "eps": "graded"},
        # the read-outs at a recorded time: energy, face and centre spectra,
        # middle section
        {"name": "readout_160", "kind": "readout", "nx": 160, "ny": 160, "nz": 160, "steps": 32,
         "npml": 8},
        # theory curves of linewidth and peak versus pump
        {"name": "theory_200", "kind": "theory", "pumps": 200, "grid": 2047, "kappa": 0.1},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(["step", "ensemble", "adjoint", "design", "readout", "theory"],
                       [10, 2, 2, 1, 2, 2])[0]
    if kind == "theory":
        return {"kind": kind, "pumps": _log_int(rng, 1, 256), "grid": _log_int(rng, 255, 2500),
                "kappa": round(rng.uniform(0.08, 0.3), 4)}
    if kind == "ensemble":
        sides = sorted(rng.randint(96, 160) for _ in range(rng.randint(1, 3)))
        return {"kind": kind, "sides": ",".join(map(str, sides)), "levels": rng.randint(1, 4),
                "steps": rng.randint(2, 40)}
    if kind == "adjoint":
        steps = _log_int(rng, 40, 300)
        return {"kind": kind, "nx": rng.randint(40, 112), "ny": rng.randint(40, 112),
                "nz": rng.randint(40, 112), "steps": steps, "ckpt": rng.randint(20, 200),
                "npml": rng.choice([4, 8]), "eps": "packed"}
    if kind == "design":
        return {"kind": kind, "nx": rng.randint(20, 64), "ny": rng.randint(20, 64),
                "nz": rng.randint(20, 64), "steps": _log_int(rng, 20, 200), "ckpt": rng.randint(10, 60),
                "npml": 4, "eps": "graded"}
    if kind == "readout":
        base = _log_int(rng, 48, 256)
        return {"kind": kind, "nx": base + rng.randint(-8, 8), "ny": base + rng.randint(-8, 8),
                "nz": base + rng.randint(-8, 8), "steps": rng.randint(4, 40), "npml": 8}
    base = math.exp(rng.uniform(math.log(20.0), math.log(320.0)))
    n = [max(18, min(400, int(base * rng.uniform(0.7, 1.4)))) for _ in range(3)]
    if rng.random() < 0.4:
        n[0] = max(32, n[0] // 16 * 16)
    cells = n[0] * n[1] * n[2]
    steps = max(1, min(_log_int(rng, 1, 100), int(1.2e9 / cells)))
    gain = rng.random() < 0.75
    if not gain:   # the source's field has to reach the sample
        steps = max(steps, 12)
    return _step(None, n[0], n[1], n[2], steps, npml=8 if min(n) >= 24 and rng.random() < 0.75 else 4,
                 eps="packed" if rng.random() < 0.75 else "graded", gain=gain,
                 source=rng.choice(["none", "pulse"]) if gain else rng.choice(["pulse", "cw"]),
                 point=rng.random() < 0.7, faces=rng.random() < 0.4, plane=rng.random() < 0.2)


# ----------------------------------------------------------------- the samples

def _tile(rng):
    """Signed distance (cells, positive inside) to the nearest sphere surface
    of a periodic packing on a TILE^3 tile."""
    d = np.clip(rng.normal(15.0, 1.5, 67), 7.5, 22.5)
    x, r = rng.random((len(d), 3)) * TILE, 0.5 * d
    for _ in range(200):
        v = x[:, None] - x[None]
        v -= TILE * np.round(v / TILE)
        dist = np.linalg.norm(v, axis=2) + 1e-9
        lap = np.maximum(r[:, None] + r[None] + 0.02 - dist, 0.0)
        np.fill_diagonal(lap, 0.0)
        if lap.max() < 0.05:
            break
        x = (x + 0.5 * (v / dist[..., None] * lap[..., None]).sum(1)) % TILE
    c = torch.arange(TILE, device="cuda", dtype=torch.float32) + 0.5
    best = torch.full((TILE,) * 3, -1e9, device="cuda")
    for (cx, cy, cz), rad in zip(x.tolist(), r.tolist()):
        q = [((c - o + TILE / 2) % TILE - TILE / 2).square() for o in (cx, cy, cz)]
        best = torch.maximum(best, rad - torch.sqrt(q[2][:, None, None] + q[1][:, None] + q[0]))
    return best


def _maps(grid, npml, eps, seed):
    """(eps_r float32, gain uint8) on the GPU, indexed [k, j, i]."""
    rng = np.random.default_rng(seed)
    tile = _tile(rng)
    ix = [((torch.arange(n, device="cuda") + int(rng.integers(TILE))) % TILE) for n in grid]
    s = tile[ix[2][:, None, None], ix[1][:, None], ix[0]]
    core = [((torch.arange(n, device="cuda") >= npml) & (torch.arange(n, device="cuda") < n - npml))
            for n in grid]
    core = core[2][:, None, None] & core[1][:, None] & core[0]
    if eps == "packed":
        e = torch.where((s > 0) & core, EPS_SPHERE, 1.0)
        gain = (s <= 0) & core
    else:   # soft edges three cells wide: every edge cell a value of its own
        e = torch.where(core, 1.0 + (EPS_SPHERE - 1.0) * (s / 3.0 + 0.5).clamp(0.0, 1.0), 1.0)
        gain = (s <= -1.5) & core
    return e.float(), gain.to(torch.uint8)


def _grid(case):
    return case["nx"], case["ny"], case["nz"]


def _mid(grid):
    return tuple(v // 2 for v in grid)


def _noise_seed(seed):
    return (0x5EED0000 + int(seed) * 2654435761) & 0xFFFFFFFFFFFF


N_A = 5e24


def _levels(n):
    return np.geomspace(5e23, 2e25, n).tolist()


def _pulse(grid):
    return _mid(grid), 2, PULSE_LAM, 1.2e-15, 0.4e-15, 1e9


def _simulation(case, seed, faces):
    grid = _grid(case)
    eps, gain = _maps(grid, case["npml"], case.get("eps", "packed"), seed)
    sim = MBSimulation(grid, DX, DT, mb_default_params(npml=case["npml"]))
    sim.set_material(eps.cpu().numpy(), gain.cpu().numpy(), N_A if case.get("gain", True) else 0.0, PUMP)
    sim.set_seed(_noise_seed(seed))
    if faces:
        sim.add_face_probes(FACE_STRIDE, FACE_EVERY, N_FREQ, LAM_MIN, LAM_MAX)
    return sim


def prepare(case, seed):
    kind = case["kind"]
    if kind == "theory":
        rng = np.random.default_rng(seed)
        lo = gp.p_threshold(case["kappa"])
        return {"case": case, "p": np.sort(lo * 1.02 + (8.0 - lo * 1.02) * rng.random(case["pumps"]))}
    if kind == "ensemble":
        sides = [int(v) for v in case["sides"].split(",")]
        grids = [(n,) * 3 for n in sides for _ in range(case["levels"])]
        b = MBBatch(grids, DX, DT, mb_default_params(npml=8))
        for s, n in enumerate(sides):
            eps, gain = _maps((n,) * 3, 8, "packed", 100 * seed + s)
            eps, gain = eps.cpu().numpy(), gain.cpu().numpy()
            for q, n_a in enumerate(_levels(case["levels"])):
                m = s * case["levels"] + q
                b.set_instance(m, eps, gain, n_a, PUMP, _noise_seed(100 * seed + m))
                b.instances[m].add_point_probe(_mid(grids[m]), N_FREQ, LAM_MIN, LAM_MAX)
        b.autotune()
        return {"case": case, "batch": b}
    if kind == "design":
        grid = _grid(case)
        eps, gain = _maps(grid, case["npml"], case["eps"], seed)
        r = Realization(grid=grid, dx=DX, dt=DT, gain_mask=gain.cpu().numpy(), N_a=N_A,
                        seed=_noise_seed(seed), n_steps=case["steps"], ckpt_every=case["ckpt"],
                        params=mb_default_params(npml=case["npml"]), sources=[_pulse(grid)])
        return {"case": case, "eps": eps, "pump": torch.tensor(PUMP, dtype=torch.float64), "run": r}
    sim = _simulation(case, seed, case.get("faces", kind == "readout"))
    st = {"case": case, "sim": sim}
    grid = _grid(case)
    if case.get("point", kind == "readout"):
        st["probe"] = sim.add_point_probe(_mid(grid), N_FREQ, LAM_MIN, LAM_MAX)
    if case.get("plane"):
        st["plane"] = sim.add_plane_probe(grid[2] // 2, 1, 1, CW_LAM, CW_LAM)
    if case.get("source") == "pulse":
        sim.set_source(*_pulse(grid))
    elif case.get("source") == "cw":
        sim.set_source_cw(_mid(grid), 2, CW_LAM, 0.0, 4e-15, 1e9, 1 << 20)
    sim.autotune()
    if kind == "readout":
        sim.step(case["steps"])
        sim.synchronize()
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "theory":
        return gp.theory_curves(state["p"], case["kappa"], case["grid"])
    if kind == "ensemble":
        b = state["batch"]
        b.step(case["steps"])
        return {"spectra": np.array([m.probe_spectrum(0)[0] for m in b.instances]),
                "fields": [[m.field_device(f)[0] for f in MEMBER] for m in b.instances]}
    if kind == "design":
        eps = state["eps"].detach().requires_grad_()
        pump = state["pump"].detach().requires_grad_()
        J = emitted_energy(eps, pump, state["run"])
        J.backward()
        return {"J": J.detach(), "eps": eps.grad, "pump": pump.grad}
    sim = state["sim"]
    if kind == "adjoint":
        J, g, gp_ = sim.adjoint_energy_zface(case["steps"], case["ckpt"])
        return {"J": J, "eps": g, "pump": gp_}
    if kind == "readout":
        return {"U": sim.energy()[0],
                "faces": np.array([sim.face_spectrum(q)[0] for q in range(6)]),
                "spectrum": sim.probe_spectrum(state["probe"])[0],
                "section": sim.plane_energy_density(case["nz"] // 2)}
    sim.step(case["steps"])
    out = {f: sim.field_device(f) for f in (STATE if case["state"] and case["gain"] else EH)}
    if "probe" in state:
        out["spectrum"] = sim.probe_spectrum(state["probe"])
    if "plane" in state:
        out["map"] = sim.plane_mode_map(state["plane"], 0)
    return out


# -------------------------------------------------------------- work of a pass

def _step_work(grid, npml, gain):
    """(bytes, flops) of one time step: E and H read and written, the material
    byte; in gain cells (55 % of the interior) P, J, n1..n3 read and written;
    four CPML memories read and written per slab axis."""
    nx, ny, nz = grid
    n = float(nx * ny * nz)
    inner = math.prod(max(0, v - 2 * npml) / v for v in grid)
    g = 0.55 * inner if gain else 0.0
    f = sum(min(1.0, 2 * npml / v) for v in grid)
    return n * (49 + 72 * g + 32 * f), n * (42 + 130 * g + 24 * f)


def work(case):
    kind = case["kind"]
    if kind == "theory":   # about 10 Newton iterations of a tridiagonal solve
        return {"bytes": 48.0 * case["pumps"], "flops": 10 * 30.0 * case["pumps"] * case["grid"]}
    if kind == "ensemble":
        by = fl = 0.0
        for n in (int(v) for v in case["sides"].split(",")):
            b, f = _step_work((n,) * 3, 8, True)
            by += case["levels"] * (case["steps"] * b + 8.0 * len(MEMBER) * n ** 3)
            fl += case["levels"] * case["steps"] * f
        return {"bytes": by, "flops": fl}
    grid = _grid(case)
    n = float(math.prod(grid))
    if kind == "readout":   # E, H and the material byte once; the face sums once
        pts = 2 * sum(math.prod(-(-(v - 16) // FACE_STRIDE) for v in pair)
                      for pair in ((grid[1], grid[2]), (grid[0], grid[2]), (grid[0], grid[1])))
        return {"bytes": 25.0 * n + 24.0 * 4 * N_FREQ * pts, "flops": 14.0 * n + 8.0 * N_FREQ * pts}
    b, f = _step_work(grid, case["npml"], case.get("gain", True))
    if kind in ("adjoint", "design"):
        # a forward step, and a reverse step of as many adjoint fields that
        # reads the forward E, J and populations once more
        inner = math.prod(max(0, v - 2 * case["npml"]) / v for v in grid)
        by = case["steps"] * (2 * b + n * (12 + 24 * 0.55 * inner)) + 4 * n
        return {"bytes": by, "flops": case["steps"] * 3 * f}
    fields = len(STATE) if case["state"] and case["gain"] else len(EH)
    return {"bytes": case["steps"] * b + 8.0 * fields * n, "flops": case["steps"] * f}


# ----------------------------------------------------------- 64-bit reference

def _mulhilo(m, b):
    """(high, low) words of the 32 x 32 bit product m b (b an int64 tensor)."""
    p0, p1 = m * (b & 0xFFFF), m * (b >> 16)
    t = p1 + (p0 >> 16)
    return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)


def _normals(cells, step, seed):
    """Three standard normals per cell: Philox4x32-10 and Box–Muller."""
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    z = torch.zeros_like(cells)
    c = [cells, z + step, z, z]
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
        h0, l0 = _mulhilo(0xD2511F53, c[0])
        h1, l1 = _mulhilo(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
    u = [((v >> 9).double() + 0.5) * 2.0 ** -23 for v in c]
    r01, r23 = torch.sqrt(-2.0 * torch.log(u[0])), torch.sqrt(-2.0 * torch.log(u[2]))
    a, b = 2.0 * math.pi * u[1], 2.0 * math.pi * u[3]
    return r01 * torch.cos(a), r01 * torch.sin(a), r23 * torch.cos(b)


X, Y, Z = 2, 1, 0   # axes of [k, j, i]


def _fwd(F, ax):
    return torch.diff(F, dim=ax, append=torch.zeros_like(F.narrow(ax, 0, 1)))


def _bwd(F, ax):
    return torch.diff(F, dim=ax, prepend=torch.zeros_like(F.narrow(ax, 0, 1)))


class _Reference:
    """The scheme in 64 bits, in units E0 (E), E0/eta0 (H), eps0 E0 (P),
    eps0 E0/dt (J) and N_a (N).  A state is a list: E, H, P, J (3 each),
    N1..N3, six psi_H and six psi_E."""

    PAIRS = (("x", Y, "z"), ("x", Z, "y"), ("y", Z, "x"), ("y", X, "z"), ("z", X, "y"), ("z", Y, "x"))

    def __init__(self, grid, npml, eps, gain, n_a, seed, source=None):
        self.grid, self.npml, self.seed, self.source = grid, npml, seed, source
        lam0, dlam, t32, t21, t10 = 590e-9, 230e-9, 100e-15, 1e-9, 100e-15
        self.w0 = w0 = 2 * math.pi * C0 / lam0
        dw = 2 * math.pi * C0 * dlam / lam0 ** 2
        self.E0 = math.sqrt(HBAR * w0 * 1e24 / EPS0)
        self.eta0 = 1.0 / (EPS0 * C0)
        self.S = C0 * DT / DX
        self.n_a, self.eps = n_a, eps.double()
        self.gain = (gain != 0) if n_a > 0 else torch.zeros_like(gain, dtype=torch.bool)
        self.mask = self.gain.double()
        self.cells = torch.nonzero(self.gain.reshape(-1)).reshape(-1)
        a = 0.5 * dw * DT
        xi = 6 * math.pi * EPS0 * C0 ** 3 / (w0 ** 2 * t21)
        a_se = w0 * (QE * 0.1e-9) * math.sqrt(2 * dw)
        self.cJ1 = (1 - a) / (1 + a)
        self.cJE = DT * DT * xi * n_a / (EPS0 * (1 + a))
        self.cJP = (w0 * DT) ** 2 / (1 + a)
        self.cJN = DT * DT * a_se * math.sqrt(max(n_a, 0.0) / (DX ** 3 * DT)) / (EPS0 * self.E0 * (1 + a))
        self.rates = (t32, t21, t10)
        self.spop = EPS0 * self.E0 ** 2 / (HBAR * w0 * n_a) if n_a > 0 else 0.0
        dev = eps.device
        self.prof = {}
        for ax, n in ((X, grid[0]), (Y, grid[1]), (Z, grid[2])):
            shape = [1, 1, 1]
            shape[ax] = n
            self.prof[ax] = [tuple(torch.tensor(v, device=dev).reshape(shape) for v in self._cpml(n, h))
                             for h in (0.0, 0.5)]
            pos = (torch.arange(n, device=dev) > 0).double().reshape(shape)
            self.prof[ax].append(pos)
        self.n = 0
        self.pump(torch.tensor(PUMP, dtype=torch.float64))

    def _cpml(self, n, half):
        L = self.npml
        x = np.arange(n) + half
        depth = np.clip(np.maximum((L - x) / L, (x - (n - L)) / L), 0.0, 1.0)
        sigma = 0.8 * 4.0 / (self.eta0 * DX) * depth ** 3
        alpha = 2 * math.pi * EPS0 * 0.1 * C0 / 590e-9 * (1.0 - depth)
        b = np.where(depth > 0, np.exp(-(sigma + alpha) * DT / EPS0), 0.0)
        return b, np.where(depth > 0, sigma / (sigma + alpha) * (b - 1.0), 0.0)

    def pump(self, W):
        """Crank–Nicolson propagator (CPU tensors, differentiable in W)."""
        t32, t21, t10 = self.rates
        A = torch.zeros(4, 4, dtype=torch.float64)
        A[0, 1], A[1, 1], A[1, 2], A[2, 2] = 1 / t10, -1 / t10, 1 / t21, -1 / t21
        A[2, 3], A[3, 3] = 1 / t32, -1 / t32
        P = torch.zeros(4, 4, dtype=torch.float64)
        P[0, 0], P[3, 0] = -1.0, 1.0
        A = A + P * W
        I = torch.eye(4, dtype=torch.float64)
        L = I - 0.5 * DT * A
        M = torch.linalg.solve(L, I + 0.5 * DT * A)
        m = DT * torch.linalg.solve(L, torch.tensor([0.0, -1.0, 1.0, 0.0], dtype=torch.float64))
        dev = self.eps.device
        self.M, self.m = M.to(dev), (m / DT * self.spop).to(dev)

    def initial(self):
        z = lambda: torch.zeros_like(self.eps)   # noqa: E731
        return [z() for _ in range(27)]

    def wave(self, n):
        """Scaled source current of step n, or None."""
        if self.source is None:
            return None
        kind, cell, comp, lam, t0, tau, amp = self.source
        t = (n + 0.5) * DT - t0
        v = amp * DT / (EPS0 * self.E0) * math.sin(2 * math.pi * C0 / lam * t)
        env = math.exp(-(t / tau) ** 2)
        return cell, comp, v * (env if kind == "pulse" else 1.0 - env)

    def step(self, s, ie):
        """(the state after the step, E of before)."""
        E, H, P, J, N = s[0:3], s[3:6], s[6:9], s[9:12], s[12:15]
        comp = {"x": 0, "y": 1, "z": 2}
        sign = (1, -1, 1, -1, 1, -1)

        def curl(F, diff, psi, side):
            out, new = [0.0, 0.0, 0.0], []
            for (c, ax, o), sg, p in zip(self.PAIRS, sign, psi):
                d = diff(F[comp[o]], ax)
                b, cc = self.prof[ax][side]
                p = b * p + cc * d
                new.append(p)
                out[comp[c]] = out[comp[c]] + sg * (d + p)
            return out, new

        cE, psH = curl(E, _fwd, s[15:21], 1)
        H = [h - self.S * c for h, c in zip(H, cE)]
        if self.n_a > 0:
            amp = self.cJN * torch.sqrt(torch.relu(N[1]) + 1e-9) * self.mask
            zeta = _normals(self.cells, self.n, self.seed)
            dn = self.cJE * (N[0] - N[1])
            newJ = []
            for c in range(3):
                z = torch.zeros_like(self.eps).reshape(-1)
                z[self.cells] = zeta[c]
                newJ.append(self.cJ1 * J[c] + dn * E[c] - self.cJP * P[c] + amp * z.reshape(self.eps.shape))
            J = newJ
            P = [p + j for p, j in zip(P, J)]
        cH, psE = curl(H, _bwd, s[21:27], 0)
        cur = list(J)
        w = self.wave(self.n)
        if w is not None:
            (i, j, k), c, v = w
            cur[c] = cur[c].clone()
            cur[c][k, j, i] = cur[c][k, j, i] + v
        E1 = [e + ie * (self.S * c - q) for e, c, q in zip(E, cH, cur)]
        x, y, z = (self.prof[a][2] for a in (X, Y, Z))
        E1 = [E1[0] * y * z, E1[1] * x * z, E1[2] * x * y]
        if self.n_a > 0:
            sp = 0.5 * sum((a + b) * j for a, b, j in zip(E, E1, J))
            n0 = self.mask - N[0] - N[1] - N[2]
            pop = [n0] + list(N)
            N = [sum(self.M[r, q] * pop[q] for q in range(4)) + self.m[r] * sp for r in (1, 2, 3)]
        self.n += 1
        return E1 + H + list(P) + list(J) + list(N) + psH + psE, E

    def flux_z(self, s, E):
        """+z Poynting term of the step just taken, over the +z face."""
        L = self.npml
        nx, ny, nz = self.grid
        p, xs, ys = nz - L, slice(L, nx - L), slice(L, ny - L)
        at = lambda F, k: F[k, ys, xs]   # noqa: E731
        return 0.5 * ((at(E[0], p) + at(s[0], p)) * at(s[4], p - 1)
                      - (at(E[1], p) + at(s[1], p)) * at(s[3], p - 1)).sum()

    def scale(self, f):
        return {"E": self.E0, "H": self.E0 / self.eta0, "P": EPS0 * self.E0,
                "J": EPS0 * self.E0 / DT, "N": self.n_a}[f[0]]


LAMS = LAM_MIN + (LAM_MAX - LAM_MIN) * np.arange(N_FREQ) / (N_FREQ - 1)


def _reference(case, seed):
    grid = _grid(case)
    eps, gain = _maps(grid, case["npml"], case.get("eps", "packed"), seed)
    src = None
    if case.get("source") == "pulse" or case["kind"] == "design":
        src = ("pulse",) + _pulse(grid)
    elif case.get("source") == "cw":
        src = ("cw", _mid(grid), 2, CW_LAM, 0.0, 4e-15, 1e9)
    return _Reference(grid, case["npml"], eps, gain, N_A if case.get("gain", True) else 0.0,
                      _noise_seed(seed), src)


def _omega(lams):
    return torch.tensor(2 * math.pi * C0 / np.atleast_1d(lams), device="cuda")


def _phase(w, t):
    return torch.exp(1j * w * t)


def _advance(ref, steps, probes=None):
    """The state after `steps` steps; probes(state, n) after each."""
    s = ref.initial()
    ie = 1.0 / ref.eps
    for _ in range(steps):
        s, _ = ref.step(s, ie)
        if probes:
            probes(s, ref.n)
    return s


def _point_dft(ref, acc):
    i, j, k = _mid(ref.grid)
    w = _omega(LAMS)

    def add(s, n):
        e = torch.stack([s[c][k, j, i] for c in range(3)])
        acc.add_(e[:, None] * (_phase(w, n * DT) * (DT * ref.E0))[None])
    return add


def _spectrum(acc):
    return (acc.real.square() + acc.imag.square()).sum(0).cpu().numpy()


def _exact_step(case, seed):
    ref = _reference(case, seed)
    point = torch.zeros(3, N_FREQ, dtype=torch.complex128, device="cuda")
    plane = torch.zeros((3,) + tuple(ref.eps.shape[1:]), dtype=torch.complex128, device="cuda")
    add_point, wc, kz = _point_dft(ref, point), _omega(CW_LAM), case["nz"] // 2

    def probes(s, n):
        if case["point"]:
            add_point(s, n)
        if case["plane"]:
            ph = _phase(wc, n * DT)[0] * (DT * ref.E0)
            plane.add_(torch.stack([s[c][kz] for c in range(3)]) * ph)

    s = _advance(ref, case["steps"], probes)
    out = {f: (s[q], ref.scale(f)) for q, f in enumerate(STATE if case["state"] and case["gain"] else EH)}
    if case["point"]:
        out["spectrum"] = (_spectrum(point), LAMS)
    if case["plane"]:
        out["map"] = (plane.real.square() + plane.imag.square()).sum(0)
    return out


def _exact_ensemble(case, seed):
    spectra, fields = [], []
    for s, n in enumerate(int(v) for v in case["sides"].split(",")):
        eps, gain = _maps((n,) * 3, 8, "packed", 100 * seed + s)
        for q, n_a in enumerate(_levels(case["levels"])):
            ref = _Reference((n,) * 3, 8, eps, gain, n_a, _noise_seed(100 * seed + s * case["levels"] + q))
            acc = torch.zeros(3, N_FREQ, dtype=torch.complex128, device="cuda")
            st = _advance(ref, case["steps"], _point_dft(ref, acc))
            spectra.append(_spectrum(acc))
            fields.append([st[STATE.index(f)] for f in MEMBER])
    return {"spectra": np.array(spectra), "fields": fields}


def _exact_gradient(case, seed):
    ref = _reference(case, seed)
    seg = 20
    steps = case["steps"]
    starts, s = [], ref.initial()
    ie = 1.0 / ref.eps
    with torch.no_grad():
        for n in range(steps):
            if n % seg == 0:
                starts.append(s)
            s, _ = ref.step(s, ie)
    K = DT * ref.E0 * (ref.E0 / ref.eta0) * DX * DX
    lam = [torch.zeros_like(v) for v in s]
    g_eps, g_w, total = torch.zeros_like(ref.eps), 0.0, 0.0
    for q in range(len(starts) - 1, -1, -1):
        leaf = [v.detach().requires_grad_() for v in starts[q]]
        eps = ref.eps.detach().requires_grad_()
        W = torch.tensor(PUMP, dtype=torch.float64, requires_grad=True)
        ref.pump(W)
        ref.n, s, J = q * seg, leaf, 0.0
        for _ in range(min(seg, steps - q * seg)):
            s, E = ref.step(s, 1.0 / eps)
            J = J + ref.flux_z(s, E)
        obj = J + sum((a * b).sum() for a, b in zip(s, lam))
        got = torch.autograd.grad(obj, leaf + [eps, W], allow_unused=True)
        lam = [torch.zeros_like(a) if g is None else g for a, g in zip(leaf, got)]
        g_eps += got[-2]
        g_w += float(got[-1])
        total += float(J.detach())
    return {"J": K * total, "eps": K * g_eps, "pump": K * g_w}


def _exact_readout(case, seed):
    ref = _reference(case, seed)
    L, (nx, ny, nz) = 8, ref.grid
    w = _omega(LAMS)
    point = torch.zeros(3, N_FREQ, dtype=torch.complex128, device="cuda")
    add_point, acc = _point_dft(ref, point), [None] * 6
    sl = [slice(L, n - L, FACE_STRIDE) for n in (nx, ny, nz)]
    wt = FACE_EVERY * DT

    def face(s, q):
        ax, p = q // 2, ((L, nx - L), (L, ny - L), (L, nz - L))[q // 2][q % 2]
        a, b = ((1, 2), (2, 0), (0, 1))[ax]

        def cut(F, at):
            ix = [sl[2], sl[1], sl[0]]
            ix[2 - ax] = at
            return F[tuple(ix)].reshape(-1)
        return [cut(s[a], p), cut(s[b], p), cut(s[3 + a], p - 1), cut(s[3 + b], p - 1)]

    def probes(s, n):
        add_point(s, n)
        if n % FACE_EVERY == 0:
            pe, ph = _phase(w, n * DT) * wt * ref.E0, _phase(w, (n - 0.5) * DT) * wt * ref.E0 / ref.eta0
            for q in range(6):
                v = [F[:, None] * p[None] for F, p in zip(face(s, q), (pe, pe, ph, ph))]
                acc[q] = v if acc[q] is None else [x + y for x, y in zip(acc[q], v)]

    s = _advance(ref, case["steps"], probes)
    faces = []
    for q in range(6):
        Ea, Eb, Ha, Hb = acc[q]
        S = (Ea * Hb.conj() - Eb * Ha.conj()).real.sum(0) * (FACE_STRIDE * DX) ** 2
        faces.append(((1 if q % 2 else -1) * S).cpu().numpy())
    e2, h2 = sum(v * v for v in s[0:3]), sum(v * v for v in s[3:6])
    u = 0.5 * EPS0 * ref.E0 ** 2 * (ref.eps * e2 + h2)
    return {"U": float(u.sum()) * DX ** 3, "faces": np.array(faces), "spectrum": _spectrum(point),
            "section": u[nz // 2]}


def _exact_theory(case, seed):
    p = prepare(case, seed)["p"]
    kappa, n = case["kappa"], case["grid"]
    E = (p - 1.0) / (kappa * np.sqrt(p))
    L = np.sqrt(E) + 8.0
    h = 2.0 * L / (n + 1)
    t2 = (-L + h * (np.arange(n)[:, None] + 1)) ** 2
    phi = np.maximum(np.sqrt(np.maximum(E - t2, 0.0)),
                     2.0 ** 0.25 * np.sqrt(E - 1.0) * np.exp(-0.5 * t2))
    off = -1.0 / h ** 2
    last = np.inf
    for _ in range(60):   # Newton with a tridiagonal elimination per step
        f = t2 * phi + phi ** 3 - E * phi - 2.0 * off * phi
        f[1:] += off * phi[:-1]
        f[:-1] += off * phi[1:]
        d = -2.0 * off + t2 + 3.0 * phi * phi - E
        for i in range(1, n):
            w = off / d[i - 1]
            d[i] -= w * off
            f[i] -= w * f[i - 1]
        f[n - 1] /= d[n - 1]
        for i in range(n - 2, -1, -1):
            f[i] = (f[i] - off * f[i + 1]) / d[i]
        phi -= f
        size = np.abs(f).max()
        if size < 1e-13 or (size < 1e-9 and size >= last):
            break
        last = size
    step = np.diff(np.concatenate([np.zeros((1, len(E))), phi, np.zeros((1, len(E)))]), axis=0)
    wphi = np.sqrt((step ** 2).sum(0) / h ** 2 / (phi ** 2).sum(0)) / (2 * math.pi)
    th = 1.0 + 0.5 * kappa ** 2 + 0.5 * kappa * math.sqrt(4.0 + kappa ** 2)
    return {"p": p, "E": E, "W_tg": wphi * math.sqrt(kappa) / p ** 0.25,
            "S_p": (h * phi.sum(0)) ** 2 / (4 * math.pi ** 2), "p_th": th}


def exact(case, seed):
    kind = case["kind"]
    if kind == "theory":
        return _exact_theory(case, seed)
    if kind == "ensemble":
        return _exact_ensemble(case, seed)
    if kind in ("adjoint", "design"):
        if case["steps"] * math.prod(_grid(case)) > 8e8:
            return None
        return _exact_gradient(case, seed)
    return _exact_readout(case, seed) if kind == "readout" else _exact_step(case, seed)
