"""Performance cases: calls that programs make on a lattice, through the package's public entry points.

A case is one of
  run        Lattice.step(n), then what the program reads back: the macroscopic fields (a monitored
             or coupled run) or the populations (a checkpoint, a coupled population solver);
  adjoint    restart from given fields, Lattice.adjoint over T steps, Lattice.adjoint_state: one
             evaluation of an objective with its gradient and the sensitivity of the initial state;
  fragments  Lattice.fragments of a broken-up state.

Every state is a developed one (red blob, droplet or jet column in a disturbed ambient), made on
the GPU from the seed.  exact() is the same run in double precision, written here in plain torch
from the method's equations (arXiv:1804.08923, Section II and IV.A); the gradients come from
torch's reverse mode through it.
"""
import math

import numpy as np
import torch

import paper_1804_08923_gb300 as lb

STORAGE = {"fp32": lb.STORE_FP32, "fp16": lb.STORE_FP16, "fp16_fit": lb.STORE_FP16_FIT}


# ------------------------------------------------------------------------------- cases
def _run(name, nx, ny, nz, scene, steps, out, storage="fp32"):
    return {"name": name, "kind": "run", "nx": nx, "ny": ny, "nz": nz, "scene": scene, "steps": steps, "out": out,
            "storage": storage}


def listed():
    return [
        # a small droplet run watched at every step: the smallest call, launches and host work count
        _run("monitor_32", 32, 32, 32, "blob", 1, "fields"),
        # the static droplet of Section III as it is run: 200 steps in one call on a lattice that
        # fits the L2 cache many times over
        _run("droplet_32", 32, 32, 32, "droplet", 200, "populations"),
        # a mixture in a box of odd extents with gravity, a few steps between looks at it
        _run("box_ragged", 45, 37, 53, "gravity", 10, "fields"),
        # a million-node jet coupled to another program, one step per call with all fields read
        _run("jet_64_coupled", 64, 64, 256, "jet", 1, "fields"),
        # the liquid-liquid jet (96 x 96 x 384) between two outputs
        _run("jet_96", 96, 96, 384, "jet", 50, "populations"),
        # the same jet in the two half-precision storages, the second on a larger lattice
        _run("jet_96_fp16", 96, 96, 384, "jet", 50, "populations", "fp16"),
        _run("jet_128_fp16_fit", 128, 128, 512, "jet", 20, "populations", "fp16_fit"),
        # the paper's own melt jet (free-slip side walls, gravity) at half its resolution
        _run("melt_jet_120", 120, 120, 600, "melt", 20, "populations"),
        # the high-Reynolds-number jet with gravity, 67 million nodes: a production-size run
        _run("jet_256", 256, 256, 1024, "fast", 20, "populations"),
        # sensitivities of the interface area of a million-node jet
        {"name": "adjoint_64", "kind": "adjoint", "nx": 64, "ny": 64, "nz": 256, "scene": "jet", "steps": 50,
         "objective": "area"},
        # sensitivities of the penetration length of a small walled jet with gravity, odd extents
        {"name": "adjoint_walls", "kind": "adjoint", "nx": 41, "ny": 38, "nz": 90, "scene": "melt", "steps": 30,
         "objective": "penetration"},
        # fragment statistics of a broken-up state on the 96 x 96 x 384 lattice
        {"name": "fragments_96", "kind": "fragments", "nx": 96, "ny": 96, "nz": 384, "connectivity": 6, "storage": "fp32"},
    ]


MAX_NODE_STEPS = 256 * 256 * 1024 * 20 // 4  # a drawn run costs at most a quarter of the largest listed one


def _extent(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run"] * 7 + ["adjoint"] * 2 + ["fragments"])
    if kind == "run":
        scene = rng.choice(["blob", "droplet", "gravity", "jet", "jet", "melt", "fast"])
        n = _extent(rng, 24, 192)
        nx, ny = n, max(20, n + rng.randint(-n // 5, n // 5))
        nz = n + rng.randint(0, 9) if scene in ("blob", "droplet", "gravity") else int(n * rng.uniform(2.5, 5.0))
        steps = min(_extent(rng, 1, 200), max(1, MAX_NODE_STEPS // (nx * ny * nz)))
        out = "fields" if steps <= 10 and scene != "droplet" and rng.random() < 0.6 else "populations"
        storage = rng.choice(["fp32", "fp32", "fp32", "fp16", "fp16_fit"])
        if storage != "fp32":
            out = "populations"
        case = _run("", nx, ny, nz, scene, steps, out, storage)
        del case["name"]
        return case
    if kind == "adjoint":
        n = _extent(rng, 28, 72)
        return {"kind": "adjoint", "nx": n, "ny": n + rng.randint(-4, 4), "nz": int(n * rng.uniform(2.0, 4.0)),
                "scene": rng.choice(["jet", "melt"]), "steps": rng.randint(8, 50),
                "objective": rng.choice(["area", "penetration"])}
    n = _extent(rng, 32, 128)
    nz = int(n * rng.uniform(1.0, 4.0))
    return {"kind": "fragments", "nx": n, "ny": n + rng.randint(-5, 5), "nz": nz, "connectivity": rng.choice([6, 26]), "storage": rng.choice(["fp32", "fp16", "fp16_fit"])}


# --------------------------------------------------------------------------- parameters
def _jet(D, u, gamma, eta, Re, We, Fr=None):
    """Lattice parameters of a jet from its dimensionless groups (Eqs. (1)-(5)), rho_r0 = 1."""
    nu = u * D / Re
    g = 0.0 if Fr is None else u * u / (Fr * D)
    return dict(rho_r0=1.0, rho_b0=1.0 / gamma, nu_r=nu, nu_b=nu / eta, sigma=u * u * D / We, g=(0.0, 0.0, g), u_in=u,
                d_in=float(D))


# regulariser of |grad phi| in the differentiated runs: with the default 1e-6 the sensitivities of
# single nodes in the interface's tails depend on the rounding of the state
ADJOINT_EPS = 1e-4


def _setup(case):
    """(params, bc) of a case: those of its scene, with the adjoint's regulariser."""
    p, bc = _scene(case)
    return (dict(p, eps_grad=ADJOINT_EPS) if case["kind"] == "adjoint" else p), bc


def _scene(case):
    """The jets keep D = nx / 6 as the 96 x 96 x 384 jet does, the melt jet D = nx / 8 as in the paper."""
    scene, nx = case.get("scene", "blob"), case["nx"]
    if scene == "droplet":
        return dict(rho_r0=1.0, rho_b0=1.0, nu_r=1 / 6, nu_b=1 / 6, sigma=0.01), (0, 0, 0, 0)
    if scene == "blob":
        return dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.05, nu_b=0.1, sigma=0.005), (0, 0, 0, 0)
    if scene == "gravity":
        return dict(rho_r0=1.0, rho_b0=0.5, nu_r=0.02, nu_b=0.08, sigma=0.003, g=(0.0, 0.0, 1e-5)), (0, 0, 0, 0)
    if scene == "jet":
        p, bc = _jet(nx / 6, 0.05, 1.5, 1.0, 2000, 100), (lb.BC_INLET, lb.BC_CONVECTIVE, 0, 0)
        return dict(p, noise_amp=0.01), bc
    if scene == "fast":
        p, bc = _jet(nx / 8, 0.04, 2.0, 1.0, 1e5, 1000, 100), (lb.BC_INLET, lb.BC_CONVECTIVE, 0, 0)
        return dict(p, noise_amp=0.005), bc
    p = _jet(nx / 8, 0.05, 8.3, 0.54, 6.1e4, 230, 64)  # melt: UT Case 1
    return p, (lb.BC_INLET, lb.BC_CONVECTIVE, lb.BC_FREESLIP, lb.BC_FREESLIP)


def _noise_seed(seed):
    return (int(seed) * 2654435761 + 12345) % (1 << 62)


def _fields(case, seed):
    """Developed initial state (rho_r, rho_b, u), float32 on the GPU, of the case's scene."""
    p, bc = _setup(case)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(int(seed))
    z = torch.arange(nz, device="cuda", dtype=torch.float32).view(nz, 1, 1)
    y = torch.arange(ny, device="cuda", dtype=torch.float32).view(1, ny, 1)
    x = torch.arange(nx, device="cuda", dtype=torch.float32).view(1, 1, nx)

    def wave(amp):  # a smooth disturbance, products of low modes that fit the lattice
        out = 0.0
        for _ in range(2):
            k, ph = rng.integers(1, 3, 3), rng.uniform(0, 2 * math.pi, 3)
            out = out + amp / 2 * (torch.cos(2 * math.pi * k[0] / nx * x + ph[0]) *
                                   torch.cos(2 * math.pi * k[1] / ny * y + ph[1]) *
                                   torch.cos(2 * math.pi * k[2] / nz * z + ph[2]))
        return out

    dx, dy = x - (nx - 1) / 2, y - (ny - 1) / 2
    u_in = p.get("u_in", 0.0)
    if u_in:  # a jet column from the inlet with a wavy surface and a round tip
        R, L = p["d_in"] / 2, nz * rng.uniform(0.45, 0.65)
        r = torch.sqrt(dx * dx + dy * dy + torch.clamp(z - L, min=0.0) ** 2)
        wavy = 1 + 0.12 * torch.sin(2 * math.pi * rng.integers(2, 5) / nz * z + rng.uniform(0, 6.28))
        s = torch.tanh((2 / 3) * (r - R * wavy))
    else:
        R = min(nx, ny, nz) * rng.uniform(0.24, 0.28)
        d0 = rng.uniform(-1, 1, 3)
        r = torch.sqrt((dx - d0[0]) ** 2 + (dy - d0[1]) ** 2 + (z - (nz - 1) / 2 - d0[2]) ** 2)
        s = torch.tanh(0.5 * (r - R) if case.get("scene") == "droplet" else (2 / 3) * (r - R * (1 + wave(0.15))))
    still = case.get("scene") == "droplet"
    dens = 1.0 if still else 1 + wave(0.005)
    rr, rb = 0.5 * p["rho_r0"] * (1 - s) * dens, 0.5 * p["rho_b0"] * (1 + s) * dens
    u = torch.zeros((3, nz, ny, nx), device="cuda", dtype=torch.float32)
    if not still:
        for d in range(3):
            u[d] = wave(0.03)
        if u_in:
            u[2] += u_in * 0.5 * (1 - s)
    return rr.contiguous(), rb.contiguous(), u


def _broken_up(case, seed):
    """Broken-up state, |phi| = 0.9: a wavy red core along z, the remains of the jet, and red balls of
    radius 1.5 to 3.5 about it, one near the middle of every 12-node cell that the core leaves free
    (so that every state has the same number of fragments)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    rng = np.random.default_rng(int(seed))
    core = min(nx, ny) / 8
    cells = np.stack(np.meshgrid(*(np.arange(n // 12) * 12 + 5.5 for n in (nz, ny, nx)), indexing="ij"), -1).reshape(-1, 3)
    axis = np.array([(ny - 1) / 2, (nx - 1) / 2])
    cells = cells[np.hypot(*(cells[:, 1:] - axis).T) > core + 8]
    n = len(cells)
    c = torch.tensor(cells + rng.uniform(-1, 1, (n, 3)), device="cuda").view(n, 3, 1)
    r = torch.tensor(rng.uniform(1.5, 3.5, n), device="cuda").view(n, 1, 1, 1)
    at = torch.floor(c).long() + torch.arange(-5, 6, device="cuda").view(1, 1, 11)  # (n, axis, 11)
    d2 = (at - c) ** 2
    b, i, j, l = (d2[:, 0, :, None, None] + d2[:, 1, None, :, None] + d2[:, 2, None, None, :] < r * r).nonzero(as_tuple=True)
    z = torch.arange(nz, device="cuda").view(nz, 1, 1)
    y = torch.arange(ny, device="cuda").view(1, ny, 1)
    x = torch.arange(nx, device="cuda").view(1, 1, nx)
    wavy = core * (0.9 + 0.1 * torch.sin(2 * math.pi * rng.integers(2, 6) / nz * z + rng.uniform(0, 6.28)))
    red = (y - axis[0]) ** 2 + (x - axis[1]) ** 2 < wavy * wavy
    red[at[b, 0, i], at[b, 1, j], at[b, 2, l]] = True
    phi = torch.where(red, 0.9, -0.9)
    rr, rb = 0.5 * (1 + phi), 0.5 * (1 - phi) / 1.5
    return rr.float().contiguous(), rb.float().contiguous(), torch.zeros((3, nz, ny, nx), device="cuda")


# --------------------------------------------------------------------------------- runs
def _objective(case):
    return (case["objective"], (1e-3,) if case["objective"] == "area" else (4.0,))


def prepare(case, seed):
    grid = (case["nx"], case["ny"], case["nz"])
    if case["kind"] == "fragments":
        p = dict(rho_r0=1.0, rho_b0=1 / 1.5, nu_r=4e-4, nu_b=4e-4, sigma=4e-4, storage=STORAGE[case["storage"]])
        lat = lb.Lattice(grid, p)
        lat.init_fields(*_broken_up(case, seed))
        return {"case": case, "lat": lat}
    p, bc = _setup(case)
    lat = lb.Lattice(grid, dict(p, seed=_noise_seed(seed), storage=STORAGE[case.get("storage", "fp32")]), bc=bc)
    fields = _fields(case, seed)
    lat.init_fields(*fields)
    state = {"case": case, "lat": lat}
    if case["kind"] == "adjoint":
        state["fields"] = fields
    return state


def run(state):
    case, lat = state["case"], state["lat"]
    if case["kind"] == "fragments":
        return lat.fragments(case["connectivity"], exclude_inlet=False)
    if case["kind"] == "adjoint":
        lat.init_fields(*state["fields"])
        J, grad = lat.adjoint(case["steps"], *_objective(case))
        # the optimiser holds its parameters in single precision
        return {"J": J, "grad": torch.tensor(grad, dtype=torch.float32), "state": lat.adjoint_state(device=True)}
    lat.step(case["steps"])
    return lat.populations() if case["out"] == "populations" else lat.fields()


# Floating-point operations of one step and of its transpose per node, in round numbers: the
# moments of the 54 populations, two gradients, the collision and 54 new populations.
FLOPS_STEP, FLOPS_ADJOINT = 800, 1600


def work(case):
    nodes = case["nx"] * case["ny"] * case["nz"]
    pops = 216 if case.get("storage", "fp32") == "fp32" else 112
    if case["kind"] == "fragments":  # the state in, one label's worth of marks out
        return {"bytes": nodes * (pops + 4), "flops": nodes * 54}
    if case["kind"] == "adjoint":  # five fields in, the sensitivity of the state out
        return {"bytes": nodes * (20 + 216), "flops": nodes * case["steps"] * (FLOPS_STEP + FLOPS_ADJOINT)}
    out = 216 if case["out"] == "populations" else 28
    # the state in, the new state out and the outputs
    return {"bytes": nodes * (2 * pops + out), "flops": nodes * case["steps"] * FLOPS_STEP}


# ------------------------------------------------------- the same in double precision
# directions of Eq. (8), as (cx, cy, cz); after the rest direction they come in opposite pairs
C = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
     (-1, 1, 0), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
     (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1)]
W = [(8 / 27, 2 / 27, 1 / 54, 1 / 216)[sum(abs(v) for v in c)] for c in C]
OMA_B = 19 / 27  # 1 - alpha_b


def _dir(c):
    return C.index(tuple(c))


def _dot(c, v):
    out = 0.0
    for k in range(3):
        if c[k]:
            out = out + c[k] * v[k]
    return out


def _varphi(i, oma):
    q = sum(abs(v) for v in C[i])
    return 1 - oma if q == 0 else oma * (0, 2 / 19, 1 / 38, 1 / 152)[q]


def _poly(cu, uu):
    return 3 * cu + 4.5 * cu * cu - 1.5 * uu + 4.5 * cu ** 3 - 4.5 * cu * uu


def _splitmix(v):
    m = (1 << 64) - 1
    v = (v + 0x9E3779B97F4A7C15) & m
    v = ((v ^ (v >> 30)) * 0xBF58476D1CE4E5B9) & m
    v = ((v ^ (v >> 27)) * 0x94D049BB133111EB) & m
    return v ^ (v >> 31)


class Exact:
    """The lattice in double precision: populations f[k][i] as (2, nz, ny, nx) tensors by direction."""

    def __init__(self, case, seed, theta=None):
        self.p, self.bc = _setup(case)
        self.n = (case["nz"], case["ny"], case["nx"])
        self.seed = _noise_seed(seed)
        p = self.p
        self.u_in, self.sigma, self.nu_r, self.nu_b = (
            (p.get("u_in", 0.0), p["sigma"], p["nu_r"], p["nu_b"]) if theta is None else (theta[0], theta[1], theta[2], theta[3]))
        self.fourier = None if theta is None else theta[4:]
        self.oma_r = OMA_B * p["rho_b0"] / p["rho_r0"]
        self.g = p.get("g", (0.0, 0.0, 0.0))
        ny, nx = case["ny"], case["nx"]
        self.rx = (torch.arange(nx, device="cuda", dtype=torch.float64) - (nx - 1) / 2).view(1, nx).expand(ny, nx)
        self.ry = (torch.arange(ny, device="cuda", dtype=torch.float64) - (ny - 1) / 2).view(ny, 1).expand(ny, nx)
        d = p.get("d_in", 0.0)
        self.disc = (4 * (self.rx ** 2 + self.ry ** 2) < d * d) if self.bc[0] == lb.BC_INLET else None

    def start(self, rr, rb, u):
        rr, rb, u = rr.double(), rb.double(), u.double()
        uu = (u * u).sum(0)
        out = []
        for i in range(27):
            pw = W[i] * _poly(_dot(C[i], u), uu)
            out.append(torch.stack([rr * (_varphi(i, self.oma_r) + pw), rb * (_varphi(i, OMA_B) + pw)]))
        return out

    # -- inlet
    def inlet(self, step):
        """Populations leaving the ghost plane z = -1 inside the disc, by direction with cz = +1."""
        ny, nx = self.n[1:]
        r = torch.sqrt(self.rx ** 2 + self.ry ** 2)
        safe = torch.where(r > 0, r, torch.ones_like(r))
        c1, s1 = torch.where(r > 0, self.rx / safe, torch.ones_like(r)), torch.where(r > 0, self.ry / safe, torch.zeros_like(r))
        amp = self.p.get("noise_amp", 0.0)
        xi = np.zeros((ny, nx))
        if amp:
            for yy, xx in self.disc.nonzero().tolist():
                xi[yy, xx] = (_splitmix(self.seed ^ _splitmix((step * ny + yy) * nx + xx)) >> 40) / 8388608.0 - 1.0
        a = self.u_in * amp * torch.tensor(xi, device="cuda") * (r > 0)
        prof = 1.0
        if self.fourier is not None:
            c, s = torch.ones_like(r), torch.zeros_like(r)
            for m in range(8):
                c, s = c * c1 - s * s1, s * c1 + c * s1
                prof = prof + self.fourier[2 * m] * c + self.fourier[2 * m + 1] * s
        v = (a * c1, a * s1, self.u_in * prof * torch.ones_like(r))
        uu = v[0] ** 2 + v[1] ** 2 + v[2] ** 2
        out = {}
        for i in range(27):
            if C[i][2] == 1:
                red = self.p["rho_r0"] * (_varphi(i, self.oma_r) + W[i] * _poly(_dot(C[i], v), uu))
                out[i] = torch.stack([red, torch.zeros_like(red)])
        return out

    # -- one step: f, hist -> f, hist
    def sides(self, get, i):
        """Direction i's plane(s) with one ghost layer on each side in x and y (get(i) without)."""
        cx, cy, cz = C[i]

        def pad_x(j):
            a = get(j)
            if self.bc[2] == lb.BC_FREESLIP:
                b = get(_dir((-C[j][0], C[j][1], C[j][2])))
                return torch.cat([b[..., :1], a, b[..., -1:]], -1)
            return torch.cat([a[..., -1:], a, a[..., :1]], -1)

        a = pad_x(i)
        if self.bc[3] == lb.BC_FREESLIP:
            b = pad_x(_dir((cx, -cy, cz)))
            return torch.cat([b[..., :1, :], a, b[..., -1:, :]], -2)
        return torch.cat([a[..., -1:, :], a, a[..., :1, :]], -2)

    def stream(self, f, step, hist):
        nz, ny, nx = self.n
        lo, hi = self.bc[0], self.bc[1]
        inflow = self.inlet(step) if lo == lb.BC_INLET else None
        out = []
        for i in range(27):
            cx, cy, cz = C[i]

            def column(j):
                """Direction j with the ghost planes its pull can need."""
                if C[j][2] == 0:
                    return f[j]
                k = _dir((C[j][0], C[j][1], -C[j][2]))
                if C[j][2] == 1:
                    below = f[j][:, -1:] if lo == lb.BC_PERIODIC else f[k][:, :1]
                    if inflow is not None:
                        below = torch.where(self.disc, inflow[j].unsqueeze(1), below)
                    return torch.cat([below, f[j][:, :-1]], 1)
                above = f[j][:, :1] if lo == lb.BC_PERIODIC else f[k][:, -1:]
                return torch.cat([f[j][:, 1:], above], 1)

            a = self.sides(column, i) if (cx or cy) else column(i)
            if cx or cy:
                a = a[:, :, 1 - cy:1 - cy + ny, 1 - cx:1 - cx + nx]
            out.append(a)
        if hi == lb.BC_CONVECTIVE:
            fm = torch.stack([a[:, -2] for a in out])  # 27, 2, ny, nx
            tot = fm.sum(1)
            rho, jz = tot.sum(0), sum(C[i][2] * tot[i] for i in range(27) if C[i][2])
            lam = torch.clamp((jz + 0.5 * (rho - self.p["rho_b0"]) * self.g[2]) / rho, 0.0, 1.0)
            hist = (hist + lam * fm) / (1 + lam)
            out = [torch.cat([a[:, :-1], hist[i].unsqueeze(1)], 1) for i, a in enumerate(out)]
        return out, hist

    def gradient(self, chi, ghost):
        def pad(a, axis, wrap):
            n = a.shape[axis]
            lo, hi = a.narrow(axis, 0, 1), a.narrow(axis, n - 1, 1)
            return torch.cat([hi, a, lo] if wrap else [lo, a, hi], axis)

        if self.bc[0] == lb.BC_PERIODIC:
            a = pad(chi, 0, True)
        else:
            below = chi[:1]
            if self.disc is not None:
                below = torch.where(self.disc, torch.full_like(below, ghost), below)
            a = torch.cat([below, chi, chi[-1:]], 0)
        a = pad(pad(a, 1, self.bc[3] != lb.BC_FREESLIP), 2, self.bc[2] != lb.BC_FREESLIP)

        def mean(v, axis):
            n = v.shape[axis] - 2
            return (v.narrow(axis, 0, n) + 4 * v.narrow(axis, 1, n) + v.narrow(axis, 2, n)) / 6

        def diff(v, axis):
            n = v.shape[axis] - 2
            return (v.narrow(axis, 2, n) - v.narrow(axis, 0, n)) / 2

        return diff(mean(mean(a, 0), 1), 2), diff(mean(mean(a, 0), 2), 1), diff(mean(mean(a, 1), 2), 0)

    def phi_of(self, rr, rb):
        a, b = rr / self.p["rho_r0"], rb / self.p["rho_b0"]
        return (a - b) / (a + b)

    def collide(self, f):
        p = self.p
        tot = [a[0] + a[1] for a in f]
        rr, rb = sum(a[0] for a in f), sum(a[1] for a in f)
        rho = rr + rb
        phi = self.phi_of(rr, rb)
        gp, gr = self.gradient(phi, 1.0), self.gradient(rho, p["rho_r0"])
        F = [(rho - p["rho_b0"]) * v for v in self.g]
        u = [(sum(C[i][k] * tot[i] for i in range(27) if C[i][k]) + 0.5 * F[k]) / rho for k in range(3)]
        uu = sum(v * v for v in u)
        hp, hm = 0.5 * (1 + phi), 0.5 * (1 - phi)
        oma = hp * self.oma_r + hm * OMA_B
        nu = 1 / (hp / self.nu_r + hm / self.nu_b)
        tau = 3 * nu + 0.5
        A = 2.25 * self.sigma / tau
        ugr = sum(a * b for a, b in zip(u, gr))
        uF = sum(a * b for a, b in zip(u, F))
        cs2 = 9 / 19 * oma
        # second central moments of f - f^e + F'/2, relaxed: bulk rate 1, shear rate 1/tau
        Q = {}
        for a in range(3):
            for b in range(a, 3):
                raw = sum(C[i][a] * C[i][b] * tot[i] for i in range(27) if C[i][a] * C[i][b])
                q = raw - rho * u[a] * u[b] - nu * (u[a] * gr[b] + u[b] * gr[a]) + 0.5 * (u[a] * F[b] + u[b] * F[a])
                Q[a, b] = q - rho * cs2 - nu * ugr if a == b else q
        tr = (Q[0, 0] + Q[1, 1] + Q[2, 2]) / 3
        K = {ab: (1 - 1 / tau) * (q - tr if ab[0] == ab[1] else q) for ab, q in Q.items()}
        g2 = sum(v * v for v in gp)
        gm = torch.sqrt(g2 + p.get("eps_grad", 1e-6) ** 2)  # |grad phi|, regularised
        # values at c = -1, 0, 1 of the inverse central-moment transform, orders 0, 1, 2
        G = [{-1: (0.5 * (v * v - v), v - 0.5, 0.5), 0: (1 - v * v, -2 * v, -1.0), 1: (0.5 * (v * v + v), v + 0.5, 0.5)}
             for v in u]
        out = []
        for i in range(27):
            c = C[i]
            q = sum(abs(v) for v in c)
            cu, cg, cF, cp = _dot(c, u), _dot(c, gr), _dot(c, F), _dot(c, gp)
            Phi = -3 * nu * ugr if q == 0 else (0, 16, 4, 1)[q] / 24 * nu * cu * cg
            s = rho * (_varphi(i, oma) + W[i] * _poly(cu, uu)) + Phi
            s = s + 0.5 * W[i] * (3 * (cF - uF) + 9 * cu * cF)
            for (a, b), k in K.items():
                o = [0, 0, 0]
                o[a] += 1
                o[b] += 1
                s = s + k * G[0][c[0]][o[0]] * G[1][c[1]][o[1]] * G[2][c[2]][o[2]]
            s = s + A / gm * (W[i] * cp * cp - (-10 / 27 if q == 0 else W[i]) * g2)
            seg = 0.0 if q == 0 else p.get("beta", 0.7) * rr * rb / rho * _varphi(i, oma) * cp / (gm * math.sqrt(q))
            out.append(torch.stack([rr / rho * s + seg, rb / rho * s - seg]))
        return out

    def step(self, f, hist, step):
        f, hist = self.stream(f, step, hist)
        return self.collide(f), hist

    def macroscopic(self, f):
        rr, rb = sum(a[0] for a in f), sum(a[1] for a in f)
        rho, phi = rr + rb, self.phi_of(rr, rb)
        u = [(sum(C[i][k] * (f[i][0] + f[i][1]) for i in range(27) if C[i][k]) - 0.5 * (rho - self.p["rho_b0"]) * self.g[k]) / rho
             for k in range(3)]
        oma = 0.5 * (1 + phi) * self.oma_r + 0.5 * (1 - phi) * OMA_B
        return {"rho_r": rr, "rho_b": rb, "phi": phi, "ux": u[0], "uy": u[1], "uz": u[2], "p": rho * 9 / 19 * oma}

    def objective(self, f, kind, args):
        nz = self.n[0]
        phi = self.phi_of(sum(a[0] for a in f), sum(a[1] for a in f))
        if kind == "area":
            g = self.gradient(phi, 1.0)
            return torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2 + args[0] ** 2)[1:nz - 1].sum()
        z = torch.arange(nz, device="cuda", dtype=torch.float64).view(nz, 1, 1)
        return nz - 1 + args[0] * torch.log((((1 + phi) / 2) ** 2 * torch.exp((z - (nz - 1)) / args[0])).sum())


def _exact_adjoint(case, seed):
    p, _ = _setup(case)
    theta = torch.tensor([p["u_in"], p["sigma"], p["nu_r"], p["nu_b"]] + [0.0] * 16, device="cuda", dtype=torch.float64,
                         requires_grad=True)
    start = torch.stack(Exact(case, seed).start(*_fields(case, seed))).requires_grad_()
    states = [(start.detach(), start.detach()[:, :, -1])]
    with torch.no_grad():
        for t in range(case["steps"]):
            f, h = Exact(case, seed, theta).step(list(states[-1][0]), states[-1][1], t)
            states.append((torch.stack(f), h))
    f = states[-1][0].requires_grad_()
    J = Exact(case, seed, theta).objective(list(f), *_objective(case))
    lf, = torch.autograd.grad(J, f)
    lh, gt = torch.zeros_like(states[-1][1]), torch.zeros_like(theta)
    for t in reversed(range(case["steps"])):
        f, h = states[t][0].requires_grad_(), states[t][1].requires_grad_()
        fo, ho = Exact(case, seed, theta).step(list(f), h, t)
        lf, lh, g = torch.autograd.grad([torch.stack(fo), ho], [f, h, theta], [lf, lh])
        gt += g
        states[t + 1] = None
    return {"J": float(J.detach()), "grad": gt.cpu(), "state": lf.transpose(0, 1).contiguous()}


def exact(case, seed):
    nodes = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "fragments" or nodes * case["steps"] > 4e8:
        return None
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        e = Exact(case, seed)
        f = e.start(*_fields(case, seed))
        hist = torch.stack([a[:, -1] for a in f])
        for t in range(case["steps"]):
            f, hist = e.step(f, hist, t)
        if case["out"] == "fields":
            return e.macroscopic(f)
        return torch.stack(f, 1)
