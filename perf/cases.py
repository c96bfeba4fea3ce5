"""The measured cases: what a user of this library has it do, through its
public entry points, and the same results in 64 bits by plain torch.

A case is one whole call sequence of a user's program: initial fields in, a
number of time steps, the diagnostics and the fields out (``march``), the same
from and to host arrays (``host``), a batch of cavities advanced and read out
(``batch``), or a Nusselt number and its gradients (``adjoint``).  Fields come
back in the precision the lattice stores (an FP32 lattice's T is an FP32
number, an FP16 one's an FP16 number of the dimensionless field), and whole.
"""
import math

import numpy as np
import torch

from paper_1505_02976_gb300 import lbm
from paper_1505_02976_gb300 import workloads as W
from paper_1505_02976_gb300.autograd import wall_nusselt

FLOPS_PER_NODE = 346  # floating-point operations of one node update (multiply-add = 2)
FIELDS = ("p", "ux", "uy", "T")


def listed():
    return [
        # the paper's own grid (Sec. 4.2): FP64, advanced between two checks of the steady criterion;
        # a run is tens of thousands of these tiny steps, so latency and launches count
        dict(name="cavity32_f64", kind="march", flow="cavity", nx=32, ny=32, precision="f64", steps=200,
             Ra=1e3, Da=1e-2, eps=0.6),
        # the table runs' grids are N + 1 nodes wide, odd and small, and check the criterion every 100 steps
        dict(name="cavity201_f32", kind="march", flow="clear", nx=201, ny=201, precision="f32", steps=100, Ra=1e5),
        # the headline lattice
        dict(name="cavity2048_f32", kind="march", flow="cavity", nx=2048, ny=2048, precision="f32", steps=100,
             Ra=1e6, Da=1e-4, eps=0.4),
        # the same lattice on the moment state
        dict(name="moments2048_f32", kind="march", flow="cavity", nx=2048, ny=2048, precision="f32", steps=100,
             Ra=1e6, Da=1e-4, eps=0.4, state="moments"),
        # the largest: 67M nodes in FP16 storage
        dict(name="cavity8192_f16", kind="march", flow="cavity", nx=8192, ny=8192, precision="f16", steps=20,
             Ra=1e5, Da=1e-3, eps=0.6, Ma=0.0156),
        # throughput of FP64 lattices, ragged size
        dict(name="cavity700x517_f64", kind="march", flow="cavity", nx=700, ny=517, precision="f64", steps=50,
             Ra=1e5, Da=1e-3, eps=0.5),
        # mixed-convection channel (Sec. 4.1): periodic in x, moving permeable walls, a driving profile
        dict(name="channel1024x513_f32", kind="march", flow="channel", nx=1024, ny=513, precision="f32", steps=100,
             Da=1e-2, eps=0.6),
        # heterogeneous medium: a porosity field, relaxation times off 1, a heat source; ragged size
        dict(name="porous1000x777_f32", kind="march", flow="porous", nx=1000, ny=777, precision="f32", steps=100,
             Ra=1e5, Da=1e-3, eps=0.5, tau_f=0.8, tau_T=1.15),
        # a sweep of independent cavities of uneven size, replayed from a CUDA graph, then read out
        dict(name="batch128_f32", kind="batch", count=128, shapes=20150511, precision="f32", steps=500, mode="graph"),
        # gradient of the hot-wall Nusselt number with respect to a porosity field (training)
        dict(name="adjoint256_f32", kind="adjoint", n=256, ny=256, precision="f32", steps=256, Ra=1e5),
        # the same in FP64 on a small ragged grid (gradient checks, small inverse problems)
        dict(name="adjoint65x49_f64", kind="adjoint", n=65, ny=49, precision="f64", steps=100, Ra=1e4),
        # fields from and to page-locked host arrays, all diagnostics: heat-generating cavity (Sec. 4.3, Table 3)
        dict(name="host1025_f32", kind="host", flow="heated", nx=1025, ny=1025, precision="f32", steps=50,
             Ra=1e6, Da=1e-2, eps=0.4),
    ]


def _size(rng, lo, hi):
    """A whole number in [lo, hi], spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("cavity_f32", "cavity_f32", "cavity_f64", "cavity_f16", "moments", "channel", "porous",
                       "batch", "adjoint", "host"))
    Ra, Da, eps = 10.0 ** rng.uniform(3.0, 6.0), 10.0 ** rng.uniform(-4.0, -2.0), rng.uniform(0.3, 0.9)
    if kind == "batch":
        return dict(kind="batch", count=_size(rng, 3, 100), shapes=rng.randrange(1 << 30), precision="f32",
                    steps=_size(rng, 100, 500), mode=rng.choice(("graph", "fused")))
    if kind == "adjoint":
        # 64 bits on the smaller grids, as a gradient check runs it
        f64 = rng.random() < 0.5
        n, ny = _size(rng, 24, 100 if f64 else 320), _size(rng, 24, 100 if f64 else 320)
        return dict(kind="adjoint", n=n, ny=ny, precision="f64" if f64 else "f32", steps=_size(rng, 40, 200),
                    Ra=10.0 ** rng.uniform(4.0, 5.5))
    base = dict(kind="march", Ra=Ra, Da=Da, eps=eps, precision="f32")
    aspect = rng.uniform(0.5, 2.0)

    def sides(lo, hi):
        n = _size(rng, lo, hi)
        nx, ny = max(8, int(n * math.sqrt(aspect))), max(8, int(n / math.sqrt(aspect)))
        # the Mach number that keeps the lattice viscosity at most 0.25, 0.1 (the paper's) where it can be
        return dict(nx=nx, ny=ny, Ma=min(0.1, 0.43 * math.sqrt(Ra) / nx))

    if kind == "cavity_f32":
        return {**base, "flow": "cavity", **sides(24, 4000), "steps": _size(rng, 20, 100)}
    if kind == "cavity_f64":
        return {**base, "flow": "cavity", "precision": "f64", **sides(16, 1200), "steps": _size(rng, 20, 100)}
    if kind == "cavity_f16":
        return {**base, "flow": "cavity", "precision": "f16", **sides(512, 5600), "steps": _size(rng, 10, 20)}
    if kind == "moments":
        return {**base, "flow": "cavity", "state": "moments", **sides(64, 3000), "steps": _size(rng, 20, 100)}
    if kind == "channel":
        return {**base, "flow": "channel", **sides(32, 1500), "steps": _size(rng, 20, 100)}
    if kind == "porous":
        off = rng.random() < 0.5
        return {**base, "flow": "porous", **sides(32, 1500), "steps": _size(rng, 20, 100),
                "tau_f": rng.uniform(0.75, 1.2) if off else 1.0, "tau_T": rng.uniform(0.75, 1.2) if off else 1.0}
    return {**base, "kind": "host", "flow": "heated", **sides(64, 1200), "steps": _size(rng, 20, 100)}


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _problem(case):
    flow, nx, ny = case["flow"], case["nx"], case["ny"]
    kw = {k: case[k] for k in ("Ma", "tau_f", "tau_T") if k in case}
    if flow == "clear":
        return W.clear_fluid_cavity(nx, case["Ra"], ny=ny, **kw)
    if flow == "channel":
        u0 = 0.02  # speed of the moving top wall; both walls are permeable (normal velocity v0)
        return W.problem(nx=nx, ny=ny, bc=("periodic", "periodic", "dirichlet", "dirichlet"), eps=case["eps"],
                         Da=case["Da"], nu=0.05, forchheimer=0, L=float(ny - 1), T_bc=(1.0, 0.0, 0.0, 1.0),
                         gbeta=u0 * u0 / ny, alpha_e=0.05,
                         u_bc=((0.0, 0.0), (0.0, 0.0), (0.0, 0.25 * u0), (u0, 0.25 * u0)))
    if flow == "heated":  # every wall at T_c, internal heat source
        return W.cavity(nx, case["Ra"], case["Da"], case["eps"], ny=ny, bc=("dirichlet",) * 4,
                        T_bc=(0.0, 0.0, 0.0, 0.0), Q=1e-4, T0=0.0, **kw)
    if flow == "porous":
        return W.cavity(nx, case["Ra"], case["Da"], case["eps"], ny=ny, Q=1e-5, **kw)
    return W.cavity(nx, case["Ra"], case["Da"], case["eps"], ny=ny, **kw)


def _smooth(g, ny, nx, modes=4):
    """A smooth random field of order 1, zero on the boundary: a few sine modes."""
    a = torch.randn(modes, modes, generator=g, device="cuda", dtype=torch.float64)
    k = torch.arange(1, modes + 1, device="cuda", dtype=torch.float64)
    y = torch.linspace(0.0, math.pi, ny, device="cuda", dtype=torch.float64)
    x = torch.linspace(0.0, math.pi, nx, device="cuda", dtype=torch.float64)
    return torch.sin(y[:, None] * k) @ (a / (k[:, None] + k)) @ torch.sin(k[:, None] * x)


def _fields(p, seed):
    """A developed state: the conduction profile with smooth disturbances, a smooth circulation."""
    g, nx, ny = _gen(seed), p["nx"], p["ny"]
    U = p["Ma"] / math.sqrt(3.0) if p["bc"][0] != "periodic" else 0.02
    T = (0.5 + 0.2 * _smooth(g, ny, nx)).contiguous()
    return T, (0.3 * U * _smooth(g, ny, nx)).contiguous(), (0.3 * U * _smooth(g, ny, nx)).contiguous()


def _porosity(seed, ny, nx, corr=16.0):
    """Gaussian random field of correlation length `corr` cells mapped into [0.3, 0.9]."""
    z = torch.randn(ny, nx, generator=_gen(seed + 77), device="cuda", dtype=torch.float64)
    ky = 2.0 * math.pi * torch.fft.fftfreq(ny, device="cuda", dtype=torch.float64)
    kx = 2.0 * math.pi * torch.fft.fftfreq(nx, device="cuda", dtype=torch.float64)
    z = torch.fft.ifft2(torch.fft.fft2(z) * torch.exp(-0.5 * corr ** 2 * (ky[:, None] ** 2 + kx ** 2))).real
    z = (z - z.mean()) / z.std()
    return (0.3 + 0.3 * (1.0 + torch.erf(z / math.sqrt(2.0)))).contiguous()


def _batch_problems(case, seed):
    """Sizes belong to the case, the groups (Ra, Da, eps) to the seed."""
    shape = np.random.Generator(np.random.PCG64(case["shapes"]))
    rng = np.random.Generator(np.random.PCG64(seed))
    sizes = (64, 96, 128, 192, 256, 384, 512)
    return [W.cavity(int(sizes[shape.integers(len(sizes))]), 10.0 ** rng.uniform(3.0, 6.0),
                     10.0 ** rng.uniform(-6.0, -2.0), rng.uniform(0.3, 0.9)) for _ in range(case["count"])]


def _adjoint_inputs(case, seed):
    p = W.cavity(case["n"], case["Ra"], 1e-3, 0.6, ny=case["ny"])
    dtype = torch.float64 if case["precision"] == "f64" else torch.float32
    eps = _porosity(seed, case["ny"], case["n"]).to(dtype)
    walls = torch.tensor([1.0, 0.0], dtype=dtype)
    walls += 0.05 * torch.rand(2, generator=torch.Generator().manual_seed(int(seed)), dtype=dtype)
    return p, eps, walls


def _force_profile(p):
    """Driving profile a_y(y) of the channel: balances the Darcy drag on v0."""
    y = np.linspace(0.0, 1.0, p["ny"])
    drag = p["nu"] / (p["Da"] * p["L"] ** 2) * p["u_bc"][2][1]
    return drag - p["gbeta"] * (y - 0.5)


def prepare(case, seed):
    if case["kind"] == "adjoint":
        p, eps, walls = _adjoint_inputs(case, seed)
        return dict(case=case, p=p, eps=eps.requires_grad_(), walls=walls.requires_grad_())
    if case["kind"] == "batch":
        return dict(case=case, b=lbm.Batch(_batch_problems(case, seed), case["precision"]))
    p = _problem(case)
    s = dict(case=case, p=p, fields=_fields(p, seed), eps=None)
    s["lat"] = lbm.Lattice(p, case["precision"], state=case.get("state", "populations"))
    if case["flow"] == "channel":
        s["lat"].set_force_profile(_force_profile(p))
    if case["flow"] == "porous":
        s["eps"] = _porosity(seed, p["ny"], p["nx"])
    if case["kind"] == "host":
        # page-locked, so that the upload runs at the link's rate
        s["pinned"] = [f.cpu().pin_memory() for f in s["fields"]]
        s["fields"] = [t.numpy() for t in s["pinned"]]
    else:
        s["out"] = {k: torch.empty(p["ny"], p["nx"], dtype=torch.float64, device="cuda") for k in FIELDS}
    return s


# -------------------------------------------------------------------- runs

def _stored(case, p, name, v):
    """A field in the precision of the lattice's storage; FP16 lattices give the dimensionless field."""
    if case["precision"] == "f64":
        return v
    if case["precision"] == "f32":
        return v.float() if isinstance(v, torch.Tensor) else np.asarray(v, np.float32)
    U = p["Ma"] / math.sqrt(3.0)
    return (v * {"p": 1.0 / U ** 2, "ux": 1.0 / U, "uy": 1.0 / U, "T": 1.0}[name]).half()


def run(state):
    case = state["case"]
    return {"march": _run_march, "host": _run_host, "batch": _run_batch, "adjoint": _run_adjoint}[case["kind"]](state)


def _run_march(s):
    case, p, lat = s["case"], s["p"], s["lat"]
    lat.set_fields(*s["fields"], eps_field=s["eps"])
    lat.step(case["steps"])
    res_u, res_T = lat.residual()
    side = "N" if p["bc"][0] == "periodic" else "W"
    mean, local = lat.nusselt(side)
    lat.moments_device(s["out"])
    out = {k: _stored(case, p, k, v) for k, v in s["out"].items()}
    if case["precision"] == "f16":
        return {**out, "nu": np.asarray(local, np.float16)}
    kind = np.float64 if case["precision"] == "f64" else np.float32
    return {**out, "nu": local.astype(kind), "mean": kind(mean), "residual": np.asarray([res_u, res_T], kind)}


def _run_host(s):
    case, p, lat = s["case"], s["p"], s["lat"]
    lat.set_fields(*s["fields"])
    lat.step(case["steps"])
    mean, local = lat.nusselt("W")
    psi, _ = lat.stream_function()
    m = lat.moments()
    out = {k: _stored(case, p, k, v) for k, v in m.items()}
    return {**out, "psi": psi.astype(np.float32), "nu": local.astype(np.float32), "mean": np.float32(mean)}


def _run_batch(s):
    case, b = s["case"], s["b"]
    b.set_fields(-1)
    b.step(case["steps"], case["mode"])
    b.sync()
    out = {k: np.empty(b.cells, np.float32) for k in FIELDS}
    at = 0
    for c in range(b.n):
        m = b.moments(c)
        n = m["T"].size
        for k in FIELDS:
            out[k][at:at + n] = m[k].reshape(-1)
        at += n
    return {**out, "nu": b.nusselt("W").astype(np.float32)}


def _run_adjoint(s):
    case = s["case"]
    loss = wall_nusselt(s["eps"], s["walls"], s["p"], case["steps"], precision=case["precision"])
    d_eps, d_walls = torch.autograd.grad(loss, (s["eps"], s["walls"]))
    return {"loss": loss.detach().to(d_eps.dtype), "d_eps": d_eps, "d_walls": d_walls}


def work(case):
    """Bytes: the initial fields read once and the outputs written once.  Operations: every node of every
    step; a gradient costs the forward steps and at least three times as much backwards."""
    width = {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
    if case["kind"] == "adjoint":
        n = case["n"] * case["ny"]
        return {"bytes": 2 * n * width, "flops": 4.0 * n * case["steps"] * FLOPS_PER_NODE}
    if case["kind"] == "batch":
        n = sum(p["nx"] * p["ny"] for p in _batch_problems(case, 0))
        return {"bytes": 4 * n * width, "flops": float(n) * case["steps"] * FLOPS_PER_NODE}
    n = case["nx"] * case["ny"]
    inputs = 4 if case["flow"] == "porous" else 3
    outputs = 5 if case["kind"] == "host" else 4
    return {"bytes": n * (8 * inputs + width * outputs), "flops": float(n) * case["steps"] * FLOPS_PER_NODE}


# ------------------------------------------------------- the same in 64 bits

class _Model:
    """The paper's evolution equations on [B, ny, nx] lattices in float64 torch (B > 1: cavities of one
    size with groups of their own), populations [9, B, ny, nx]; every operation is differentiable."""

    CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
    CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)

    def __init__(self, problems, eps=None, ay=None, walls=None):
        p = problems[0]
        self.p, self.nx, self.ny = p, p["nx"], p["ny"]

        def col(values):
            return torch.tensor([float(v) for v in values], dtype=torch.float64, device="cuda").reshape(-1, 1, 1)

        d = [self._derived(q) for q in problems]
        self.w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64, device="cuda")
        self.L, self.dT, self.T0 = d[0]["L"], d[0]["dT"], d[0]["T0"]
        for k in ("gbeta", "nu", "A", "B", "K", "Q"):
            setattr(self, k, col([q[k] for q in d]))
        self.rho0, self.sigma = p["rho0"], p["sigma"]
        self.tf, self.tT = p["tau_f"], p["tau_T"]
        ref = col([q["eps"] for q in problems])
        self.eps = ref if eps is None else eps.reshape(1, self.ny, self.nx)
        K = self.K
        if eps is not None:  # Kozeny-Carman permeability of each node
            K = K * (self.eps ** 3 / (1 - self.eps) ** 2) / (ref ** 3 / (1 - ref) ** 2)
        F = 1.75 / torch.sqrt(150 * self.eps ** 3) if p["forchheimer"] else torch.zeros_like(self.eps)
        none = torch.zeros_like(self.eps)
        self.drag0 = none if p["da_infinite"] else self.eps * self.nu / K
        self.drag1 = none if p["da_infinite"] else self.eps * F / torch.sqrt(K)
        self.ay = p["ay"] if ay is None else p["ay"] + torch.tensor(ay, device="cuda").reshape(1, -1, 1)
        self._walls(p, walls)

    @staticmethod
    def _derived(p):
        own = lambda v, other: other if math.isnan(v) else v  # noqa: E731
        L = own(p["L"], float(p["nx"] - 1))
        dT, U = p["Th"] - p["Tc"], p["Ma"] / math.sqrt(3.0)
        nu = own(p["nu"], U * L * math.sqrt(p["Pr"] / p["Ra"]))
        alpha = own(p["alpha_e"], nu / p["Pr"])
        return dict(L=L, dT=dT, T0=own(p["T0"], 0.5 * (p["Th"] + p["Tc"])), nu=nu,
                    gbeta=own(p["gbeta"], U * U / (dT * L) if dT else 0.0),
                    A=own(p["A"], p["tau_f"] - 0.5 - 3 * p["J"] * nu), B=own(p["B"], p["tau_T"] - 0.5 - 3 * alpha / p["sigma"]),
                    K=own(p["K"], p["Da"] * L * L), Q=own(p["Q"], p["Ra_I"] * alpha * dT / (p["Ra"] * L * L)))

    def _walls(self, p, walls):
        """For every wall node: its x_f and x_ff, the side that gives T (or none) and u."""
        nx, ny = self.nx, self.ny
        on = [b != "periodic" for b in p["bc"]]
        T_bc = list(p["T_bc"])
        node, f, ff, T_side, u, fix = [], [], [], [], [], []
        border = {(x, y) for x in range(nx) for y in (0, ny - 1)} | {(x, y) for x in (0, nx - 1) for y in range(ny)}
        for x, y in sorted(border):
            dx = 1 if on[0] and x == 0 else -1 if on[1] and x == nx - 1 else 0
            dy = 1 if on[2] and y == 0 else -1 if on[3] and y == ny - 1 else 0
            if not dx and not dy:
                continue
            xs, ys = (0 if dx > 0 else 1) if dx else -1, (2 if dy > 0 else 3) if dy else -1
            node.append(y * nx + x)
            f.append((y + dy) * nx + x + dx)
            ff.append((y + 2 * dy) * nx + x + 2 * dx)
            T_side.append(next((s for s in (xs, ys) if s >= 0 and p["bc"][s] == "dirichlet"), -1))
            u.append(p["u_bc"][xs if xs >= 0 else ys])
            fix.append((1.0 if xs >= 0 else 0.0, 1.0 if ys >= 0 else 0.0))
        dev = dict(device="cuda")
        self.at, self.xf, self.xff = (torch.tensor(v, dtype=torch.long, **dev) for v in (node, f, ff))
        side = torch.tensor(T_side, **dev)
        self.given = side >= 0
        temps = torch.tensor(T_bc, dtype=torch.float64, **dev)
        if walls is not None:
            temps = torch.cat([walls.to(temps), temps[2:]])
        self.T_wall = temps[side.clamp(min=0)]
        self.u_wall = torch.tensor(u, dtype=torch.float64, **dev)
        self.keep = 1.0 - torch.tensor(fix, dtype=torch.float64, **dev)

    def _dirs(self):
        c = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda").reshape(9, 1, 1, 1)  # noqa: E731
        return c(self.CX), c(self.CY), self.w.reshape(9, 1, 1, 1)

    def equilibria(self, m, sources=True):
        """f^eq (without the rest population, which no moment reads), g^eq and the source terms F_i, P_i + Q_i."""
        cx, cy, w = self._dirs()
        e, rho0, sg = self.eps, self.rho0, self.sigma
        T, p, ux, uy = m["T"], m["p"], m["ux"], m["uy"]
        uu = ux * ux + uy * uy
        cu = cx * ux + cy * uy
        quad = (4.5 * cu * cu - 1.5 * uu) / e
        tr = cx * cx * m["Sxx"] + 2 * cx * cy * m["Sxy"] + cy * cy * m["Syy"] - (m["Sxx"] + m["Syy"]) / 3
        fe = w * (3 * e * p + rho0 * (3 * cu + quad) + 1.5 * rho0 * self.A * tr)
        vp = w.clone()
        vp[0] = -5 / 9
        ge = w * (sg * T + T * (3 * cu + quad) + sg * self.B * (cx * m["gx"] + cy * m["gy"])) + vp * 3 * T * e * p / rho0
        if not sources:
            return fe, ge, 0.0, 0.0
        cF = cx * m["Fx"] + cy * m["Fy"]
        uF = ux * m["Fx"] + uy * m["Fy"]
        Fi = w * rho0 * (1 - 0.5 / self.tf) * (3 * cF + (9 * cu * cF - 3 * uF) / e)
        Wx, Wy = T * m["Fx"] + e * p * m["gx"] / rho0, T * m["Fy"] + e * p * m["gy"] / rho0
        ug = ux * m["gx"] + uy * m["gy"]
        PQ = w * (1 - 0.5 / self.tT) * (3 * (cx * Wx + cy * Wy) + 3 * (1 / e - 1 / sg) * cu * ug + (1 + 3 * cu / sg) * self.Q)
        return fe, ge, Fi, PQ

    def start(self, T, ux, uy):
        z = torch.zeros_like(T + self.eps + self.Q)
        m = dict(T=T + z, ux=ux + z, uy=uy + z, p=z, Sxx=z, Sxy=z, Syy=z, gx=z, gy=z)
        fe, ge, _, _ = self.equilibria(m, sources=False)
        return fe, ge

    def stream(self, f, g):
        pull = lambda h: torch.stack([torch.roll(h[i], (self.CY[i], self.CX[i]), (-2, -1)) for i in range(9)])  # noqa: E731
        return pull(f), pull(g)

    def force(self, m):
        speed = m["ux"] ** 2 + m["uy"] ** 2
        speed = torch.sqrt(torch.where(speed > 0, speed, torch.ones_like(speed))) * (speed > 0)
        drag = self.drag0 + self.drag1 * speed
        Gy = self.gbeta * (m["T"] - self.T0) + self.ay
        m["Fx"] = self.eps * self.p["ax"] - drag * m["ux"]
        m["Fy"] = self.eps * Gy - drag * m["uy"]

    def moments(self, f, g):
        """Moments of every node from its pulled populations, wall nodes as in Sec. 3.4: (as pulled, with walls)."""
        cx, cy, _ = self._dirs()
        e, rho0, sg = self.eps, self.rho0, self.sigma
        m = {}
        T = m["T"] = (g.sum(0) + 0.5 * self.Q) / sg
        f = torch.cat([torch.zeros_like(f[:1]), f[1:]])
        Gy = self.gbeta * (T - self.T0) + self.ay
        vx = (cx * f).sum(0) / rho0 + 0.5 * e * self.p["ax"]
        vy = (cy * f).sum(0) / rho0 + 0.5 * e * Gy
        c0 = 0.5 * (1 + 0.5 * self.drag0)
        vv = vx * vx + vy * vy
        v = torch.sqrt(torch.where(vv > 0, vv, torch.ones_like(vv))) * (vv > 0)
        den = c0 + torch.sqrt(c0 * c0 + 0.5 * self.drag1 * v)
        ux, uy = m["ux"], m["uy"] = vx / den, vy / den
        self.force(m)
        Fx, Fy = m["Fx"], m["Fy"]
        uu, uF = ux * ux + uy * uy, ux * Fx + uy * Fy
        F0 = -(4 / 3) * rho0 * (1 - 0.5 / self.tf) * uF / e
        p = m["p"] = 3 / (5 * e) * (f.sum(0) + self.tf * F0 - rho0 * (2 / 3) * uu / e)
        D = 1 / (rho0 * (self.A - self.tf) / 3)
        r = rho0 / e
        m["Sxx"] = ((cx * cx * f).sum(0) - e * p - r * ux * ux + r * ux * Fx) * D
        m["Syy"] = ((cy * cy * f).sum(0) - e * p - r * uy * uy + r * uy * Fy) * D
        m["Sxy"] = ((cx * cy * f).sum(0) - r * ux * uy + 0.5 * r * (ux * Fy + uy * Fx)) * D
        Nx = (cx * g).sum(0) - T * ux + 0.5 * (T * Fx + ux * self.Q / sg)
        Ny = (cy * g).sum(0) - T * uy + 0.5 * (T * Fy + uy * self.Q / sg)
        b = 0.5 * (1 / e - 1 / sg)
        a = -e * p / (2 * rho0) + sg * (self.B - self.tT) / 3
        # (a I - b u u^T) grad T = N, by Cramer's rule
        mxx, mxy, myy = a - b * ux * ux, -b * ux * uy, a - b * uy * uy
        det = mxx * myy - mxy * mxy
        m["gx"] = (myy * Nx - mxy * Ny) / det
        m["gy"] = (mxx * Ny - mxy * Nx) / det
        if not len(self.at):
            return m, m
        flat = {k: v.expand(T.shape).flatten(1) for k, v in m.items()}
        wall = {k: flat[k][:, self.xf] for k in ("p", "Sxx", "Sxy", "Syy", "gx", "gy", "T")}
        n = wall["T"].shape
        free = (4 * wall["T"] - flat["T"][:, self.xff]) / 3
        wall["T"] = torch.where(self.given, self.T_wall, free)
        for k, j in (("gx", 0), ("gy", 1)):
            wall[k] = torch.where(self.given, wall[k], wall[k] * self.keep[:, j])
        wall["ux"], wall["uy"] = self.u_wall[:, 0].expand(n), self.u_wall[:, 1].expand(n)
        out = {k: flat[k].index_copy(1, self.at, v).reshape(T.shape) for k, v in wall.items()}
        self.force(out)
        return m, out

    def step(self, f, g):
        f, g = self.stream(f, g)
        m, b = self.moments(f, g)
        fb, gb, Fi, PQ = self.equilibria(b)
        f2, g2 = fb + Fi, gb + PQ
        if self.tf != 1.0 or self.tT != 1.0:  # the part of the distance to equilibrium that is left
            fe, ge, _, _ = self.equilibria(m)
            df, dg = (1 - 1 / self.tf) * (f - fe), (1 - 1 / self.tT) * (g - ge)
            if len(self.at):
                flat = lambda v: v.flatten(2).index_copy(2, self.at, v.flatten(2)[:, :, self.xf]).reshape(v.shape)  # noqa: E731
                df, dg = flat(df), flat(dg)
            f2, g2 = f2 + df, g2 + dg
        return f2, g2

    def now(self, f, g):
        return self.moments(*self.stream(f, g))[1]

    def nusselt(self, T, side):
        t = {"W": (T[..., :, 0], T[..., :, 1], T[..., :, 2]), "N": (T[..., -1, :], T[..., -2, :], T[..., -3, :])}[side]
        inward = (-3 * t[0] + 4 * t[1] - t[2]) / 2
        local = -self.L * (inward if side == "W" else -inward) / self.dT
        ends = 0.5 * (local[..., 0] + local[..., -1])
        return (local.sum(-1) - ends) / (local.shape[-1] - 1), local


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        return _exact_batch(case, seed) if case["kind"] == "batch" else _exact_march(case, seed)


def _exact_march(case, seed):
    if case["nx"] * case["ny"] * case["steps"] > 2e9:
        return None
    p = _problem(case)
    eps = _porosity(seed, p["ny"], p["nx"]) if case["flow"] == "porous" else None
    M = _Model([p], eps, _force_profile(p) if case["flow"] == "channel" else None)
    f, g = M.start(*(v[None] for v in _fields(p, seed)))
    first = M.now(f, g)
    for _ in range(case["steps"]):
        f, g = M.step(f, g)
    m = M.now(f, g)
    mean, local = M.nusselt(m["T"][0], "N" if p["bc"][0] == "periodic" else "W")
    out = {k: m[k][0] for k in FIELDS}
    if case["precision"] == "f16":
        U = p["Ma"] / math.sqrt(3.0)
        return {"p": out["p"] / U ** 2, "ux": out["ux"] / U, "uy": out["uy"] / U, "T": out["T"], "nu": local}
    if case["kind"] == "host":
        u = out["ux"]
        psi = torch.cat([torch.zeros_like(u[:1]), torch.cumsum(0.5 * (u[1:] + u[:-1]), 0)])
        return {**out, "psi": psi, "nu": local, "mean": mean}
    du = torch.sqrt((m["ux"] - first["ux"]) ** 2 + (m["uy"] - first["uy"]) ** 2).sum()
    res = torch.stack([du / torch.sqrt(m["ux"] ** 2 + m["uy"] ** 2).sum(),
                       (m["T"] - first["T"]).abs().sum() / m["T"].abs().sum()])
    return {**out, "nu": local, "mean": mean, "residual": res}


def _exact_batch(case, seed):
    problems = _batch_problems(case, seed)
    found = [None] * len(problems)
    for n in sorted({p["nx"] for p in problems}):
        which = [c for c, p in enumerate(problems) if p["nx"] == n]
        M = _Model([problems[c] for c in which])
        z = torch.zeros(len(which), n, n, dtype=torch.float64, device="cuda")
        f, g = M.start(z + 0.5, z, z)
        for _ in range(case["steps"]):
            f, g = M.step(f, g)
        m = M.now(f, g)
        nu = M.nusselt(m["T"], "W")[0]
        for j, c in enumerate(which):
            found[c] = ({k: m[k][j].reshape(-1) for k in FIELDS}, nu[j])
    return {**{k: torch.cat([v[0][k] for v in found]) for k in FIELDS}, "nu": torch.stack([v[1] for v in found])}


def _exact_adjoint(case, seed):
    if case["steps"] > 300:
        return None
    p, eps, walls = _adjoint_inputs(case, seed)
    eps, walls = eps.double().requires_grad_(), walls.double().requires_grad_()
    with torch.no_grad():
        M = _Model([p], eps, walls=walls)
        z = torch.zeros(1, case["ny"], case["n"], dtype=torch.float64, device="cuda")
        kept = [M.start(z + 0.5, z, z)]
        for _ in range(case["steps"]):
            kept.append(M.step(*kept[-1]))
    # the derivative of each step by itself, from the last one back
    f, g = (v.detach().requires_grad_() for v in kept.pop())
    M = _Model([p], eps, walls=walls)
    loss = M.nusselt(M.now(f, g)["T"][0], "W")[0]
    df, dg, de, dw = torch.autograd.grad(loss, (f, g, eps, walls), allow_unused=True)
    total = [torch.zeros_like(eps) if de is None else de, torch.zeros_like(walls) if dw is None else dw]
    z = torch.zeros_like(f)
    df = z if df is None else df
    while kept:
        f, g = (v.detach().requires_grad_() for v in kept.pop())
        M = _Model([p], eps, walls=walls)
        f2, g2 = M.step(f, g)
        df, dg, de, dw = torch.autograd.grad((f2, g2), (f, g, eps, walls), (df, dg))
        total[0] += de
        total[1] += dw
    # the initial state is given: its own dependence on the porosity is not part of the gradient
    return {"loss": loss.detach(), "d_eps": total[0], "d_walls": total[1]}
