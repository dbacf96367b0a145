"""Workloads of the projection library, each one pass through its public entry
points: inputs drawn on the GPU from a seed, the plan (or batch) a program
keeps, the call, and the same result in plain FP64 torch.

A case is one of
  project     ppe.Plan.project: Eqs. (32)-(34) of one grid (the solver's step);
  constraint  divergence_constraint (Eq. (31)) then project, as a time step that
              forms S and rho from its phase-wise quantities does;
  steps       rhs, solve, correct called one by one (a solver with its own
              scheduling, or one that needs f);
  unsplit     project_unsplit, the iterative baseline (Eqs. (29)-(30));
  batch       many uneven grids in one launch (ensembles, parameter studies).
Fields follow the package's synthetic recipe (tanh density layer around a
wavy interface, N(0, 1) predicted velocities and old pressures, S in the
interface band), on boxes of any side lengths.
"""
import math

import numpy as np
import torch

from paper_2103_01874_gb300 import fields, ppe

TWO_PI = 2.0 * math.pi
# side lengths the library takes (2^a 3^b); nx even
SIZES = [n for n in range(16, 513) if 2 ** 9 * 3 ** 6 % n == 0]


def _case(name, kind, nx, ny, nz, prec, **kw):
    c = dict(name=name, kind=kind, nx=nx, ny=ny, nz=nz, prec=prec, lx=TWO_PI, ly=TWO_PI, lz=TWO_PI,
             face="arithmetic", top="wall", modes=8, width=6.0, rho_g=60.0, given_rho0=False)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest workload: one small single-mode interface, called every step; launches and latency count
        _case("project fp32 32", "project", 32, 32, 32, "fp32", modes=1, width=2.0, rho_g=120.0),
        # the smallest served grid, in the plain FP64 form
        _case("project fp64 64", "project", 64, 64, 64, "fp64"),
        # a time step that assembles Eq. (31) first (with under-resolved cells masked); radix-3 lines
        _case("constraint fp32 96", "constraint", 96, 96, 96, "fp32"),
        # the middle workload (128^3, 640/120)
        _case("project fp32 128", "project", 128, 128, 128, "fp32", rho_g=120.0),
        # ragged, anisotropic grid through the separate entry points, harmonic faces, rho_0 given
        _case("steps fp64 144x81x108", "steps", 144, 81, 108, "fp64", lx=3.0, ly=2.0, lz=5.0, face="harmonic",
              given_rho0=True),
        # a jet with an open top: no zero mode, tridiagonal y solve
        _case("outflow fp32 128x192x128", "project", 128, 192, 128, "fp32", top="outflow"),
        # a served grid in the FP64 form, radix-3 lines
        _case("project fp64 192", "project", 192, 192, 192, "fp64"),
        # the headline workload: 256^3, 8 modes, 640/60, FP32 solve + refinement
        _case("project fp32 256", "project", 256, 256, 256, "fp32"),
        # the same in the plain FP64 form
        _case("project fp64 256", "project", 256, 256, 256, "fp64"),
        # the largest served grid
        _case("project fp32 384x256x384", "project", 384, 256, 384, "fp32"),
        # the unsplit baseline that the split is compared with
        _case("unsplit fp32 128", "unsplit", 128, 128, 128, "fp32", rho_g=120.0),
        # 64 uneven grids, every dimension from {32, 48, 64, 96, 128, 192}, one launch
        _case("batch fp32 64 grids", "batch", 0, 0, 0, "fp32", modes=1, width=2.0, rho_g=120.0, grids=64,
              shape_seed=3),
    ]


def draw(rng):
    kind = rng.choices(["project", "constraint", "steps", "unsplit", "batch"], [10, 2, 3, 2, 2])[0]
    prec = rng.choice(["fp32", "fp32", "fp64"])
    kw = dict(face=rng.choice(["arithmetic", "arithmetic", "harmonic"]), modes=rng.choice([1, 8]),
              width=rng.choice([2.0, 4.0, 6.0]), rho_g=rng.choice([60.0, 120.0, 300.0]))
    if kind == "batch":
        return {k: v for k, v in _case("", "batch", 0, 0, 0, "fp32", grids=rng.randint(8, 48),
                                       shape_seed=rng.randrange(1 << 20), **kw).items() if k != "name"}
    cap = math.log(2.1e6 if kind == "unsplit" else 1.7e7)
    want = rng.uniform(math.log(16 ** 3), cap)  # cells, over their logarithm
    while True:
        nx, ny, nz = (rng.choice(SIZES) for _ in range(3))
        if nx % 2 == 0 and abs(math.log(nx * ny * nz) - want) < 0.25 and math.log(nx * ny * nz) <= cap:
            break
    # cells within a factor of three of cubic, as a mesh that resolves an interface is
    h = [rng.uniform(0.5, 1.5) for _ in range(3)]
    scale = TWO_PI / max(nx * h[0], ny * h[1], nz * h[2])
    kw.update(lx=nx * h[0] * scale, ly=ny * h[1] * scale, lz=nz * h[2] * scale)
    if kind in ("project", "steps"):
        kw["top"] = rng.choice(["wall", "wall", "wall", "outflow"])
        kw["given_rho0"] = rng.random() < 0.25
    return {k: v for k, v in _case("", kind, nx, ny, nz, prec, **kw).items() if k != "name"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _centres(n, length, dev):
    return (torch.arange(n, dtype=torch.float64, device=dev) + 0.5) * (length / n)


def _inputs(case, seed, dev="cuda"):
    """The fields of one grid: u, v, w, S, rho, p_n, p_nm1 (and, for Eq. (31), its phase-wise inputs)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    lx, ly, lz = case["lx"], case["ly"], case["lz"]
    gen = torch.Generator(device=dev).manual_seed(seed)
    host = np.random.default_rng(seed)

    def normal(*shape):
        return torch.randn(shape, generator=gen, dtype=torch.float64, device=dev)

    x = _centres(nx, lx, dev)[None, None, :] * (TWO_PI / lx)
    z = _centres(nz, lz, dev)[:, None, None] * (TWO_PI / lz)
    y = _centres(ny, ly, dev)[None, :, None]
    dy = ly / ny
    eta = torch.zeros((nz, 1, nx), dtype=torch.float64, device=dev)
    for _ in range(case["modes"]):  # wavy interface around mid height
        kx, kz = int(host.integers(0, 9)), int(host.integers(1, 9))
        eta += torch.cos(kx * x + kz * z + float(host.uniform(0.0, TWO_PI)))
    eta = ly * (0.5 + (0.016 if case["modes"] == 1 else 0.008) * eta)
    rho_l, rho_g = 640.0, case["rho_g"]
    C = 0.5 * (1.0 - torch.tanh(2.0 * (y - eta) / (case["width"] * dy)))
    band = ((y - eta).abs() <= 3.0 * dy).expand(nz, ny, nx)
    d = dict(rho=(rho_g + (rho_l - rho_g) * C).expand(nz, ny, nx).contiguous(), u=normal(nz, ny, nx),
             v=normal(nz, ny + 1, nx), w=normal(nz, ny, nx))
    d["v"][:, 0] = 0.0
    d["v"][:, ny] = 0.0
    S = torch.where(band, 0.1 * normal(nz, ny, nx), torch.zeros((), dtype=torch.float64, device=dev))
    d["S"] = torch.where(band, S - S.sum() / band.sum().clamp(min=1), S)
    for k in ("p_n", "p_nm1"):
        p = normal(nz, ny, nx)
        d[k] = p - p.mean()
    if case["kind"] == "constraint":
        d["C"] = C.expand(nz, ny, nx).contiguous()
        d["comp_g"], d["comp_l"] = 0.1 * normal(nz, ny, nx), 0.01 * normal(nz, ny, nx)
        d["mdot"] = torch.where(band, 5.0 * normal(nz, ny, nx), 0.0 * C)
        d["rho_gas"] = rho_g * (1.0 + 0.02 * normal(nz, ny, nx).clamp(-3, 3))
        d["rho_liq"] = rho_l * (1.0 + 0.01 * normal(nz, ny, nx).clamp(-3, 3))
        d["mask"] = (torch.rand((nz, ny, nx), generator=gen, device=dev) < 0.02).to(torch.uint8)
    d["dt"] = 1e-3
    d["rho0"] = 0.95 * rho_g if case["given_rho0"] else -1.0
    return d


def _plan(case):
    return ppe.Plan(case["nx"], case["ny"], case["nz"], case["lx"], case["ly"], case["lz"],
                    precision=ppe.FP32_REFINE if case["prec"] == "fp32" else ppe.FP64,
                    face_rule=ppe.FACE_HARMONIC if case["face"] == "harmonic" else ppe.FACE_ARITHMETIC,
                    bc_top=ppe.BC_OUTFLOW if case["top"] == "outflow" else ppe.BC_WALL)


def _grids(case):
    """The cases of a batch's grids."""
    for nx, ny, nz in fields.batch_shapes(case["grids"], seed=case["shape_seed"]):
        yield dict(case, kind="project", nx=nx, ny=ny, nz=nz)


def prepare(case, seed):
    if case["kind"] == "batch":
        grids = list(_grids(case))
        cells = [g["nx"] * g["ny"] * g["nz"] for g in grids]
        faces = [g["nx"] * (g["ny"] + 1) * g["nz"] for g in grids]
        # outputs of all grids in one array each
        out = {k: torch.empty(sum(faces if k == "v" else cells), dtype=torch.float64, device="cuda")
               for k in ("p", "u", "v", "w")}
        parts = {k: out[k].split(faces if k == "v" else cells) for k in out}
        items = []
        for i, g in enumerate(grids):
            d = _inputs(g, seed * 1000 + i)
            c, vs = d["u"].shape, d["v"].shape
            items.append((_plan(g), dict(d, p=parts["p"][i].view(c), u_out=parts["u"][i].view(c),
                                         v_out=parts["v"][i].view(vs), w_out=parts["w"][i].view(c))))
        return dict(case=case, items=items, batch=ppe.Batch(items), out=out)
    d = _inputs(case, seed)
    out = {k: torch.empty_like(d[s]) for k, s in (("p", "rho"), ("u", "u"), ("v", "v"), ("w", "w"))}
    if case["kind"] in ("steps", "constraint"):
        out["f" if case["kind"] == "steps" else "S"] = torch.empty_like(d["rho"])
    if case["kind"] == "constraint":
        out["rho"] = torch.empty_like(d["rho"])
    return dict(case=case, plan=_plan(case), d=d, out=out)


def run(state):
    kind, o = state["case"]["kind"], state["out"]
    if kind == "batch":
        state["batch"].launch()
        return o
    plan, d = state["plan"], state["d"]
    if kind == "project":
        plan.project(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], d["dt"], o["p"], o["u"], o["v"],
                     o["w"], rho0=d["rho0"])
    elif kind == "constraint":
        plan.divergence_constraint(d["C"], d["comp_g"], d["comp_l"], d["mdot"], d["rho_gas"], d["rho_liq"], o["S"],
                                   rho=o["rho"], under_resolved=d["mask"])
        plan.project(d["u"], d["v"], d["w"], o["S"], o["rho"], d["p_n"], d["p_nm1"], d["dt"], o["p"], o["u"], o["v"],
                     o["w"])
    elif kind == "steps":
        plan.rhs(d["u"], d["v"], d["w"], d["S"], d["rho"], d["p_n"], d["p_nm1"], d["dt"], o["f"], rho0=d["rho0"])
        plan.solve(o["f"], o["p"])
        plan.correct(d["u"], d["v"], d["w"], d["rho"], o["p"], d["p_n"], d["p_nm1"], d["dt"], o["u"], o["v"], o["w"],
                     rho0=d["rho0"])
    else:
        plan.project_unsplit(d["u"], d["v"], d["w"], d["S"], d["rho"], d["dt"], o["p"], o["u"], o["v"], o["w"],
                             tol=1e-10, max_iter=500)
    return o


# ---------------------------------------------------------------------------
# what one pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        w = [work(g) for g in _grids(case)]
        return {k: sum(x[k] for x in w) for k in ("bytes", "flops")}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    n, nv = nx * ny * nz, nx * (ny + 1) * nz
    # u, w, S, rho, p_n, p_nm1, v in; p, u, w, v out
    doubles = 9 * n + 2 * nv
    # right-hand side 30, correction 25, tridiagonal solve and scaling 10, real FFTs in x and z both ways
    flops = n * (65 + 5.0 * math.log2(nx * nz))
    if case["kind"] == "unsplit":  # no old pressures; at least one solve
        doubles -= 2 * n
    if case["kind"] == "steps":  # f is an output too
        doubles += n
    nbytes = 8 * doubles
    if case["kind"] == "constraint":  # six phase-wise fields and the mask in; S and rho out instead of in
        nbytes += 8 * 6 * n + n
        flops += 12 * n
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in plain FP64 torch
# ---------------------------------------------------------------------------
def _up(q, dim):
    """q of the lower neighbour (periodic)."""
    return q.roll(1, dim)


class _Ops:
    """Finite-volume operators and the constant-coefficient solve of one grid."""

    def __init__(self, case, dev):
        self.nx, self.ny, self.nz = case["nx"], case["ny"], case["nz"]
        self.h = (case["lx"] / self.nx, case["ly"] / self.ny, case["lz"] / self.nz)
        self.open = case["top"] == "outflow"
        self.harmonic = case["face"] == "harmonic"
        ny = self.ny
        j = torch.arange(ny, dtype=torch.int64, device=dev)
        kk = j[:, None]
        if self.open:  # cos(pi (k + 1/2)(j + 1/2)/ny)
            num, freq = (2 * kk + 1) * (2 * j[None, :] + 1), (2 * j + 1).double() / (4 * ny)
        else:          # cos(pi k (j + 1/2)/ny)
            num, freq = 2 * kk * (2 * j[None, :] + 1), j.double() / (2 * ny)
        basis = torch.cos((num % (8 * ny)).double() * (math.pi / (4 * ny)))
        norm = torch.full((ny, 1), 2.0 / ny, dtype=torch.float64, device=dev)
        if not self.open:
            norm[0] = 1.0 / ny
        self.basis, self.inv = basis, (norm * basis).T.contiguous()

        def lam(frac, h):
            return -(4.0 / h ** 2) * torch.sin(math.pi * frac) ** 2

        kx = torch.arange(self.nx // 2 + 1, device=dev).double() / self.nx
        kz = torch.arange(self.nz, device=dev).double() / self.nz
        self.lam = lam(kx, self.h[0])[None, None, :] + lam(freq, self.h[1])[None, :, None] \
            + lam(kz, self.h[2])[:, None, None]

    def faces(self, rho):
        """Densities on the x, y (ny + 1 planes) and z faces."""
        def mean(a, b):
            return 2.0 / (1.0 / a + 1.0 / b) if self.harmonic else 0.5 * (a + b)
        inner = mean(rho[:, :-1], rho[:, 1:])
        return (mean(_up(rho, 2), rho), torch.cat([rho[:, :1], inner, rho[:, -1:]], 1), mean(_up(rho, 0), rho))

    def grad(self, q):
        gy = torch.zeros((self.nz, self.ny + 1, self.nx), dtype=q.dtype, device=q.device)
        gy[:, 1:-1] = (q[:, 1:] - q[:, :-1]) / self.h[1]
        if self.open:  # ghost -q above the top cell
            gy[:, -1] = -2.0 * q[:, -1] / self.h[1]
        return (q - _up(q, 2)) / self.h[0], gy, (q - _up(q, 0)) / self.h[2]

    def div(self, a, b, c):
        return (a.roll(-1, 2) - a) / self.h[0] + (b[:, 1:] - b[:, :-1]) / self.h[1] + (c.roll(-1, 0) - c) / self.h[2]

    def solve(self, f):
        """L p = f - mean(f), zero mean (walls); L p = f (open top)."""
        s = torch.fft.fft(torch.fft.rfft(f, dim=2), dim=0)

        def along_y(m, t):
            return torch.complex(torch.matmul(m, t.real), torch.matmul(m, t.imag))
        s = along_y(self.basis, s)
        if self.open:
            s = s / self.lam
        else:
            lam = self.lam.clone()
            lam[0, 0, 0] = 1.0
            s = s / lam
            s[0, 0, 0] = 0.0
        s = along_y(self.inv, s)
        return torch.fft.irfft(torch.fft.ifft(s, dim=0), n=self.nx, dim=2)


def _exact_split(case, d, S, rho):
    ops = _Ops(case, rho.device)
    rho0 = d["rho0"] if d["rho0"] > 0 else float(rho.min())
    phat = 2.0 * d["p_n"] - d["p_nm1"]
    gh = ops.grad(phat)
    rf = ops.faces(rho)
    flux = [(1.0 - rho0 / r) * g for r, g in zip(rf, gh)]
    f = ops.div(*flux) + (rho0 / d["dt"]) * (ops.div(d["u"], d["v"], d["w"]) - S)
    p = ops.solve(f)
    gp = ops.grad(p)
    vel = [q - d["dt"] * (a / rho0 + (1.0 / r - 1.0 / rho0) * b) for q, a, r, b in
           zip((d["u"], d["v"], d["w"]), gp, rf, gh)]
    return dict(f=f, p=p, u=vel[0], v=vel[1], w=vel[2])


def _exact_unsplit(case, d):
    ops = _Ops(case, d["rho"].device)
    rf = ops.faces(d["rho"])

    def K(q):
        return -ops.div(*[g / r for g, r in zip(ops.grad(q), rf)])

    b = -(ops.div(d["u"], d["v"], d["w"]) - d["S"]) / d["dt"]
    b = b - b.mean()
    x = torch.zeros_like(b)
    r, p, rz, best, stale = b.clone(), None, None, math.inf, 0
    top = float(b.abs().max())
    for _ in range(400):  # conjugate gradients down to the rounding of the residual
        z = -ops.solve(r)
        rz_new = float((r * z).sum())
        p = z if p is None else z + (rz_new / rz) * p
        rz = rz_new
        q = K(p)
        a = rz / float((p * q).sum())
        x += a * p
        r -= a * q
        now = float(r.abs().max()) / top
        stale = 0 if now < 0.9 * best else stale + 1
        best = min(best, now)
        if best < 1e-15 or stale > 6:
            break
    x -= x.mean()
    gp = ops.grad(x)
    u, v, w = [q - d["dt"] * g / r for q, g, r in zip((d["u"], d["v"], d["w"]), gp, rf)]
    return dict(p=x, u=u, v=v, w=w)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        parts = [exact(g, seed * 1000 + i) for i, g in enumerate(_grids(case))]
        return {k: torch.cat([q[k].reshape(-1) for q in parts]) for k in ("p", "u", "v", "w")}
    d = _inputs(case, seed)
    if kind == "unsplit":
        return _exact_unsplit(case, d)
    if kind == "constraint":
        C = d["C"]
        S = -(1.0 - C) * d["comp_g"] - C * d["comp_l"] + d["mdot"] * (1.0 / d["rho_gas"] - 1.0 / d["rho_liq"])
        S = torch.where((d["mask"] != 0) & (C > 0) & (C < 1), torch.zeros_like(S), S)
        rho = d["rho_gas"] * (1.0 - C) + d["rho_liq"] * C
        r = _exact_split(case, dict(d, rho0=-1.0), S, rho)
        return dict(p=r["p"], u=r["u"], v=r["v"], w=r["w"], S=S, rho=rho)
    r = _exact_split(case, d, d["S"], d["rho"])
    if kind == "project":
        r.pop("f")
    return r
