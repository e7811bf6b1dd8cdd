"""The solver's work as its users' programs run it: the calls, sizes and options that are timed.

A case is one program: ``prepare`` builds what it holds before the call (the lattice and
flow on the GPU, the solver handles), ``run`` is its one pass through the public entry
points of ``paper_2502_08034_gb300``, and ``exact`` gives the same outputs from plain torch
in FP64 (the face-by-face operator assembled here and iterated to its rounding floor).

Kinds:
  step      explicit sweeps from a given field, outputs and field read back (a program that
            follows the pseudo-time, e.g. for a residual curve)
  solve     steady state from a cold start, outputs and field read back
  gradient  differentiable objective, forward and backward: I_tot, U, U_mt and their
            gradients by the per-voxel area field and the velocity scale
  batch     lattices of uneven size at their own operating points, solved together
  upsample  coarse-to-fine chain over refinement levels with U_mt on the finest
  nernst    steady state by the Nernst model, with the overpotential field
  bv        Butler-Volmer model with electromigration, refined from the SBV state

Lattices are the repository's fiber recipe (random straight cylinders of 4 or 8 cells'
diameter, porosity 0.75 to 0.9, unreachable pockets filled, potential flow), built on the
GPU; constants are those of its workloads.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2502_08034_gb300 import rfb, synth, workflows
from paper_2502_08034_gb300.autograd import soc_objective

R_GAS, FARADAY = 8.314462618, 96485.33212
H, D = 1.25e-6, 4e-10                    # cell size [m], diffusivity [m^2/s]
ALPHA, N_E, T, C0 = 0.5, 2, 298.0, 20.0  # kinetics of the workloads
CFL = 0.4

BASE = dict(precision="fp64", porosity=0.80, fiber=8.0, u=0.01, eta=-0.10, s_in=0.5, k0=1e-7,
            tol=1e-10, inlet="face", area_mult=False)


def _case(name, kind, dims, **over):
    return dict(BASE, name=name, kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], **over)


def listed():
    return [
        # a few sweeps of a coarse lattice: launches and host waits are all of it
        _case("step fp64 24x20x37", "step", (24, 20, 37), fiber=4.0, sweeps=8),
        # the plain FP64 workload
        _case("solve fp64 48x48x96", "solve", (48, 48, 96)),
        # the FP64 path where it streams from memory, on the differentiation lattice
        _case("solve fp64 128x128x256", "solve", (128, 128, 256)),
        # mixed precision on the smallest lattice of the batched design study
        _case("solve mixed 64x64x64", "solve", (64, 64, 64), precision="mixed", porosity=0.85,
              u=0.02, eta=-0.05, s_in=0.3),
        # a ragged lattice (an imaged sample cropped to no round size), ghost-cell inlet
        _case("solve mixed 75x61x118", "solve", (75, 61, 118), precision="mixed",
              inlet="ghost"),
        # mid-size, narrower than a tile's multiple in both directions, fitted wall areas
        _case("solve mixed 160x160x200", "solve", (160, 160, 200), precision="mixed",
              porosity=0.82, eta=-0.05, s_in=0.3, area_mult=True),
        # the benchmark lattice and operating point
        _case("solve mixed 256x256x512", "solve", (256, 256, 512), precision="mixed",
              porosity=0.85, u=0.005, eta=-0.05, s_in=0.3),
        # the differentiation workload with mixed-precision adjoints
        _case("gradient mixed 128x128x256", "gradient", (128, 128, 256), precision="mixed",
              area_mult=True, tol=1e-11),
        # a gradient at test size, FP64 throughout
        _case("gradient fp64 32x32x64", "gradient", (32, 32, 64), fiber=4.0, area_mult=True,
              tol=1e-12),
        # a geometry / flow-rate / voltage study, the batched recipe at half size
        _case("batch 16 of 32..96", "batch", (96, 96, 192), precision="mixed", fiber=4.0,
              lattices=16),
        # the paper's fast kinetics by the Nernst model
        _case("nernst fp64 48x48x96", "nernst", (48, 48, 96), k0=7.2e-5),
        # model refinement from SBV to Butler-Volmer on a small lattice
        _case("bv 20x14x26", "bv", (20, 14, 26), fiber=4.0, u=0.002, s_in=0.2, k0=2e-5,
              tol=1e-8),
    ]


def draw(rng):
    def size(lo, hi, q=1):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / q)) * q

    kind = rng.choice(["step", "solve", "solve", "solve", "solve", "solve", "gradient", "batch",
                       "upsample", "nernst", "bv"])
    c = dict(BASE, kind=kind, porosity=round(rng.uniform(0.76, 0.9), 3),
             u=float("%.3g" % math.exp(rng.uniform(math.log(0.003), math.log(0.03)))),
             eta=round(rng.uniform(-0.15, -0.02), 3), s_in=round(rng.uniform(0.1, 0.9), 2),
             inlet=rng.choice(["face", "face", "ghost"]))
    if kind == "step":
        c.update(nx=size(9, 200), ny=size(9, 200), nz=size(12, 240), sweeps=rng.randint(1, 64))
    elif kind == "solve":
        c["precision"] = rng.choice(["fp64", "mixed", "mixed", "mixed"])
        hi = 256 if c["precision"] == "mixed" else 128
        q = rng.choice([1, 4, 4, 16])     # any width, or one that the vector kernels take
        c.update(nx=size(24, hi, q), ny=size(24, hi), nz=size(32, hi),
                 area_mult=rng.random() < 0.3)
    elif kind == "gradient":
        c["precision"] = rng.choice(["fp64", "mixed"])
        hi = 128 if c["precision"] == "mixed" else 48
        c.update(nx=size(16, hi, 4), ny=size(16, hi), nz=size(24, hi), area_mult=True, tol=1e-11,
                 inlet="face")
    elif kind == "batch":
        n = rng.randint(3, 12)
        c.update(nx=size(32, 96, 4), nz=size(48, 160), precision="mixed", lattices=n,
                 inlet="face")
        c["ny"] = c["nx"]
    elif kind == "upsample":
        c.update(nx=2 * size(16, 64, 4), ny=2 * size(16, 64), nz=2 * size(24, 96), precision="mixed",
                 inlet="face")
    elif kind == "nernst":
        c.update(nx=size(16, 80), ny=size(16, 80), nz=size(24, 120), k0=7.2e-5)
    else:
        c.update(nx=size(9, 20), ny=size(9, 20), nz=size(12, 28), u=0.002, s_in=0.2, k0=2e-5,
                 tol=1e-8, eta=-0.10)
    c["fiber"] = 8.0 if min(c["nx"], c["ny"]) >= 48 else 4.0
    return c


# ---- inputs

def _stamp(solid, f, scale):
    """OR one fiber (z0, x0, y0, angle, diameter; fine-cell units) into solid (nz, ny, nx)."""
    z0, x0, y0, th, d = f
    nz, ny, nx = solid.shape
    k0 = max(0, int((z0 - d / 2) / scale) - 1)
    k1 = min(nz, int((z0 + d / 2) / scale) + 2)
    dev, f8 = solid.device, torch.float64
    x = (torch.arange(nx, device=dev, dtype=f8) + 0.5) * scale - x0
    y = (torch.arange(ny, device=dev, dtype=f8) + 0.5) * scale - y0
    z = (torch.arange(k0, k1, device=dev, dtype=f8) + 0.5) * scale - z0
    across = x[None, :] * math.sin(th) - y[:, None] * math.cos(th)
    solid[k0:k1] |= z[:, None, None] ** 2 + (across ** 2)[None] <= (d / 2) ** 2


def _reachable(fluid):
    """Fluid cells 6-connected to the inlet plane: along each line, a reached cell reaches
    every later fluid cell up to the next solid one; repeated until nothing is added."""
    reach = torch.zeros_like(fluid)
    reach[0] = fluid[0]
    n = -1
    while int(reach.sum()) != n:
        n = int(reach.sum())
        for ax in (0, 1, 2):
            for back in (False, True):
                f = fluid.flip(ax) if back else fluid
                r = reach.flip(ax) if back else reach
                pos = torch.arange(1, f.shape[ax] + 1, device=f.device, dtype=torch.int32)
                pos = pos.view([-1 if a == ax else 1 for a in range(3)])
                wall = (pos * ~f).cummax(ax).values
                seen = (pos * r).cummax(ax).values
                r = f & (seen > wall)
                reach = r.flip(ax) if back else r
    return reach


def _lattice(case, seed, levels=1, dims=None):
    """The fibers of ``seed`` at ``levels`` refinement levels, coarsest first, each with its
    flow: face velocities of the potential flow at mean velocity u."""
    nx, ny, nz = dims or (case["nx"], case["ny"], case["nz"])
    for attempt in range(20):             # a lattice whose fibers block the flow is redrawn
        rng = np.random.default_rng([seed, attempt])
        fine = torch.zeros((nz, ny, nx), dtype=torch.bool, device="cuda")
        fibers = []
        while int(fine.sum()) < (1.0 - case["porosity"]) * fine.numel():
            f = (rng.uniform(0, nz), rng.uniform(0, nx), rng.uniform(0, ny),
                 rng.uniform(0, math.pi), case["fiber"])
            fibers.append(f)
            _stamp(fine, f, 1.0)
        out = []
        for lev in range(levels):
            s = 2 ** (levels - 1 - lev)
            solid = fine
            if s > 1:
                solid = torch.zeros((nz // s, ny // s, nx // s), dtype=torch.bool, device="cuda")
                for f in fibers:
                    _stamp(solid, f, float(s))
            fluid = _reachable(~solid)
            if not bool(fluid[-1].any()):
                break
            U, V, W, _ = synth.potential_flow((~fluid).cpu().numpy(), H * s, case["u"],
                                              tol=1e-10, device="cuda")
            out.append(SimpleNamespace(
                dims=(nx // s, ny // s, nz // s), h=H * s, solid=(~fluid).to(torch.uint8),
                U=torch.from_numpy(U).cuda(), V=torch.from_numpy(V).cuda(),
                W=torch.from_numpy(W).cuda(), m=None, s_in=case["s_in"], eta=case["eta"]))
        if len(out) == levels:
            if case["area_mult"]:         # lognormal wall areas, median 1
                g = torch.Generator("cuda").manual_seed(seed)
                x = out[-1]
                z = torch.randn(x.solid.shape, generator=g, device="cuda", dtype=torch.float64)
                x.m = torch.where(_walls(x)[1] > 0, torch.exp(0.3 * z), 1.0).reshape(-1)
            return out
    raise RuntimeError("no open lattice in 20 draws")


def _batch(case, seed):
    """Lattices of a third to all of the case's extents (the case's own), each with its own
    porosity, flow rate and operating point (of the seed)."""
    extent = np.random.default_rng([case["nx"], case["nz"], case["lattices"]])
    rng = np.random.default_rng([seed, 99])
    out = []
    for q in range(case["lattices"]):
        nx = max(16, 4 * int(round(case["nx"] * extent.uniform(1 / 3, 1) / 4)))
        nz = int(min(case["nz"], max(24, nx * extent.uniform(1, 2))))
        c = dict(case, porosity=rng.uniform(0.76, 0.9), u=0.003 * 10 ** rng.uniform(0, 1),
                 s_in=rng.uniform(0.1, 0.9), eta=rng.uniform(-0.15, -0.02))
        out.append(_lattice(c, 1000 * seed + q, dims=(nx, nx, nz))[0])
    return out


def _solver(case, x):
    return rfb.Solver(x.dims, x.h, x.solid, x.U, x.V, x.W, D, case["k0"], ALPHA, N_E, T, C0,
                      area_mult=x.m)


def _step_field(case, x, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    s = torch.rand(x.solid.shape, generator=g, device="cuda", dtype=torch.float64)
    return torch.where(x.solid == 0, s, 0.0)


def prepare(case, seed):
    kind = case["kind"]
    st = SimpleNamespace(case=case)
    if kind == "batch":
        st.lattices = _batch(case, seed)
    else:
        st.lattices = _lattice(case, seed, levels=2 if kind == "upsample" else 1)
    st.solvers = [_solver(case, x) for x in st.lattices]
    st.sv, x = st.solvers[-1], st.lattices[-1]
    st.s = [torch.empty(v.n_cells, dtype=torch.float64, device="cuda") for v in st.solvers]
    if kind == "step":
        st.s0 = _step_field(case, x, seed)
    elif kind == "batch":
        st.batch = rfb.Batch(st.solvers)
    elif kind == "gradient":
        st.m = x.m.clone().requires_grad_()
        st.beta = torch.tensor(1.0, dtype=torch.float64, device="cuda", requires_grad=True)
        st.weights = [torch.tensor(w, dtype=torch.float64, device="cuda")
                      for w in (1e5, 1.0, 1.0)]
    elif kind == "nernst":
        st.eta_t = torch.empty_like(st.s[-1])
    return st


# ---- the passes

def _numbers(r):
    return {k: r[k] for k in ("I_tot", "F_in", "F_out", "U", "outlet_mean")}


def run(st):
    c, sv = st.case, st.sv
    kind, s_in, eta, tol = c["kind"], c["s_in"], c["eta"], c["tol"]
    opts = dict(precision=c["precision"], inlet_bc=c["inlet"])
    if kind == "step":
        sv.set_state(st.s0)
        r = sv.step(s_in, eta, c["sweeps"], **opts)
        return {"s": sv.get_state(out=st.s[0]), **_numbers(r)}
    if kind == "gradient":
        sv.reset_state()
        y = soc_objective(sv, st.m, st.beta, s_in, eta, tol, c["precision"])
        gm, gb = torch.autograd.grad(y, (st.m, st.beta), grad_outputs=st.weights)
        return {"I_tot": y[0], "U": y[1], "U_mt": y[2], "grad_m": gm, "grad_beta": gb}
    if kind == "upsample":
        out, (u_mt, _) = workflows.upsample_chain(st.solvers, st.lattices, tol,
                                                  precision=c["precision"])
        return {"s": sv.get_state(out=st.s[-1]), "U_mt": u_mt, **_numbers(out[-1])}
    for v in st.solvers:                  # the others start cold
        v.reset_state()
    if kind == "batch":
        x = st.lattices
        # a fixed check interval, so that a run stops at the same sweep every time
        r, _ = st.batch.solve([q.s_in for q in x], [q.eta for q in x], [tol] * len(x),
                              check_every=200, inlet_bc=c["inlet"])
        return {"s": [v.get_state(out=s) for v, s in zip(st.solvers, st.s)],
                **{k: np.array([n[k] for n in r]) for k in _numbers(r[0])}}
    if kind == "nernst":
        r = sv.solve_nernst(s_in, eta, tol, **opts)
        return {"s": sv.get_state(out=st.s[0]),
                "eta_t": sv.get_overpotential(out=st.eta_t), **_numbers(r)}
    r = sv.solve(s_in, eta, tol, **opts)
    if kind == "bv":
        b = sv.solve_bv(s_in, eta, tol, start="sbv", **opts)
        return {**sv.get_bv_state(), **{k: b[k] for k in ("I_tot", "U", "s_out", "I_membrane",
                                                          "phi_mean")}}
    return {"s": sv.get_state(out=st.s[0]), **_numbers(r)}


def work(case):
    """Bytes: mask, three face velocities (and the area field) in, the field out, once.
    Operations: an explicit update is 7 multiply-adds a cell and sweep; the local-step
    iteration takes about 8 sweeps per plane along the flow to carry the inlet's state
    through, as many again for each adjoint or transport problem solved beside it."""
    n = case["nx"] * case["ny"] * case["nz"]
    if case["kind"] == "batch":           # mean extent two thirds, squared, times 1.5 along z
        n = case["lattices"] * int((0.67 * case["nx"]) ** 2 * min(case["nz"], case["nx"]))
    sweeps = case.get("sweeps", 8 * case["nz"])
    solves = {"gradient": 5, "upsample": 2, "bv": 4, "nernst": 1}.get(case["kind"], 1)
    fields = {"gradient": 2, "nernst": 2, "bv": 4}.get(case["kind"], 1)
    return {"bytes": n * (25 + 8 * fields + (8 if case["area_mult"] else 0)),
            "flops": 14.0 * n * sweeps * solves}


# ---- the same in plain torch, FP64

def _walls(x):
    """Fluid mask, fiber 6-neighbours and fluid 6-neighbours per direction (-x, +x, ..)."""
    fluid = x.solid == 0
    pad = torch.zeros([n + 2 for n in fluid.shape], dtype=torch.bool, device=fluid.device)
    inside = torch.zeros_like(pad)
    pad[1:-1, 1:-1, 1:-1] = fluid
    inside[1:-1, 1:-1, 1:-1] = True
    nz, ny, nx = fluid.shape
    at = [(1, 1, 0), (1, 1, 2), (1, 0, 1), (1, 2, 1), (0, 1, 1), (2, 1, 1)]
    cut = [(slice(a, a + nz), slice(b, b + ny), slice(q, q + nx)) for a, b, q in at]
    nbr = [fluid & pad[q] for q in cut]
    n_wall = sum((inside[q] & ~pad[q]).to(torch.float64) for q in cut) * fluid
    return fluid, n_wall, nbr


class _Operator:
    """RHS(s) = L s + b on the unknown cells, face by face (upwind advection, 7-point
    diffusion, wall reaction; ``umt``: cells at a wall held at 1, no reaction)."""

    def __init__(self, case, x, umt=False):
        self.shape = x.solid.shape
        nz, ny, nx = self.shape
        self.n = nx * ny * nz
        fluid, n_wall, nbr = _walls(x)
        self.fluid, self.n_wall = fluid, n_wall
        self.unknown = fluid & (n_wall == 0) if umt else fluid
        q = [x.U[:, :, :-1], -x.U[:, :, 1:], x.V[:, :-1, :], -x.V[:, 1:, :], x.W[:-1], -x.W[1:]]
        q = [f / x.h for f in q]              # inflow through each face, per cell volume
        dh = D / x.h ** 2
        vt = N_E * -case["eta"] / (R_GAS * T / FARADAY)
        A = math.exp(ALPHA * vt)
        self.A, self.B = A, A * (1 + math.exp(-vt))
        m = 1.0 if x.m is None else x.m.view(self.shape)
        self.kap = m * case["k0"] / x.h * n_wall * (0.0 if umt else 1.0)
        self.s_in = 0.0 if umt else case["s_in"]
        self.adv = [f.clamp(min=0) * self.unknown for f in q]
        self.out = sum((-f).clamp(min=0) for f in q) * self.unknown
        a = [(p + dh * k) * self.unknown for p, k in zip(self.adv, nbr)]
        a[4][0] = 0.0
        self.g_in = torch.zeros(self.shape, dtype=torch.float64, device=fluid.device)
        self.g_in[0] = (2 if case["inlet"] == "face" else 1) * dh
        self.q_in = torch.zeros_like(self.g_in)
        self.q_in[0] = x.W[0] / x.h * fluid[0]
        self.diag = (self.out + dh * sum(k.to(torch.float64) for k in nbr) + self.g_in +
                     self.kap * self.B) * self.unknown
        self.b = ((self.q_in + self.g_in) * self.s_in + self.kap * self.A) * self.unknown
        self.a = [f.reshape(-1) for f in a]
        self.off = [-1, 1, -nx, nx, -nx * ny, nx * ny]
        self.pinned = (fluid & ~self.unknown).to(torch.float64).reshape(-1)

    def transposed(self):
        """Neighbour weights of L^T: the neighbour's coefficient that points back here."""
        at = []
        for f in range(6):
            o, back = self.off[f], self.a[f ^ 1]
            z = torch.zeros_like(back)
            if o > 0:
                z[:-o] = back[o:]
            else:
                z[-o:] = back[:o]
            at.append(z * self.unknown.reshape(-1))
        return at

    def rhs(self, a, b, s, pad):
        m = self.off[5]
        pad[m:-m] = s
        r = torch.addcmul(b, self.diag.reshape(-1), s, value=-1)
        for w, o in zip(a, self.off):
            r.addcmul_(w, pad[m + o:m + o + self.n])
        return r

    def solve(self, a, b, s, eps=1e-15, most=60000):
        """Damped Jacobi from s until the update stalls at rounding."""
        pad = torch.zeros(self.n + 2 * self.off[5], dtype=torch.float64, device=s.device)
        step = torch.where(self.unknown, 0.8 / self.diag.clamp(min=1e-300), 0.0).reshape(-1)
        for _ in range(0, most, 200):
            for _ in range(200):
                s.addcmul_(step, self.rhs(a, b, s, pad))
            if float((step * self.rhs(a, b, s, pad)).norm() / s.norm()) < eps:
                break
        return s

    def steady(self):
        b = self.b.reshape(-1)
        return self.solve(self.a, b, (self.s_in * self.fluid.reshape(-1) +
                                      (1 - self.s_in) * self.pinned).contiguous())

    def numbers(self, x, s):
        s = s.view(self.shape)
        scale = N_E * FARADAY * C0 * x.h ** 3
        i_tot = scale * float((self.kap * (self.A - self.B * s)).sum())
        fl = self.fluid
        f_in = float((self.q_in * self.s_in + self.g_in * (self.s_in - s) * fl).sum())
        w_out = x.W[-1] / x.h * fl[-1]
        q = float(x.W[0][fl[0]].sum()) * x.h ** 2
        return {"I_tot": i_tot, "F_in": scale * f_in,
                "F_out": scale * float((w_out * s[-1]).sum()),
                "U": i_tot / (N_E * FARADAY * C0 * q * (1 - self.s_in)),
                "outlet_mean": float((w_out * s[-1]).sum() / w_out.sum())}

    def advection(self, s):
        """Advective part of RHS(s), cell by cell (the velocity scale's derivative at 1)."""
        m = self.off[5]
        pad = torch.zeros(self.n + 2 * m, dtype=torch.float64, device=s.device)
        pad[m:-m] = s
        r = self.q_in.reshape(-1) * self.s_in * self.unknown.reshape(-1) - self.out.reshape(-1) * s
        for f, o in enumerate(self.off):
            w = self.adv[f].clone()
            if f == 4:
                w[0] = 0.0
            r.addcmul_(w.reshape(-1), pad[m + o:m + o + self.n])
        return r


def _exact_gradient(case, x):
    op = _Operator(case, x)
    s = op.steady()
    v = op.numbers(x, s)
    at = op.transposed()
    mult = x.m
    rate = (op.kap.reshape(-1) / mult) * (op.A - op.B * s)      # d(source) / d(multiplier)
    scale = N_E * FARADAY * C0 * x.h ** 3
    lam = op.solve(at, -(op.kap * op.B).reshape(-1), torch.zeros_like(s) - 1e-3)
    per_i = 1e5 + v["U"] / v["I_tot"]     # weights of I_tot and of U through I_tot
    grad_m = per_i * scale * (1 + lam) * rate
    grad_b = per_i * scale * float(lam @ op.advection(s)) - v["U"]
    tr = _Operator(case, x, umt=True)
    t = tr.steady()
    u_mt = tr.numbers(x, t)["outlet_mean"]
    g = torch.zeros(tr.shape, dtype=torch.float64, device=s.device)
    g[-1] = x.W[-1] * tr.unknown[-1] / (x.W[-1] * tr.fluid[-1]).sum()
    lam = tr.solve(tr.transposed(), g.reshape(-1), torch.full_like(s, 1e-6) * tr.unknown.reshape(-1))
    grad_b += float(lam @ tr.advection(t))
    return {"I_tot": v["I_tot"], "U": v["U"], "U_mt": u_mt, "grad_m": grad_m,
            "grad_beta": torch.tensor(grad_b, dtype=torch.float64)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "bv":
        return None                       # nonlinear and coupled: minutes in plain torch
    if kind == "batch":
        s, r = [], []
        for x in _batch(case, seed):
            op = _Operator(dict(case, s_in=x.s_in, eta=x.eta), x)
            s.append(op.steady())
            r.append(op.numbers(x, s[-1]))
        return {"s": s, **{k: np.array([n[k] for n in r]) for k in r[0]}}
    x = _lattice(case, seed, levels=2 if kind == "upsample" else 1)[-1]
    if kind == "gradient":
        return _exact_gradient(case, x)
    op = _Operator(case, x)
    if kind == "step":
        # the local step is a 32-bit field, rounded down
        want = torch.where(op.unknown, CFL / op.diag.clamp(min=1e-300), 0.0).reshape(-1)
        dt = want.float()
        dt = torch.where(dt.double() > want, torch.nextafter(dt, torch.zeros_like(dt)), dt).double()
        s = _step_field(case, x, seed).reshape(-1)
        pad = torch.zeros(op.n + 2 * op.off[5], dtype=torch.float64, device=s.device)
        for _ in range(case["sweeps"]):
            s = torch.addcmul(s, dt, op.rhs(op.a, op.b.reshape(-1), s, pad))
    else:
        s = op.steady()
    out = {"s": s, **op.numbers(x, s)}
    if kind == "nernst":
        vt = N_E * -case["eta"] / (R_GAS * T / FARADAY)
        wall = (op.n_wall.reshape(-1) > 0)
        out["eta_t"] = torch.where(wall, vt - torch.log(s / (1 - s)), 0.0)
    if kind == "upsample":
        tr = _Operator(case, x, umt=True)
        out["U_mt"] = tr.numbers(x, tr.steady())["outlet_mean"]
    return out
