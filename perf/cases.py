"""The work that users of this library have it do, as measurable cases.

Every case goes through the public entry points (``lbve.Simulation``, the C
entry points of the same names, ``lbve.force_to_fields``) on the workloads of
``workloads.py`` with the parameters of the tests and the benchmark:

* ``frm``       one four-roll mill: small and long (64^2, FP64), ordinary
                (512^2), large (2048^2);
* ``channels``  the Wi-sweep Poiseuille channels stepped towards the steady
                state with the residual read after each call;
* ``mix``       the batched mix of uneven channels and mills, per precision;
* ``transfer``  the mix end to end: forces and initial fields from pinned host
                memory, steps, fields back to pinned host memory;
* ``cylinder``  the open channel past a cylinder (solid mask, curved walls,
                inlet and outlet columns) with its drag;
* ``adjoint``   a gradient with respect to the per-node force.

``exact`` restates the coupled step in plain float64 torch.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2508_16997_gb300 import lbve
from paper_2508_16997_gb300 import workloads as wl

PRECISION = {"fp64": lbve.LBVE_FP64, "fp32": lbve.LBVE_FP32_DEV, "df32": lbve.LBVE_DF32}
SWEEP = (1.0, 10.0, 100.0, 1e3, 1e4)  # Wi of the channel sweep

# Independent values of a node's state: the collided populations span 8 (hydrodynamic lattice) and
# 3 x 6 (conformation lattices) Hermite coefficients, the source's backward difference needs 3 more.
STATE_VALUES = 8 + 3 * 6 + 3
FLOPS_PER_UPDATE = 659  # float32 step kernel, additions, multiplications and 2 per FMA
ON_CHIP_BYTES = 129e6   # a state below the L2 size is read and written once per call, above it every step


def listed():
    return [
        # the smallest configuration as specified: 64^2, FP64, 2000 steps from rest
        {"name": "frm64_fp64", "kind": "frm", "N": 64, "precision": "fp64", "steps": 2000},
        # the Wi sweep to steady state advances by H / U_c = 1108 steps and looks at the residual
        {"name": "channels64_fp64", "kind": "channels", "H": 64, "nx": 4, "n": 5, "precision": "fp64", "steps": 1108},
        {"name": "channels64_fp32", "kind": "channels", "H": 64, "nx": 4, "n": 5, "precision": "fp32", "steps": 1108},
        # an ordinary single grid, resident in L2
        {"name": "frm512_fp32", "kind": "frm", "N": 512, "precision": "fp32", "steps": 100},
        # one large grid
        {"name": "frm2048_fp32", "kind": "frm", "N": 2048, "precision": "fp32", "steps": 20},
        # the batched mix: 256 uneven instances in FP32 storage, and smaller batches in the two
        # precisions for long horizons
        {"name": "mix256_fp32", "kind": "mix", "n": 256, "precision": "fp32", "steps": 20},
        {"name": "mix64_fp64", "kind": "mix", "n": 64, "precision": "fp64", "steps": 20},
        {"name": "mix64_df32", "kind": "mix", "n": 64, "precision": "df32", "steps": 20},
        # host to host through the batched entry points
        {"name": "transfer64_fp32", "kind": "transfer", "n": 64, "precision": "fp32", "steps": 20},
        # flow past a cylinder: the benchmark's R = 64 in FP32, a small one in FP64
        {"name": "cylinder64_fp32", "kind": "cylinder", "R": 64, "precision": "fp32", "steps": 200},
        {"name": "cylinder16_fp64", "kind": "cylinder", "R": 16, "precision": "fp64", "steps": 200},
        # the 512^2 gradient of the differentiation workload, shortened
        {"name": "adjoint512_fp32", "kind": "adjoint", "N": 512, "precision": "fp32", "steps": 200},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frm", "frm", "channels", "mix", "transfer", "cylinder", "adjoint"])
    if kind == "frm":
        N, precision = _log_int(rng, 16, 2048), rng.choice(["fp64", "fp32", "df32"])
        most = {"fp64": 4e6, "df32": 1e7, "fp32": 6e7}[precision] / (N * N)
        return {"kind": kind, "N": N, "precision": precision, "steps": max(1, min(_log_int(rng, 5, 2000), int(most)))}
    if kind == "channels":
        return {"kind": kind, "H": _log_int(rng, 8, 512), "nx": _log_int(rng, 3, 48), "n": rng.randint(1, 5),
                "precision": rng.choice(["fp64", "fp32", "df32"]), "steps": _log_int(rng, 20, 1500)}
    if kind in ("mix", "transfer"):
        return {"kind": kind, "n": _log_int(rng, 4, 48), "precision": rng.choice(["fp64", "fp32", "df32"]),
                "steps": rng.randint(1, 20)}
    if kind == "cylinder":
        return {"kind": kind, "R": _log_int(rng, 4, 40), "precision": rng.choice(["fp64", "fp32"]),
                "steps": _log_int(rng, 10, 200)}
    return {"kind": kind, "N": _log_int(rng, 12, 320), "precision": rng.choice(["fp64", "fp32"]),
            "steps": _log_int(rng, 5, 100)}


# ---- inputs ------------------------------------------------------------------------------------


@functools.lru_cache(maxsize=3)
def _base(kind, size, nx, n):
    """The instances of a case before the seed's part (a cylinder's link search takes seconds; the
    list of links is kept with its instance)."""
    if kind in ("frm", "adjoint"):
        return [wl.frm(size, Wi=5.0)]
    if kind == "channels":
        return [wl.channel(size, nx=nx, Wi=w) for w in SWEEP[:n]]
    if kind == "cylinder":
        inst = wl.cylinder_channel(size, Wi=0.5, open_x=True)
        links = inst.wall_links()
        inst.wall_links = lambda: links
        return [inst]
    return wl.batch_mix(n)


def _instances(case, seed):
    """The case's instances, each driven at its own strength (mean 1, 10 %), a mill's per-node force
    with 1 % noise where the case is a single one."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    out = []
    for base in _base(kind, case.get("N", case.get("H", case.get("R", 0))), case.get("nx", 0), case.get("n", 1)):
        inst = wl.Instance(**{k: v for k, v in base.__dict__.items() if k != "wall_links"})
        amp = float(1.0 + 0.1 * rng.uniform(-1.0, 1.0))
        inst.Fx *= amp
        if inst.force_field is not None:
            inst.force_field = inst.force_field * amp
            if kind in ("frm", "adjoint"):
                inst.force_field += 0.01 * np.abs(inst.force_field).max() * rng.standard_normal(inst.force_field.shape)
        if kind == "cylinder":
            inst.wall_links = base.wall_links
            inst.inlet = inst.inlet.copy()
            inst.inlet[0] *= amp
        out.append(inst)
    return out


def _initial_fields(inst, i, seed):
    """Smooth initial fields near rest: an eighth of the velocity scale and 5 % of stretch."""
    rng = np.random.default_rng([seed, i])
    U = wl.velocity_scale(inst.Ma)
    X = 2.0 * math.pi * np.arange(inst.nx) / inst.nx
    Y = (math.pi if not inst.periodic_y else 2.0 * math.pi) * np.arange(inst.ny) / max(1, inst.ny - (not inst.periodic_y))
    a = rng.uniform(0.5, 1.0, 4)
    sx, sy = np.sin(X + a[0])[None, :], np.sin(Y)[:, None]
    f = np.empty((6, inst.ny, inst.nx))
    f[0] = 1.0 + 1e-2 * U * U * a[1] * sx * sy
    f[1] = 0.125 * U * a[2] * sx * sy
    f[2] = -0.125 * U * a[3] * sx * sy
    f[3] = 1.0 + 0.05 * a[1] * (sx * sy) ** 2
    f[4] = 0.02 * a[2] * sx * sy
    f[5] = 1.0 + 0.05 * a[3] * (sx * sy) ** 2
    return f


def _developed(inst):
    """The inlet profile on every column, as initial fields of an open channel."""
    f = np.ones((6, inst.ny, inst.nx))
    f[1:] = inst.inlet[:, :, None]
    return f


def _views(insts, flat):
    """Each instance's [6, ny, nx] part of a flat buffer."""
    out, at = [], 0
    for inst in insts:
        out.append(flat[at:at + 6 * inst.n_nodes].view(6, inst.ny, inst.nx))
        at += 6 * inst.n_nodes
    return out


def prepare(case, seed):
    insts = _instances(case, seed)
    state = {"case": case, "insts": insts}
    nodes = sum(i.n_nodes for i in insts)
    if case["kind"] == "transfer":
        # a program that keeps its arrays in pinned host memory
        inputs = torch.empty(6 * nodes, dtype=torch.float64, pin_memory=True)
        forces = []
        for i, (inst, view) in enumerate(zip(insts, _views(insts, inputs))):
            view.numpy()[:] = _initial_fields(inst, i, seed)
            forces.append(None if inst.force_field is None else torch.from_numpy(inst.force_field).pin_memory())
        state |= {"inputs": [v.numpy() for v in _views(insts, inputs)], "keep": (inputs, forces),
                  "forces": [None if f is None else f.numpy() for f in forces]}
    init = [_developed(insts[0])] if case["kind"] == "cylinder" else None
    state["sim"] = lbve.Simulation(insts, precision=PRECISION[case["precision"]], init_fields=init)
    if case["kind"] == "adjoint":
        rng = np.random.default_rng([seed, 1])
        shape = (insts[0].ny, insts[0].nx)
        g = np.zeros((6, *shape))
        g[1:3] = rng.standard_normal((2, *shape))
        g[3:] = 1e-6 * rng.standard_normal((3, *shape))
        state["grad"] = torch.from_numpy(g).cuda()
        state["force"] = torch.from_numpy(insts[0].force_field).cuda().requires_grad_(True)
    else:
        state["out"] = torch.empty(6 * nodes, dtype=torch.float64, device="cpu" if case["kind"] == "transfer" else "cuda",
                                   pin_memory=case["kind"] == "transfer")
        state["ptrs"] = [v.data_ptr() for v in _views(insts, state["out"])]
    return state


def _split(views):
    """Density, velocity and conformation of each [6, ny, nx] as outputs of their own: their scales
    lie decades apart."""
    return [{"density": v[0], "velocity": v[1:3], "conformation": v[3:]} for v in views]


# ---- one pass -----------------------------------------------------------------------------------


def run(state):
    sim, case = state["sim"], state["case"]
    ids = range(len(state["insts"]))
    if case["kind"] == "adjoint":
        state["force"].grad = None
        fields = lbve.force_to_fields(sim, 0, state["force"], case["steps"])
        fields.backward(state["grad"])
        return {"fields": _split([fields.detach()]), "gradient": state["force"].grad}
    if case["kind"] == "transfer":
        lbve.lbve_set_geometry_many(sim.h, ids, None, state["forces"], state["inputs"],
                                    n_nodes=[i.n_nodes for i in state["insts"]])
        sim.step(case["steps"])
        lbve.lbve_fields_many(sim.h, ids, state["ptrs"], False)
        return {"fields": state["out"]}
    sim.step(case["steps"])
    lbve.lbve_fields_many(sim.h, ids, state["ptrs"], True)
    if case["kind"] == "mix":
        return {"fields": state["out"]}
    out = {"fields": _split(_views(state["insts"], state["out"]))}
    if case["kind"] == "channels":
        out["residual"] = np.array([sim.residual(i) for i in ids])
    if case["kind"] == "cylinder":
        out["totals"] = sim.totals(0)
    return out


def work(case):
    """State values, forces and fields that must move, and the floating-point operations."""
    insts = _base(case["kind"], case.get("N", case.get("H", case.get("R", 0))), case.get("nx", 0), case.get("n", 1))
    es = 4 if case["precision"] == "fp32" else 8
    state = force = fields = 0
    for inst in insts:
        state += inst.n_nodes * STATE_VALUES * es
        force += inst.n_nodes * 2 * es if inst.force_field is not None else 0
        fields += inst.n_nodes * 6 * 8
    sweeps = case["steps"] if state + force > ON_CHIP_BYTES else 1
    once = sweeps * (2 * state + force)
    flops = FLOPS_PER_UPDATE * case["steps"] * sum(i.n_nodes for i in insts)
    if case["kind"] == "adjoint":
        # forward, checkpointed forward again, reverse sweep: the adjoint state is as large as the state
        nodes = insts[0].n_nodes
        return {"bytes": 2 * once + sweeps * 2 * state + nodes * (8 * 8 + 2 * 8), "flops": 4 * flops}
    extra = 0
    if case["kind"] == "transfer":
        extra = fields + sum(i.n_nodes * 16 for i in insts if i.force_field is not None)
    return {"bytes": once + fields + extra, "flops": flops}


# ---- the same in plain float64 torch ----------------------------------------------------------------

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


class _Reference:
    """The coupled step (two-relaxation-time regularised hydrodynamic lattice, three conformation
    lattices, flat and masked walls, open columns) on deviations f_i - w_i, g_i - w_i delta."""

    def __init__(self, inst, device):
        self.inst, self.dev = inst, device
        nx, ny, n = inst.nx, inst.ny, inst.n_nodes
        self.n = n
        t = functools.partial(torch.tensor, dtype=torch.float64, device=device)
        ex, ey, w = np.array(EX, float), np.array(EY, float), np.array(W)
        xx, yy, xy = ex * ex - 1 / 3, ey * ey - 1 / 3, ex * ey
        xxy, xyy = ey * xx, ex * yy
        one = np.ones(9)
        self.M = t(np.stack([one, ex, ey, ex * ex, ey * ey, xy, ex * ex * ey, ex * ey * ey]))
        self.B = t((w * np.stack([one, 3 * ex, 3 * ey, 4.5 * xx, 4.5 * yy, 9 * xy, 13.5 * xxy, 13.5 * xyy])).T.copy())
        y, x = np.divmod(np.arange(n), nx)
        self.src = torch.tensor(np.stack([((y - EY[i]) % ny) * nx + (x - EX[i]) % nx for i in range(9)]), device=device)
        Uc = inst.Ma * math.sqrt(1 / 3)
        nu0 = Uc * inst.Lc / inst.Re
        nus, mup = inst.beta * nu0, (1 - inst.beta) * nu0
        ts1 = 3 * nus + 0.5
        tp1 = 3 * nus / inst.Sc + 0.5
        ts2, tp2 = inst.Lambda_s / (ts1 - 0.5) + 0.5, inst.Lambda_p / (tp1 - 0.5) + 0.5
        lam = inst.Wi * inst.Lc / Uc
        self.Uc, self.il, self.mpl = Uc, 1 / lam, mup / lam
        self.cs1, self.cs2, self.hs1, self.ws1 = 1 - 1 / ts1, 1 - 1 / ts2, (ts1 - 0.5) / ts1, 1 / ts1
        self.e1, self.cp2, self.hp1 = (tp1 - 1.0) / tp1, 1 - 1 / tp2, (tp1 - 0.5) / tp1
        self.delta = t([1.0, 0.0, 1.0])[:, None]
        self.solid = inst.solid
        self.fluid = torch.tensor(np.ones(n, bool) if inst.solid is None else inst.solid.reshape(-1) == 0, device=device)
        # difference coefficients and neighbours along each axis
        s = np.zeros((ny, nx), bool) if inst.solid is None else inst.solid != 0
        self.diff = []
        for axis in (0, 1):
            def shift(j, axis=axis):
                X, Y = (x + j, y) if axis == 0 else (x, y + j)
                return (Y % ny) * nx + X % nx
            sp, sm = s.reshape(-1)[shift(1)], s.reshape(-1)[shift(-1)]
            end = (x if axis == 0 else y, nx if axis == 0 else ny)
            closed = inst.open_x if axis == 0 else not inst.periodic_y
            if closed:
                sp, sm = sp | (end[0] == end[1] - 1), sm | (end[0] == 0)
            two_p, two_m = ~s.reshape(-1)[shift(2)], ~s.reshape(-1)[shift(-2)]
            c = np.zeros((5, n))
            for sel, v in ((~sp & ~sm, (0, -0.5, 0, 0.5, 0)), (sp & ~sm & two_m, (0.5, -2, 1.5, 0, 0)),
                           (sp & ~sm & ~two_m, (0, -1, 1, 0, 0)), (sm & ~sp & two_p, (0, 0, -1.5, 2, -0.5)),
                           (sm & ~sp & ~two_p, (0, 0, -1, 1, 0))):
                c[:, sel] = np.array(v, float)[:, None]
            used = [j for j in range(5) if np.any(c[j])]
            self.diff.append([(t(c[j]), torch.tensor(shift(j - 2), device=device)) for j in used])
        self.rows = []
        if not inst.periodic_y:
            self.rows = [(torch.arange(nx, device=device), 1, (2, 5, 6)),
                         (torch.arange(n - nx, n, device=device), -1, (4, 7, 8))]
        # mask wall nodes: per direction the nodes whose neighbour x - e_i is solid
        self.links = []
        if inst.solid is not None:
            sf = s.reshape(-1)
            for i in range(1, 9):
                Y = y - EY[i]
                ok = np.ones(n, bool) if inst.periodic_y else (Y >= 0) & (Y < ny)
                k = np.nonzero(~sf & ok & sf[(Y % ny) * nx + (x - EX[i]) % nx])[0]
                q = np.full(k.size, 0.5) if inst.wall_q is None else inst.wall_q[i].reshape(-1)[k]
                kf = ((y[k] + EY[i]) % ny) * nx + (x[k] + EX[i]) % nx
                self.links.append((i, torch.tensor(k, device=device), t(q), torch.tensor(kf, device=device),
                                   torch.tensor(~sf[kf], device=device)))

    def equilibrium(self, rho0, rho, ux, uy, third):
        z = rho * ux * ux * uy if third else torch.zeros_like(ux * rho)
        v = rho * ux * uy * uy if third else z
        return self.B @ torch.stack([rho0, rho * ux, rho * uy, rho * ux * ux, rho * uy * uy, rho * ux * uy, z, v])

    def start(self, force, init=None):
        n, inst = self.n, self.inst
        if force is None:
            force = torch.tensor([[inst.Fx], [inst.Fy]], dtype=torch.float64, device=self.dev).expand(2, n)
        self.F = force
        if init is None:
            init = torch.tensor([1.0, 0, 0, 1, 0, 1], dtype=torch.float64, device=self.dev)[:, None].expand(6, n)
        u = init[1:3]
        d = torch.stack([self.equilibrium(init[0] - 1, init[0], u[0], u[1], True)] +
                        [self.equilibrium(init[3 + l] - self.delta[l], init[3 + l], u[0], u[1], False) for l in range(3)])
        self.first = True
        self.u_prev = u
        self.fields = init
        return self.collide(d, torch.zeros(5, n, dtype=torch.float64, device=self.dev), self.F)

    def macroscopic(self, d, F):
        m = self.M @ d[0]
        rho = 1 + m[0]
        return m, rho, (m[1] + 0.5 * F[0]) / rho, (m[2] + 0.5 * F[1]) / rho

    def grad(self, axis, q):
        return sum(c * q[..., k] for c, k in self.diff[axis])

    def collide(self, d, hist, F):
        m, rho, ux, uy = self.macroscopic(d, F)
        c = torch.matmul(self.M, d[1:])
        A0 = c[:, 0]
        A = A0 + self.delta
        gx = self.grad(0, torch.stack([ux, uy, rho * ux ** 3]))
        gy = self.grad(1, torch.stack([ux, uy, rho * uy ** 3]))
        div = gx[0] + gy[1]
        S = torch.stack([2 * (A[0] * gx[0] + A[1] * gy[0]), A[0] * gx[1] + A[1] * gy[1] + A[1] * gx[0] + A[2] * gy[0],
                         2 * (A[1] * gx[1] + A[2] * gy[1])]) - A0 * self.il + A * div
        So, uo = (S, (ux, uy)) if self.first else (hist[:3], hist[3:])
        self.first = False
        self.fields = torch.cat([torch.stack([rho, ux, uy]), A])
        cs2 = 1 / 3
        ruu = (rho * ux * ux, rho * uy * uy, rho * ux * uy)
        t = self.mpl * A0
        post = [self.B @ torch.stack([
            m[0], m[1] + F[0], m[2] + F[1],
            ruu[0] + self.cs1 * (m[3] - cs2 * m[0] - ruu[0]) - self.hs1 * gx[2] - self.ws1 * t[0],
            ruu[1] + self.cs1 * (m[4] - cs2 * m[0] - ruu[1]) - self.hs1 * gy[2] - self.ws1 * t[2],
            ruu[2] + self.cs1 * (m[5] - ruu[2]) - self.ws1 * t[1],
            ruu[0] * uy + self.cs2 * (m[6] - cs2 * m[2] - ruu[0] * uy),
            ruu[1] * ux + self.cs2 * (m[7] - cs2 * m[1] - ruu[1] * ux)])]
        z = torch.zeros_like(rho)
        for l in range(3):
            flux = [self.hp1 * (A[l] / rho * F[a] + u * S[l] + 0.5 * (u * S[l] - uo[a] * So[l]))
                    for a, u in ((0, ux), (1, uy))]
            post.append(self.B @ torch.stack([
                A0[l] + 1.5 * S[l] - 0.5 * So[l],
                A[l] * ux + self.e1 * (c[l, 1] - A[l] * ux) + flux[0],
                A[l] * uy + self.e1 * (c[l, 2] - A[l] * uy) + flux[1],
                A[l] * ux * ux + self.cp2 * (c[l, 3] - cs2 * A0[l] - A[l] * ux * ux),
                A[l] * uy * uy + self.cp2 * (c[l, 4] - cs2 * A0[l] - A[l] * uy * uy),
                A[l] * ux * uy + self.cp2 * (c[l, 5] - A[l] * ux * uy), z, z]))
        return torch.stack(post), torch.cat([S, torch.stack([ux, uy])])

    def complete_cnebb(self, p, post, k, unknown, ux, uy):
        """Conservative completion of the conformation lattices at nodes k (unknown: [9, m] bool)."""
        own = torch.stack([post[1:, OPP[i], k] for i in range(9)], 1)
        g = p[1:, :, k]
        have = torch.where(unknown, own, g)
        total = have.sum(1)
        phi = total + self.delta
        new = [None] * 9
        for i in range(1, 9):
            new[i] = torch.where(unknown[i], g[:, OPP[i]] + 6 * W[i] * phi * (EX[i] * ux + EY[i] * uy), g[:, i])
        new[0] = total - sum(new[1:])
        p[1:, :, k] = torch.stack(new, 1)
        weights = torch.tensor(W, dtype=torch.float64, device=self.dev)[:, None]
        full = lambda v: torch.where(unknown, v + weights * self.delta[:, None], torch.zeros_like(v)).sum((1, 2))  # noqa: E731
        self.wall[0] += full(p[1:, :, k]) + (new[0] - g[:, 0]).sum(1)
        self.wall[1] += full(own)

    def step(self, post, hist, F):
        inst, n = self.inst, self.n
        p = torch.gather(post, 2, self.src.expand(4, 9, n))
        self.wall = torch.zeros(2, 3, dtype=torch.float64, device=self.dev)
        self.drag = torch.zeros(2, dtype=torch.float64, device=self.dev)
        for k, side, unknown in self.rows:
            if inst.open_x:
                k = k[1:-1]
            self.row(p, post, k, side, unknown, F)
        if self.solid is not None:
            nodes = torch.unique(torch.cat([k for _, k, *_ in self.links]))
            at = torch.full((n,), -1, dtype=torch.long, device=self.dev)
            at[nodes] = torch.arange(nodes.numel(), device=self.dev)
            unknown = torch.zeros(9, nodes.numel(), dtype=torch.bool, device=self.dev)
            for i, k, q, kf, fluid in self.links:
                toward, same, nxt = post[0, OPP[i], k], post[0, i, k], post[0, OPP[i], kf]
                nxt = torch.where(fluid, nxt, toward)
                v = torch.where(q < 0.5, 2 * q * toward + (1 - 2 * q) * nxt, toward / (2 * q) + (1 - 1 / (2 * q)) * same)
                p[0, i, k] = v
                unknown[i, at[k]] = True
                total = (2 * W[i] + toward + v).sum()
                self.drag -= torch.stack([EX[i] * total, EY[i] * total])
            _, _, ux, uy = self.macroscopic(p[:, :, nodes], F[:, nodes])
            self.complete_cnebb(p, post, nodes, unknown, ux, uy)
        if inst.open_x:
            self.columns(p, F)
        p = torch.where(self.fluid, p, torch.zeros_like(p))
        return self.collide(p, hist, F)

    def row(self, p, post, k, side, unknown, F):
        a, b, c = unknown
        h = 0.5 * (p[0, 1, k] - p[0, 3, k])
        qx, qy = 0.25 * F[0, k], 0.25 * F[1, k]
        if side > 0:
            p[0, 2, k] = p[0, 4, k]
            p[0, 5, k] = p[0, 7, k] - h - qx - qy
            p[0, 6, k] = p[0, 8, k] + h + qx - qy
        else:
            p[0, 4, k] = p[0, 2, k]
            p[0, 7, k] = p[0, 5, k] + h + qx + qy
            p[0, 8, k] = p[0, 6, k] - h - qx + qy
        _, _, ux, uy = self.macroscopic(p[:, :, k], F[:, k])
        mask = torch.zeros(9, k.numel(), dtype=torch.bool, device=self.dev)
        mask[[a, b, c]] = True
        self.complete_cnebb(p, post, k, mask, ux, uy)

    def columns(self, p, F):
        """Non-equilibrium extrapolation into the inlet and outlet columns."""
        nx, ny = self.inst.nx, self.inst.ny
        y = torch.arange(ny, device=self.dev)
        inlet = torch.tensor(self.inst.inlet, dtype=torch.float64, device=self.dev)
        for side in (0, 1):
            k, kf = y * nx + (nx - 1 if side else 0), y * nx + (nx - 2 if side else 1)
            f = p[:, :, kf]
            _, rho, ux, uy = self.macroscopic(f, F[:, kf])
            if side == 0:
                bx, by = inlet[0], inlet[1]
                e = self.equilibrium(rho - 1, rho, bx, by, True) - self.equilibrium(rho - 1, rho, ux, uy, True)
                p[0, :, k] = f[0] + e
                for l in range(3):
                    phi, phib = f[1 + l].sum(0) + self.delta[l], inlet[2 + l]
                    p[1 + l, :, k] = f[1 + l] + (self.equilibrium(phib - self.delta[l], phib, bx, by, False) -
                                                 self.equilibrium(phi - self.delta[l], phi, ux, uy, False))
            else:
                one = torch.ones_like(rho)
                p[0, :, k] = f[0] + (self.equilibrium(one - 1, one, ux, uy, True) -
                                     self.equilibrium(rho - 1, rho, ux, uy, True))
                p[1:, :, k] = f[1:]

    def advance(self, steps, force=None, init=None):
        """Fields after `steps` steps, [6, n]; the residual and wall sums of the last stay in self."""
        post, hist = self.start(force, init)
        u0 = self.fields[1:3]
        for _ in range(steps):
            post, hist = self.step(post, hist, self.F)
        fields = torch.where(self.fluid, self.fields, torch.zeros_like(self.fields))
        self.residual = float((self.fields[1:3] - u0)[:, self.fluid].abs().max() / self.Uc)
        return fields


def _flat(a, device):
    return None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(device).reshape(a.shape[0], -1)


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    insts = _instances(case, seed)
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, insts[0], seed, device)
    with torch.no_grad():
        parts, residuals = [], []
        for i, inst in enumerate(insts):
            ref = _Reference(inst, device)
            init = None
            if case["kind"] == "transfer":
                init = _flat(_initial_fields(inst, i, seed), device)
            elif case["kind"] == "cylinder":
                init = _flat(_developed(inst), device)
            parts.append(ref.advance(case["steps"], _flat(inst.force_field, device), init).reshape(-1))
            residuals.append(ref.residual)
        flat = torch.cat(parts)
        if case["kind"] in ("mix", "transfer"):
            return {"fields": flat.cpu() if case["kind"] == "transfer" else flat}
        out = {"fields": _split(_views(insts, flat))}
        if case["kind"] == "channels":
            out["residual"] = np.array(residuals)
        if case["kind"] == "cylinder":
            rho, ux, uy, a, b, c = (v[ref.fluid] for v in parts[0].view(6, -1))
            sums = torch.stack([v.sum() for v in (rho, rho * ux, rho * uy, a, b, c)])
            out["totals"] = torch.cat([sums, ref.wall[0], ref.wall[1], ref.drag]).cpu().numpy()
    return out


def _exact_adjoint(case, inst, seed, device):
    from torch.utils.checkpoint import checkpoint
    ref = _Reference(inst, device)
    rng = np.random.default_rng([seed, 1])
    g = np.zeros((6, inst.ny, inst.nx))
    g[1:3] = rng.standard_normal((2, inst.ny, inst.nx))
    g[3:] = 1e-6 * rng.standard_normal((3, inst.ny, inst.nx))
    force = _flat(inst.force_field, device).requires_grad_(True)
    post, hist = ref.start(force)
    fields = None

    def one(post, hist, F):
        post, hist = ref.step(post, hist, F)
        return post, hist, ref.fields

    for _ in range(case["steps"]):
        post, hist, fields = checkpoint(one, post, hist, force, use_reentrant=False)
    fields.backward(_flat(g, device))
    shape = (inst.ny, inst.nx)
    return {"fields": _split([fields.detach().reshape(6, *shape)]), "gradient": force.grad.reshape(2, *shape)}
