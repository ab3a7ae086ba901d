"""The work that users of this library have it do, as cases to be timed.

Every case goes through the public entry points: ``Lattice`` (one lattice, one
context), ``Batch`` (many lattices per launch, its populations read through the
C entry point with a device pointer) and ``CdWindow`` (the differentiable drag
window).  Kernels are chosen by the library (no tuning calls), as in a program
that does not tune.

Lattice units throughout: dh = dt = 1, density 1, inflow speed 0.05 (0.02 in
the 40D x 40D domain).  Flows start impulsively from a uniform stream with
seeded Gaussian noise of 1e-4 on both velocity components.
"""
import math
import random

import numpy as np
import torch

from paper_1806_09403_gb300 import btdf as B
from paper_1806_09403_gb300.autograd import CdWindow, DragWindow

STORAGE = {"f32": B.BTDF_F32, "f16": B.BTDF_F16DEV, "bf16": B.BTDF_BF16DEV}
BCX = {"periodic": B.BTDF_BCX_PERIODIC, "inout": B.BTDF_BCX_INOUT, "convective": B.BTDF_BCX_CONVECTIVE}
BCY = {"periodic": B.BTDF_BCY_PERIODIC, "freeslip": B.BTDF_BCY_FREESLIP, "noslip": B.BTDF_BCY_NOSLIP}
LAYOUT = {"rows": B.LAYOUT_ROWS, "planes": B.LAYOUT_PLANES}

# One lattice advanced by `steps` steps: the base of the single-lattice cases.
SINGLE = {"kind": "single", "nx": 0, "ny": 0, "storage": "f32", "delta": 3, "nf": 1, "bcx": "inout", "bcy": "freeslip",
          "layout": "rows", "tau": 0.53, "u": 0.05, "gx": 0.0, "bodies": 1, "D": 20.0, "cx": 0.25, "cy": 0.5, "steps": 100}


def _tau(re, d, u=0.05):
    return 0.5 + 3.0 * u * d / re


def listed():
    return [
        # The validation cylinder at Re = 40 (4-point cosine delta), 1000 steps: the short runs that
        # parameter studies and parity checks are made of.  Every launch counts.
        dict(SINGLE, name="cyl-160x80-f32", nx=160, ny=80, delta=5, tau=_tau(40, 16), D=16.0, cy=0.5, steps=1000),
        # An oscillating cylinder driven from the host: new marker velocities, one step and the
        # force on the body back on the host, every step (control, fluid-structure coupling).
        dict(SINGLE, name="control-320x160-f32", kind="control", nx=320, ny=160, tau=_tau(100, 20), steps=32),
        # The headline cylinder, 1600 x 800 at Re = 200, stepped between two read-outs; also with FP16 storage.
        dict(SINGLE, name="cyl-1600x800-f32", nx=1600, ny=800, tau=_tau(200, 40), D=40.0, steps=200),
        dict(SINGLE, name="cyl-1600x800-f16", nx=1600, ny=800, tau=_tau(200, 40), D=40.0, steps=200, storage="f16"),
        # The paper's 40D x 40D domain (odd sizes) with the convective outlet, in BF16 storage: the
        # long runs that give Strouhal number and mean drag.
        dict(SINGLE, name="domain-1601x1601-bf16", nx=1601, ny=1601, tau=_tau(200, 40, 0.02), u=0.02, D=40.0, cx=0.45,
             bcx="convective", storage="bf16", steps=100),
        # A body-force-driven no-slip channel with four bodies, three forcing passes per step (MDF)
        # and the 4-point delta; ragged sizes.
        dict(SINGLE, name="channel-mdf-1201x401-f32", nx=1201, ny=401, tau=0.6, u=0.02, gx=1e-7, delta=4, nf=3, bodies=4,
             bcx="periodic", bcy="noslip", steps=100),
        # Many bodies on a lattice far beyond L2 (8192 x 4096, 400 cylinders), FP32 and FP16 storage.
        dict(SINGLE, name="cyl-8192x4096-f32", nx=8192, ny=4096, tau=_tau(200, 20), bodies=400, steps=50),
        dict(SINGLE, name="cyl-8192x4096-f16", nx=8192, ny=4096, tau=_tau(200, 20), bodies=400, steps=50, storage="f16"),
        # Many independent cylinders of uneven lattice sizes per launch (sweeps over Re and D): a
        # large FP32 batch and a small FP16 one.
        {"name": "batch-128-f32", "kind": "batch", "count": 128, "mix": 7, "kmin": 8, "kmax": 64, "storage": "f32", "delta": 3,
         "layout": "rows", "steps": 100},
        {"name": "batch-24-f16", "kind": "batch", "count": 24, "mix": 7, "kmin": 8, "kmax": 32, "storage": "f16", "delta": 3,
         "layout": "rows", "steps": 100},
        # The gradient of the window-averaged drag with respect to the inflow speed and every marker's
        # radial offset, 800 x 400 at Re = 100: one evaluation and its backward pass in an optimization.
        {"name": "adjoint-800x400", "kind": "adjoint", "nx": 800, "ny": 400, "delta": 3, "tau": _tau(100, 24), "u": 0.05,
         "D": 24.0, "steps": 500, "every": 50},
    ]


def draw(rng):
    kind = rng.choice(["single", "single", "single", "single", "control", "batch", "adjoint"])
    if kind == "batch":
        kmin = rng.randint(8, 24)
        return {"kind": "batch", "count": int(round(math.exp(rng.uniform(math.log(4), math.log(128))))), "mix": rng.randint(1, 999),
                "kmin": kmin, "kmax": rng.randint(kmin + 1, 64), "storage": rng.choice(["f32", "f32", "f16", "bf16"]),
                "delta": rng.choice([3, 4]), "layout": rng.choice(["rows", "rows", "planes"]), "steps": rng.randint(33, 100)}
    if kind == "adjoint":
        ny = int(round(math.exp(rng.uniform(math.log(96), math.log(400)))))
        d = rng.uniform(12.0, min(24.0, ny / 6.0))
        return {"kind": "adjoint", "nx": 2 * ny + rng.randint(-17, 0), "ny": ny, "delta": rng.choice([3, 4, 5]),
                "tau": max(0.53, _tau(rng.uniform(40, 120), d)), "u": 0.05, "D": round(d, 2), "steps": rng.randint(60, 300),
                "every": rng.choice([20, 50, 64])}
    top = 320 * 160 * 4 if kind == "control" else 8192 * 4096
    nodes = math.exp(rng.uniform(math.log(160 * 80), math.log(top)))
    ny = max(72, int(round(math.sqrt(nodes / rng.choice([1.0, 2.0, 2.0, 3.0])))))
    nx = min(8192, max(ny, int(round(nodes / ny))))
    d = rng.uniform(10.0, min(40.0, ny / 6.0))
    bcx = rng.choice(["inout", "inout", "inout", "convective", "periodic"])
    c = dict(SINGLE, kind=kind, nx=nx, ny=ny, storage=rng.choice(["f32", "f32", "f16", "bf16"]), delta=rng.choice([3, 3, 4, 5]),
             nf=rng.choice([1, 1, 1, 1, 2]), bcx=bcx, bcy=rng.choice(["freeslip", "freeslip", "noslip", "periodic"]),
             layout=rng.choice(["rows", "rows", "rows", "planes"]), tau=max(0.53, _tau(math.exp(rng.uniform(0.0, math.log(200))), d)),
             gx=1e-7 if bcx == "periodic" else 0.0, D=round(d, 2), cx=rng.uniform(0.25, 0.5), cy=rng.uniform(0.4, 0.6),
             bodies=1 if nx * ny < 200_000 or kind == "control" else max(1, min(400, int(nx * ny / (30 * d) ** 2))),
             steps=rng.randint(16, 32) if kind == "control" else max(20, min(1000, int(1.2e9 / (nx * ny)))))
    return c


# ---- inputs ---------------------------------------------------------------------------------

def _circle(cx, cy, d, n):
    th = 2.0 * np.pi * np.arange(n) / n
    return cx + 0.5 * d * np.cos(th), cy + 0.5 * d * np.sin(th)


def _bodies(c, seed):
    """Centres: one body at (cx nx, cy ny); several on a jittered grid of cells, clear of the boundaries."""
    nx, ny, d, nb = c["nx"], c["ny"], c["D"], c["bodies"]
    rng = np.random.default_rng(seed)
    if nb == 1:
        at = [(c["cx"] * nx + rng.uniform(-0.5, 0.5), c["cy"] * ny + rng.uniform(-0.5, 0.5))]
    else:
        w, h = nx - 6.0 * d, ny - 4.0 * d
        cols = max(1, min(nb, int(round(math.sqrt(nb * w / h)))))
        rows = -(-nb // cols)
        sx, sy = w / cols, h / rows
        jx, jy = max(0.0, 0.5 * sx - d), max(0.0, 0.5 * sy - d)
        at = [(3.5 * d + (k % cols + 0.5) * sx + rng.uniform(-jx, jx), 2.0 * d + (k // cols + 0.5) * sy + rng.uniform(-jy, jy))
              for k in range(nb)]
    n = max(8, int(round(math.pi * d)))
    return [_circle(x, y, d, n) for x, y in at], math.pi * d / n


def _fields(nx, ny, u, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = 1e-4 * torch.randn((2, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    return np.ones((ny, nx)), (u + noise[0]).cpu().numpy(), noise[1].cpu().numpy()


class _BatchCase:
    """One lattice of a batch, with the attributes that ``Batch`` reads."""

    def __init__(self, nx, ny, tau, delta, seed):
        self.nx, self.ny, self.tau, self.u_in, self.delta, self.nf = nx, ny, tau, 0.05, delta, 1
        self.bc_x, self.bc_y, self.gx, self.gy, self.drs, self.seed = B.BTDF_BCX_INOUT, B.BTDF_BCY_FREESLIP, 0.0, 0.0, 0.0, seed


def _batch_cases(c, seed):
    """nx = 16 k with k uniform in kmin..kmax, ny = nx / 2, D uniform in [10, min(40, ny / 5)], Re from {0.1, 40, 200}."""
    rng = np.random.default_rng([c["mix"], 3])   # sizes and flows belong to the case, the noise to the seed
    out = []
    for i in range(c["count"]):
        nx = 16 * int(rng.integers(c["kmin"], c["kmax"] + 1))
        ny = nx // 2
        d = float(rng.uniform(10.0, min(40.0, ny / 5.0)))
        k = _BatchCase(nx, ny, max(0.53, _tau(float(rng.choice([0.1, 40.0, 200.0])), d)), c["delta"], seed * 1009 + i)
        n = max(8, int(round(math.pi * d)))
        k.markers, k.ds = _circle(nx / 4.0 + 0.31, ny / 2.0 + 0.17, d, n), math.pi * d / n
        out.append(k)
    return out


def _offsets(c, seed):
    """Inflow speed and radial offsets of the differentiated window, in single precision as optimizers keep them."""
    rng = np.random.default_rng([seed, 5])
    n = max(8, int(round(math.pi * c["D"])))
    return np.float32(c["u"] * (1.0 + 0.02 * rng.uniform(-1, 1))), rng.uniform(-0.05, 0.05, n).astype(np.float32)


def _velocity(c, k, n):
    """Marker velocity of the oscillating cylinder in step k."""
    return np.zeros(n), np.full(n, 0.01 * math.sin(2.0 * math.pi * k / 400.0))


def prepare(case, seed):
    c = case
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "batch":
        cases = _batch_cases(c, seed)
        bt = B.Batch(cases, storage=STORAGE[c["storage"]], history_len=1024, stream=stream, layout=LAYOUT[c["layout"]])
        for i, k in enumerate(cases):
            bt.init_fields(i, *_fields(k.nx, k.ny, k.u_in, k.seed))
            bt.add_markers(i, *k.markers, k.ds)
        pops = [torch.empty((9, k.ny, k.nx), device="cuda") for k in cases]
        return {"case": c, "batch": bt, "pops": pops}
    if c["kind"] == "adjoint":
        n = max(8, int(round(math.pi * c["D"])))
        cx, cy = 0.25 * c["nx"], 0.5 * c["ny"]
        lat = B.Lattice(c["nx"], c["ny"], c["tau"], c["u"], c["delta"], bc_x=B.BTDF_BCX_INOUT, bc_y=B.BTDF_BCY_FREESLIP,
                        history_len=1024, stream=stream)
        lat.init_fields(*_fields(c["nx"], c["ny"], c["u"], seed))
        lat.add_markers(*_circle(cx, cy, c["D"], n), math.pi * c["D"] / n)
        u, dr = _offsets(c, seed)
        return {"case": c, "window": DragWindow.for_lattice(lat, cx, cy, 0.5 * c["D"], c["steps"], every=c["every"], dref=c["D"]),
                "u": torch.tensor(u, device="cuda", requires_grad=True), "dr": torch.tensor(dr, device="cuda", requires_grad=True)}
    lat = B.Lattice(c["nx"], c["ny"], c["tau"], c["u"], c["delta"], c["nf"], STORAGE[c["storage"]], BCX[c["bcx"]], BCY[c["bcy"]],
                    gx=c["gx"], history_len=4096, stream=stream, layout=LAYOUT[c["layout"]])
    lat.init_fields(*_fields(c["nx"], c["ny"], c["u"], seed))
    bodies, ds = _bodies(c, seed)
    for X, Y in bodies:
        lat.add_markers(X, Y, ds)
    return {"case": c, "lattice": lat, "pops": torch.empty((9, c["ny"], c["nx"]), device="cuda")}


def run(state):
    c = state["case"]
    n = c["steps"]
    if c["kind"] == "batch":
        bt = state["batch"]
        bt.step(n)
        first = bt.steps - n
        forces = [bt.forces(b, first, n) for b in range(c["count"])]
        for i, t in enumerate(state["pops"]):
            bt._check(B.lib().btdf_batch_read_field(bt._b, i, B.FIELD_POPS, t.data_ptr(), 1), "btdf_batch_read_field")
        return {"forces": np.array(forces), "pops": torch.cat([t.view(-1) for t in state["pops"]])}
    if c["kind"] == "adjoint":
        u, dr = state["u"], state["dr"]
        u.grad = dr.grad = None
        J = CdWindow.apply(u, dr, state["window"])
        J.backward()
        return {"J": J.detach(), "dU": u.grad, "ddr": dr.grad}
    lat = state["lattice"]
    if c["kind"] == "control":
        m = lat.marker_count
        forces = []
        for _ in range(n):
            lat.set_marker_velocity(-1, *_velocity(c, lat.steps, m))
            lat.step(1)
            forces.append(lat.forces(-1, lat.steps - 1, 1))
        forces = np.concatenate(forces, axis=1)
    else:
        lat.step(n)
        forces = np.array(lat.forces(-1, lat.steps - n, n))
    lat.field_to_device(B.FIELD_POPS, state["pops"].data_ptr())
    return {"forces": forces, "pops": state["pops"]}


def work(case):
    """The state is read once and written once (populations of the storage type) and read out once
    in single precision; 120 operations per node and step.  The window also writes and reads one
    state per step (its reverse sweep needs every state), with about four times the operations."""
    c = case
    if c["kind"] == "batch":
        nodes = sum(k.nx * k.ny for k in _batch_cases(c, 0))
    else:
        nodes = c["nx"] * c["ny"]
    if c["kind"] == "adjoint":
        return {"bytes": 72.0 * nodes * c["steps"], "flops": 480.0 * nodes * c["steps"]}
    elem = 4 if c["storage"] == "f32" else 2
    return {"bytes": (18.0 * elem + 36.0) * nodes, "flops": 120.0 * nodes * c["steps"]}


# ---- the same in 64 bits ----------------------------------------------------------------------

EX, EY = [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]
WT = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
MIRROR, OPPOSITE = [0, 1, 4, 3, 2, 8, 7, 6, 5], [0, 3, 4, 1, 2, 7, 8, 5, 6]
WIDTH, SHELL = {3: 3, 4: 4, 5: 4}, {3: 1.9, 4: 2.6, 5: 2.6}


def _delta(kind, r):
    a = r.abs()
    if kind == 5:
        return torch.where(a < 2.0, 0.25 * (1.0 + torch.cos(0.5 * math.pi * a)), torch.zeros_like(a))
    # each branch on arguments clamped to its own range, so that both stay differentiable
    if kind == 3:
        lo, hi = a.clamp(max=0.5), a.clamp(0.5, 1.5)
        inner = (1.0 + torch.sqrt(1.0 - 3.0 * lo * lo)) / 3.0
        outer = (5.0 - 3.0 * hi - torch.sqrt(1.0 - 3.0 * (1.0 - hi) ** 2)) / 6.0
        return torch.where(a <= 0.5, inner, torch.where(a < 1.5, outer, torch.zeros_like(a)))
    lo, hi = a.clamp(max=1.0), a.clamp(1.0, 2.0)
    inner = (3.0 - 2.0 * lo + torch.sqrt(1.0 + 4.0 * lo - 4.0 * lo * lo)) / 8.0
    outer = (5.0 - 2.0 * hi - torch.sqrt(-7.0 + 12.0 * hi - 4.0 * hi * hi)) / 8.0
    return torch.where(a < 1.0, inner, torch.where(a < 2.0, outer, torch.zeros_like(a)))


class _Flow:
    """Algorithm 1 of the method on one lattice, in FP64 tensor operations."""

    def __init__(self, nx, ny, tau, u, delta, nf, bcx, bcy, gx, X, Y, ds):
        t = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")  # noqa: E731
        self.nx, self.ny, self.tau, self.u, self.delta, self.nf = nx, ny, tau, u, delta, nf
        self.bcx, self.bcy, self.gx, self.ds, self.drs = bcx, bcy, gx, ds, SHELL[delta]
        self.ex, self.ey, self.w = t(EX).view(9, 1, 1), t(EY).view(9, 1, 1), t(WT).view(9, 1, 1)
        self.mom = t([[1.0] * 9, [float(v) for v in EX], [float(v) for v in EY]])
        self.place(X, Y)

    def place(self, X, Y):
        S = WIDTH[self.delta]
        k = torch.arange(S, device="cuda")
        i = torch.floor(X.detach() - 0.5 * S).long()[:, None] + 1 + k
        j = torch.floor(Y.detach() - 0.5 * S).long()[:, None] + 1 + k
        wx, wy = _delta(self.delta, i - X[:, None]), _delta(self.delta, j - Y[:, None])
        self.W = (wy[:, :, None] * wx[:, None, :]).flatten(1)
        self.node = ((j % self.ny)[:, :, None] * self.nx + (i % self.nx)[:, None, :]).flatten(1)

    def equilibrium(self, rho, ux, uy):
        eu = self.ex * ux + self.ey * uy
        return self.w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))

    def step(self, f, ubx=0.0, uby=0.0):
        """Post-streaming populations one step on, and the Lagrangian forces of the step."""
        m = (self.mom @ f.flatten(1)).view(3, self.ny, self.nx)
        rho = m[0]
        ux, uy = m[1] / rho, m[2] / rho
        W, node = self.W, self.node
        rl = (W * rho.flatten()[node]).sum(1)
        zero = torch.zeros(self.ny * self.nx, dtype=torch.float64, device="cuda")
        Fx = Fy = 0.0
        fx = fy = zero
        vx, vy = ux.flatten(), uy.flatten()
        for _ in range(self.nf):
            Fx = Fx + 2.0 * rl * (ubx - (W * vx[node]).sum(1))
            Fy = Fy + 2.0 * rl * (uby - (W * vy[node]).sum(1))
            c = W * (self.ds * self.drs)
            fx = zero.index_add(0, node.flatten(), (c * Fx[:, None]).flatten())
            fy = zero.index_add(0, node.flatten(), (c * Fy[:, None]).flatten())
            vx, vy = ux.flatten() + 0.5 * fx / rho.flatten(), uy.flatten() + 0.5 * fy / rho.flatten()
        fx, fy = fx.view_as(rho) + self.gx, fy.view_as(rho)
        ux, uy = ux + 0.5 * fx / rho, uy + 0.5 * fy / rho
        eu, eF = self.ex * ux + self.ey * uy, self.ex * fx + self.ey * fy
        guo = (1.0 - 0.5 / self.tau) * self.w * (3.0 * (eF - (ux * fx + uy * fy)) + 9.0 * eu * eF)
        g = f + (self.equilibrium(rho, ux, uy) - f) / self.tau + guo
        n = []
        for a in range(9):
            s = torch.roll(g[a], (EY[a], EX[a]), (0, 1))
            if EY[a] and self.bcy != "periodic":
                y = 0 if EY[a] > 0 else self.ny - 1
                row = torch.roll(g[MIRROR[a]][y], EX[a], 0) if self.bcy == "freeslip" else g[OPPOSITE[a]][y]
                s = torch.cat([row[None], s[1:]]) if y == 0 else torch.cat([s[:-1], row[None]])
            n.append(s)
        n = torch.stack(n)
        if self.bcx != "periodic":
            f1 = n[:, :, 1:2]
            r1 = f1.sum(0)
            u1, v1 = (self.ex * f1).sum(0) / r1, (self.ey * f1).sum(0) / r1
            inlet = f1 + self.equilibrium(r1, self.u + 0.0 * r1, 0.0 * r1) - self.equilibrium(r1, u1, v1)
            out = n[:, :, -2:-1]
            if self.bcx == "convective":
                out = (f[:, :, -1:] + self.u * out) / (1.0 + self.u)
            n = torch.cat([inlet, n[:, :, 1:-1], out], 2)
        return n, Fx, Fy


def _start(flow, c, seed):
    rho, ux, uy = (torch.from_numpy(v).cuda() for v in _fields(flow.nx, flow.ny, c["u"], seed))
    return flow.equilibrium(rho, ux, uy)


def _exact_single(c, seed):
    bodies, ds = _bodies(c, seed)
    X, Y = (torch.tensor(np.concatenate([b[k] for b in bodies]), device="cuda") for k in (0, 1))
    flow = _Flow(c["nx"], c["ny"], c["tau"], c["u"], c["delta"], c["nf"], c["bcx"], c["bcy"], c["gx"], X, Y, ds)
    f = _start(flow, c, seed)
    nb, hist = len(bodies), []
    for k in range(c["steps"]):
        vb = float(_velocity(c, k, 1)[1][0]) if c["kind"] == "control" else 0.0
        f, Fx, Fy = flow.step(f, 0.0, vb)
        hist.append(torch.stack([Fx.view(nb, -1).sum(1), Fy.view(nb, -1).sum(1)]) * (-ds * flow.drs))
    return {"forces": torch.stack(hist).transpose(0, 1).contiguous(), "pops": f}


def _exact_batch(c, seed):
    forces, pops = [], []
    for k in _batch_cases(c, seed):
        X, Y = (torch.tensor(v, device="cuda") for v in k.markers)
        flow = _Flow(k.nx, k.ny, k.tau, k.u_in, k.delta, 1, "inout", "freeslip", 0.0, X, Y, k.ds)
        f = _start(flow, {"u": k.u_in}, k.seed)
        hist = []
        for _ in range(c["steps"]):
            f, Fx, Fy = flow.step(f)
            hist.append(torch.stack([Fx.sum(), Fy.sum()]) * (-k.ds * flow.drs))
        forces.append(torch.stack(hist).T)
        pops.append(f.flatten())
    return {"forces": torch.stack(forces), "pops": torch.cat(pops)}


def _exact_adjoint(c, seed):
    from torch.utils.checkpoint import checkpoint
    u0, dr0 = _offsets(c, seed)
    n = len(dr0)
    U = torch.tensor(float(u0), dtype=torch.float64, device="cuda", requires_grad=True)
    dr = torch.tensor(dr0.astype(np.float64), device="cuda", requires_grad=True)
    th = torch.tensor(2.0 * np.pi * np.arange(n) / n, device="cuda")
    r = 0.5 * c["D"] + dr
    X, Y = 0.25 * c["nx"] + r * torch.cos(th), 0.5 * c["ny"] + r * torch.sin(th)
    ds = math.pi * c["D"] / n
    flow = _Flow(c["nx"], c["ny"], c["tau"], c["u"], c["delta"], 1, "inout", "freeslip", 0.0, X, Y, ds)
    f = _start(flow, c, seed).detach()
    flow.u = U

    def segment(f, W, U, k):
        flow.W, flow.u = W, U
        total = 0.0
        for _ in range(k):
            f, Fx, _ = flow.step(f)
            total = total + Fx.sum()
        return f, total

    W, total, k = flow.W, 0.0, 0
    while k < c["steps"]:
        m = min(10, c["steps"] - k)
        f, part = checkpoint(segment, f, W, U, m, use_reentrant=False)
        total = total + part
        k += m
    J = -total * (ds * flow.drs) / (0.5 * U * U * c["D"] * c["steps"])
    J.backward()
    return {"J": J.detach(), "dU": U.grad, "ddr": dr.grad}


def exact(case, seed):
    if case["kind"] == "adjoint":
        return _exact_adjoint(case, seed)
    with torch.no_grad():
        if case["kind"] == "batch":
            return _exact_batch(case, seed) if case["count"] <= 32 else None
        return _exact_single(case, seed)


if __name__ == "__main__":
    print([c["name"] for c in listed()], [draw(random.Random(s)) for s in range(3)])
