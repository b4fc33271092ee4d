"""Workloads whose speed matters to users of the library, each through its public calls.

A case is one pass of a user's program: a number of coupled steps and the read-out that
follows them, a batched launch, or one gradient. The flows, capsules and parameters are
those of ``paper_1903_03356_gb300.workloads`` (the paper's set-ups), so a case only holds
sizes, the scheme, the storage type and the step count.

  single      one capsule in shear, body-force Poiseuille flow or the open channel. The
              capsule is put back on its start (``set_capsule_positions``) before every
              pass, as a program does that runs many starts through one developed flow
              (so it never reaches an outlet, however many passes are made).
  suspension  many biconcave capsules in a channel, stepped on from pass to pass.
  dense       a packed suspension with the capsule-capsule repulsion, put back likewise.
  rigid       the suspension's shapes as rigid particles.
  lattice     the flow alone (developing a flow before capsules are added).
  batch       many independent small shear cases in one persistent launch.
  adjoint     J = D(T) and its gradient in the membrane constants and the body force.

Outputs are the populations (the zero-copy view, in the storage type) and the capsules'
positions and velocities, or their observables where there are many; what the library
computes in single precision is handed on in single precision. The last forces are left
out: in single precision they are small differences of rounded pressures.

``exact`` steps the same problem in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_1903_03356_gb300 import lbmib as L
from paper_1903_03356_gb300 import workloads as W

SCHEMES = {"kinematic": W.KINEMATIC, "dynamic": W.DYNAMIC}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2}
REPULSION_RANGE = 2.0


def listed():
    return [
        # the smallest calls: a program that reads the capsule every few steps (a controller,
        # a plot) on the 100 x 100 shear box, in the binding's default storage
        {"name": "shear_100_fp64", "kind": "shear", "nx": 100, "ny": 100, "radius": 10.0, "n": 64,
         "scheme": "kinematic", "storage": "fp64", "steps": 10},
        # the inertial capsule of the 600 x 120 channel, read every 200 of its 20000 steps
        {"name": "poiseuille_600x120", "kind": "poiseuille", "nx": 600, "ny": 120, "radius": 12.0, "n": 96,
         "scheme": "dynamic", "storage": "fp32", "steps": 200},
        # the paper's open channel: large finely resolved capsule (586 vertices), inlet and outlet
        {"name": "open_360x120", "kind": "open", "nx": 360, "ny": 120, "diameter": 56.0, "scheme": "dynamic",
         "storage": "fp32", "steps": 100},
        # the precision workload, 256 capsules, in both precisions people compare
        {"name": "suspension_4096x512", "kind": "suspension", "nx": 4096, "ny": 512, "count": 256, "n": 128,
         "scheme": "dynamic", "storage": "fp32", "steps": 100},
        {"name": "suspension_4096x512_fp64", "kind": "suspension", "nx": 4096, "ny": 512, "count": 256, "n": 128,
         "scheme": "dynamic", "storage": "fp64", "steps": 20},
        # FP16 storage and the Kinematic scheme, as a long run with halved traffic uses them
        {"name": "suspension_2048x1024_fp16", "kind": "suspension", "nx": 2048, "ny": 1024, "count": 256, "n": 128,
         "scheme": "kinematic", "storage": "fp16", "steps": 50},
        # the largest: the benchmark's channel and capsule density, far above L2
        {"name": "suspension_8192x4096", "kind": "suspension", "nx": 8192, "ny": 4096, "count": 4096, "n": 128,
         "scheme": "dynamic", "storage": "fp32", "steps": 20},
        # packed suspension, 16000 markers at 30 % hematocrit, with the repulsion
        {"name": "dense_1200x450", "kind": "dense", "nx": 1200, "ny": 450, "count": 16, "n": 1000,
         "hematocrit": 0.30, "scheme": "dynamic", "storage": "fp32", "steps": 200},
        # rigid particles in the channel of the precision workload
        {"name": "rigid_4096x512", "kind": "rigid", "nx": 4096, "ny": 512, "count": 256, "n": 128,
         "scheme": "dynamic", "storage": "fp32", "steps": 100},
        # a flow without capsules on a lattice whose rows fit no vector width
        {"name": "lattice_4099x2053", "kind": "lattice", "nx": 4099, "ny": 2053, "walls": True, "storage": "fp32",
         "steps": 20},
        # a parameter study: 512 independent shear cases in one launch
        {"name": "batch_512", "kind": "batch", "count": 512, "storage": "fp32", "steps": 300},
        # one gradient of D(T) on the 512 x 128 channel, with checkpoints
        {"name": "adjoint_512x128", "kind": "adjoint", "nx": 512, "ny": 128, "radius": 16.0, "n": 128,
         "scheme": "dynamic", "storage": "fp32", "steps": 400, "ckpt_every": 100},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["shear", "poiseuille", "open", "suspension", "suspension", "dense", "rigid", "lattice",
                       "lattice", "batch", "adjoint"])
    scheme = rng.choice(["kinematic", "dynamic"])
    storage = rng.choice(["fp64", "fp32", "fp32", "fp16"])
    c = {"kind": kind, "storage": storage}
    if kind in ("shear", "poiseuille"):
        ny = _log(rng, 60, 240)
        radius = round(rng.uniform(0.08, 0.14) * ny, 2) + 0.0037   # no vertex on a half-integer line
        c.update(nx=rng.randint(ny, 5 * ny), ny=ny, radius=radius, n=int(rng.uniform(6.4, 8.0) * radius),
                 scheme=scheme, storage=rng.choice(["fp64", "fp32"]), steps=_log(rng, 10, 200))
    elif kind == "open":
        ny = rng.randint(80, 160)
        c.update(nx=3 * ny, ny=ny, diameter=round(7.0 / 15.0 * ny, 2), scheme=scheme,
                 storage=rng.choice(["fp64", "fp32"]), steps=_log(rng, 20, 200))
    elif kind in ("suspension", "rigid"):
        nx, ny = _log(rng, 300, 8192), _log(rng, 130, 2048)
        # one capsule per 4600 nodes and up: the placement's cells hold about half of that
        count = max(1, min(2048, int(nx * ny / rng.uniform(4600, 16000)), ((ny - 6) // 24) * (nx // 24) // 2))
        if kind == "rigid":
            count, scheme, storage = min(count, 256), "dynamic", rng.choice(["fp64", "fp32"])
        c.update(nx=nx, ny=ny, count=count, n=2 * rng.randint(52, 72), scheme=scheme, storage=storage,
                 steps=_log(rng, 10, 60))
    elif kind == "dense":
        ny = rng.randint(300, 450)
        c.update(nx=rng.randint(2 * ny, 3 * ny), ny=ny, count=rng.randint(8, 16), n=rng.randint(500, 1000),
                 hematocrit=round(rng.uniform(0.15, 0.25), 3), scheme=scheme, storage="fp32", steps=_log(rng, 20, 100))
    elif kind == "lattice":
        c.update(nx=_log(rng, 64, 8192), ny=_log(rng, 64, 4096), walls=rng.random() < 0.7, steps=_log(rng, 10, 100))
    elif kind == "batch":
        c.update(count=_log(rng, 16, 512), storage=rng.choice(["fp32", "fp32", "fp64"]), steps=_log(rng, 20, 100))
    else:
        ny = rng.randint(64, 128)
        radius = round(rng.uniform(0.09, 0.125) * ny, 2) + 0.0037
        c.update(nx=rng.randint(2 * ny, 4 * ny), ny=ny, radius=radius, n=int(8 * radius), scheme=scheme,
                 storage=rng.choice(["fp64", "fp32"]), steps=_log(rng, 40, 300), ckpt_every=rng.choice([20, 50, 400]))
    # no dearer than the largest listed cases: the lattice updates of a pass, fewer in FP64
    nodes = c["count"] * 21700 if c["kind"] == "batch" else c["nx"] * c["ny"]
    most = 1.2e8 if c["storage"] == "fp64" else 1.1e9 if c["kind"] == "batch" else 6.0e8
    c["steps"] = max(1, min(c["steps"], int(most / nodes)))
    return c


# ---------------------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------------------
def _flow(case, seed):
    """The case's W.Case and its initial fields (rho, ux, uy), from the seed alone."""
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "lattice":
        nx, ny, tau = case["nx"], case["ny"], 0.7
        p = rng.uniform(0, 2 * np.pi, 6)
        m = rng.integers(1, 5, 4)
        x, y = 2 * np.pi * np.arange(nx) / nx, 2 * np.pi * np.arange(ny) / ny
        u0 = rng.uniform(0.01, 0.03)
        rho = 1.0 + 2e-3 * np.outer(np.sin(m[0] * y + p[0]), np.cos(m[1] * x + p[1]))
        ux = u0 * np.outer(np.cos(m[2] * y + p[2]), np.sin(m[1] * x + p[3]))
        uy = 0.5 * u0 * np.outer(np.sin(m[0] * y + p[4]), np.cos(m[3] * x + p[5]))
        w = W.Case("lattice", nx, ny, tau, case["walls"], -0.01, 0.01, gx=W.poiseuille_force(tau, 0.02, ny))
        return w, (rho, ux, uy)
    scheme = SCHEMES[case["scheme"]]
    ca = float(10.0 ** rng.uniform(-2.2, -1.8))
    if kind == "shear":
        centre = (0.5 * case["nx"] + rng.uniform(0.05, 0.45), 0.5 * case["ny"] - 0.5 + rng.uniform(0.05, 0.45))
        w = W.shear_capsule(case["nx"], case["ny"], radius=case["radius"], n=case["n"], ca=ca, scheme=scheme,
                            centre=centre)
    elif kind == "poiseuille":
        w = W.poiseuille_capsule(case["nx"], case["ny"], radius=case["radius"], n=case["n"], ca=ca, scheme=scheme,
                                 y_frac=float(rng.uniform(0.3, 0.5)))
    elif kind == "open":
        w = W.open_channel_capsule(case["ny"], case["nx"] / case["ny"], diameter=case["diameter"], ca=ca,
                                   scheme=scheme, y_frac=float(rng.uniform(0.43, 0.57)))
    elif kind == "adjoint":
        w = W.poiseuille_capsule(case["nx"], case["ny"], radius=case["radius"], n=case["n"], ca=2 * ca,
                                 scheme=scheme, y_frac=float(rng.uniform(0.29, 0.31)))
    elif kind == "dense":
        w = W.dense_biconcave(case["nx"], case["ny"], case["count"], case["n"], case["hematocrit"], seed=seed,
                              scheme=scheme)
    else:
        w = W.poiseuille_biconcave(case["nx"], case["ny"], count=case["count"], n=case["n"], a=case["n"] / 16.0,
                                   seed=seed, scheme=scheme, placement="grid")
    return w, w.fields()


def _study(case, seed):
    """The batch's cases: the sizes of one study, every capsule's place and constants from the seed."""
    rng = np.random.default_rng(seed)
    study = W.batch_cases(case["count"])
    for w in study:
        cap = w.capsules[0]
        cap.xy = cap.xy + rng.uniform(-0.3, 0.3, 2)
        stiffer = float(10.0 ** rng.uniform(-0.3, 0.3))
        cap.ks, cap.kb = stiffer * cap.ks, stiffer * cap.kb
    return study


def _single(v, storage):
    """What the library computed in single precision, handed on as such."""
    return v if storage == "fp64" else v.astype(np.float32)


def prepare(case, seed):
    if case["kind"] == "batch":
        return {"case": case, "batch": L.Batch(_study(case, seed), storage=case["storage"], autotune_steps=20)}
    w, fields = _flow(case, seed)
    ctx = L.Context(w.nx, w.ny, w.tau, w.walls, w.u_bottom, w.u_top, w.gx, w.gy, storage=case["storage"],
                    max_capsules=len(w.capsules), max_nodes=w.n_nodes)
    ctx.init_fields(*fields)
    if w.u_in is not None:
        ctx.set_inflow(w.u_in, w.rho_out)
    for c in w.capsules:
        if case["kind"] == "rigid":
            A, _, _, J = W.polygon_inertia(c.xy)
            ctx.add_rigid(c.xy, A, J)
        else:
            ctx.add_capsule(c.xy, c.ks, c.kb, c.ka, c.mass)
    if case["kind"] == "dense":
        ctx.set_repulsion(REPULSION_RANGE)
    return {"case": case, "ctx": ctx, "flow": w}


def run(state):
    case = state["case"]
    steps, storage, kind = case["steps"], case["storage"], case["kind"]
    if kind == "batch":
        b = state["batch"]
        b.step(steps)
        rings = [b.read_capsule(k) for k in range(min(case["count"], 16))]
        return {"observables": b.observables(), "xy": np.concatenate([r[0] for r in rings]),
                "velocity": _single(np.concatenate([r[1] for r in rings]), storage)}
    ctx, w = state["ctx"], state["flow"]
    if kind in ("shear", "poiseuille", "open", "adjoint", "dense"):
        for k, c in enumerate(w.capsules):
            ctx.set_capsule_positions(k, c.xy)
    if kind == "adjoint":
        J, grad = ctx.adjoint(steps, L.OBJ_TAYLOR_D, 0, case["ckpt_every"], w.scheme)
        xy = ctx.read_capsule(0)[0]
        return {"J": J, "gradient": _single(grad, storage), "xy": xy}
    ctx.step(steps, W.KINEMATIC if kind == "lattice" else w.scheme)
    out = {}
    if kind in ("shear", "poiseuille", "open"):
        out["xy"], vel, _, _ = ctx.read_capsule(0)
        out["velocity"] = _single(vel, storage)
    elif kind != "lattice":
        out["observables"] = ctx.observables_all()
    else:
        ctx.sync()
    out["populations"] = ctx.field_view(L.FIELD_POPULATIONS)[:, :, :case["nx"]]   # without the rows' padding
    return out


def work(case):
    """Bytes and operations of one pass: every lattice update reads and writes nine
    populations once, every vertex its positions, velocities and constants; a gradient
    also reads the states again and carries the populations' adjoints in 64 bits."""
    s, steps = BYTES[case["storage"]], case["steps"]
    if case["kind"] == "batch":
        nodes = case["count"] * float(np.mean(W.BATCH_SIZES)) ** 2
        vertices = case["count"] * float(np.mean(W.BATCH_NODES))
    else:
        nodes = case["nx"] * case["ny"]
        vertices = 0 if case["kind"] == "lattice" else _vertices(case)
    b = steps * (nodes * 18.0 * s + vertices * 160.0)
    f = steps * (nodes * 130.0 + vertices * 1500.0)
    if case["kind"] == "adjoint":
        b += steps * (nodes * (9.0 * s + 18.0 * 8.0) + vertices * 320.0)
        f += steps * (nodes * 260.0 + vertices * 6000.0)
    return {"bytes": b, "flops": f}


def _vertices(case):
    if case["kind"] == "open":
        return int(round(math.pi * case["diameter"] / 0.3))
    return case.get("count", 1) * case["n"]


# ---------------------------------------------------------------------------------------
# The same problems in 64 bits, in plain torch
# ---------------------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


class _Flow:
    """Lattice and rings. f: populations before the collision, less the rest weights."""

    def __init__(self, w, fields, dev, repulsion=0.0, rigid=False):
        self.w, self.dev, self.rc, self.rigid = w, dev, repulsion, rigid
        self.g = [torch.tensor(w.gx, device=dev, dtype=torch.float64), torch.tensor(w.gy, device=dev, dtype=torch.float64)]
        rho, ux, uy = (torch.as_tensor(a, device=dev) for a in fields)
        self.f = self.equilibrium(rho, ux, uy)
        self.post = None
        self.u_in = None if w.u_in is None else torch.as_tensor(w.u_in, device=dev)
        self.close()
        if w.capsules:
            caps, M = w.capsules, w.n_nodes
            n = [c.xy.shape[0] for c in caps]
            off = np.concatenate([[0], np.cumsum(n)])
            right, left = np.arange(1, M + 1), np.arange(-1, M - 1)
            right[off[1:] - 1], left[off[:-1]] = off[:-1], off[1:] - 1
            self.right, self.left = (torch.as_tensor(a, device=dev) for a in (right, left))
            self.ring = torch.as_tensor(np.repeat(np.arange(len(caps)), n), device=dev)
            self.n, self.off = n, off
            per = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device=dev)  # noqa: E731
            self.ks, self.kb, self.ka = (per([getattr(c, k) for c in caps]) for k in ("ks", "kb", "ka"))
            self.m = per([c.mass for c in caps])
            self.X = per(np.concatenate([c.xy for c in caps]))
            self.Xm = self.X
            self.uv = torch.zeros_like(self.X)
            self.age = 0
            e, turn = self.edges(self.X)
            self.L0, self.th0, self.A0 = e.norm(dim=1), turn, self.area(self.X)
            if rigid:
                body = np.array([W.polygon_inertia(c.xy) for c in caps])
                self.mass, self.inertia = per(body[:, 0]), per(body[:, 3])
                self.body = torch.cat([per(body[:, 1:3]), torch.zeros(len(caps), 4, device=dev, dtype=torch.float64)], 1)
                self.prev = self.body
                self.R0 = self.X - self.body[self.ring, :2]

    # lattice
    def equilibrium(self, rho, ux, uy):
        usq = 1.5 * (ux * ux + uy * uy)
        out = []
        for i in range(9):
            eu = EX[i] * ux + EY[i] * uy
            out.append(WT[i] * ((rho - 1.0) + rho * (3.0 * eu + 4.5 * eu * eu - usq)))
        return torch.stack(out)

    def moments(self, fx, fy):
        f = self.f
        rho = 1.0 + f.sum(0)
        ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8] + 0.5 * fx) / rho
        uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8] + 0.5 * fy) / rho
        return rho, ux, uy

    def advance(self, fib):
        w = self.w
        fx, fy = (self.g[0], self.g[1]) if fib is None else (self.g[0] + fib[0], self.g[1] + fib[1])
        rho, ux, uy = self.moments(fx, fy)
        usq, uF = 1.5 * (ux * ux + uy * uy), ux * fx + uy * fy
        post = []
        for i in range(9):
            eu, eF = EX[i] * ux + EY[i] * uy, EX[i] * fx + EY[i] * fy
            feq = WT[i] * ((rho - 1.0) + rho * (3.0 * eu + 4.5 * eu * eu - usq))
            guo = (1.0 - 0.5 / w.tau) * WT[i] * (3.0 * (eF - uF) + 9.0 * eu * eF)
            post.append(self.f[i] - (self.f[i] - feq) / w.tau + guo)
        self.post = torch.stack(post)
        f = []
        for i in range(9):
            p = torch.roll(post[i], (EY[i], EX[i]), (0, 1))
            if w.walls and EY[i] > 0:
                p = torch.cat([post[OPP[i]][:1] - 6.0 * WT[i] * EX[OPP[i]] * w.u_bottom, p[1:]])
            if w.walls and EY[i] < 0:
                p = torch.cat([p[:-1], post[OPP[i]][-1:] - 6.0 * WT[i] * EX[OPP[i]] * w.u_top])
            f.append(p)
        self.f = torch.stack(f)
        self.close()

    def close(self):
        """Zou-He inlet and outlet columns of an open channel."""
        if self.u_in is None:
            return
        f, (gx, gy) = self.f.clone(), self.g
        for x in (0, -1):
            c = [f[i, :, x] for i in range(9)]
            if x == 0:
                rho = (1.0 + c[0] + c[2] + c[4] + 2.0 * (c[3] + c[6] + c[7]) - 0.5 * gx) / (1.0 - self.u_in)
                jx = rho * self.u_in - 0.5 * gx
            else:
                rho = torch.full_like(self.u_in, self.w.rho_out)
                jx = c[0] + c[2] + c[4] + 2.0 * (c[1] + c[5] + c[8]) - (rho - 1.0)
            q = self.equilibrium(rho, jx / rho, -0.5 * gy / rho)
            nt = 0.5 * ((c[2] - q[2]) - (c[4] - q[4]))
            if x == 0:
                f[1, :, 0], f[5, :, 0], f[8, :, 0] = c[3] + q[1] - q[3], c[7] + q[5] - q[7] - nt, c[6] + q[8] - q[6] + nt
            else:
                f[3, :, -1], f[7, :, -1], f[6, :, -1] = (c[1] + q[3] - q[1], c[5] + q[7] - q[5] + nt,
                                                         c[8] + q[6] - q[8] - nt)
        self.f = f

    # rings
    def edges(self, X):
        b = X[self.right] - X
        a = b[self.left]
        return b, torch.atan2(a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0], (a * b).sum(1))

    def per_ring(self, v):
        return torch.zeros((len(self.n),) + v.shape[1:], device=v.device, dtype=v.dtype).index_add(0, self.ring, v)

    def area(self, X):
        X = X - X[torch.as_tensor(self.off[:-1], device=self.dev)][self.ring]
        r = X[self.right]
        return 0.5 * self.per_ring(X[:, 0] * r[:, 1] - r[:, 0] * X[:, 1])

    def internal(self, X):
        k, R, Lf = self.ring, self.right, self.left
        b, turn = self.edges(X)
        a = b[Lf]
        ln = b.norm(dim=1)
        s = (self.ks[k] * (ln - self.L0) / ln)[:, None] * b
        F = s - s[Lf]
        t = (self.kb[k] * torch.sin(turn - self.th0))[:, None]
        dl = torch.stack([-a[:, 1], a[:, 0]], 1) / (a * a).sum(1)[:, None]
        dr = torch.stack([-b[:, 1], b[:, 0]], 1) / (b * b).sum(1)[:, None]
        F = F + t * (dl + dr) - (t * dl)[R] - (t * dr)[Lf]
        q = (self.ka * (1.0 - self.area(X) / self.A0) / 6.0)[k]
        d = a + b
        return F + q[:, None] * torch.stack([d[:, 1], -d[:, 0]], 1)

    def repulsion(self, X):
        if self.rc <= 0.0 or len(self.n) < 2:
            return 0.0
        e = X[self.right] - X
        nb = torch.stack([e[:, 1], -e[:, 0]], 1) / e.norm(dim=1)[:, None]
        nrm = nb + nb[self.left]
        nrm = nrm / nrm.norm(dim=1)[:, None]
        f = []
        for k, n in enumerate(self.n):
            o = self.off[k]
            d = X[o:o + n, None, :] - X[None, :, :]
            px, py = self.w.nx if self.u_in is None else 0, 0 if self.w.walls else self.w.ny
            dx = d[..., 0] - px * torch.floor(d[..., 0] / px + 0.5) if px else d[..., 0]
            dy = d[..., 1] - py * torch.floor(d[..., 1] / py + 0.5) if py else d[..., 1]
            d = torch.sqrt(dx * dx + dy * dy)
            near = (d < self.rc) & (self.ring != k)[None, :]
            f.append(torch.where(near, d, torch.inf).pow(-2.5).sum(1))
        return -(1e-4 / (8.0 * math.sqrt(2.0)) * torch.cat(f))[:, None] * nrm

    def shapes(self, P):
        """Support nodes (flat index), values and gradients of the linear MLS fit at P."""
        w = self.w
        c = torch.floor(P.detach() + 0.5)
        o = torch.tensor([(a, b) for b in (-1.0, 0.0, 1.0) for a in (-1.0, 0.0, 1.0)], device=self.dev,
                         dtype=torch.float64)
        k = c[:, None, :] + o[None]
        d = k - P[:, None, :]
        wt = torch.exp(-(d * d).sum(2) / (2.6 * 0.3) ** 2)
        p = torch.cat([torch.ones_like(d[..., :1]), d], 2)
        wp = wt[..., None] * p
        A = wp.transpose(1, 2) @ p
        # inverse of the symmetric 3 x 3 moment matrices by cofactors
        a, b, e = A[:, 0], A[:, 1], A[:, 2]
        r = torch.stack([torch.linalg.cross(b, e), torch.linalg.cross(e, a), torch.linalg.cross(a, b)], 1)
        inv = r / (a * r[:, 0]).sum(1)[:, None, None]
        phi = wp @ inv.transpose(1, 2)
        x, y = k[..., 0].long() % w.nx, k[..., 1].long()
        y = y.clamp(0, w.ny - 1) if w.walls else y % w.ny
        return y * w.nx + x, phi

    def at(self, field, shape):
        node, phi = shape
        v = field.reshape(-1)[node]
        return (v * phi[..., 0]).sum(1), (v * phi[..., 1]).sum(1), (v * phi[..., 2]).sum(1)

    def spread(self, shape, F):
        node, phi = shape
        out = []
        for a in range(2):
            v = torch.zeros(self.w.nx * self.w.ny, device=self.dev, dtype=torch.float64)
            out.append(v.index_add(0, node.reshape(-1), (phi[..., 0] * F[:, a:a + 1]).reshape(-1)).view(self.w.ny, -1))
        return out

    def stress(self, P, rho, ux, uy):
        """Density and rho nu (grad u + its transpose) at the probes P."""
        s = self.shapes(P)
        r = self.at(rho - 1.0, s)[0]
        _, uxx, uxy = self.at(ux, s)
        _, uyx, uyy = self.at(uy, s)
        m = (1.0 + r) * (self.w.tau - 0.5) / 3.0
        return r, 2.0 * m * uxx, 2.0 * m * uyy, m * (uxy + uyx)

    def step(self, scheme):
        w = self.w
        if not w.capsules:
            self.advance(None)
            return
        X, left = self.X, self.left
        rep = self.repulsion(X)
        s = self.shapes(X)
        if scheme == W.KINEMATIC:
            fib = self.spread(s, self.internal(X) + rep)
            self.advance(fib)
            _, ux, uy = self.moments(self.g[0] + fib[0], self.g[1] + fib[1])
            u = torch.stack([self.at(ux, s)[0], self.at(uy, s)[0]], 1)
            new = X + u if self.age == 0 else (2.0 * X - 0.5 * self.Xm + u) * (2.0 / 3.0)
            self.uv = u
        else:
            _, ux, uy = self.moments(*self.g)
            U = torch.stack([self.at(ux, s)[0], self.at(uy, s)[0]], 1)
            if self.rigid:
                d = X - self.body[self.ring, :2]
                om = self.body[self.ring, 5:6]
                self.uv = self.body[self.ring, 3:5] + om * torch.stack([-d[:, 1], d[:, 0]], 1)
            elif self.age == 0:
                self.uv, self.Xm = U, X - U
            e = X[self.right] - X
            ln = e.norm(dim=1)
            cl = 0.5 * (ln + ln[left])
            self.advance(self.spread(s, cl[:, None] * (self.uv - U)))
            rho, ux, uy = self.moments(*self.g)
            nrm = torch.stack([e[:, 1], -e[:, 0]], 1) / ln[:, None]
            mid = X + 0.5 * e
            load = 0.0
            for side in (1.0,) if self.rigid else (1.0, -1.0):
                r, xx, yy, xy = self.stress(mid + 1.2 * side * nrm, rho, ux, uy)
                t = torch.stack([xx * nrm[:, 0] + xy * nrm[:, 1], xy * nrm[:, 0] + yy * nrm[:, 1]], 1)
                load = load + side * (t - (r / 3.0)[:, None] * nrm) * ln[:, None]
            if self.rigid:
                d = mid - self.body[self.ring, :2]
                mom = d[:, 0] * load[:, 1] - d[:, 1] * load[:, 0]
                acc = torch.cat([self.per_ring(load) / self.mass[:, None], (self.per_ring(mom) / self.inertia)[:, None]], 1)
                v = (2.0 * self.body[:, 3:] - 0.5 * self.prev[:, 3:] + acc) * (2.0 / 3.0)
                q = (2.0 * self.body[:, :3] - 0.5 * self.prev[:, :3] + v) * (2.0 / 3.0)
                self.prev, self.body = self.body, torch.cat([q, v], 1)
                cs, sn = torch.cos(q[self.ring, 2]), torch.sin(q[self.ring, 2])
                new = q[self.ring, :2] + torch.stack([cs * self.R0[:, 0] - sn * self.R0[:, 1],
                                                      sn * self.R0[:, 0] + cs * self.R0[:, 1]], 1)
            else:
                F = self.internal(X) + 0.5 * (load + load[left]) + rep
                new = X + U + 0.5 * F / self.m[self.ring][:, None]
                self.uv = 1.5 * new - 2.0 * X + 0.5 * self.Xm
        self.Xm, self.X = X, new
        self.age += 1

    def area_sums(self, X, k):
        x = X[self.off[k]:self.off[k] + self.n[k]]
        x0 = x[:1].detach()
        a = x - x0
        b = a.roll(-1, 0)
        c = a[:, 0] * b[:, 1] - b[:, 0] * a[:, 1]
        A = 0.5 * c.sum()
        xc = ((a + b) * c[:, None]).sum(0) / (6.0 * A)
        xx, yy = ((a * a + a * b + b * b) * c[:, None]).sum(0) / 12.0 - A * xc * xc
        xy = ((a[:, 0] * b[:, 1] + 2 * a[:, 0] * a[:, 1] + 2 * b[:, 0] * b[:, 1] + b[:, 0] * a[:, 1]) * c).sum() / 24.0
        return A, xc + x0[0], xx, yy, xy - A * xc[0] * xc[1]

    def taylor(self, X, k):
        A, _, xx, yy, xy = self.area_sums(X, k)
        mid, dev = 0.5 * (xx + yy), torch.sqrt(0.25 * (xx - yy) ** 2 + xy * xy)
        a, b = torch.sqrt((mid + dev) / A), torch.sqrt((mid - dev) / A)
        return (a - b) / (a + b)

    def observables(self):
        ln = (self.X[self.right] - self.X).norm(dim=1)
        per, per0 = self.per_ring(ln), self.per_ring(self.L0)
        out = []
        for k in range(len(self.n)):
            A, c, xx, yy, xy = self.area_sums(self.X, k)
            out.append(torch.stack([A, per[k], self.taylor(self.X, k), c[0], c[1], A * 4.0 * math.pi / per[k] ** 2,
                                    0.5 * torch.atan2(2.0 * xy, xx - yy), per[k] / per0[k] - 1.0]))
        return torch.stack(out)


def _seconds(case):
    """About what exact() takes: launches, lattice nodes, vertices, pairs of the repulsion."""
    if case["kind"] == "batch":
        return case["count"] * case["steps"] * 6e-3
    per = 6e-3 + 4e-9 * case["nx"] * case["ny"] + 5e-8 * _vertices(case) if case["kind"] != "lattice" else \
        2e-3 + 4e-9 * case["nx"] * case["ny"]
    if case["kind"] == "dense":
        per += 2e-10 * _vertices(case) ** 2
    if case["kind"] == "adjoint":
        per *= 5
    return per * case["steps"] + 2e-3 * case.get("count", 1)


def exact(case, seed):
    if _seconds(case) > 15.0:
        return None
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        obs, xy, vel = [], [], []
        for w in _study(case, seed):
            s = _Flow(w, w.fields(), dev)
            for _ in range(steps):
                s.step(W.KINEMATIC)
            obs.append(s.observables())
            xy.append(s.X.reshape(-1))
            vel.append(s.uv.reshape(-1))
        return {"observables": torch.cat(obs), "xy": torch.cat(xy[:16]), "velocity": torch.cat(vel[:16])}
    w, fields = _flow(case, seed)
    s = _Flow(w, fields, dev, REPULSION_RANGE if kind == "dense" else 0.0, kind == "rigid")
    if kind == "adjoint":
        return _exact_gradient(s, w.scheme, steps)
    for _ in range(steps):
        s.step(w.scheme)
    out = {"populations": s.post * (1024.0 if case["storage"] == "fp16" else 1.0)}
    if kind in ("shear", "poiseuille", "open"):
        out["xy"], out["velocity"] = s.X.reshape(-1), s.uv.reshape(-1)
    elif kind != "lattice":
        out["observables"] = s.observables()
    return out


def _exact_gradient(s, scheme, steps, chunk=20):
    """J and dJ/d(k_s, k_b, g_x, g_y): chunks of steps are run again for their reverse sweep."""
    par = [s.ks, s.kb, s.g[0], s.g[1]]
    state, starts = (s.f, s.X, s.Xm, s.uv), []

    def go(state, par, n0):
        s.f, s.X, s.Xm, s.uv = state
        s.ks, s.kb, s.g = par[0], par[1], [par[2], par[3]]
        for n in range(n0, min(n0 + chunk, steps)):
            s.age = n
            s.step(scheme)
        return s.f, s.X, s.Xm, s.uv

    with torch.no_grad():
        for n0 in range(0, steps, chunk):
            starts.append((n0, state))
            state = go(state, par, n0)
    X = state[1].clone().requires_grad_()
    J = s.taylor(X, 0)
    (gX,) = torch.autograd.grad(J, X)
    bar = [torch.zeros_like(state[0]), gX, torch.zeros_like(gX), torch.zeros_like(gX)]
    total = [torch.zeros_like(p) for p in par]
    for n0, st in reversed(starts):
        leaf = [v.detach().clone().requires_grad_() for v in st]
        p = [v.detach().clone().requires_grad_() for v in par]
        end = go(leaf, p, n0)
        got = torch.autograd.grad(end, leaf + p, bar, allow_unused=True)
        got = [torch.zeros_like(v) if q is None else q for q, v in zip(got, leaf + p)]
        bar, total = got[:4], [a + b for a, b in zip(total, got[4:])]
    grad = torch.cat([total[0], total[1], total[2][None], total[3][None]])
    return {"J": J.detach(), "gradient": grad, "xy": state[1].reshape(-1)}
