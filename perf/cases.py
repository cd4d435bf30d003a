"""Performance cases of the VP-LBM library: whole solver calls through the public
entry points, over the range of lattices its users run.

A pass is what a solver loop does between two looks at the flow: a run of time
steps, every step's forces read into host memory, and the flow fields of the
current level.  The lattices, bodies and step counts come from the workloads of
`paper_2110_00967_gb300.workloads` (the disk channel, the airfoil grids of the
benchmark and of the serving mix, the paper's airfoil grid, the two sedimentation
set-ups) and from the parity tests' ragged and body-force-driven lattices.

A case's "lattices" is a text of comma-separated lattice descriptions
`kind:nx:ny:dtype:parameter` (see `_workload`); several lattices are stepped
together as one batch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_00967_gb300 import vplbm as V
from paper_2110_00967_gb300 import workloads as W

CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
FLIPY = (0, 1, 4, 3, 2, 8, 7, 6, 5)
WT = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2, "f16sr": 2, "bf16sr": 2}
# floating-point operations of one node update: moments, velocity, equilibrium
# and TRT collision of nine populations
FLOPS_PER_NODE = 160


def _grids(kind, sizes, dtype, params):
    return ",".join(f"{kind}:{nx}:{ny}:{dtype}:{p:g}" for (nx, ny), p in zip(sizes, params))


def listed():
    return [
        # a caller that couples each step to its own model: one step per call and
        # both force estimates after it, on the smallest grid of the serving mix
        {"name": "coupled steps 512x256 f32", "mode": "coupled", "lattices": "naca:512:256:f32:10", "steps": 8},
        # the FP64 reference case: disk channel, BGK, Re 20
        {"name": "disk channel 256x128 f64", "mode": "run", "lattices": "disk:256:128:f64:20", "steps": 100},
        # one airfoil solve on a small grid, as the long time-mean runs step it
        {"name": "airfoil 512x256 f32", "mode": "run", "lattices": "naca:512:256:f32:15", "steps": 256},
        # an FP64 airfoil on a ragged middle-sized lattice (reference runs)
        {"name": "airfoil 1001x487 f64", "mode": "run", "lattices": "naca:1001:487:f64:7", "steps": 16},
        # a window of the serving loop: one lattice per grid of its mix, in the
        # storage form that it serves
        {"name": "serving mix f16sr", "mode": "run",
         "lattices": _grids("naca", W.SERVING_GRIDS, "f16sr", (3, 8, 12, 16, 19)), "steps": 128},
        # the benchmark's batch: five angles on 2048 x 1024
        {"name": "airfoil batch 5x2048x1024 f32", "mode": "run",
         "lattices": _grids("naca", [(2048, 1024)] * 5, "f32", W.NACA_ANGLES), "steps": 100},
        # the same in 16-bit storage, rounded to nearest
        {"name": "airfoil batch 5x2048x1024 f16", "mode": "run",
         "lattices": _grids("naca", [(2048, 1024)] * 5, "f16", W.NACA_ANGLES), "steps": 100},
        # the paper's airfoil case, one lattice
        {"name": "paper airfoil 3614x1946 f32", "mode": "run", "lattices": "paper:3614:1946:f32:12", "steps": 100},
        # the large single lattice
        {"name": "airfoil 8192x4096 f32", "mode": "run", "lattices": "naca:8192:4096:f32:10", "steps": 50},
        # the falling disk in the closed box, driven by either estimator side by side
        {"name": "sedimentation 2x400x1600 f32", "mode": "run",
         "lattices": "sed:400:1600:f32:mem,sed:400:1600:f32:sim", "steps": 64},
        # the paper's sedimentation channel (inlet above, free outlet below)
        {"name": "falling disk 1560x104 f32", "mode": "run", "lattices": "sedpaper:1560:104:f32:sim", "steps": 64},
        # a disk between no-slip walls in a flow driven by a body force, ragged, 16-bit
        {"name": "driven channel 777x395 f16", "mode": "run", "lattices": "driven:777:395:f16:40", "steps": 64},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("coupled", "disk", "naca", "naca", "batch", "batch", "sed", "sedpaper", "driven"))
    if kind == "coupled":
        nx = _log(rng, 256, 1600)
        return {"mode": "coupled", "steps": rng.randint(2, 12),
                "lattices": f"naca:{nx}:{nx // 2 + rng.randint(-9, 9)}:{rng.choice(('f32', 'f16sr'))}:{rng.uniform(1, 20):.2f}"}
    if kind == "disk":
        ny = _log(rng, 90, 400)
        return {"mode": "run", "steps": _log(rng, 10, 100),
                "lattices": f"disk:{2 * ny + rng.randint(0, 15)}:{ny}:{rng.choice(('f64', 'f32'))}:{rng.uniform(12, 0.25 * ny):.2f}"}
    if kind == "naca":
        nx = _log(rng, 300, 6000)
        dtype = rng.choice(("f32", "f32", "f16", "bf16", "f16sr", "bf16sr", "f64" if nx < 1500 else "f32"))
        ny = int(nx * rng.uniform(0.4, 0.6))
        return {"mode": "run", "steps": max(16, min(250, int(5e8 / (nx * ny)))),
                "lattices": f"naca:{nx}:{ny}:{dtype}:{rng.uniform(0, 20):.2f}"}
    if kind == "batch":
        n = rng.randint(2, 6)
        dtype = rng.choice(("f32", "f16", "bf16", "f16sr"))
        same = rng.random() < 0.5
        grids = [rng.choice(W.SERVING_GRIDS)] * n if same else [rng.choice(W.SERVING_GRIDS) for _ in range(n)]
        return {"mode": "run", "steps": rng.randint(20, 100),
                "lattices": _grids("naca", grids, dtype, [round(rng.uniform(0, 20), 2) for _ in grids])}
    if kind == "sed":
        nx = _log(rng, 200, 700)
        est = rng.choice(("mem", "sim"))
        return {"mode": "run", "steps": _log(rng, 16, 100),
                "lattices": f"sed:{nx}:{_log(rng, nx, 4 * nx)}:{rng.choice(('f32', 'f32', 'f64' if nx < 300 else 'f32'))}:{est}"}
    if kind == "sedpaper":
        return {"mode": "run", "steps": _log(rng, 16, 100),
                "lattices": f"sedpaper:{_log(rng, 400, 3000)}:{_log(rng, 100, 300)}:f32:{rng.choice(('mem', 'sim'))}"}
    nx = _log(rng, 200, 3000)
    return {"mode": "run", "steps": _log(rng, 10, 80),
            "lattices": f"driven:{nx}:{max(100, nx // 2 + rng.randint(-7, 7))}:"
                        f"{rng.choice(('f32', 'f16', 'bf16sr'))}:{rng.uniform(20, 45):.2f}"}


# ---------------------------------------------------------------------------
# a lattice description as a workload
# ---------------------------------------------------------------------------
def _workload(text, seed):
    """`kind:nx:ny:dtype:parameter` as a Workload.  naca, paper: parameter = angle
    of attack; disk, driven: diameter; sed, sedpaper: the estimator that drives the
    falling disk.  The seed shifts the body by a fraction of a node (the disks) or
    turns it by a fraction of a degree (the airfoils)."""
    kind, nx, ny, dtype, par = text.split(":")
    nx, ny = int(nx), int(ny)
    rng = np.random.default_rng(seed)
    a, b = (float(v) for v in rng.uniform(-0.4, 0.4, 2))
    if kind in ("naca", "paper"):
        if kind == "paper":
            w = W.naca_paper(float(par) + a, dtype=dtype)
        else:
            # tau+ for Re 1000 on chords other than 200 nodes, as the library's
            # own large lattice takes it
            w = W.naca(float(par) + a, dtype=dtype, nx=nx, ny=ny,
                       tau_plus=0.62 if nx >= 6000 else 0.53)
        return w
    if kind == "disk":
        d = float(par)
        w = W.disk_channel()
        u_ref = (0.0, 0.0) if dtype == "f64" else (0.05, 0.0)
        body = W.Body("disk", length=d, x_c=0.25 * nx + a, y_c=0.5 * ny + b)
        return w.with_(nx=nx, ny=ny, dtype=dtype, u_ref=u_ref, body=body, tau_plus=0.5 + 3.0 * 0.05 * d / 20.0)
    if kind == "driven":
        d = float(par)
        body = W.Body("disk", length=d, x_c=0.3 * nx + a, y_c=0.5 * ny + b)
        return W.Workload(name="driven", nx=nx, ny=ny, dtype=dtype, collision="trt", tau_plus=0.6,
                          u_in=(0.03, 0.0), bc=("periodic", "periodic", "noslip", "noslip"), body=body,
                          steps=1, body_force=(1e-5, 0.0), u_ref=(0.03, 0.0))
    if kind == "sed":
        w = W.sedimentation(par)
        body = W.Body("disk", length=50.0, x_c=60.0 + a, y_c=ny - 90.0 + b, moving=True, density_ratio=1.03,
                      gravity=w.body.gravity, estimator=par)
        return w.with_(nx=nx, ny=ny, dtype=dtype, body=body)
    w = W.sedimentation_paper(1.03, par)
    body = W.Body("disk", length=26.0, x_c=103.5 + a, y_c=40.0 + b, moving=True, density_ratio=1.03,
                  gravity=w.body.gravity, estimator=par)
    return w.with_(nx=nx, ny=ny, dtype=dtype, body=body)


def _workloads(case, seed):
    return [_workload(t, 1000 * seed + k) for k, t in enumerate(case["lattices"].split(","))]


def _body_velocity(w):
    """A falling disk is already falling: a fraction of a node per step along gravity."""
    if not w.body.moving:
        return (0.0, 0.0)
    g = math.hypot(*w.body.gravity)
    return tuple(0.01 * v / g for v in w.body.gravity)


def _initial(w, seed):
    """Pre-collision populations [9][ny][nx] (FP64, on the GPU): equilibrium at the
    free stream slowed to the body's velocity over a boundary layer, with a seeded
    large-scale disturbance of density and velocity."""
    dev = "cuda"
    x = torch.arange(w.nx, dtype=torch.float64, device=dev)[None, :]
    y = torch.arange(w.ny, dtype=torch.float64, device=dev)[:, None]
    b = w.body
    if b.kind == "naca":
        ca, sa = math.cos(b.angle), math.sin(b.angle)
        s = (x - b.x_c) * ca - (y - b.y_c) * sa
        t = (x - b.x_c) * sa + (y - b.y_c) * ca
        s = s - s.clamp(-b.pivot_chord_frac * b.length, (1 - b.pivot_chord_frac) * b.length)
        dist = (torch.sqrt(s * s + t * t) - 0.06 * b.length).clamp(min=0.0)
    else:
        dist = (torch.sqrt((x - b.x_c) ** 2 + (y - b.y_c) ** 2) - 0.5 * b.length).clamp(min=0.0)
    layer = torch.exp(-dist / (0.1 * b.length + 2.0))
    del dist
    rng = np.random.default_rng(seed + 77)
    u0 = max(abs(w.u_in[0]), 0.01)
    ub = _body_velocity(w)
    field = []
    for q in range(3):  # rho - 1, u_x, u_y
        v = torch.zeros((w.ny, w.nx), dtype=torch.float64, device=dev)
        for m in range(2):
            kx, ky = (int(k) for k in rng.integers(1, 6, 2))
            px, py = (float(p) for p in rng.uniform(0, 2 * math.pi, 2))
            v += torch.sin(2 * math.pi * kx / w.nx * x + px) * torch.sin(2 * math.pi * ky / w.ny * y + py)
        field.append(v * (u0 * (0.01 if q == 0 else 0.04)))
    rho, ux, uy = field
    rho += 1.0
    ux = (ux + w.u_in[0]) * (1 - layer) + ub[0] * layer
    uy = (uy + w.u_in[1]) * (1 - layer) + ub[1] * layer
    return _feq(rho, ux, uy)


def _feq(rho, ux, uy):
    f = torch.empty((9,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
    uu = 1.5 * (ux * ux + uy * uy)
    for a in range(9):
        cu = CX[a] * ux + CY[a] * uy
        f[a] = WT[a] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - uu)
    return f


# ---------------------------------------------------------------------------
# preparation and one pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    """Lattices with their bodies placed, a developed start state, the first step
    taken, and the runs of this length announced to the library, as the benchmark
    does; page-locked memory for the force histories, device memory for the
    fields."""
    works = _workloads(case, seed)
    lats, hist, fields = [], [], []
    n = case["steps"]
    for k, w in enumerate(works):
        lat = V.Lattice(V.config_of(w))
        body = V.body_of(w)
        body.u[0], body.u[1] = _body_velocity(w)
        lat.set_body(body)
        f = _initial(w, 1000 * seed + k)
        V.vplbm_set_state(lat.ctx, f.data_ptr(), None, 0)
        torch.cuda.synchronize()
        del f
        lats.append(lat)
        hist.append(torch.empty((n, 9), dtype=torch.float64, pin_memory=True))
        fields.append(torch.empty((3, w.ny, w.nx), dtype=torch.float64, device="cuda"))
    batch = V.Batch(lats) if len(lats) > 1 else None
    stepper = batch if batch is not None else lats[0]
    stepper.step(1)
    if case["mode"] == "run":
        stepper.prepare(n)
    torch.cuda.synchronize()
    return {"case": case, "works": works, "lats": lats, "batch": batch, "stepper": stepper,
            "hist": hist, "fields": fields}


def run(state):
    """The steps, each step's forces in host memory, and the flow fields.  Values
    come in the lattice's compute type (FP64 lattices FP64, the others FP32)."""
    case, lats = state["case"], state["lats"]
    out = []
    if case["mode"] == "coupled":
        mem, sim = [], []
        lat = lats[0]
        for _ in range(case["steps"]):
            lat.step(1)
            mem.append(lat.force_mem())
            sim.append(lat.force_sim())
        out.append({"mem": _typed(np.array(mem), state["works"][0]),
                    "sim": _typed(np.array(sim), state["works"][0])})
    else:
        n = case["steps"]
        state["stepper"].step(n)
        for lat, h in zip(lats, state["hist"]):
            V.vplbm_force_history_async(lat.ctx, n, h.data_ptr())
    for lat, fl in zip(lats, state["fields"]):
        V.vplbm_get_fields_dev(lat.ctx, fl[0].data_ptr(), fl[1].data_ptr(), fl[2].data_ptr())
    if case["mode"] != "coupled":
        lats[0].stream.synchronize()  # the forces are in host memory now
        for w, h in zip(state["works"], state["hist"]):
            rows = h.numpy()
            out.append({"mem": _typed(rows[:, 0:3], w), "sim": _typed(rows[:, 3:6], w)})
    for w, fl, d in zip(state["works"], state["fields"], out):
        d["rho"], d["ux"], d["uy"] = (fl[q] if w.dtype == "f64" else fl[q].float() for q in range(3))
    return out


def _typed(a, w):
    return np.array(a, dtype=np.float64 if w.dtype == "f64" else np.float32)


def work(case):
    """The state read once and written once, the fields and force rows written;
    and the node updates of all steps."""
    bytes_, flops = 0.0, 0.0
    for text in case["lattices"].split(","):
        _, nx, ny, dtype, _ = text.split(":")
        n = int(nx) * int(ny)
        bytes_ += n * (2 * 9 * BYTES[dtype] + 3 * 8) + case["steps"] * 72
        flops += float(n) * case["steps"] * FLOPS_PER_NODE
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same pass in plain FP64 torch
# ---------------------------------------------------------------------------
def _polygon(b):
    """SIM points (x - x_G, y - y_G, n_x, n_y, S): the midpoints of a closed
    polygon on the body."""
    if b.kind == "disk":
        n = math.ceil(2.0 * math.pi * (0.5 * b.length) / 0.5)
        th = 2.0 * np.pi * np.arange(n) / n
        vx, vy = 0.5 * b.length * np.cos(th), 0.5 * b.length * np.sin(th)
    else:
        m = 424
        k = np.concatenate([np.arange(m, -1, -1), np.arange(1, m + 1)])
        sign = np.concatenate([np.ones(m + 1), -np.ones(m)])
        xi = 0.5 * (1.0 - np.cos(np.pi * k / m))
        yt = 5.0 * b.thickness * (0.2969 * np.sqrt(xi) - 0.1260 * xi - 0.3516 * xi ** 2 + 0.2843 * xi ** 3
                                  - 0.1015 * xi ** 4)
        s, z = (xi - b.pivot_chord_frac) * b.length, sign * yt * b.length
        ca, sa = math.cos(b.angle), math.sin(b.angle)
        vx, vy = s * ca + z * sa, -s * sa + z * ca
    ex, ey = np.roll(vx, -1) - vx, np.roll(vy, -1) - vy
    ln = np.sqrt(ex * ex + ey * ey)
    return np.stack([0.5 * (vx + np.roll(vx, -1)), 0.5 * (vy + np.roll(vy, -1)), ey / ln, -ex / ln, ln])


class _Exact:
    """One lattice of the method (D2Q9 BGK/TRT with volume penalization, MEM and SIM
    forces, rigid disk) stepped in FP64."""

    def __init__(self, w, f):
        self.w, self.f = w, f
        b = w.body
        self.x, self.y = b.x_c, b.y_c
        self.u = list(_body_velocity(w))
        self.om = 0.0
        self.pts = _polygon(b)
        cl = np.array([(CX[a] * self.pts[2] + CY[a] * self.pts[3]) / (1.0 if a <= 4 else math.sqrt(2.0))
                       for a in range(1, 9)])
        self.dirs = 1 + np.argmax(cl, axis=0)
        tp = w.tau_plus
        tm = tp if w.collision == "bgk" else w.lambda_trt / (tp - 0.5) + 0.5
        self.sp, self.sm, self.af = 1.0 / tp, 1.0 / tm, 1.0 - 0.5 / tp
        self.chi = None

    def mask(self):
        b, w = self.w.body, self.w
        if self.chi is not None and not b.moving:
            return self.chi
        i = np.arange(w.nx, dtype=np.float64)[None, :] - self.x
        j = np.arange(w.ny, dtype=np.float64)[:, None] - self.y
        if b.kind == "disk":
            r = 0.5 * b.length
            self.chi = i * i + j * j <= r * r
        else:
            ca, sa = math.cos(b.angle), math.sin(b.angle)
            xi = (i * ca - j * sa) / b.length + b.pivot_chord_frac
            ze = (i * sa + j * ca) / b.length
            x = np.clip(xi, 0.0, 1.0)
            x2 = x * x
            t = 0.2969 * np.sqrt(x) - 0.1260 * x - 0.3516 * x2 + 0.2843 * (x2 * x) - 0.1015 * (x2 * x * x)
            self.chi = (xi >= 0) & (xi <= 1) & (np.abs(ze) <= 5.0 * b.thickness * t)
        r0, r1 = (np.flatnonzero(self.chi.any(axis=k))[[0, -1]] for k in (1, 0))
        w = self.w
        self.box = (max(0, r0[0] - 6), min(w.ny, r0[1] + 7), max(0, r1[0] - 6), min(w.nx, r1[1] + 7))
        return self.chi

    def us(self, xx, yy):
        return self.u[0] - self.om * (yy - self.y), self.u[1] + self.om * (xx - self.x)

    def moments(self):
        """rho and u of Eqs. updatestep, updatestepm, and the force density."""
        w, f = self.w, self.f
        chi = self.mask()
        rho = f.sum(0)
        jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]) + 0.5 * w.body_force[0]
        jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]) + 0.5 * w.body_force[1]
        j0, j1, i0, i1 = self.box
        sl = (slice(j0, j1), slice(i0, i1))
        m = torch.from_numpy(chi[sl]).to(f.device)
        xx = torch.arange(i0, i1, dtype=torch.float64, device=f.device)[None, :]
        yy = torch.arange(j0, j1, dtype=torch.float64, device=f.device)[:, None]
        usx, usy = self.us(xx, yy)
        k = 0.5 / w.eta
        ux, uy = jx / rho, jy / rho
        r, gx, gy = rho[sl], torch.zeros_like(rho[sl]), torch.zeros_like(rho[sl])
        dx, dy = jx[sl] - r * usx, jy[sl] - r * usy
        ux[sl] = torch.where(m, usx + dx / (r * (1 + k)), ux[sl])
        uy[sl] = torch.where(m, usy + dy / (r * (1 + k)), uy[sl])
        gx = torch.where(m, -2 * k * dx / (1 + k), gx)
        gy = torch.where(m, -2 * k * dy / (1 + k), gy)
        return rho, ux, uy, sl, m, gx, gy, xx, yy

    def sim(self):
        """Eq. defFf on the pre-collision populations."""
        w, f = self.w, self.f
        chi = self.mask()
        dx, dy, nx, ny, s = self.pts
        x, y = self.x + dx, self.y + dy
        rx, ry = np.floor(x + 0.5), np.floor(y + 0.5)
        sig, count = np.zeros((3, len(x))), np.zeros(len(x))
        cxd, cyd = np.array(CX)[self.dirs], np.array(CY)[self.dirs]
        for u in range(2):
            for v in range(2):
                use = ((u == 0) | (ry == y + 0.5)) & ((v == 0) | (rx == x + 0.5))
                qi, qj = rx.astype(int) - v, ry.astype(int) - u
                done = np.zeros(len(x), bool)
                fi, fj = qi.copy(), qj.copy()
                for k in range(4):
                    ii = np.clip(qi + k * cxd, 0, w.nx - 1)
                    jj = np.clip(qj + k * cyd, 0, w.ny - 1)
                    hit = ~done & ~chi[jj, ii]
                    fi[hit], fj[hit] = ii[hit], jj[hit]
                    done |= hit
                if not use.any():
                    continue
                fl = f[:, torch.from_numpy(fj).to(f.device), torch.from_numpy(fi).to(f.device)].cpu().numpy()
                rho = fl.sum(0)
                ux = (sum(CX[a] * fl[a] for a in range(9)) + 0.5 * w.body_force[0]) / rho
                uy = (sum(CY[a] * fl[a] for a in range(9)) + 0.5 * w.body_force[1]) / rho
                p = np.zeros((3, len(x)))
                for a in range(9):
                    cu = CX[a] * ux + CY[a] * uy
                    d = fl[a] - WT[a] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))
                    p += np.array([[CX[a] * CX[a]], [CX[a] * CY[a]], [CY[a] * CY[a]]]) * d
                st = -self.af * p
                st[0] -= rho / 3
                st[2] -= rho / 3
                sig += np.where(use, st, 0.0)
                count += use
        sig /= count
        tx, ty = s * (sig[0] * nx + sig[1] * ny), s * (sig[1] * nx + sig[2] * ny)
        return np.array([tx.sum(), ty.sum(), (dx * ty - dy * tx).sum()])

    def step(self):
        """One time step; the MEM and SIM forces (F_x, F_y, T) of it."""
        w, f, dev = self.w, self.f, self.f.device
        rho, ux, uy, sl, m, gx, gy, xx, yy = self.moments()
        sim = self.sim()
        uu = ux * ux + uy * uy
        o = torch.empty_like(f)
        bfx, bfy = w.body_force
        forced = bfx != 0.0 or bfy != 0.0
        for a in (0, 1, 2, 5, 6):
            b = OPP[a]
            cu = CX[a] * ux + CY[a] * uy
            ep = WT[a] * rho * (1.0 + 4.5 * cu * cu - 1.5 * uu)
            em = WT[a] * rho * 3.0 * cu
            dp = -self.sp * (0.5 * (f[a] + f[b]) - ep)
            dm = -self.sm * (0.5 * (f[a] - f[b]) - em)
            del ep, em
            if forced:
                cg, ug = CX[a] * bfx + CY[a] * bfy, ux * bfx + uy * bfy
                dp += self.af * WT[a] * (9.0 * cu * cg - 3.0 * ug)
                dm += self.af * WT[a] * 3.0 * cg
            cg, ug = CX[a] * gx + CY[a] * gy, ux[sl] * gx + uy[sl] * gy
            dp[sl] += self.af * WT[a] * (9.0 * cu[sl] * cg - 3.0 * ug)
            dm[sl] += self.af * WT[a] * 3.0 * cg
            o[a] = f[a] + dp + dm
            if a:
                o[b] = f[b] + dp - dm
        del rho, uu, cu, dp, dm
        # MEM on the links of the box
        j0, j1, i0, i1 = self.box
        mem = torch.zeros(3, dtype=torch.float64, device=dev)
        for a in range(1, 9):
            js, jd = (slice(max(0, -CY[a]), m.shape[0] - max(0, CY[a])),
                      slice(max(0, CY[a]), m.shape[0] - max(0, -CY[a])))
            is_, id_ = (slice(max(0, -CX[a]), m.shape[1] - max(0, CX[a])),
                        slice(max(0, CX[a]), m.shape[1] - max(0, -CX[a])))
            me, nb = m[js, is_], m[jd, id_]
            sg = torch.where(me, -1.0, 1.0).double() * (me != nb)
            rx = xx[:, is_] - self.x + 0.5 * CX[a]
            ry = yy[js] - self.y + 0.5 * CY[a]
            q = sg * o[a][sl][js, is_]
            lx, ly = (CX[a] - (self.u[0] - self.om * ry)) * q, (CY[a] - (self.u[1] + self.om * rx)) * q
            mem += torch.stack([lx.sum(), ly.sum(), (rx * ly - ry * lx).sum()])
        mem = mem.cpu().numpy()
        self.f = self.stream(f, o)
        if w.body.moving:
            self.move(sim if w.body.estimator == "sim" else mem)
        return mem, sim

    def move(self, F):
        b = self.w.body
        r = 0.5 * b.length
        mass = b.density_ratio * math.pi * r * r
        buoy = 1.0 - 1.0 / b.density_ratio
        u0, w0 = list(self.u), self.om
        self.u = [u0[q] + F[q] / mass + buoy * b.gravity[q] for q in range(2)]
        self.om = w0 + F[2] / (0.5 * mass * r * r)
        self.x += 0.5 * (u0[0] + self.u[0])
        self.y += 0.5 * (u0[1] + self.u[1])

    def stream(self, pre, o):
        w = self.w
        xl, xh, yl, yh = w.bc
        f = torch.empty_like(o)
        for a in range(9):
            f[a] = torch.roll(o[a], (CY[a], CX[a]), (0, 1))
            for row, kind, inward in ((0, yl, 1), (w.ny - 1, yh, -1)):
                if CY[a] != inward or kind == "periodic":
                    continue
                if kind == "symmetry":
                    f[a][row] = torch.roll(o[FLIPY[a]][row], CX[a], 0)
                else:
                    f[a][row] = o[OPP[a]][row]
            if CX[a] == 1 and xl != "periodic":
                cin = 6 * WT[a] * (CX[a] * w.u_in[0] + CY[a] * w.u_in[1]) if xl == "inlet" else 0.0
                f[a][:, 0] = o[OPP[a]][:, 0] + cin
            if CX[a] == -1 and xh != "periodic":
                if xh == "outlet":
                    uc = math.hypot(*w.u_in)
                    f[a][:, -1] = (pre[a][:, -1] + uc * f[a][:, -2]) / (1 + uc)
                elif xh == "outlet_free":
                    f[a][:, -1] = f[a][:, -2]
                else:
                    f[a][:, -1] = o[OPP[a]][:, -1]
        return f


def exact(case, seed):
    out = []
    for k, w in enumerate(_workloads(case, seed)):
        e = _Exact(w, _initial(w, 1000 * seed + k))
        e.step()
        rows = [e.step() for _ in range(case["steps"])]
        rho, ux, uy = e.moments()[:3]
        # one step's forces on a lattice stored in 16 bits carry the storage rounding
        # at full size (unless FP16 is rounded stochastically): no value to hold them to
        forces = w.dtype in ("f64", "f32", "f16sr")
        out.append({"mem": np.array([r[0] for r in rows]) if forces else None,
                    "sim": np.array([r[1] for r in rows]) if forces else None,
                    "rho": rho, "ux": ux, "uy": uy})
    return out
