"""The solves that users of this library run, as timed passes with an independent 64-bit answer.

A pass is what a program does between two looks at its solution: advance a solver by a
block of time steps, read the residual, read the fields.  Meshes and handles belong to
`prepare`, as in a program that keeps them for the whole run.  FP32-compute solvers hand
their fields on in FP32 (the program's snapshots), FP64 solvers in FP64.

`exact` restates the scheme (face-based finite volumes, paper Sec. II-III) with plain
torch in FP64 and does not use this library's code.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2007_07347_gb300 import meshes as M
from paper_2007_07347_gb300 import sdugks as S

U_LID = 0.1

PERIODIC, WALL, MOVING, FARFIELD = M.BC_PERIODIC, M.BC_WALL, M.BC_MOVING_WALL, M.BC_FARFIELD


def listed():
    return [
        # the accuracy study: FP64 plane Couette channel, a few hundred cells, checkpointed
        # whole (f and W) after every thousand steps; each step is one small launch
        dict(name="couette_4x64_fp64", flow="couette", nx=4, ny=64, re=10.0, precision="fp64", steps=1000),
        # the longest channel of the serving mix: narrow and tall, far below one wave
        dict(name="couette_4x1024_fp32", flow="couette", nx=4, ny=1024, re=10.0, precision="fp32", steps=1000),
        # the headline benchmark: lid-driven cavity, Re 1000, residual every thousand steps
        dict(name="cavity_256_fp32", flow="cavity", nx=256, ny=256, re=1000.0, precision="fp32", steps=1000),
        # a request of the serving mix with an odd, ragged size and a high Reynolds number
        dict(name="cavity_723_fp32", flow="cavity", nx=723, ny=723, re=3200.0, precision="fp32", steps=200),
        # the largest grid of the benchmark's size sweep, its state in HBM
        dict(name="cavity_2048_fp32", flow="cavity", nx=2048, ny=2048, re=5000.0, precision="fp32", steps=50),
        # the parity mode on the headline grid
        dict(name="cavity_256_fp64", flow="cavity", nx=256, ny=256, re=1000.0, precision="fp64", steps=50),
        # half-size storage on a uniform grid
        dict(name="cavity_1024_bf16dev", flow="cavity", nx=1024, ny=1024, re=2000.0, precision="bf16dev", steps=100),
        # the body-fitted validation: shuffled O-mesh, bf16 storage, drag read with the residual
        dict(name="cylinder_512x256_bf16dev", flow="cylinder", nx=512, ny=256, re=40.0, precision="bf16dev", steps=500),
        # a small cylinder of the serving mix in FP32
        dict(name="cylinder_208x104_fp32", flow="cylinder", nx=208, ny=104, re=60.0, precision="fp32", steps=500),
        # many uneven cavities at once, drawn log-uniformly from 32 to 512, each retired once
        dict(name="batch_32_fp32", flow="batch", count=32, n_lo=32, n_hi=512, draw_seed=1, precision="fp32", steps=500),
        # the rarefied micro cavity on the paper's grids
        dict(name="micro_40_nv100_fp32", flow="micro", nx=40, nv=100, kn=1.0, precision="fp32", steps=50),
        # a small rarefied cavity on sizes that divide nothing
        dict(name="micro_23_nv50_fp32", flow="micro", nx=23, nv=50, kn=0.1, precision="fp32", steps=200),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more solve of the same ranges."""
    flow = rng.choice(["cavity", "cavity", "cavity", "couette", "cylinder", "batch", "micro", "micro"])
    if flow == "cavity":
        prec = rng.choice(["fp32", "fp32", "fp32", "bf16dev", "fp16dev", "fp64"])
        n = int(round(_log(rng, 32, 1024 if prec == "fp64" else 2048)))
        if n > 128 and rng.random() < 0.5:
            n += 1 - n % 2                        # odd
        cost = 30.0 if prec == "fp64" else 1.0    # steps so that the pass stays below the largest listed one
        steps = int(min(1000, max(4, 2.0e8 / (n * n * cost))))
        return dict(flow="cavity", nx=n, ny=n, re=round(_log(rng, 100, 5000), 1), precision=prec, steps=steps)
    if flow == "couette":
        return dict(flow="couette", nx=4, ny=int(round(_log(rng, 64, 1024))), re=10.0,
                    precision=rng.choice(["fp32", "fp64"]), steps=rng.randint(300, 1000))
    if flow == "cylinder":
        nt = 16 * int(round(_log(rng, 128, 512) / 16))
        return dict(flow="cylinder", nx=nt, ny=max(16, nt // 2), re=round(_log(rng, 10, 100), 1),
                    precision=rng.choice(["fp32", "bf16dev"]), steps=rng.randint(100, 500))
    if flow == "batch":
        case = dict(flow="batch", count=rng.randint(4, 32), n_lo=32, n_hi=rng.choice([128, 256, 512]),
                    draw_seed=rng.randint(2, 10 ** 6), precision=rng.choice(["fp32", "fp32", "bf16dev"]))
        return dict(case, steps=int(min(rng.randint(100, 500), 8.0e8 / sum(n * n for n, _ in _sizes(case)))))
    n, nv = int(round(_log(rng, 8, 40))), int(round(_log(rng, 16, 100)))
    return dict(flow="micro", nx=n, nv=nv, kn=round(_log(rng, 0.1, 8.0), 2), precision=rng.choice(["fp32", "fp32", "fp64"]),
                steps=int(min(200, max(5, 4.0e8 / (n * n * nv * nv)))))


# ---------------------------------------------------------------- grids and starting fields

def _geometry(case):
    """(lx, ly, tau, dt) of a uniform-grid case in lattice units."""
    nx, ny, re = case["nx"], case["ny"], case["re"]
    if case["flow"] == "couette":
        h = 1.0 / ny
        return nx * h, 1.0, 3.0 * U_LID / re, 0.5 * h / math.sqrt(2.0)
    return float(nx), float(ny), 3.0 * U_LID * nx / re, 0.5 / math.sqrt(2.0)


def _sizes(case):
    """(edge, Reynolds number) of each cavity of a batch."""
    rng = np.random.default_rng(case["draw_seed"])
    ns = np.rint(np.exp(rng.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]), case["count"]))).astype(int)
    res = np.exp(rng.uniform(math.log(100.0), math.log(5000.0), case["count"]))
    return [(int(n), float(r)) for n, r in zip(ns, res)]


def _start(nx, ny, seed, periodic_x=False):
    """Smooth seeded fields on a grid: rho 1 +- 1 %, u of a few large eddies that vanish at
    the walls; [nx * ny] and [nx * ny, 2], cell i + nx j."""
    rng = np.random.default_rng(seed)
    x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
    rho, u, v = np.ones((ny, nx)), np.zeros((ny, nx)), np.zeros((ny, nx))
    for _ in range(3):
        kx, ky = int(rng.integers(1, 4)), int(rng.integers(1, 4))
        a, b, c = rng.normal(size=3) / 3.0
        cx = np.cos(2 * math.pi * (kx * x + rng.random())) if periodic_x else np.sin(math.pi * kx * x)
        sy = np.sin(math.pi * ky * y)
        rho += 0.01 * a * np.outer(np.cos(math.pi * ky * y), np.cos(2 * math.pi * kx * x))
        u += 0.05 * b * np.outer(sy, cx)
        v += 0.05 * c * np.outer(sy, cx)
    return rho.ravel(), np.stack([u.ravel(), v.ravel()], 1)


def _cylinder_mesh(nt, nr, seed=7):
    """O-mesh around a cylinder of diameter 1 out to 50 diameters, first cell 0.005, cells and
    faces in a random order, as face-owner/neighbour arrays (patches: 0 wall, 1 far field),
    with each cell's polar position."""
    r0, first, far = 0.5, 0.005, 50.0
    lo, hi = 1.0 + 1e-12, 2.0
    for _ in range(200):
        q = 0.5 * (lo + hi)
        lo, hi = (q, hi) if r0 + first * (q ** nr - 1.0) / (q - 1.0) < far else (lo, q)
    radii = r0 + first * (q ** np.arange(nr + 1) - 1.0) / (q - 1.0)
    radii[-1] = far
    th = 2.0 * math.pi * np.arange(nt) / nt
    pts = np.stack([np.outer(radii, np.cos(th)).ravel(), np.outer(radii, np.sin(th)).ravel()], 1)
    k, i = (a.ravel() for a in np.meshgrid(np.arange(nr), np.arange(nt), indexing="ij"))
    fp = [np.stack([i + nt * k, i + nt * (k + 1)], 1)]
    own, nbr = [(i - 1) % nt + nt * k], [i + nt * k]
    k, i = (a.ravel() for a in np.meshgrid(np.arange(nr + 1), np.arange(nt), indexing="ij"))
    fp.append(np.stack([i + nt * k, (i + 1) % nt + nt * k], 1))
    own.append(np.where(k == 0, i, i + nt * (k - 1)))
    nbr.append(np.where(k == 0, -1, np.where(k == nr, -2, i + nt * k)))
    fp, own, nbr = np.concatenate(fp), np.concatenate(own), np.concatenate(nbr)
    rng = np.random.default_rng(seed)
    cp, fo = rng.permutation(nt * nr), rng.permutation(len(own))
    own, nbr, fp = cp[own[fo]], np.where(nbr[fo] >= 0, cp[np.maximum(nbr[fo], 0)], nbr[fo]), fp[fo]
    pos = np.empty((nt * nr, 2))
    pos[cp, 0] = np.repeat(0.5 * (radii[:-1] + radii[1:]), nt)
    pos[cp, 1] = np.tile(2.0 * math.pi * (np.arange(nt) + 0.5) / nt, nr)
    return pts, fp.astype(np.int64), own.astype(np.int64), nbr.astype(np.int64), pos


def _cylinder_numbers(case):
    d = min(0.005, math.pi / case["nx"])
    return 3.0 * U_LID / case["re"], 0.5 * d / math.sqrt(2.0)


def _cylinder_start(pos, seed):
    """The free stream with a seeded kick in the near wake, and a faint pressure pattern."""
    rng = np.random.default_rng(seed)
    x, y = pos[:, 0] * np.cos(pos[:, 1]), pos[:, 0] * np.sin(pos[:, 1])
    u = np.zeros((len(x), 2))
    u[:, 0] = U_LID
    for _ in range(3):
        cx, cy, a, b = rng.uniform(1.0, 3.0), rng.uniform(-1.0, 1.0), *rng.normal(size=2)
        g = np.exp(-((x - cx) ** 2 + (y - cy) ** 2))
        u[:, 0] += 0.1 * U_LID * a * g
        u[:, 1] += 0.1 * U_LID * b * g
    return 1.0 + 0.002 * rng.normal() * np.exp(-0.1 * (x * x + y * y)), u


def _micro_start(n, seed):
    rho, u = _start(n, n, seed)
    rng = np.random.default_rng(seed + 1)
    x = (np.arange(n) + 0.5) / n
    rt = 0.5 + 0.02 * rng.normal() * np.outer(np.sin(math.pi * x), np.sin(math.pi * x)).ravel()
    return rho, u, rt


# ---------------------------------------------------------------- the passes

@functools.lru_cache(maxsize=2)
def _library_mesh(key):
    """The library's mesh handles of a case: a program builds them once and keeps them."""
    case = dict(key)
    if case["flow"] == "batch":
        made = [M.cavity(n, U=U_LID, Re=r) for n, r in _sizes(case)]
    elif case["flow"] == "cavity":
        made = [M.cavity(case["nx"], U=U_LID, Re=case["re"])]
    elif case["flow"] == "couette":
        made = [M.couette(case["ny"], nx=case["nx"], U=U_LID, Re=case["re"])]
    elif case["flow"] == "micro":
        made = [M.micro_cavity(case["nx"], case["kn"], U=U_LID, nv=case["nv"])]
    else:
        pts, fp, own, nbr, pos = _cylinder_mesh(case["nx"], case["ny"])
        tau, dt = _cylinder_numbers(case)
        mesh = M.Mesh(pts, fp, own, nbr, case["nx"] * case["ny"], dict(wall=0, farfield=1))
        made = [M.Case("cylinder", mesh, [(0, WALL, (0.0, 0.0, 0.0)), (1, FARFIELD, (1.0, U_LID, 0.0))], tau, dt,
                       meta=dict(pos=pos))]
    return [(c, S.Mesh(c.mesh, c.bcs)) for c in made]


def _mesh(case):
    key = tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "steps", "precision")))
    return _library_mesh(key)


def prepare(case, seed):
    flow, prec = case["flow"], case["precision"]
    made = _mesh(case)
    c, mesh = made[0]
    st = dict(case)
    if flow == "batch":
        pool = sum(32 * (n + 32) * (n + 32) * 9 for n, _ in _sizes(case)) + (1 << 20)
        b = S.Batch(pool, prec, max_instances=case["count"])
        st["ids"] = [b.add(m, k.tau, k.dt, *_start(k.mesh.meta["nx"], k.mesh.meta["ny"], seed + q))
                     for q, (k, m) in enumerate(made)]
        st["solver"] = b
        return st
    if flow == "micro":
        k = c.meta
        st["solver"] = S.Dvm(mesh, k["nv"], k["vmax"], k["RT0"], c.tau, c.dt, prec).init(*_micro_start(case["nx"], seed))
        return st
    if flow == "cylinder":
        start = _cylinder_start(c.meta["pos"], seed)
    else:
        start = _start(case["nx"], case["ny"], seed, flow == "couette")
    st["solver"] = S.Solver(mesh, c.tau, c.dt, prec).init(*start)
    n = c.mesh.n_cells
    st["mesh"] = mesh
    st["rho"] = torch.empty(n, dtype=torch.float64, device="cuda")
    st["u"] = torch.empty(n, 2, dtype=torch.float64, device="cuda")
    return st


def run(st):
    s, wide = st["solver"], st["precision"] == "fp64"
    if st["flow"] == "batch":
        s.step(st["steps"])
        res = s.residual()
        out = [s.macros(i) for i in st["ids"]]
        return dict(eps=np.array([res[i][0] for i in st["ids"]], np.float32),
                    mass=np.array([res[i][1] for i in st["ids"]], np.float32),
                    rho=np.concatenate([o[0] for o in out]).astype(np.float32),
                    u=np.concatenate([o[1] for o in out]).astype(np.float32))
    if st["flow"] == "micro":
        s.step(st["steps"])
        out = s.macros()
        return list(out) if wide else [x.astype(np.float32) for x in out]
    if st["flow"] == "cylinder":
        s.step(st["steps"] - 1)
        force = s.step_forces()[:1].astype(np.float32)      # drag and lift
    else:
        s.step(st["steps"])
        force = None
    eps, mass = s.residual()
    if st["flow"] == "couette" and wide:       # the study's checkpoint
        f, w = s.get_state()
        return dict(eps=eps, mass=mass, f=f, W=w)
    s.macros_device(st["rho"], st["u"])
    if wide:
        return dict(eps=eps, mass=mass, rho=st["rho"], u=st["u"])
    return dict(eps=eps, mass=mass, force=force, rho=st["rho"].float(), u=st["u"].float())


def work(case):
    """Bytes: the state (f and the FP64 conserved variables) read and written once a step,
    and on unstructured meshes each face's cells and geometry; flops: the scheme's own."""
    steps = case["steps"]
    fs = {"fp64": 8, "fp32": 4, "bf16dev": 2, "fp16dev": 2}[case["precision"]]
    if case["flow"] == "micro":
        n, q = case["nx"] ** 2, case["nv"] ** 2
        return dict(bytes=steps * n * (2 * q * fs + 64), flops=steps * n * q * 60.0)
    cells = sum(n * n for n, _ in _sizes(case)) if case["flow"] == "batch" else case["nx"] * case["ny"]
    mesh = 64 if case["flow"] == "cylinder" else 0
    return dict(bytes=steps * cells * (18 * fs + 48 + mesh), flops=steps * cells * 400.0)


# ---------------------------------------------------------------- the same passes in 64 bits

def _faces(case):
    """Face-based description of a case: points, face points, owners, neighbours (-1 - patch on
    the boundary), the cell count, and {patch: (kind, parameters)}."""
    if case["flow"] == "cylinder":
        pts, fp, own, nbr, _ = _cylinder_mesh(case["nx"], case["ny"])
        return pts, fp, own, nbr, case["nx"] * case["ny"], {0: (WALL, None), 1: (FARFIELD, (1.0, U_LID, 0.0))}
    if case["flow"] == "micro":
        nx = ny = case["nx"]
        lx = ly = 1.0
    else:
        nx, ny = case["nx"], case["ny"]
        lx, ly = _geometry(case)[:2]
    j, i = (a.ravel() for a in np.meshgrid(np.arange(ny + 1), np.arange(nx + 1), indexing="ij"))
    pts = np.stack([i * (lx / nx), j * (ly / ny)], 1)
    j, i = (a.ravel() for a in np.meshgrid(np.arange(ny), np.arange(nx + 1), indexing="ij"))
    fp = [np.stack([i + (nx + 1) * j, i + (nx + 1) * (j + 1)], 1)]
    own = [np.where(i == 0, nx * j, i - 1 + nx * j)]
    nbr = [np.where(i == 0, -4, np.where(i == nx, -2, i + nx * j))]
    j, i = (a.ravel() for a in np.meshgrid(np.arange(ny + 1), np.arange(nx), indexing="ij"))
    fp.append(np.stack([i + (nx + 1) * j, i + 1 + (nx + 1) * j], 1))
    own.append(np.where(j == 0, i, i + nx * (j - 1)))
    nbr.append(np.where(j == 0, -1, np.where(j == ny, -3, i + nx * j)))
    bcs = {0: (WALL, None), 1: (WALL, None), 2: (MOVING, (U_LID, 0.0)), 3: (WALL, None)}
    if case["flow"] == "couette":
        bcs[1], bcs[3] = (PERIODIC, (3, -lx, 0.0)), (PERIODIC, (1, lx, 0.0))
    return pts, np.concatenate(fp), np.concatenate(own), np.concatenate(nbr), nx * ny, bcs


class _Plain:
    """Geometry of a face-based mesh in plain FP64 torch: n l, offsets, volumes, LLSR inverse."""

    def __init__(self, faces):
        pts, fp, own, nbr, n, bcs = faces
        p, q = pts[fp[:, 0]], pts[fp[:, 1]]
        xf, nl = 0.5 * (p + q), np.stack([q[:, 1] - p[:, 1], -(q[:, 0] - p[:, 0])], 1)
        inner = nbr >= 0

        def gather(w):
            """Sum over a cell's faces of a per-face value (owner side, neighbour side)."""
            o, k = w
            s = np.zeros((n,) + o.shape[1:])
            np.add.at(s, own, o)
            np.add.at(s, nbr[inner], k[inner])
            return s
        ones = np.ones(len(own))
        mid = gather((xf, xf)) / gather((ones, ones))[:, None]
        nb0 = np.where(inner, nbr, own)
        # outward from the owner: away from the owner's mean point
        nl[np.einsum("fd,fd->f", xf - mid[own], nl) < 0] *= -1.0
        at = 0.5 * np.einsum("fd,fd->f", xf - mid[own], nl), -0.5 * np.einsum("fd,fd->f", xf - mid[nb0], nl)
        vol = gather(at)
        xc = mid + gather((at[0][:, None] * (xf - mid[own]), at[1][:, None] * (xf - mid[nb0]))) * (2.0 / 3.0) / vol[:, None]
        other, pos, kind = np.where(inner, nbr, -1), xc[nb0].copy(), np.zeros(len(own), int)
        self.patch = np.where(inner, -1, -1 - nbr)
        par = np.zeros((len(own), 3))
        for p_, (k_, v) in bcs.items():
            sel = np.where(nbr == -1 - p_)[0]
            if k_ != PERIODIC:
                kind[sel] = k_
                if v is not None:
                    par[sel, :len(v)] = v
                continue
            far = np.where(nbr == -1 - v[0])[0]
            a, b = xf[sel] + np.array(v[1:]), xf[far]
            sa, sb = np.lexsort(np.round(a, 9).T), np.lexsort(np.round(b, 9).T)
            other[sel[sa]] = own[far[sb]]
            pos[sel[sa]] = xc[own[far[sb]]] - np.array(v[1:])
        link = other >= 0
        d = np.where(link[:, None], pos - xc[own], 0.0)
        dd = np.stack([d[:, 0] ** 2, d[:, 0] * d[:, 1], d[:, 1] ** 2], 1)
        xx, xy, yy = gather((dd, np.where(inner[:, None], dd, 0.0))).T
        det = xx * yy - xy * xy
        dev = torch.device("cuda")
        t = lambda v: torch.from_numpy(np.ascontiguousarray(v)).to(dev)  # noqa: E731
        self.n, self.own, self.other, self.inner, self.link = n, t(own), t(np.maximum(other, 0)), t(np.where(inner)[0]), t(link)
        self.nl, self.ro, self.rk, self.d, self.vol = t(nl), t(xf - xc[own]), t(xf - pos), t(d), t(vol)
        self.inv = t(np.stack([yy, -xy, xx], 1) / det[:, None])
        self.kind, self.par = t(kind), t(par)

    def gather(self, o, k):
        s = torch.zeros(self.n, o.shape[1], dtype=torch.float64, device=o.device)
        s.index_add_(0, self.own, o)
        return s.index_add_(0, self.other[self.inner], k[self.inner])

    def gradients(self, phi):
        diff = torch.where(self.link[:, None], phi[self.other] - phi[self.own], 0.0)
        bx, by = diff * self.d[:, :1], diff * self.d[:, 1:]
        bx, by = self.gather(bx, bx), self.gather(by, by)
        return self.inv[:, :1] * bx + self.inv[:, 1:2] * by, self.inv[:, 1:2] * bx + self.inv[:, 2:] * by

    def interface(self, phi, xi, dt, s, tie=1e-12):
        """The distribution that arrives at each face along the characteristics, and the owner's own."""
        sx, sy = self.gradients(phi)

        def side(cell, r):
            return phi[cell] + (r[:, :1] - dt * xi[:, 0]) * sx[cell] + (r[:, 1:] - dt * xi[:, 1]) * sy[cell]
        a = side(self.own, self.ro)
        b = side(self.other, self.rk)
        up = torch.where(s > tie, a, torch.where(s < -tie, b, 0.5 * (a + b)))
        return torch.where(self.link[:, None], up, a), a


def _d2q9(case):
    """(f, W, eps, mass, force on patch 0) after the pass; a batch is one mesh of separate parts."""
    dev = torch.device("cuda")
    parts = [dict(flow="cavity", nx=n, ny=n, re=r) for n, r in _sizes(case)] if case["flow"] == "batch" else [case]
    all_, taus, dts, starts, at = [], [], [], [], [0]
    for q, c in enumerate(parts):
        faces = _faces(c)
        tau, dt = _cylinder_numbers(c) if c["flow"] == "cylinder" else _geometry(c)[2:]
        all_.append(faces)
        taus.append(tau)
        dts.append(dt)
        at.append(at[-1] + faces[4])
        if c["flow"] == "cylinder":
            starts.append(_cylinder_start(_cylinder_mesh(c["nx"], c["ny"])[4], case["seed"]))
        else:
            starts.append(_start(c["nx"], c["ny"], case["seed"] + q, c["flow"] == "couette"))
    if len(parts) > 1:
        po = np.cumsum([0] + [len(f[0]) for f in all_])
        # the parts side by side, far enough apart that no point is shared
        merged = (np.concatenate([f[0] for f in all_]), np.concatenate([f[1] + o for f, o in zip(all_, po)]),
                  np.concatenate([f[2] + o for f, o in zip(all_, at)]),
                  np.concatenate([np.where(f[3] >= 0, f[3] + o, f[3]) for f, o in zip(all_, at)]), at[-1], all_[0][5])
    else:
        merged = all_[0]
    g = _Plain(merged)
    each = lambda v: torch.cat([torch.full((b - a, 1), x, dtype=torch.float64, device=dev)  # noqa: E731
                                for x, a, b in zip(v, at, at[1:])])
    tau, dt = each(taus), each(dts)
    xi = torch.tensor([[0, 0], [1, 0], [0, 1], [-1, 0], [0, -1], [1, 1], [-1, 1], [-1, -1], [1, -1]],
                      dtype=torch.float64, device=dev)
    w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64, device=dev)

    def feq(rho, ux, uy):
        eu = ux * xi[:, 0] + uy * xi[:, 1]
        return w * rho * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))

    def moments(f):
        return torch.stack([f.sum(1), f @ xi[:, 0], f @ xi[:, 1]], 1)

    def feq_w(W):
        r = W[:, :1]
        return feq(r, W[:, 1:2] / r, W[:, 2:] / r)
    rho = torch.from_numpy(np.concatenate([r for r, _ in starts])).to(dev)[:, None]
    u = torch.from_numpy(np.concatenate([v for _, v in starts])).to(dev)
    W = torch.cat([rho, rho * u], 1)
    f = feq_w(W)
    ef, tf = dt[g.own], tau[g.own]
    s = g.nl @ xi.T
    bound = torch.where(~g.link)[0]
    ob, kb, pb = g.own[bound], g.kind[bound][:, None], g.par[bound]
    sb, force, u0 = s[bound], None, u
    for _ in range(case["steps"]):
        fe = feq_w(W)
        plus = ((2 * tau - dt) * f + dt * fe) / (2 * tau)
        up, _ = g.interface(plus, xi, ef, s)
        fb = (up + ef / (2 * tf) * feq_w(moments(up))) * (2 * tf / (2 * tf + ef))
        if len(bound):
            r = torch.where(kb == FARFIELD, pb[:, :1], W[ob, :1])
            off = (kb == FARFIELD)
            ux = torch.where(kb == WALL, 0.0, torch.where(off, pb[:, 1:2], pb[:, :1]))
            uy = torch.where(kb == WALL, 0.0, torch.where(off, pb[:, 2:], pb[:, 1:2]))
            eb = feq(r, ux, uy)
            out = (up[bound] + ef[bound] / (2 * tf[bound]) * eb) * (2 * tf[bound] / (2 * tf[bound] + ef[bound]))
            fb[bound] = torch.where(sb < -1e-12, eb + f[ob] - fe[ob], out)
        flux = s * fb
        force = flux @ xi
        F = g.gather(flux, -flux) * (dt / g.vol[:, None])
        W = W - moments(F)
        f = (f - F + dt / tau * feq_w(W)) / (1.0 + dt / tau)
    u = W[:, 1:] / W[:, :1]
    eps, mass = [], []
    for a, b in zip(at, at[1:]):
        eps.append(float((u[a:b] - u0[a:b]).norm() / u0[a:b].norm()))
        mass.append(float((g.vol[a:b] * W[a:b, 0]).sum()))
    wall = force[torch.from_numpy(g.patch == 0).to(dev)].sum(0, keepdim=True)
    return f, W, eps, mass, wall


def _micro(case):
    """(rho, u, R T) after the pass."""
    dev = torch.device("cuda")
    n, nv, rt0, vmax = case["nx"], case["nv"], 0.5, 2.0
    g = _Plain(_faces(case))
    h = 2.0 * vmax / nv
    node = -vmax + (torch.arange(nv, dtype=torch.float64, device=dev) + 0.5) * h
    xi = torch.stack([node.repeat(nv), node.repeat_interleave(nv)], 1)
    psi = torch.stack([torch.ones(nv * nv, dtype=torch.float64, device=dev), xi[:, 0], xi[:, 1], 0.5 * (xi * xi).sum(1)], 1)
    tau = case["kn"] * math.sqrt(2.0 / (math.pi * rt0))
    dt = 0.5 * (1.0 / n) / (math.sqrt(2.0) * (vmax - 0.5 * h))

    def maxwell(rho, ux, uy, rt):
        c2 = (xi[:, 0] - ux) ** 2 + (xi[:, 1] - uy) ** 2
        return h * h * rho / (2.0 * math.pi * rt) * torch.exp(-c2 / (2.0 * rt))

    def feq_w(W):
        r, ux, uy = W[:, :1], W[:, 1:2] / W[:, :1], W[:, 2:3] / W[:, :1]
        return maxwell(r, ux, uy, W[:, 3:] / r - 0.5 * (ux * ux + uy * uy))
    rho, u, rt = (torch.from_numpy(v).to(dev) for v in _micro_start(n, case["seed"]))
    W = torch.cat([rho[:, None], rho[:, None] * u, (rho * (0.5 * (u * u).sum(1) + rt))[:, None]], 1)
    f = feq_w(W)
    b, c, tie = dt / (2 * tau), 2 * tau / (2 * tau + dt), 1e-12
    s = g.nl @ xi.T
    wall = torch.where(~g.link)[0]
    sw = s[wall]
    into = sw < -tie
    gw = maxwell(torch.ones(len(wall), 1, dtype=torch.float64, device=dev),
                 torch.where(g.kind[wall] == MOVING, g.par[wall, 0], 0.0)[:, None],
                 torch.where(g.kind[wall] == MOVING, g.par[wall, 1], 0.0)[:, None], rt0)
    for _ in range(case["steps"]):
        plus = ((2 * tau - dt) * f + dt * feq_w(W)) / (2 * tau)
        up, _ = g.interface(plus, xi, dt, s)
        fb = (up + b * feq_w(up @ psi)) * c
        so = torch.where(into, 0.0, sw * up[wall]).sum(1)
        go, gin = torch.where(into, 0.0, sw * gw).sum(1), torch.where(into, sw * gw, 0.0).sum(1)
        rw = (-c * so / (c * b * go + gin))[:, None]
        fb[wall] = torch.where(into, rw * gw, (up[wall] + b * rw * gw) * c)
        flux = s * fb
        F = g.gather(flux, -flux) * (dt / g.vol[:, None])
        W = W - F @ psi
        f = (f - F + dt / tau * feq_w(W)) / (1.0 + dt / tau)
    u = W[:, 1:3] / W[:, :1]
    return [W[:, 0], u, W[:, 3] / W[:, 0] - 0.5 * (u * u).sum(1)]


def exact(case, seed):
    case = dict(case, seed=seed)
    if case["flow"] == "micro":
        return _micro(case)
    f, W, eps, mass, force = _d2q9(case)
    u = W[:, 1:] / W[:, :1]
    if case["flow"] == "batch":
        return dict(eps=np.array(eps), mass=np.array(mass), rho=W[:, 0].cpu().numpy(), u=u.cpu().numpy())
    if case["flow"] == "couette" and case["precision"] == "fp64":
        return dict(eps=eps[0], mass=mass[0], f=f.cpu().numpy(), W=W.cpu().numpy())
    return dict(eps=eps[0], mass=mass[0], force=force if case["flow"] == "cylinder" else None, rho=W[:, 0], u=u)
