"""Measured cases: wave propagation through the package's public entry points.

Five kinds of call that a user's program makes, over the sizes, meshes,
degrees and arithmetics that the package is used with:

  erk      one shot stepped explicitly on the device, receivers recorded after
           every step, then a canonical snapshot (hho_erk_step_record,
           hho_state_unpack); with ``energy`` the run is cut into pieces and the
           discrete energy is read between them (hho_energy);
  shots    many shots advanced together (hho_batch_erk_step, hho_batch_unpack);
  host     one step end to end from a pinned host vector (hho_erk_run_host);
  adjoint  the gradient of recorded traces with respect to the materials and
           the wavelet (hho_adjoint_vjp, hho_adjoint_vjp_f32);
  sdirk    implicit steps beyond the explicit limit (hho_sdirk_step).

Meshes lie on [0, width] x [0, 1] with a solid below a water layer: ``quad``
(rectangles), ``tri`` (split squares), ``hybrid`` (squares below y = 0.7, split
squares above) and ``hanging`` (every fourth row refined twice, so that its
neighbours are pentagons with a hanging node).  The solid carries a smooth
random field of +-20 %; every state has a point force with a Ricker wavelet.

``exact`` states the scheme again in plain 64-bit torch, with nodal face values
at Gauss points, dense cell matrices and autograd for the gradients.
"""
import math

import numpy as np
import torch

from paper_2505_15771_gb300 import hho
from paper_2505_15771_gb300.solver import Problem

# largest stable dt c_max / h of classical ERK4 on squares and on split squares
_CFL = {"quad": {1: 0.233, 2: 0.122, 3: 0.082}, "hanging": {1: 0.19, 2: 0.10, 3: 0.066},
        "tri": {1: 0.135, 2: 0.07, 3: 0.045}, "hybrid": {1: 0.135, 2: 0.07, 3: 0.045}}
_OF_STAGES = {2: 0.7, 3: 0.88, 4: 1.0}
_PREC = {"f64": hho.HHO_F64, "f32": hho.HHO_F32, "f32x2": hho.HHO_F32X2}
_F0 = 10.0


def _case(kind, mesh, nx, ny, k, stages, steps, arith="f64", shots=1, receivers=16, width=0.0, **more):
    return dict(kind=kind, mesh=mesh, nx=nx, ny=ny, width=float(width or nx / ny), k=k, stages=stages, steps=steps,
                arith=arith, shots=shots, receivers=receivers, **more)


def listed():
    return [
        # the 512-triangle academic run, whole: a mesh for teaching and convergence tables, all latency
        dict(_case("erk", "tri", 16, 16, 1, 4, 200, receivers=8, at_interface=True), name="academic_tri512_k1"),
        # the paper's 64 x 64 run with three sensors, the energy read every tenth of the run
        dict(_case("erk", "quad", 64, 64, 2, 4, 40, receivers=3, energy=4), name="squares64_k2_energy"),
        # local refinement on an odd grid: pentagons, ERK3 at the highest degree
        dict(_case("erk", "hanging", 101, 67, 3, 3, 12, receivers=33), name="hanging_k3_erk3"),
        # the benchmark's bilayer at full size in FP64 and in double-float
        dict(_case("erk", "quad", 1024, 512, 2, 4, 4, receivers=256), name="bilayer_k2_f64"),
        dict(_case("erk", "quad", 1024, 512, 2, 4, 4, "f32x2", receivers=256), name="bilayer_k2_f32x2"),
        # squares and triangles at the highest degree in FP64, the hybrid recipe at half its resolution
        dict(_case("erk", "hybrid", 680, 340, 3, 4, 2, receivers=256), name="hybrid_k3_f64"),
        # a survey: 16 shots in FP32 on the same mesh (the largest case)
        dict(_case("shots", "hybrid", 680, 340, 3, 4, 2, "f32", shots=16, receivers=256), name="shots16_hybrid_k3_f32"),
        # a survey on a locally refined mesh, an odd number of shots
        dict(_case("shots", "hanging", 331, 167, 2, 4, 3, "f32", shots=21, receivers=128),
             name="shots21_hanging_k2_f32"),
        # one step from and to pinned host memory: a solver driven by a host program
        dict(_case("host", "quad", 1024, 512, 2, 4, 1, receivers=0), name="host_bilayer_k2_f64"),
        # full-waveform inversion: the gradient of one shot's misfit on the 256 x 256 two-layer model
        dict(_case("adjoint", "quad", 256, 256, 2, 4, 40, receivers=128, checkpoint=20, at_interface=True),
             name="adjoint_k2_f64"),
        dict(_case("adjoint", "quad", 256, 256, 2, 4, 40, "f32", receivers=128, checkpoint=20, at_interface=True),
             name="adjoint_k2_f32"),
        # implicit stepping at four times the explicit limit
        dict(_case("sdirk", "quad", 256, 128, 2, 3, 1, receivers=0, ratio=4.0, tol=1e-8, restart=10),
             name="sdirk_bilayer_k2"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["erk", "erk", "erk", "shots", "shots", "host", "adjoint", "sdirk"])
    k = rng.choice([1, 2, 2, 3])
    mesh = rng.choice(["quad", "quad", "tri", "hybrid", "hanging"])
    top = {"erk": 200_000, "shots": 40_000, "host": 200_000, "adjoint": 40_000, "sdirk": 16_000}[kind]
    squares = _log(rng, 100, top)
    ny = max(6, int(math.sqrt(squares / rng.uniform(1.0, 2.5))))
    nx = max(8, squares // ny)
    width = nx / ny * rng.choice([1.0, 1.0, 1.25]) if mesh == "quad" else nx / ny
    stages = rng.choice([2, 3, 4, 4])
    steps = max(1, min(rng.randint(2, 40), 1_500_000 // squares))
    receivers = rng.choice([1, 5, 37, 128])
    if kind == "erk":
        return _case(kind, mesh, nx, ny, k, stages, steps, rng.choice(["f64", "f64", "f32x2"]), receivers=receivers,
                     width=width, at_interface=rng.random() < 0.3)
    if kind == "shots":
        shots = rng.randint(2, max(3, min(40, 400_000 // squares)))
        return _case(kind, mesh, nx, ny, k, stages, min(steps, 3), rng.choice(["f32", "f32", "f32x2", "f64"]),
                     shots=shots, receivers=receivers, width=width)
    if kind == "host":
        return _case(kind, mesh, nx, ny, k, stages, 1, rng.choice(["f64", "f32x2"]), receivers=0, width=width)
    if kind == "adjoint":
        steps = max(2, min(steps, 20))
        return _case(kind, mesh, nx, ny, k, stages, steps, rng.choice(["f64", "f32"]), receivers=receivers,
                     width=width, checkpoint=rng.randint(max(1, steps // 3), steps),
                     at_interface=rng.random() < 0.5)
    return _case(kind, mesh, nx, ny, min(k, 2), rng.choice([1, 2, 3]), 1, receivers=0, width=width,
                 ratio=rng.choice([2.0, 4.0]), tol=1e-8, restart=rng.choice([10, 20]))


# ---- inputs ---------------------------------------------------------------------------


class _Mesh:
    """Vertices, counter-clockwise cells and domains, as Problem takes them."""

    def __init__(self, xy, ptr, vtx, y_water):
        self.xy, self.cell_ptr, self.cell_vtx = xy, ptr, vtx
        count = np.diff(ptr)
        self.mid = np.stack([np.add.reduceat(xy[vtx, a], ptr[:-1]) / count for a in (0, 1)], axis=1)
        self.cell_domain = (self.mid[:, 1] < y_water).astype(np.uint8)
        self.y_water = y_water


def _y_water(c):
    return (c["ny"] // 2) / c["ny"]


def _grid(c):
    nx, ny, fine = c["nx"], c["ny"], 2 if c["mesh"] == "hanging" else 1
    X, Y = np.meshgrid(c["width"] * np.arange(fine * nx + 1) / (fine * nx), np.arange(fine * ny + 1) / (fine * ny))
    xy, row = np.stack([X.ravel(), Y.ravel()], axis=1), fine * nx + 1
    cells = []                                            # (cells, vertices of one cell) arrays, row by row
    for j in range(ny):
        a = fine * j * row + fine * np.arange(nx)
        up = fine * row
        quad = [a, a + fine, a + fine + up, a + up]
        if c["mesh"] == "tri" or (c["mesh"] == "hybrid" and j + 0.5 > 0.7 * ny):
            cells.append(np.stack([quad[0], quad[1], quad[2], quad[0], quad[2], quad[3]], axis=1).reshape(-1, 3))
        elif c["mesh"] == "hanging" and j % 4 == 0:
            for half in (0, 1):
                b = (2 * j + half) * row + np.arange(2 * nx)
                cells.append(np.stack([b, b + 1, b + 1 + row, b + row], axis=1))
        elif c["mesh"] == "hanging" and j % 4 == 1:
            cells.append(np.stack([a, a + 1, a + 2, a + 2 + up, a + up], axis=1))
        elif c["mesh"] == "hanging" and j % 4 == 3 and j + 1 < ny:
            cells.append(np.stack([a, a + 2, a + 2 + up, a + 1 + up, a + up], axis=1))
        else:
            cells.append(np.stack(quad, axis=1))
    vtx = np.concatenate([b.ravel() for b in cells])
    count = np.concatenate([np.full(len(b), b.shape[1]) for b in cells])
    if fine == 2:                                         # drop the fine lattice's unused vertices
        used = np.zeros(len(xy), bool)
        used[vtx] = True
        vtx, xy = (np.cumsum(used) - 1)[vtx], xy[used]
    ptr = np.concatenate([[0], np.cumsum(count)]).astype(np.int64)
    return _Mesh(xy, ptr, vtx.astype(np.int64), _y_water(c))


def _media(c, mesh, seed):
    """rho, lambda, mu, kappa per cell: water over a solid with a smooth random field (+-20 %)."""
    rng = np.random.default_rng([seed, 1])
    field = []
    for _ in range(2):
        g = np.zeros(len(mesh.mid))
        for _ in range(6):
            kx, ky, phase = rng.uniform(-25, 25), rng.uniform(-25, 25), rng.uniform(0, 6.28)
            g += np.cos(kx * mesh.mid[:, 0] + ky * mesh.mid[:, 1] + phase)
        field.append(1.0 + 0.2 * g / 6)
    solid = mesh.cell_domain == 1
    rho = np.where(solid, 2.5 * field[1], 1.0)
    vp, vs = 3.0 * field[0], 1.7 * field[0]
    return (rho, np.where(solid, rho * (vp ** 2 - 2 * vs ** 2), 0.0), np.where(solid, rho * vs ** 2, 0.0),
            np.where(solid, 0.0, 1.5 ** 2))


def _dt(c):
    h = min(1.0 / c["ny"], c["width"] / c["nx"]) / (2 if c["mesh"] == "hanging" else 1)
    dt = 0.8 * _CFL[c["mesh"]][c["k"]] * h / 3.6
    return dt * c["ratio"] if c["kind"] == "sdirk" else dt * _OF_STAGES[c["stages"]]


def _points(c, seed):
    """Sources (solid), one per shot, and receivers, off the mesh lines but for those on the interface."""
    rng = np.random.default_rng([seed, 2])
    yw, w = _y_water(c), c["width"]
    src = np.stack([w * rng.uniform(0.1, 0.9, c["shots"]), yw * rng.uniform(0.3, 0.9, c["shots"])], axis=1)
    x = w * (np.arange(c["receivers"]) + 0.41421356) / max(1, c["receivers"])
    y = yw if c.get("at_interface") else yw + (1 - yw) * 0.5382
    return src, np.stack([x, np.full(len(x), y)], axis=1)


def _state(c, mesh, seed):
    """Canonical vectors [shots][n_canonical] on the GPU: a rough wave field whose coefficients fall with degree."""
    n = (c["k"] + 1) * (c["k"] + 2) // 2
    fall = torch.tensor([0.3 ** d for d in range(c["k"] + 1) for _ in range(d + 1)], dtype=torch.float64, device="cuda")
    fields = np.where(mesh.cell_domain == 1, 5, 3).sum()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.randn((c["shots"], int(fields), n), generator=gen, dtype=torch.float64, device="cuda") * fall
    return u.reshape(c["shots"], -1)


def _cotangent(c, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed + 7919)
    return torch.randn((c["steps"], c["receivers"], 5), generator=gen, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    c, mesh = case, _grid(case)
    p = Problem(mesh, _media(c, mesh, seed), c["k"])
    src, rec = _points(c, seed)
    force = np.tile([0.6, 0.8], (len(src), 1))
    prec = _PREC[c["arith"]]
    s = {"case": c, "problem": p, "dt": _dt(c), "prec": prec}
    if c["receivers"]:
        p.set_receivers(rec)
    if c["kind"] == "shots":
        p.set_shot_sources(src, force, _F0)
    else:
        p.set_sources(src, force, _F0)
    canon = _state(c, mesh, seed)
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] in ("erk", "host"):
        p.set_arithmetic(prec)
    if c["kind"] == "host":
        s["host"] = canon[0].cpu().pin_memory()
        return s
    if c["kind"] == "shots":
        s["state"], s["work"] = p.batch_buffers(c["stages"], c["shots"], prec)
        hho.hho_batch_pack(p.ops, c["shots"], prec, canon.data_ptr(), s["state"].data_ptr(), stream)
        s["snapshot"] = canon                                # the snapshot's buffer from here on
        s["seismogram"] = torch.zeros((c["steps"], c["shots"], c["receivers"], 5), device="cuda",
                                      dtype=torch.float32 if c["arith"] == "f32" else torch.float64)
        return s
    s["state"] = p.empty_state()
    hho.hho_state_pack(p.ops, canon.data_ptr(), s["state"].data_ptr(), stream)
    if c["kind"] == "adjoint":
        tab, size = hho.hho_tableau_erk(c["stages"]), hho.hho_adjoint_work_size
        g = _cotangent(c, seed)
        if c["arith"] == "f32":
            size, g = hho.hho_adjoint_work_size_f32, g.float()
            s["state"] = torch.zeros(p.layout.n_state, dtype=torch.float32, device="cuda")
            hho.hho_batch_pack(p.ops, 1, prec, canon.data_ptr(), s["state"].data_ptr(), stream)
        s["cotangent"] = g
        s["work"] = torch.empty(size(p.ops, tab, c["steps"], c["checkpoint"]), dtype=g.dtype, device="cuda")
        s["cells"] = len(mesh.cell_domain)
        return s
    s["snapshot"] = canon[0]
    s["seismogram"] = torch.zeros((c["steps"], c["receivers"], 5), dtype=torch.float64, device="cuda")
    return s


def run(state):
    s = state
    c, p, dt = s["case"], s["problem"], s["dt"]
    stream = torch.cuda.current_stream().cuda_stream
    if c["kind"] == "sdirk":
        p.sdirk_step(s["state"], c["stages"], 0.0, dt, c["steps"], tol=c["tol"], restart=c["restart"], max_iter=5000)
        hho.hho_state_unpack(p.ops, s["state"].data_ptr(), s["snapshot"].data_ptr(), stream)
        return [s["snapshot"]]
    tab = hho.hho_tableau_erk(c["stages"])
    if c["kind"] == "host":
        hho.hho_erk_run_host(p.ops, tab, 0.0, dt, c["steps"], s["host"].data_ptr(), stream)
        return [s["host"]]
    if c["kind"] == "shots":
        hho.hho_batch_erk_step(p.ops, tab, c["shots"], s["prec"], 0.0, dt, c["steps"], s["state"].data_ptr(),
                               s["work"].data_ptr(), s["seismogram"].data_ptr(), stream)
        hho.hho_batch_unpack(p.ops, c["shots"], s["prec"], s["state"].data_ptr(), s["snapshot"].data_ptr(), stream)
        return [s["snapshot"].float() if c["arith"] == "f32" else s["snapshot"], s["seismogram"]]
    if c["kind"] == "adjoint":
        vjp = hho.hho_adjoint_vjp if c["arith"] == "f64" else hho.hho_adjoint_vjp_f32
        grad, wavelet = vjp(p.ops, tab, 0.0, dt, c["steps"], c["checkpoint"], s["state"].data_ptr(),
                            s["cotangent"].data_ptr(), s["work"].data_ptr(), s["work"].numel(), s["cells"], n_src=1,
                            stream=stream)
        return [grad, wavelet] if c["arith"] == "f64" else [grad.astype(np.float32), wavelet.astype(np.float32)]
    pieces = c.get("energy", 0)
    energies, each = [], c["steps"] // max(1, pieces)
    for i in range(max(1, pieces)):
        seis = s["seismogram"][i * each:]
        hho.hho_erk_step_record(p.ops, tab, i * each * dt, dt, each, s["state"].data_ptr(), p.work(tab).data_ptr(),
                                seis.data_ptr(), stream)
        if pieces:
            energies.append(p.energy(s["state"]))
    hho.hho_state_unpack(p.ops, s["state"].data_ptr(), s["snapshot"].data_ptr(), stream)
    return [s["snapshot"], s["seismogram"], energies]


def _counts(c):
    """(cells, values of the state of one shot)."""
    solid = c["ny"] // 2
    per = {"quad": lambda j: 1, "tri": lambda j: 2, "hybrid": lambda j: 2 if j + 0.5 > 0.7 * c["ny"] else 1,
           "hanging": lambda j: 4 if j % 4 == 0 else 1}[c["mesh"]]
    rows = [c["nx"] * per(j) for j in range(c["ny"])]
    n = (c["k"] + 1) * (c["k"] + 2) // 2
    return sum(rows), n * (5 * sum(rows[:solid]) + 3 * sum(rows[solid:]))


def work(case):
    """Bytes: the state read and written once a step (once a Krylov vector or adjoint stage where the
    method needs the whole vector), the materials and the exchange between cells at their stated types.
    Flops: the sparse operator, about ten multiply-adds a value and stage on squares."""
    c = case
    cells, values = _counts(c)
    size = 4 if c["arith"] == "f32" else 8
    stages = c["stages"] * c["steps"]
    flops = 20.0 * values * c["shots"] * stages
    move = 2.0 * values * c["shots"] * size * c["steps"] + 40.0 * cells
    if c["kind"] == "adjoint":
        return {"bytes": 2.0 * move + 2.0 * values * size * stages, "flops": 4.0 * flops}
    if c["kind"] == "sdirk":
        inner = 15 * stages                                   # operator applications, at the least
        return {"bytes": 2.0 * 8 * values * inner, "flops": 20.0 * values * inner}
    if c["kind"] == "host":
        return {"bytes": move + 16.0 * values, "flops": flops}
    return {"bytes": move + 8.0 * values * c["shots"], "flops": flops}


# ---- the scheme in plain 64 bits -----------------------------------------------------------


class _Plain:
    """The semi-discrete operator on padded per-cell tensors.  Faces of a cell are its edges in order; a face
    value is held at k + 1 Gauss points of the edge, which the other cell passes in reverse order."""

    def __init__(self, c, mesh, dev="cuda"):
        k = self.k = c["k"]
        self.exps = [(d - b, b) for d in range(k + 1) for b in range(d + 1)]
        n, f = len(self.exps), k + 1
        count = np.diff(mesh.cell_ptr)
        nc, nf = len(count), int(count.max())
        at = np.minimum(np.arange(nf)[None], count[:, None] - 1)
        vid = mesh.cell_vtx[mesh.cell_ptr[:-1, None] + at]                       # the last vertex repeats as padding
        nxt = mesh.cell_vtx[mesh.cell_ptr[:-1, None] + (at + 1) % count[:, None]]
        real = np.arange(nf)[None] < count[:, None]
        T = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)       # noqa: E731
        P, Q, real_t = T(mesh.xy[vid]), T(mesh.xy[nxt]), T(real)
        O = P[:, :1]
        a, b = P - O, Q - O
        cr = (a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0]) * real_t
        self.centre = O[:, 0] + ((a + b) * cr[..., None]).sum(1) / (3 * cr.sum(1))[:, None]
        self.h = torch.cdist(P, P).flatten(1).max(1).values
        X, Y = (P - self.centre[:, None]) / self.h[:, None, None], (Q - self.centre[:, None]) / self.h[:, None, None]
        gx, gw = (T(v) for v in np.polynomial.legendre.leggauss(k + 2))
        M = torch.zeros((nc, n, n), dtype=torch.float64, device=dev)
        for t in range(nf):
            det = (X[:, t, 0] * Y[:, t, 1] - X[:, t, 1] * Y[:, t, 0]) * real_t[:, t]
            for u, wu in zip(gx, gw):
                for v, wv in zip(gx, gw):
                    r, q = 0.5 * (u + 1), 0.5 * (v + 1)
                    phi = self.basis(r * X[:, t] + r * q * (Y[:, t] - X[:, t]))
                    M += (0.25 * wu * wv * r * det)[:, None, None] * phi[:, :, None] * phi[:, None]
        fx, fw = (T(v) for v in np.polynomial.legendre.leggauss(f))
        edge = Y - X
        length = edge.norm(dim=-1)
        self.normal = torch.stack([edge[..., 1], -edge[..., 0]], -1) / length.clamp_min(1e-300)[..., None]
        pts = X[:, :, None] + 0.5 * (fx + 1)[:, None] * edge[:, :, None]
        phi = self.basis(pts)                                                    # [cell, face, point, n]
        wt = (0.5 * length[..., None] * fw) * real_t[..., None]
        self.M0 = M
        self.trace = phi.reshape(nc, nf * f, n)
        lift = torch.linalg.solve(M, (wt[..., None] * phi).reshape(nc, nf * f, n).transpose(1, 2))
        self.lift = lift                                                         # [cell, n, face * point]
        D = np.zeros((2, n, n))
        for i, (ex, ey) in enumerate(self.exps):
            if ex:
                D[0, self.exps.index((ex - 1, ey)), i] = ex
            if ey:
                D[1, self.exps.index((ex, ey - 1)), i] = ey
        self.dx, self.dy = T(D[0]), T(D[1])
        # the edge on the other side, by its two vertices
        lo, hi = np.minimum(vid, nxt), np.maximum(vid, nxt)
        key = np.where(real, lo * (mesh.cell_vtx.max() + 1) + hi, -1).ravel()
        order = np.argsort(key, kind="stable")
        same = (key[order][1:] == key[order][:-1]) & (key[order][1:] >= 0)
        other = np.full(nc * nf, -1, np.int64)
        i, j = order[:-1][same], order[1:][same]
        other[i], other[j] = j, i
        dom = mesh.cell_domain.astype(np.int64)
        has = other >= 0
        oc = np.where(has, other // nf, 0)
        mine = np.repeat(dom, nf)
        self.inside = T((has & (dom[oc] == mine)).reshape(nc, nf)[..., None])
        self.across = T((has & (dom[oc] != mine)).reshape(nc, nf)[..., None])
        self.oc = T(oc.reshape(nc, nf))
        flat = np.where(has, other, np.arange(nc * nf))
        self.gather = T((flat[:, None] * f + np.arange(f)[None, ::-1]).ravel())
        self.solid = T(dom == 1)
        self.S, self.F = torch.nonzero(self.solid)[:, 0], torch.nonzero(~self.solid)[:, 0]
        self.shape = (nc, nf, f)
        self.n = n
        self.verts, self.real = P, real_t
        # canonical places of the values of fluid and solid cells
        size = np.where(dom == 1, 5, 3) * n
        off = T(np.cumsum(size) - size)
        self.at_f = off[self.F, None] + torch.arange(3 * n, device=dev)
        self.at_s = off[self.S, None] + torch.arange(5 * n, device=dev)

    def basis(self, p):
        x, y = p[..., 0], p[..., 1]
        return torch.stack([x ** a * y ** b for a, b in self.exps], -1)

    def split(self, canon):
        return canon[self.at_f].reshape(-1, 3, self.n), canon[self.at_s].reshape(-1, 5, self.n)

    def join(self, U):
        out = torch.empty(self.at_f.numel() + self.at_s.numel(), dtype=torch.float64, device=self.h.device)
        out[self.at_f.reshape(-1)] = U[0].reshape(-1)
        out[self.at_s.reshape(-1)] = U[1].reshape(-1)
        return out

    def media(self, rho, lam, mu, kappa):
        """Materials (differentiable) and the stabilisation weights that follow them."""
        solid = self.solid
        one = torch.ones_like(rho)
        cp = torch.sqrt(torch.where(solid, lam + 2 * mu, kappa) / rho)
        self.tau = torch.where(solid, 1.5 * rho * cp, 0.8 / (rho * cp))
        self.rho, self.lam, self.mu, self.kappa = rho, lam, mu, torch.where(solid, one, kappa)

    def rate(self, U):
        (nc, nf, f), F, S = self.shape, self.F, self.S
        fl, so = U
        tr = lambda ids, x: torch.bmm(self.trace[ids], x.transpose(1, 2)).reshape(len(ids), nf, f, -1)  # noqa: E731
        tf, ts = tr(F, fl), tr(S, so)
        nF, nS = self.normal[F][:, :, None], self.normal[S][:, :, None]
        wf = self.tau[F][:, None, None] * tf[..., 2] - (tf[..., :2] * nF).sum(-1)
        sn = torch.stack([ts[..., 0] * nS[..., 0] + ts[..., 2] * nS[..., 1],
                          ts[..., 2] * nS[..., 0] + ts[..., 1] * nS[..., 1]], -1)
        ws = self.tau[S][:, None, None, None] * ts[..., 3:] - sn
        zero = torch.zeros((nc, nf, f, 2), dtype=torch.float64, device=fl.device)
        w = zero.index_put((F,), torch.stack([wf, torch.zeros_like(wf)], -1)).index_put((S,), ws)
        wn = w.reshape(-1, 2)[self.gather].reshape(nc, nf, f, 2)
        to = self.tau[self.oc][..., None]
        tfc, tsc = self.tau[F][:, None, None], self.tau[S][:, None, None]
        # interior: (w + w') / (tau + tau'); interface: [tau_f, n; -n, tau_s] [p; v] = [w_f; w_s], n out of the solid
        pf = self.inside[F] * (wf + wn[F][..., 0]) / (tfc + to[F])
        ns = -nF
        pf = pf + self.across[F] * (wf - (ns * wn[F]).sum(-1) / to[F]) / (tfc + 1 / to[F])
        vf = (self.inside[S] / (tsc + to[S]))[..., None] * (ws + wn[S])
        pi = (wn[S][..., 0] - (nS * ws).sum(-1) / tsc) / (to[S] + 1 / tsc)
        vf = vf + self.across[S][..., None] * (ws + nS * pi[..., None]) / tsc[..., None]
        jp = (pf - tf[..., 2]).unsqueeze(-1)
        jv = vf - ts[..., 3:]
        up = lambda ids, x: torch.bmm(self.lift[ids], x.reshape(len(ids), nf * f, -1)).transpose(1, 2)  # noqa: E731
        lf = up(F, torch.cat([jp * nF, jp * self.tau[F][:, None, None, None]], -1))
        x, y = jv[..., 0], jv[..., 1]
        ls = up(S, torch.stack([x * nS[..., 0], y * nS[..., 1], x * nS[..., 1] + y * nS[..., 0],
                                x * tsc, y * tsc], -1))
        dx, dy = self.dx.T, self.dy.T
        hf, hs = self.h[F][:, None], self.h[S][:, None]
        m, p = self.rho[F][:, None] * hf, self.kappa[F][:, None] / hf
        kf = torch.stack([(fl[:, 2] @ dx + lf[:, 0]) / m, (fl[:, 2] @ dy + lf[:, 1]) / m,
                          (fl[:, 0] @ dx + fl[:, 1] @ dy + lf[:, 2]) * p], 1)
        exx, eyy = so[:, 3] @ dx + ls[:, 0], so[:, 4] @ dy + ls[:, 1]
        exy = so[:, 3] @ dy + so[:, 4] @ dx + ls[:, 2]
        la, mu = (self.lam[S] / self.h[S])[:, None], (self.mu[S] / self.h[S])[:, None]
        r = self.rho[S][:, None] * hs
        ks = torch.stack([(la + 2 * mu) * exx + la * eyy, (la + 2 * mu) * eyy + la * exx, mu * exy,
                          (so[:, 0] @ dx + so[:, 2] @ dy + ls[:, 3]) / r,
                          (so[:, 2] @ dx + so[:, 1] @ dy + ls[:, 4]) / r], 1)
        return kf, ks

    def owner(self, pts, solid=None):
        """The first cell that holds each point (of the given domain)."""
        out = []
        nxt = torch.roll(self.verts, -1, 1)
        last = (self.real.sum(1) - 1)
        nxt[torch.arange(len(last), device=nxt.device), last] = self.verts[:, 0]
        e = nxt - self.verts
        for q in pts:
            d = torch.as_tensor(q, device=e.device) - self.verts
            ok = ((e[..., 0] * d[..., 1] - e[..., 1] * d[..., 0] >= -1e-11 * self.h[:, None]) | ~self.real).all(1)
            if solid is not None:
                ok &= self.solid == solid
            out.append(int(torch.nonzero(ok)[0, 0]))
        return torch.tensor(out, device=e.device)

    def at(self, cells, pts):
        p = torch.as_tensor(pts, device=self.h.device)
        return self.basis((p - self.centre[cells]) / self.h[cells][:, None])

    def load(self, src, force):
        """The load vector of a point force, before its wavelet: values of the velocities of its cell."""
        cell = self.owner([src])
        g = torch.linalg.solve(self.M0[cell], self.at(cell, src[None])[..., None])[0, :, 0]
        at = torch.nonzero(self.S == cell)[0, 0]
        return at, torch.as_tensor(force, device=g.device)[:, None] * g / self.h[cell] ** 2, cell

    def recorder(self, c, rec):
        if not len(rec):
            return lambda U: None
        inv = torch.zeros(self.shape[0], dtype=torch.int64, device=self.h.device)
        inv[self.F] = torch.arange(len(self.F), device=inv.device)
        inv[self.S] = torch.arange(len(self.S), device=inv.device)
        fc = self.owner(rec, solid=False)
        pf, fi = self.at(fc, rec), inv[fc]
        if not c.get("at_interface"):
            def fluid(U):
                v = (U[0][fi] * pf[:, None]).sum(-1)
                return torch.stack([v[:, 2], v[:, 0], v[:, 1], 0 * v[:, 0], 0 * v[:, 0]], 1)
            return fluid
        sc = self.owner(rec, solid=True)
        ps, si = self.at(sc, rec), inv[sc]
        # the face of the solid cell that the point lies on: horizontal, or the one whose line it is nearest to
        q = torch.as_tensor(rec, device=ps.device)[:, None] - self.verts[sc]
        dist = (q * self.normal[sc]).sum(-1).abs().masked_fill(~self.real[sc], 1e9)
        n = self.normal[sc, dist.argmin(1)]

        def interface(U):
            a, b = (U[0][fi] * pf[:, None]).sum(-1), (U[1][si] * ps[:, None]).sum(-1)
            tf, ts = self.tau[fc], self.tau[sc]
            wf = tf * a[:, 2] + a[:, 0] * n[:, 0] + a[:, 1] * n[:, 1]
            wx = ts * b[:, 3] - b[:, 0] * n[:, 0] - b[:, 2] * n[:, 1]
            wy = ts * b[:, 4] - b[:, 2] * n[:, 0] - b[:, 1] * n[:, 1]
            p = (wf - (n[:, 0] * wx + n[:, 1] * wy) / ts) / (tf + 1 / ts)
            return torch.stack([p, (wx + n[:, 0] * p) / ts, (wy + n[:, 1] * p) / ts, 0 * p, 0 * p], 1)
        return interface

    def energy(self, U):
        fl, so = U
        q = lambda ids, a, b: (a * torch.bmm(self.M0[ids], b[..., None])[..., 0]).sum(-1)  # noqa: E731
        F, S = self.F, self.S
        hf, hs = self.h[F] ** 2, self.h[S] ** 2
        e = hf * (self.rho[F] * (q(F, fl[:, 0], fl[:, 0]) + q(F, fl[:, 1], fl[:, 1])) + q(F, fl[:, 2], fl[:, 2]) / self.kappa[F])
        la, mu = self.lam[S], self.mu[S]
        be = la / (2 * (la + mu))
        xx, yy, xy = q(S, so[:, 0], so[:, 0]), q(S, so[:, 1], so[:, 1]), q(S, so[:, 0], so[:, 1])
        g = hs * (((1 - be) * (xx + yy) - 2 * be * xy + 2 * q(S, so[:, 2], so[:, 2])) / (2 * mu)
                  + self.rho[S] * (q(S, so[:, 3], so[:, 3]) + q(S, so[:, 4], so[:, 4])))
        return float(0.5 * (e.sum() + g.sum()))


def _ricker(t):
    a = (math.pi * _F0 * (t - 1.0 / _F0)) ** 2
    return (1 - 2 * a) * math.exp(-a)


_ERK = {2: ([[], [0.5]], [0, 1], [0, 0.5]),
        3: ([[], [0.5], [-1, 2]], [1 / 6, 2 / 3, 1 / 6], [0, 0.5, 1]),
        4: ([[], [0.5], [0, 0.5], [0, 0, 1]], [1 / 6, 1 / 3, 1 / 3, 1 / 6], [0, 0.5, 0.5, 1])}


def _add(U, terms):
    for a, k in terms:
        if a:
            U = (U[0] + a * k[0], U[1] + a * k[1])
    return U


def _forced(op, load, w, k):
    at, g, cell = load
    v = k[1].clone()
    v[at, 3:] = v[at, 3:] + w * g / op.rho[cell]
    return k[0], v


def _erk_step(op, load, tab, dt, w, U):
    """One step; w: the wavelet's values at the stages."""
    A, b, _ = tab
    ks = []
    for i, row in enumerate(A):
        Y = _add(U, [(dt * a, k) for a, k in zip(row, ks)])
        ks.append(_forced(op, load, w[i], op.rate(Y)))
    return _add(U, [(dt * x, k) for x, k in zip(b, ks)])


def _krylov(op, x0, b, a, tol=1e-13):
    """(I - a J) x = b by GMRES(60), vectors of both domains laid end to end."""
    cut = [b[0].numel()]
    flat = lambda U: torch.cat([U[0].reshape(-1), U[1].reshape(-1)])  # noqa: E731
    back = lambda v: (v[:cut[0]].reshape(b[0].shape), v[cut[0]:].reshape(b[1].shape))  # noqa: E731
    A = lambda v: v - a * flat(op.rate(back(v)))  # noqa: E731
    x, rhs, m = flat(x0), flat(b), 60
    for _ in range(40):
        r = rhs - A(x)
        beta = r.norm()
        if beta <= tol * rhs.norm():
            break
        V, H = torch.empty((m + 1, len(r)), dtype=r.dtype, device=r.device), torch.zeros((m + 1, m), dtype=r.dtype, device=r.device)
        V[0] = r / beta
        for j in range(m):
            w = A(V[j])
            for _ in range(2):
                y = V[:j + 1] @ w
                H[:j + 1, j] += y
                w = w - y @ V[:j + 1]
            H[j + 1, j] = w.norm()
            V[j + 1] = w / H[j + 1, j]
        e = torch.zeros(m + 1, dtype=r.dtype, device=r.device)
        e[0] = beta
        x = x + torch.linalg.lstsq(H.cpu(), e.cpu()[:, None], driver="gelsd").solution[:, 0].to(x.device) @ V[:m]
    return back(x)


def _sdirk(c):
    if c["stages"] == 1:
        return [[0.5]], [1.0], [0.5]
    if c["stages"] == 2:
        return [[0.25], [0.5, 0.25]], [0.5, 0.5], [0.25, 0.75]
    nu = math.cos(math.pi / 18) / math.sqrt(3) + 0.5
    xi = 1 / (6 * (2 * nu - 1) ** 2)
    return [[nu], [0.5 - nu, nu], [2 * nu, 1 - 4 * nu, nu]], [xi, 1 - 2 * xi, xi], [nu, 0.5, 1 - nu]


def exact(case, seed):
    c, mesh, dt = case, _grid(case), _dt(case)
    op = _Plain(c, mesh)
    grad = c["kind"] == "adjoint"
    mats = [torch.as_tensor(np.array(m, dtype=np.float64), device="cuda").requires_grad_(grad) for m in _media(c, mesh, seed)]
    op.media(*mats)
    src, rec = _points(c, seed)
    canon = _state(c, mesh, seed)
    loads = [op.load(p, np.array([0.6, 0.8])) for p in src]
    if c["kind"] == "sdirk":
        A, b, nodes = _sdirk(c)
        U, ks = op.split(canon[0]), []
        for i, row in enumerate(A):
            a = dt * row[i]
            Z = _add(U, [(dt * x, k) for x, k in zip(row[:i], ks)])
            force = lambda k: _forced(op, loads[0], _ricker(nodes[i] * dt), k)  # noqa: E731
            Y = _krylov(op, Z, _add(Z, [(a, force((0 * U[0], 0 * U[1])))]), a)
            ks.append(force(op.rate(Y)))
        return [op.join(_add(U, [(dt * x, k) for x, k in zip(b, ks)]))]
    tab = _ERK[c["stages"]]
    times = [[n * dt + x * dt for x in tab[2]] for n in range(c["steps"])]
    record = op.recorder(c, rec)
    if grad:
        from torch.utils.checkpoint import checkpoint
        w = torch.tensor([[_ricker(t) for t in row] for row in times], dtype=torch.float64, device="cuda").requires_grad_(True)
        G, U, loss = _cotangent(c, seed), op.split(canon[0]), 0.0

        def step(w_n, fl, so, *_):
            return _erk_step(op, loads[0], tab, dt, w_n, (fl, so))
        for n in range(c["steps"]):
            U = checkpoint(step, w[n], *U, *mats, use_reentrant=False)
            loss = loss + (record(U) * G[n]).sum()
        g = torch.autograd.grad(loss, [*mats, w])
        zero = torch.zeros_like(g[0])
        solid = op.solid
        cells = torch.stack([g[0], torch.where(solid, zero, g[3]), torch.where(solid, g[1], zero), torch.where(solid, g[2], zero)], 1)
        return [cells, g[4][..., None]]
    states, seismogram, energies = [], [], []
    each = c["steps"] // max(1, c.get("energy", 0) or 1)
    for u, load in zip(canon, loads):
        U, traces = op.split(u), []
        for n in range(c["steps"]):
            U = _erk_step(op, load, tab, dt, [_ricker(t) for t in times[n]], U)
            if len(rec):
                traces.append(record(U))
            if c.get("energy") and (n + 1) % each == 0:
                energies.append(op.energy(U))
        states.append(op.join(U))
        seismogram.append(torch.stack(traces) if traces else None)
    if c["kind"] == "host":
        return [states[0]]
    if c["kind"] == "shots":
        return [torch.stack(states), torch.stack(seismogram, 1)]
    return [states[0], seismogram[0], energies]
