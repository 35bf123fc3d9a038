"""The work that users of this library have it do, as cases that can be timed.

A case is a run in progress: a mesh and a state are kept (``prepare``), and one
pass (``run``) advances the state by the steps between two outputs and reads
the fields back, as a simulation loop does.  Passes on one state continue each
other.  Single-precision runs keep their output in single precision; the host
buffers that receive the fields are pinned and kept.

The physics is that of the package's workloads, with flows in motion (the
middle of a run, not its first steps from rest): drops carried through a
periodic box, and Rayleigh-Taylor layers between walls.  Interface width and
viscosity are those at which runs of hundreds of thousands of steps stay
bounded, so that a case can be timed for as long as one likes; velocity and
ambient pressure are of a size that single precision resolves to a few parts
in a million.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1608_01906_gb300 import configs, felbm, inputs


def listed():
    drop = dict(ratio=10.0, xi=24.0, tau=0.5, dt=0.5)
    return [
        # the smallest mesh of the batched and served ranges, on its own:
        # a step is one short launch
        dict(name="lattice_32_fp32", mesh="lattice", nx=32, ny=32, precision="fp32", steps=200, **drop),
        # the static-droplet workload (64 x 64, FP64), the reference precision
        # in which a user validates a set-up
        dict(name="lattice_64_fp64", mesh="lattice", nx=64, ny=64, precision="fp64", steps=100, **drop),
        # an ordinary served mesh: odd width and height, rows that are not a
        # multiple of the tile nor of 16 bytes
        dict(name="lattice_357x203_fp32", mesh="lattice", nx=357, ny=203, precision="fp32", steps=150, **drop),
        # the benchmark's default workload: Rayleigh-Taylor between walls
        dict(name="rt_512x2048_fp32", mesh="walled", nx=512, ny=2048, precision="fp32", steps=200),
        # the largest single lattice of the benchmark
        dict(name="lattice_2048_fp32", mesh="lattice", nx=2048, ny=2048, precision="fp32", steps=100,
             **{**drop, "ratio": 20.0, "tau": 0.1}),
        # the same Rayleigh-Taylor physics in FP64, on a quarter of the mesh
        dict(name="rt_256x1024_fp64", mesh="walled", nx=256, ny=1024, precision="fp64", steps=50),
        # many drops of uneven size in one launch per step (the batched
        # workload's sides and parameters)
        dict(name="batch_24_fp32", mesh="batch", count=24, lo=32, hi=512, sides_seed=1609, precision="fp32",
             steps=100, ratio=20.0, xi=24.0, tau=0.1, dt=0.5),
        # the unstructured droplet workload's mesh (Delaunay, 65,536 nodes)
        dict(name="delaunay_256_fp32", mesh="delaunay", nx=256, ny=256, precision="fp32", steps=100, ratio=10.0,
             xi=24.0, tau=0.1, dt=0.4, lap_fp64=False),
        # the same beyond the caches (Delaunay, 1,048,576 nodes)
        dict(name="delaunay_1024_fp32", mesh="delaunay", nx=1024, ny=1024, precision="fp32", steps=50, ratio=10.0,
             xi=24.0, tau=0.1, dt=0.4, lap_fp64=False),
        # the paper's own setting, D3Q19 on a lattice of tetrahedra: a mesh
        # that stays in the caches, and one that does not
        dict(name="kuhn_64_fp32", mesh="kuhn", nx=64, ny=64, nz=64, precision="fp32", steps=100, **{**drop, "xi": 16.0}),
        dict(name="kuhn_96_fp32", mesh="kuhn", nx=96, ny=96, nz=96, precision="fp32", steps=60, **{**drop, "xi": 16.0}),
        # general tetrahedra (every element of its own shape)
        dict(name="tets_40_fp32", mesh="tets", nx=40, ny=40, nz=40, precision="fp32", steps=50,
             **{**drop, "xi": 16.0, "dt": 0.4}),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def steps(nodes, per_second, lo=10):
        # about a millisecond to a few tens of milliseconds a pass
        return max(lo, min(200, int(rng.uniform(0.004, 0.02) * per_second / nodes)))

    drop = dict(ratio=rng.choice([5.0, 10.0, 20.0]), xi=rng.choice([24.0, 28.0, 32.0]),
                tau=rng.choice([0.1, 0.25, 0.5]), dt=0.5)
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    mesh = rng.choice(["lattice", "lattice", "lattice", "walled", "batch", "delaunay", "delaunay", "kuhn", "kuhn",
                       "tets"])
    if mesh == "lattice":
        nx, ny = log(32, 2048), log(32, 2048)
        if precision == "fp64":
            nx, ny = min(nx, 700), min(ny, 700)
        return dict(mesh=mesh, nx=nx, ny=ny, precision=precision,
                    steps=steps(nx * ny + 60000, 1e10 if precision == "fp32" else 6e8), **drop)
    if mesh == "walled":
        nx, ny = log(64, 512), log(96, 2048)
        if precision == "fp64":
            ny = min(ny, 700)
        return dict(mesh=mesh, nx=nx, ny=ny, precision=precision,
                    steps=steps(nx * ny + 60000, 1e10 if precision == "fp32" else 6e8))
    if mesh == "batch":
        return dict(mesh=mesh, count=rng.randint(2, 24), lo=32, hi=rng.choice([96, 200, 512]),
                    sides_seed=rng.randrange(1 << 20), precision="fp32", steps=rng.randint(20, 100), ratio=20.0,
                    xi=24.0, tau=0.1, dt=0.5)
    if mesh == "delaunay":
        nx, ny = log(48, 800), log(48, 800)
        if precision == "fp64":
            nx, ny = min(nx, 400), min(ny, 400)
        return dict(mesh=mesh, nx=nx, ny=ny, precision=precision,
                    steps=steps(nx * ny + 30000, 2e9 if precision == "fp32" else 4e8),
                    lap_fp64=precision == "fp32" and rng.random() < 0.3, **{**drop, "dt": 0.4})
    hi = (100 if precision == "fp32" else 48) if mesh == "kuhn" else 44
    nx, ny, nz = log(12, hi), log(12, hi), log(12, hi)
    d = dict(mesh=mesh, nx=nx, ny=ny, nz=nz, precision=precision, **{**drop, "xi": 16.0, "ratio": 10.0, "tau": 0.5})
    if mesh == "tets":
        d["dt"] = 0.4
    d["steps"] = steps(nx * ny * nz + 20000, (4e9 if mesh == "kuhn" else 1e9) / (1 if precision == "fp32" else 15))
    return d


# ---- the inputs -----------------------------------------------------------

def _sides(case):
    rng = np.random.default_rng(case["sides_seed"])
    lo, hi = math.log(case["lo"]), math.log(case["hi"])
    return [int(round(math.exp(s))) for s in rng.uniform(lo, hi, size=case["count"])]


@functools.lru_cache(maxsize=40)
def _mesh_arrays(kind, nx, ny, nz):
    """(coordinates, cells, box, tags) of a mesh."""
    if kind == "lattice":
        return inputs.structured_mesh(nx, ny)
    if kind == "walled":
        return inputs.structured_mesh(nx, ny, periodic_y=False)
    if kind == "delaunay":
        return inputs.jittered_delaunay_mesh(nx, ny, 0.25, 1608)
    if kind == "kuhn":
        return inputs.structured_tet_mesh(nx, ny, nz)
    return inputs.jittered_tet_mesh(nx, ny, nz, 0.1, 1608)


@functools.lru_cache(maxsize=40)
def _mesh(kind, nx, ny, nz):
    """The library's mesh: made once for all runs on it."""
    xy, cells, box, tag = _mesh_arrays(kind, nx, ny, nz)
    return felbm.Mesh(xy, cells, box, tag if kind == "walled" else None)


def _key(case):
    return case["mesh"], case["nx"], case["ny"], case.get("nz", 0)


def _params(case):
    if case["mesh"] == "walled":
        g, _, tau = configs.rt_params(512, Re=500.0)
        return dict(rho_l=1.0, rho_v=1.0 / 3.0, sigma=1e-4, xi=4.0, tau_l=tau, tau_v=tau, dt=0.5, gravity=(0.0, -g))
    return dict(rho_l=1.0, rho_v=1.0 / case["ratio"], sigma=0.01, xi=case["xi"], tau_l=case["tau"],
                tau_v=case["tau"], dt=case["dt"], gravity=(0.0, 0.0, 0.0))


def _fields(case, rng):
    """Density, velocity and pressure on the mesh's nodes: a drop somewhere in
    the box moving in some direction, or a perturbed layer with a solenoidal
    flow around its interface and the pressure of its weight."""
    xy, _, box, _ = _mesh_arrays(*_key(case))
    P = _params(case)
    if case["mesh"] == "walled":
        W, H = case["nx"], case["ny"]
        k = 2.0 * math.pi / W
        rho, u, p = inputs.rayleigh_taylor_fields(xy, W, H, P["rho_l"], P["rho_v"], P["xi"],
                                                  rng.uniform(0.05, 0.1) * min(W, 0.5 * H), -P["gravity"][1])
        phase, amp, s = rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.03, 0.05), W / 6.0
        y = xy[:, 1] - 0.5 * (H - 1)
        bump = np.exp(-0.5 * (y / s) ** 2) * np.sin(math.pi * xy[:, 1] / (H - 1)) ** 2
        ph = k * xy[:, 0] + phase
        # stream function amp / k sin(ph) bump(y), differentiated on the rows
        dbump = np.gradient(bump.reshape(H, W)[:, 0], edge_order=2)
        u[:, 0] = amp / k * np.sin(ph) * np.repeat(dbump, W)
        u[:, 1] = -amp * np.cos(ph) * bump
        return rho, u, p
    dim = xy.shape[1]
    side = float(np.min(box[:dim]))
    center = rng.uniform(0.0, 1.0, size=dim) * box[:dim]
    radius = rng.uniform(0.2, 0.35) * side
    v = rng.normal(size=dim)
    v *= rng.uniform(0.04, 0.08) / np.linalg.norm(v)
    f = inputs.droplet_fields if dim == 2 else inputs.droplet_fields3
    rho, u, p = f(xy, box, tuple(center), radius, P["rho_l"], P["rho_v"], P["xi"], u0=tuple(v))
    # ambient pressure, and Laplace's jump inside
    p += 0.01 + P["sigma"] * (dim - 1) / radius * (rho - P["rho_v"]) / (P["rho_l"] - P["rho_v"])
    return rho, u, p


def _runs(case):
    """The single runs of a case (a batch has many)."""
    if case["mesh"] != "batch":
        return [case]
    return [{**case, "mesh": "lattice", "nx": s, "ny": s} for s in _sides(case)]


class _Run:
    pass


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    s = _Run()
    s.steps, s.single = case["steps"], case["precision"] == "fp32"
    s.states, sizes = [], []
    for c in _runs(case):
        mesh = _mesh(*_key(c))
        params = felbm.make_params(precision=c["precision"], lap_fp64=bool(c.get("lap_fp64")), **_params(c))
        s.states.append(felbm.State(mesh, params, *_fields(c, rng)))
        sizes.append(mesh.n_nodes)
    s.batch = felbm.Batch(s.states) if case["mesh"] == "batch" else None
    dim, total = s.states[0].mesh.dim, sum(sizes)
    pin = torch.cuda.is_available()
    s.out = {"rho": torch.empty(total, dtype=torch.float64, pin_memory=pin),
             "u": torch.empty(total, dim, dtype=torch.float64, pin_memory=pin),
             "p": torch.empty(total, dtype=torch.float64, pin_memory=pin),
             "totals": torch.empty(len(sizes), 1 + dim, dtype=torch.float64, pin_memory=pin)}
    s.views, at = [], 0
    for k, n in enumerate(sizes):  # the part of the buffers that each state fills
        s.views.append({"rho": s.out["rho"][at:at + n].numpy(), "u": s.out["u"][at:at + n].numpy(),
                        "p": s.out["p"][at:at + n].numpy(), "totals": s.out["totals"][k].numpy()})
        at += n
    return s


def run(s):
    if s.batch is not None:
        s.batch.step(s.steps)
    else:
        s.states[0].step(s.steps)
    for st, v in zip(s.states, s.views):
        status = felbm.felbm_moments_get(st.handle, rho=v["rho"], u=v["u"], p=v["p"], totals=v["totals"])
        if status != felbm.FELBM_OK:
            raise felbm.FelbmError(status, "felbm_moments_get")
    if s.single:
        return {k: v.to(torch.float32) for k, v in s.out.items()}
    return s.out


def work(case):
    """Per step every population read once and written once and, on general
    meshes, the neighbour lists and operator coefficients read once; per pass
    the fields read back."""
    size = 4 if case["precision"] == "fp32" else 8
    three = case["mesh"] in ("kuhn", "tets")
    nodes = sum(c["nx"] * c["ny"] * c.get("nz", 1) for c in _runs(case))
    q, dim, per_node = (19, 3, 2900) if three else (9, 2, 850)
    bytes_step = nodes * 4 * q * size
    if case["mesh"] == "delaunay":
        bytes_step += nodes * 6 * (4 + 5 * size)
    if case["mesh"] == "tets":
        bytes_step += nodes * 14 * (4 + 9 * size)
    return {"bytes": case["steps"] * bytes_step + nodes * (2 + dim) * size, "flops": case["steps"] * nodes * per_node}


# ---- the same runs in plain torch, 64 bits --------------------------------

_E2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_E3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]


def _assemble(x, cells, box):
    """Linear elements with the lumped mass: per pair of neighbours i != j,
    a = sum |T| grad N_j / ((dim + 1) m_i) and the symmetric part of
    b = sum |T| / m_i grad N_i (x) grad N_j.  Returns (i, j, a, b, mass)."""
    n, dim = x.shape
    cells = cells.astype(np.int64)
    e = x[cells[:, 1:]] - x[cells[:, :1]]
    for c in range(dim):
        if box[c] > 0:
            e[..., c] -= box[c] * np.round(e[..., c] / box[c])
    vol = np.linalg.det(e) / math.factorial(dim)
    g = np.swapaxes(np.linalg.inv(e), 1, 2)
    g = np.concatenate([-g.sum(1, keepdims=True), g], 1)  # (cell, vertex, component)
    mass = np.bincount(cells.ravel(), np.repeat(vol / (dim + 1), dim + 1), n)
    keys, val = [], []
    for s in range(dim + 1):
        for t in range(dim + 1):
            if s == t:
                continue
            w = (vol / mass[cells[:, s]])[:, None]
            o = g[:, s, :, None] * g[:, t, None, :]
            o = 0.5 * (o + np.swapaxes(o, 1, 2)) * w[:, :, None]
            keys.append(cells[:, s] * n + cells[:, t])
            val.append(np.concatenate([w * g[:, t] / (dim + 1), o.reshape(len(vol), -1)], 1))
    key, inv = np.unique(np.concatenate(keys), return_inverse=True)
    inv, val = inv.ravel(), np.concatenate(val)
    val = np.stack([np.bincount(inv, val[:, c], len(key)) for c in range(val.shape[1])], 1)
    return key // n, key % n, val[:, :dim], val[:, dim:].reshape(-1, dim, dim), mass


def _operators(case, dev):
    """Neighbours idx (slot, node) with a (slot, dim, node or 1) and
    b (slot, dim, dim, node or 1), and the lumped mass.  On a lattice they are
    assembled on a small one of the same kind."""
    kind, nx, ny, nz = _key(case)
    if kind in ("delaunay", "tets"):
        xy, cells, box, _ = _mesh_arrays(kind, nx, ny, nz)
        i, j, a, b, mass = _assemble(xy, cells, box)
        n, dim = xy.shape
        first = np.searchsorted(i, np.arange(n))
        slot = np.arange(len(i)) - first[i]
        slots = int(slot.max()) + 1
        idx = np.tile(np.arange(n), (slots, 1))
        A, B = np.zeros((slots, dim, n)), np.zeros((slots, dim, dim, n))
        idx[slot, i] = j
        A[slot, :, i], B[slot, :, :, i] = a, b
    else:
        small = (5, 5, 5 if kind == "kuhn" else 0)
        xy, cells, box, _ = _mesh_arrays(kind, *small)
        dim = xy.shape[1]
        i, j, a, b, m = _assemble(xy, cells, box)
        size = np.array([nx, ny, nz][:dim])
        n = int(size.prod())
        cells_of = np.stack(np.unravel_index(np.arange(n), size[::-1])[::-1])  # x fastest
        offsets = sorted({tuple(((xy[q] - xy[p] + 2.5) % 5 - 2.5).astype(int)) for p, q in zip(i, j)
                          if p == 12 + (50 if dim == 3 else 0)})
        # rows 0, 2 and 4 of the small mesh stand for the first, the inner and the last rows
        kinds = [(0, 0), (2, 1), (4, 2)] if kind == "walled" else [(2, 1)]
        A, B = np.zeros((len(offsets), dim, 3)), np.zeros((len(offsets), dim, dim, 3))
        mass = np.zeros(3)
        for row, k in kinds:
            node = 2 + 5 * row + (50 if dim == 3 else 0)
            mass[k] = m[node]
            for q in np.nonzero(i == node)[0]:
                d = xy[j[q]] - xy[node]
                if not (kind == "walled" and abs(d[1]) > 2):
                    o = offsets.index(tuple(((d + 2.5) % 5 - 2.5).astype(int)))
                    A[o, :, k], B[o, :, :, k] = a[q], b[q]
        idx = np.stack([np.ravel_multi_index(tuple(((cells_of[c] + o[c]) % size[c]) for c in range(dim))[::-1],
                                             tuple(size[::-1])) for o in offsets])
        if kind == "walled":
            of = np.where(cells_of[1] == 0, 0, np.where(cells_of[1] == ny - 1, 2, 1))
            A, B, mass = A[..., of], B[..., of], mass[of]
        else:
            A, B, mass = A[..., 1:2], B[..., 1:2], np.full(n, mass[1])
    return [torch.from_numpy(np.ascontiguousarray(v)).to(dev) for v in (idx, A, B, mass)]


class _Exact:
    """The scheme on one mesh: Taylor-Galerkin streaming with the lumped mass,
    recovered gradients, chemical potential, stress force, and the split
    collision with exact-difference gravity."""

    def __init__(self, case, dev):
        self.P, self.dev = _params(case), dev
        self.idx, self.a, b, self.mass = _operators(case, dev)
        P, dt = self.P, self.P["dt"]
        self.dim = self.a.shape[1]
        e = _E2 if self.dim == 2 else _E3
        self.e = torch.tensor(e, dtype=torch.float64, device=dev)
        w = {0: 4 / 9, 1: 1 / 9, 2: 1 / 36} if self.dim == 2 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}
        self.w = torch.tensor([w[sum(abs(v) for v in q)] for q in e], dtype=torch.float64, device=dev)[:, None]
        self.opp = [e.index(tuple(-v for v in q)) for q in e]
        self.c = -dt * (torch.einsum("qc,kcn->kqn", self.e, self.a) +
                        0.5 * dt * torch.einsum("qc,qd,kcdn->kqn", self.e, self.e, b))
        d = P["rho_l"] - P["rho_v"]
        self.beta, self.kappa = 12.0 * P["sigma"] / (P["xi"] * d ** 4), 1.5 * P["xi"] * P["sigma"] / d ** 2
        self.g = torch.tensor(P["gravity"][:self.dim], dtype=torch.float64, device=dev)[:, None]
        self.walls = []
        if case["mesh"] == "walled":
            n, nx = self.idx.shape[1], case["nx"]
            self.walls = [(slice(0, nx), 1), (slice(n - nx, n), -1)]

    def recover(self, f):
        out = 0
        for k in range(len(self.idx)):
            out = out + self.a[k] * (f[self.idx[k]] - f)
        return out

    def stream(self, psi):
        out = psi.clone()
        for k in range(len(self.idx)):
            out += self.c[k] * (psi[:, self.idx[k]] - psi)
        for rows, normal in self.walls:
            old = out[:, rows].clone()
            for q in range(len(self.e)):
                if float(self.e[q, 1]) * normal > 0:
                    out[q, rows] = old[self.opp[q]]
        return out

    def forces(self, rho):
        P, dim = self.P, self.dim
        dr = self.recover(rho)
        lap = 0
        for c in range(dim):
            lap = lap + self.recover(dr[c])[c]
        K = self.recover((dr * dr).sum(0))
        for c in range(dim):
            for d in range(c, dim):
                r = self.recover(dr[c] * dr[d])
                K[c] -= r[d]
                if d != c:
                    K[d] -= r[c]
        mu = 4.0 * self.beta * (rho - P["rho_v"]) * (rho - P["rho_l"]) * (rho - 0.5 * (P["rho_v"] + P["rho_l"]))
        return dr, self.kappa * K, self.recover(mu - self.kappa * lap)

    def gamma(self, u):
        eu = self.e @ u
        return self.w * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(0))

    def terms(self, rho, u, p, dr, K, dm):
        """Equilibria and sources."""
        dt, ga = self.P["dt"], self.gamma(u)
        X = dr / 3.0 - rho * dm

        def rel(v):  # (e - u) . v
            return self.e @ v - (u * v).sum(0)

        F = 0.5 * dt * rel(X) * 3.0 * ga
        S = 0.5 * dt * rel(dr) * (ga - self.w) + 0.5 * dt * rel(K) * 3.0 * ga
        if bool((self.g != 0).any()):
            S = S + 0.5 * rho * (self.gamma(u + self.g * dt) - ga)
        return rho * ga, 3.0 * self.w * p + rho * (ga - self.w), F, S

    def start(self, rho, u, p):
        rho, p = (torch.from_numpy(np.ascontiguousarray(v)).to(self.dev) for v in (rho, p))
        u = torch.from_numpy(np.ascontiguousarray(u.T)).to(self.dev)
        he, ge, F, S = self.terms(rho, u, p, *self.forces(rho))
        self.h, self.gg = he + F, ge + S

    def step(self):
        P, dt = self.P, self.P["dt"]
        h, g = self.stream(self.h), self.stream(self.gg)
        rho = h.sum(0)
        dr, K, dm = self.forces(rho)
        u = (self.e.T @ g + 0.5 * dt * K + 0.5 * dt * rho * self.g) / rho
        p = (g.sum(0) + 0.5 * dt * (u * dr).sum(0)) / 3.0
        C = ((rho - P["rho_v"]) / (P["rho_l"] - P["rho_v"])).clamp(0.0, 1.0)
        tau = 1.0 / (C / P["tau_l"] + (1.0 - C) / P["tau_v"])
        he, ge, F, S = self.terms(rho, u, p, dr, K, dm)
        post = 2.0 * tau / (2.0 * tau + 1.0)
        for v, eq, s, name in ((h, he, F, "h"), (g, ge, S, "gg")):
            v = v + post * ((eq - v) / (2.0 * tau) + s)
            setattr(self, name, v + ((eq - v) / (2.0 * tau) + s))
        self.moments = rho, u, p

    def fields(self):
        rho, u, p = self.moments
        mr = self.mass * rho
        totals = torch.cat([mr.sum()[None], (mr * u).sum(1)])
        return {"rho": rho, "u": u.T, "p": p, "totals": totals[None]}


def exact(case, seed):
    runs = _runs(case)
    nodes = sum(c["nx"] * c["ny"] * c.get("nz", 1) for c in runs)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    three = 6 if case["mesh"] in ("kuhn", "tets") else 1
    if len(runs) * case["steps"] > 3000 or nodes * case["steps"] * three > (7e8 if dev == "cuda" else 2e6):
        return None
    rng = np.random.default_rng(seed)
    got = []
    for c in runs:
        x = _Exact(c, dev)
        x.start(*_fields(c, rng))
        for _ in range(c["steps"]):
            x.step()
        got.append(x.fields())
    return {k: torch.cat([f[k] for f in got]).cpu() for k in got[0]}
