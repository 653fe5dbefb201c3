"""Performance cases: what a user of the library has it do, through its public entry points.

A case is a dict of plain values.  The kinds:

* ``sweep``       one sweep on one mesh (``Mesh.sweep``);
* ``solve``       a quasistatic solve or a backward Euler step of a fixed number of sweeps
                  (``Mesh.solve_step``), with graph replay, restarts or the line search where asked;
* ``concurrent``  several meshes solved side by side (``solve_concurrent``);
* ``batch``       many small meshes solved as one union (``Mesh.solve_batch``);
* ``forward``     the subspace network's inference (``MLP.forward``);
* ``train``       steps of the network's training (``MLP.train``).

Meshes are boxes of ``nx x ny x nz`` cells, six tets to a cell (Kuhn split), as in the library's
tests and benchmark.  Starting positions are a small load increment away from rest: a pull of the
clamped face or a twist, plus a smooth displacement drawn from the seed, so a sweep's update is
small against the body, as in all but the first sweeps of a solve.
"""
import itertools
import math

import numpy as np
import torch

import paper_2510_12053_gb300 as cc

D_IN, LDX, D_OUT = cc.LEARNED_D_IN, cc.LEARNED_LDX, cc.LEARNED_D_OUT
NET = {"hidden": 256, "layers": 3}


# ---------------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------------
def _mesh_case(kind, nx, ny, nz, **kw):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "jitter": 0.05, "scene": "stretch", "E": 1e5, "nu": 0.3,
         "model": "snh", "precision": "mixed", "update": "cc", "schedule": "colored", "colors": "lattice", "k": 2,
         "corotated": False, "h": 0.0, "sweeps": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest body of the tests and the benchmark: launches and latency are what counts
        dict(_mesh_case("sweep", 8, 8, 8), name="sweep_cube8"),
        # the benchmark's body, one sweep as a program with its own outer loop calls it
        dict(_mesh_case("sweep", 32, 32, 32), name="sweep_cube32"),
        # a body whose state does not fit the caches (regular grid, as large grids mostly are)
        dict(_mesh_case("sweep", 64, 64, 64, jitter=0.0), name="sweep_cube64"),
        # everything in float64: the precision that the mixed sweep is checked against in use
        dict(_mesh_case("sweep", 24, 23, 25, precision="fp64"), name="sweep_box24_fp64"),
        # the ordinary call: a solve with graph replay and a residual check every 8 sweeps
        dict(_mesh_case("solve", 32, 32, 32, sweeps=24, check_every=8, graph=True), name="solve_cube32"),
        # the benchmark's headline: the four stiffnesses of one body side by side
        dict(_mesh_case("concurrent", 32, 32, 32, sweeps=16, check_every=8, graph=True, count=4),
             name="concurrent_cube32"),
        # many small bodies of unlike sizes and materials in one union (sides 4 to 24)
        dict(_mesh_case("batch", 0, 0, 0, sweeps=8, check_every=4, graph=True, count=24, side_lo=4, side_hi=24),
             name="batch_boxes"),
        # the corotational material on a twisted bar, rotated bases, greedy colouring, energy line search
        dict(_mesh_case("solve", 9, 11, 37, scene="twist", model="fcr", corotated=True, colors="greedy", sweeps=3,
                        line_search=True), name="twist_fcr_corotated"),
        # one time step of a cantilever with 3-ring bases
        dict(_mesh_case("solve", 16, 16, 64, scene="beam", jitter=0.0, E=1e6, k=3, h=1.0 / 120.0, sweeps=2),
             name="beam_step_ring3"),
        # restarted bases: every patch of the body solved again at the current positions
        dict(_mesh_case("solve", 16, 16, 16, sweeps=4, check_every=2, restart_every=2), name="restart_cube16"),
        # the learned bases of the 48^3 cube (112 847 free vertices): one inference
        {"kind": "forward", "rows": 112847, "name": "forward_cube48"},
        # training of the subspace network at the benchmark's batch
        {"kind": "train", "samples": 65536, "batch": 8192, "steps": 8, "name": "train_8192"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sweep", "sweep", "sweep64", "solve", "solve", "concurrent", "batch", "twist", "beam",
                       "restart", "forward", "train"])
    colors = rng.choice(["lattice", "lattice", "greedy"])
    jit = rng.choice([0.05, 0.05, 0.0])
    E = 10.0 ** rng.uniform(4, 7)

    def sides(lo, hi, most):
        while True:
            s = [_log_int(rng, lo, hi) for _ in range(3)]
            if s[0] * s[1] * s[2] <= most:
                return s

    if kind == "sweep":
        return _mesh_case("sweep", *sides(5, 64, 110000), jitter=jit, E=E, colors=colors,
                          update=rng.choice(["cc", "cc", "cc", "jgs2", "cd"]),
                          schedule=rng.choice(["colored", "colored", "colored", "jacobi"]))
    if kind == "sweep64":
        return _mesh_case("sweep", *sides(5, 26, 14000), jitter=jit, E=E, colors=colors, precision="fp64",
                          update=rng.choice(["cc", "cc", "jgs2", "cd"]))
    if kind == "solve":
        every = rng.choice([1, 4, 8])
        return _mesh_case("solve", *sides(5, 34, 33000), jitter=jit, E=E, colors=colors, sweeps=every * rng.choice([2, 3]),
                          check_every=every, graph=rng.random() < 0.7, k=rng.choice([1, 2, 2]))
    if kind == "concurrent":
        return _mesh_case("concurrent", *sides(6, 33, 30000), jitter=jit, sweeps=16, check_every=8, graph=True,
                          count=rng.choice([2, 3, 4]), colors=colors)
    if kind == "batch":
        return _mesh_case("batch", 0, 0, 0, sweeps=8, check_every=rng.choice([2, 4]), graph=True, colors=colors,
                          count=rng.randrange(3, 25), side_lo=4, side_hi=rng.randrange(8, 25))
    if kind == "twist":
        return _mesh_case("solve", rng.randrange(4, 12), rng.randrange(4, 12), rng.randrange(13, 41), scene="twist",
                          model=rng.choice(["fcr", "fcr", "snh"]), corotated=rng.random() < 0.7, E=E, colors=colors,
                          precision=rng.choice(["mixed", "mixed", "fp64"]), sweeps=rng.choice([2, 3]),
                          line_search=rng.random() < 0.5)
    if kind == "beam":
        return _mesh_case("solve", rng.randrange(4, 17), rng.randrange(4, 17), rng.randrange(17, 65), scene="beam",
                          jitter=0.0, E=1e6, k=rng.choice([2, 2, 3]), h=1.0 / 120.0, sweeps=rng.choice([1, 2]))
    if kind == "restart":
        return _mesh_case("solve", *sides(5, 20, 4096), jitter=0.05, E=E, colors=colors, sweeps=4, check_every=2,
                          restart_every=2)
    if kind == "forward":
        return {"kind": "forward", "rows": _log_int(rng, 500, 112000)}
    return {"kind": "train", "samples": 32768, "batch": rng.choice([1000, 2048, 4096, 5000, 8192]),
            "steps": rng.choice([2, 4, 8])}


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
class _Material:
    def __init__(self, E, nu, rho):
        self.E, self.nu, self.rho = E, nu, rho


class _Scene:
    """What ``Mesh.from_scenes`` reads of a mesh, and the starting positions."""


def _grid(nx, ny, nz, cell):
    k, j, i = np.meshgrid(np.arange(nz + 1), np.arange(ny + 1), np.arange(nx + 1), indexing="ij")
    ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1)
    sx, sy = nx + 1, (nx + 1) * (ny + 1)
    ck, cj, ci = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    base = ci.ravel() + sx * cj.ravel() + sy * ck.ravel()
    step = (1, sx, sy)
    tets = np.empty((base.size, 6, 4), dtype=np.int32)
    for p, (a, b, c) in enumerate(itertools.permutations(range(3))):
        v1, v2 = base + step[a], base + step[a] + step[b]
        if (a, b, c) in ((0, 2, 1), (1, 0, 2), (2, 1, 0)):  # odd: swapped to positive volume
            v1, v2 = v2, v1
        tets[:, p, 0], tets[:, p, 1], tets[:, p, 2], tets[:, p, 3] = base, v1, v2, base + sum(step)
    return ijk, ijk * float(cell), tets.reshape(-1, 4)


def _smooth(X, rng, size, amount):
    """A displacement of ``amount``: three sine waves of the body's length."""
    d = np.zeros_like(X)
    for _ in range(3):
        wave, phase = rng.normal(size=(3, 3)) * (2.0 / size), rng.uniform(0, 2 * np.pi, 3)
        d += np.sin(X @ wave + phase) * (amount / 3.0)
    return d


def _scene(case, rng, *, E=None, nu=None, axis=None, factor=1.01):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    beam, twist = case["scene"] == "beam", case["scene"] == "twist"
    cell = 1.0 / 16.0 if beam else 1.0 / max(nx, ny, nz)
    ijk, X, tets = _grid(nx, ny, nz, cell)
    dims = np.array([nx, ny, nz])
    if case["jitter"]:
        inner = ((ijk > 0) & (ijk < dims)).all(axis=1)
        X[inner] += rng.uniform(-1.0, 1.0, (int(inner.sum()), 3)) * (case["jitter"] * cell)
    ax = 2 if beam or twist else (0 if axis is None else axis)
    lo, hi = ijk[:, ax] == 0, ijk[:, ax] == dims[ax]
    s = _Scene()
    s.pinned = (lo if beam else lo | hi).astype(np.uint8)
    x = X.copy()
    if twist:
        th = 0.3 * X[:, 2] / (nz * cell)
        mx, my = 0.5 * nx * cell, 0.5 * ny * cell
        x[:, 0] = mx + np.cos(th) * (X[:, 0] - mx) - np.sin(th) * (X[:, 1] - my)
        x[:, 1] = my + np.sin(th) * (X[:, 0] - mx) + np.cos(th) * (X[:, 1] - my)
    elif not beam:
        x[:, ax] *= factor
    # the smooth part, faded out towards the clamped faces
    u = ijk[:, ax] / dims[ax]
    fade = np.where(s.pinned > 0, 0.0, np.sin(0.5 * np.pi * u) if beam else np.sin(np.pi * u))
    x += fade[:, None] * _smooth(X, rng, cell * dims.max(), 0.01 * cell)
    s.X, s.tets, s.x0, s.h = X, tets, x, case["h"]
    s.gravity = np.array([0.0, -9.8, 0.0]) if case["h"] else np.zeros(3)
    s.v0 = _smooth(X, rng, cell * dims.max(), 0.02) * fade[:, None] if case["h"] else None
    s.material = _Material(case["E"] if E is None else E, case["nu"] if nu is None else nu, 1000.0)
    s.n, s.T = X.shape[0], tets.shape[0]
    s.lattice = (ijk.sum(axis=1) % 4).astype(np.int32)
    return s


def _scenes(case, seed):
    rng = np.random.default_rng([seed, 11])
    if case["kind"] == "concurrent":
        return [_scene(case, rng, E=10.0 ** (4 + k)) for k in range(case["count"])]
    if case["kind"] == "batch":
        # the sizes are the case's own (every seed has the same amount of work)
        size = np.random.default_rng([case["count"], case["side_lo"], case["side_hi"]])
        out = []
        for _ in range(case["count"]):
            nx, ny, nz = (int(v) for v in size.integers(case["side_lo"], case["side_hi"] + 1, 3))
            out.append(_scene(dict(case, nx=nx, ny=ny, nz=nz), rng, E=10.0 ** rng.uniform(4, 7),
                              nu=rng.uniform(0.30, 0.35), axis=int(rng.integers(3)), factor=rng.uniform(1.002, 1.01)))
        return out
    return [_scene(case, rng)]


def _soa(x):
    return torch.as_tensor(np.ascontiguousarray(x.T), device="cuda")


def _network(seed):
    """He-normal weights, layer by layer, as one float32 vector."""
    rng = np.random.default_rng([seed, 7])
    dims = [D_IN] + [NET["hidden"]] * NET["layers"] + [D_OUT]
    parts = []
    for n_in, n_out in zip(dims[:-1], dims[1:]):
        parts.append((rng.standard_normal(n_out * n_in) * math.sqrt(2.0 / n_in)).astype(np.float32))
        parts.append((rng.standard_normal(n_out) * 0.1).astype(np.float32))
    return dims, np.concatenate(parts)


def _net_inputs(case, seed):
    """Rows as the library's inputs are: small deviations, a state channel of -1, 0 or 1, the material."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    rows = case["rows"] if case["kind"] == "forward" else case["samples"]
    X = torch.zeros((rows, LDX), dtype=torch.bfloat16, device="cuda")
    dev = torch.randn((rows, 64, 4), generator=g, device="cuda") * 0.4
    dev[:, :, 3] = torch.randint(-1, 2, (rows, 64), generator=g, device="cuda").float()
    X[:, :256] = dev.reshape(rows, 256).to(torch.bfloat16)
    X[:, 256:D_IN] = torch.randn((rows, 2), generator=g, device="cuda").to(torch.bfloat16)
    return X, g


def prepare(case, seed):
    if case["kind"] in ("forward", "train"):
        X, g = _net_inputs(case, seed)
        _, params = _network(seed)
        net = cc.MLP(max_batch=case.get("batch", 64), **NET)
        net.set_params(params)
        st = {"case": case, "net": net, "X": X}
        if case["kind"] == "train":
            st["T"] = torch.randn((case["samples"], D_OUT), generator=g, device="cuda") * 0.07
            st["idx"] = torch.randint(0, case["samples"], (case["steps"], case["batch"]), generator=g, device="cuda",
                                      dtype=torch.int32)
        return st
    st = {"case": case}
    scenes = _scenes(case, seed)
    if case["kind"] == "batch":
        stream = torch.cuda.Stream()
        m = cc.Mesh.from_scenes(scenes, stream=stream, model=case["model"])
        groups = [(m, scenes, stream)]
    else:
        groups = []
        for s in scenes:
            # a mesh whose solves are replayed as graphs or run side by side has a stream of its own
            stream = torch.cuda.Stream() if case["kind"] == "concurrent" or case.get("graph") else None
            groups.append((cc.Mesh.from_scene(s, stream=stream, model=case["model"]), [s], stream))
    st["meshes"], st["streams"], st["x0"], st["x"], st["v0"], st["v"] = [], [], [], [], [], []
    for m, part, stream in groups:
        if case["colors"] == "lattice":
            m.set_colors(np.concatenate([s.lattice for s in part]), 4)
        else:
            m.color()
        m.build_subspace(case["k"])
        x0 = _soa(np.concatenate([s.x0 for s in part]))
        st["meshes"].append(m)
        st["streams"].append(stream)
        st["x0"].append(x0)
        st["x"].append(torch.empty_like(x0))
        if case["h"]:
            v0 = _soa(np.concatenate([s.v0 for s in part]))
            st["v0"].append(v0)
            st["v"].append(torch.empty_like(v0))
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def _start(st):
    """Every mesh's positions (and velocities) back at the start, on the mesh's stream."""
    for k, s in enumerate(st["streams"]):
        with torch.cuda.stream(s):
            st["x"][k].copy_(st["x0"][k])
            if st["v"]:
                st["v"][k].copy_(st["v0"][k])


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "forward":
        return st["net"].forward(st["X"])
    if kind == "train":
        losses = st["net"].train(st["X"], st["T"], st["idx"], case["batch"])
        return {"losses": losses.tolist(), "params": st["net"].get_params()}
    _start(st)
    m, x = st["meshes"][0], st["x"][0]
    if kind == "sweep":
        m.sweep(x, update=case["update"], schedule=case["schedule"], precision=case["precision"],
                corotated=case["corotated"])
        return x
    kw = dict(update=case["update"], schedule=case["schedule"], precision=case["precision"], tol=0.0,
              max_iters=case["sweeps"], check_every=case.get("check_every", 1), use_graph=case.get("graph", False),
              corotated=case["corotated"], line_search=case.get("line_search", False),
              restart_every=case.get("restart_every", 0))
    if kind == "solve":
        r = m.solve_step(x, st["v"][0] if st["v"] else None, **kw)
        out = {"x": x, "g0": r.g0, "g_final": r.g_final, "iterations": r.iterations}
        if st["v"]:
            out["v"] = st["v"][0]
        return out
    if kind == "concurrent":
        res = cc.solve_concurrent(st["meshes"], st["x"], **kw)
        return [{"x": xk, "g_final": r.g_final, "iterations": r.iterations} for xk, r in zip(st["x"], res)]
    r = m.solve_batch(x, **kw)
    return {"x": x, "iterations": r["iterations"], "status": r["status"], "g_final": r["g_final"].tolist()}


# ---------------------------------------------------------------------------------------------
# the work that a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _ring(k):
    """Offsets of the k-ring of a grid vertex of the Kuhn split, itself excluded."""
    one = [d for d in itertools.product((0, 1), repeat=3) if any(d)]
    one = one + [tuple(-v for v in d) for d in one]
    at, seen = {(0, 0, 0)}, {(0, 0, 0)}
    for _ in range(k):
        at = {tuple(a + b for a, b in zip(p, d)) for p in at for d in one} - seen
        seen |= at
    return seen - {(0, 0, 0)}


def _pairs(dims, offsets):
    return sum(math.prod(max(0, n - abs(o)) for n, o in zip(dims, off)) for off in offsets)


def _mesh_work(case, nx, ny, nz, ax):
    """(bytes, flops) of one sweep: the bases, the supports, the tets and the positions each once; the local
    solves' products and every tet's derivatives once for each colour."""
    e = 8 if case["precision"] == "fp64" else 4
    n, tets = (nx + 1) * (ny + 1) * (nz + 1), 6 * nx * ny * nz
    free = [nx + 1, ny + 1, nz + 1]
    free[ax] -= 1 if case["scene"] == "beam" else 2
    sup = _pairs(free, _ring(case["k"])) if case["update"] != "cd" else 0
    colours = 1 if case["schedule"] == "jacobi" else (4 if case["colors"] == "lattice" else 8)
    blocks = sup * 4.0 if case["k"] > 1 else sup * 2.5  # upper blocks inside the supports
    nbytes = sup * (9 * e + 4) + tets * (16 + 10 * e) + 2 * 24 * n
    flops = 54.0 * (blocks + sup) + 36.0 * sup + 400.0 * tets * colours + 300.0 * math.prod(free)
    return nbytes, flops


def work(case):
    if case["kind"] in ("forward", "train"):
        dims = [D_IN] + [NET["hidden"]] * NET["layers"] + [D_OUT]
        weights = sum(a * b for a, b in zip(dims[:-1], dims[1:]))
        if case["kind"] == "forward":
            return {"bytes": case["rows"] * (2.0 * D_IN + 4.0 * D_OUT) + 4.0 * weights, "flops": 2.0 * case["rows"] * weights}
        rows = case["steps"] * case["batch"]
        return {"bytes": rows * (2.0 * D_IN + 4.0 * D_OUT + 4.0) + case["steps"] * 24.0 * weights,
                "flops": rows * (6.0 * weights - 2.0 * dims[0] * dims[1])}
    if case["kind"] == "batch":
        size = np.random.default_rng([case["count"], case["side_lo"], case["side_hi"]])
        parts = [_mesh_work(case, *(int(v) for v in size.integers(case["side_lo"], case["side_hi"] + 1, 3)), 0)
                 for _ in range(case["count"])]
    else:
        ax = 2 if case["scene"] in ("beam", "twist") else 0
        parts = [_mesh_work(case, case["nx"], case["ny"], case["nz"], ax)] * case.get("count", 1)
    nbytes, flops = sum(p[0] for p in parts) * case["sweeps"], sum(p[1] for p in parts) * case["sweeps"]
    if case.get("restart_every"):
        times = (case["sweeps"] - 1) // case["restart_every"]
        free = (case["nx"] - 1) * (case["ny"] + 1) * (case["nz"] + 1)
        unknowns = 3.0 * _pairs([case["nx"] - 1, case["ny"] + 1, case["nz"] + 1], _ring(case["k"])) / free
        flops += times * free * (unknowns ** 3 / 3 + 6 * unknowns ** 2)
        nbytes += times * free * unknowns * 24.0
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------------------------
# the results in 64 bits, by plain torch
# ---------------------------------------------------------------------------------------------
class _Exact:
    """Energy, derivatives, bases and sweeps of one mesh in float64, every sum written out plainly."""

    def __init__(self, scenes, case):
        f8 = dict(dtype=torch.float64, device="cuda")
        off = np.cumsum([0] + [s.n for s in scenes])
        self.X = torch.as_tensor(np.concatenate([s.X for s in scenes]), **f8)
        self.tets = torch.as_tensor(np.concatenate([s.tets.astype(np.int64) + o for s, o in zip(scenes, off)])).cuda()
        self.free = torch.as_tensor(np.concatenate([s.pinned for s in scenes]) == 0).cuda()
        self.n, self.h, self.case = int(off[-1]), scenes[0].h, case
        E = torch.as_tensor(np.concatenate([np.full(s.T, s.material.E) for s in scenes]), **f8)
        nu = torch.as_tensor(np.concatenate([np.full(s.T, s.material.nu) for s in scenes]), **f8)
        self.mu, self.lam = E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))
        p = self.X[self.tets]
        Dm = (p[:, 1:] - p[:, :1]).transpose(1, 2)
        self.vol = torch.linalg.det(Dm) / 6.0
        B = torch.linalg.inv(Dm)
        self.G = torch.cat([-B.sum(dim=1, keepdim=True), B], dim=1)  # shape vectors [T, 4, 3]
        self.w = self.h ** 2 if self.h else 1.0
        self.mass = torch.zeros(self.n, **f8).index_add_(0, self.tets.reshape(-1), (scenes[0].material.rho * self.vol / 4)
                                                         .repeat_interleave(4))
        # block pattern: keys row * n + column, ascending
        rows, cols = self.tets[:, :, None].expand(-1, 4, 4), self.tets[:, None, :].expand(-1, 4, 4)
        self.keys, self.at = torch.unique(rows * self.n + cols, return_inverse=True)
        self.brow, self.bcol = self.keys // self.n, self.keys % self.n
        self.bptr = torch.searchsorted(self.brow, torch.arange(self.n + 1, device="cuda"))
        self.eps = torch.zeros((3, 3, 3), **f8)
        for a, b, c in ((0, 1, 2), (1, 2, 0), (2, 0, 1)):
            self.eps[a, b, c], self.eps[b, a, c] = 1.0, -1.0
        self.eye = torch.eye(3, **f8)

    def energy(self, x, xt=None):
        F, J, _ = self._kinematics(x)
        if self.case["model"] == "fcr":
            psi = self.mu * (F - self._polar(F)[0]).square().sum((1, 2)) + 0.5 * self.lam * (J - 1) ** 2
        else:
            psi = 0.5 * self.mu * (F.square().sum((1, 2)) - 3) - self.mu * (J - 1) + 0.5 * (self.lam + self.mu) * (J - 1) ** 2
        e = self.w * (self.vol * psi).sum()
        return e if xt is None else e + 0.5 * (self.mass[:, None] * (x - xt) ** 2).sum()

    def _kinematics(self, x):
        F = torch.einsum("tva,tvb->tab", x[self.tets], self.G)
        C = torch.linalg.det(F)[:, None, None] * torch.linalg.inv(F).transpose(1, 2)
        return F, torch.linalg.det(F), C

    @staticmethod
    def _polar(F):
        U, s, Vh = torch.linalg.svd(F)
        flip = torch.where(torch.linalg.det(U @ Vh) < 0, -1.0, 1.0).to(F.dtype)
        U = torch.cat([U[:, :, :2], U[:, :, 2:] * flip[:, None, None]], dim=2)
        return U @ Vh, U, torch.cat([s[:, :2], s[:, 2:] * flip[:, None]], dim=1), Vh

    def derivatives(self, x, xt=None):
        """Gradient [n, 3] and Hessian blocks in the order of the pattern."""
        F, J, C = self._kinematics(x)
        eye2 = torch.einsum("ik,jl->ijkl", self.eye, self.eye)
        curl = torch.einsum("ikm,jln,tmn->tijkl", self.eps, self.eps, F)
        mu, lam = self.mu[:, None, None], self.lam[:, None, None]
        if self.case["model"] == "fcr":
            R, U, s, Vh = self._polar(F)
            P = 2 * mu * (F - R) + lam * (J - 1)[:, None, None] * C
            # dR = U [(U^T dF V - V^T dF^T U) / (s_i + s_j)] V^T for the nine unit directions dF
            M = torch.einsum("tki,tjl->tijkl", U, Vh)
            M = (M - M.transpose(1, 2)) / (s[:, :, None] + s[:, None, :])[:, :, :, None, None]
            dR = torch.einsum("tai,tijkl,tjb->tabkl", U, M, Vh)
            D = 2 * mu[..., None, None] * (eye2 - dR)
            lh, sJ = self.lam, self.lam * (J - 1)
        else:
            lh, sJ = self.lam + self.mu, (self.lam + self.mu) * (J - 1) - self.mu
            P = mu * F + sJ[:, None, None] * C
            D = mu[..., None, None] * eye2
        D = D + lh[:, None, None, None, None] * torch.einsum("tij,tkl->tijkl", C, C) + sJ[:, None, None, None, None] * curl
        wv = (self.w * self.vol)
        g = torch.zeros_like(x).index_add_(0, self.tets.reshape(-1), (torch.einsum("tab,tvb->tva", P, self.G) *
                                                                       wv[:, None, None]).reshape(-1, 3))
        half = torch.einsum("tijkl,tbl->tijkb", D, self.G)
        K = torch.einsum("tijkb,taj->tabik", half, self.G) * wv[:, None, None, None, None]
        H = torch.zeros((self.keys.numel(), 3, 3), dtype=torch.float64, device="cuda")
        H.index_add_(0, self.at.reshape(-1), K.reshape(-1, 3, 3))
        if xt is not None:
            g = g + self.mass[:, None] * (x - xt)
        if self.h:
            diag = self.brow == self.bcol
            H[diag] += self.mass[:, None, None] * self.eye
        return g * self.free[:, None], H

    def supports(self, k):
        """Support lists (CSR over vertices) and, per block product inside a support, (vertex's list, row, column, block)."""
        n, free = self.n, torch.nonzero(self.free).flatten()
        pairs = free * n + free
        seen = pairs
        for _ in range(k):
            i, j = pairs // n, pairs % n
            cnt = self.bptr[j + 1] - self.bptr[j]
            rep = torch.repeat_interleave(torch.arange(j.numel(), device="cuda"), cnt)
            pos = torch.arange(rep.numel(), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[rep] + self.bptr[j][rep]
            pairs = torch.unique(torch.cat([seen, i[rep] * n + self.bcol[pos]]))
            seen = pairs
        i, j = seen // n, seen % n
        keep = self.free[j] & (i != j)
        self.sup = seen[keep]
        self.si, self.sj = self.sup // n, self.sup % n
        self.sptr = torch.searchsorted(self.si, torch.arange(n + 1, device="cuda"))
        cnt = self.bptr[self.sj + 1] - self.bptr[self.sj]
        a = torch.repeat_interleave(torch.arange(self.sj.numel(), device="cuda"), cnt)
        blk = torch.arange(a.numel(), device="cuda") - (torch.cumsum(cnt, 0) - cnt)[a] + self.bptr[self.sj][a]
        key = self.si[a] * n + self.bcol[blk]
        b = torch.searchsorted(self.sup, key).clamp(max=self.sup.numel() - 1)
        inside, own = self.sup[b] == key, self.bcol[blk] == self.si[a]
        self.pa, self.pb, self.pblk = a[inside], b[inside], blk[inside]   # block (S_a, S_b)
        self.oa, self.oblk = a[own], blk[own]                             # block (S_a, i)
        self.diag = torch.searchsorted(self.keys, torch.arange(n, device="cuda") * (n + 1))

    def bases(self, x):
        """U [support entries, 3, 3]: -H_PP^{-1} H_Pi with the Hessian at x."""
        _, H = self.derivatives(x)
        size = self.sptr[1:] - self.sptr[:-1]
        m, U = int(size.max()), torch.zeros((self.sup.numel(), 3, 3), dtype=torch.float64, device="cuda")
        who = torch.nonzero(size > 0).flatten()
        start = torch.searchsorted(self.si[self.pa], torch.arange(self.n + 1, device="cuda"))
        step = max(1, int(2 ** 31 // (9 * m * m * 8)))
        for c0 in range(0, who.numel(), step):
            v = who[c0:c0 + step]
            lo, hi = int(v[0]), int(v[-1]) + 1
            loc = torch.full((self.n,), -1, device="cuda")
            loc[v] = torch.arange(v.numel(), device="cuda")
            e0, e1 = int(start[lo]), int(start[hi])
            a, b, blk = self.pa[e0:e1], self.pb[e0:e1], self.pblk[e0:e1]
            i = self.si[a]
            A = torch.zeros((v.numel(), m, m, 3, 3), dtype=torch.float64, device="cuda")
            A[loc[i], a - self.sptr[i], b - self.sptr[i]] = H[blk]
            pad = torch.arange(m, device="cuda")[None] >= size[v][:, None]
            pv, pm = torch.nonzero(pad, as_tuple=True)
            A[pv, pm, pm] = self.eye
            s0, s1 = int(self.sptr[lo]), int(self.sptr[hi])
            rhs = torch.zeros((v.numel(), m, 3, 3), dtype=torch.float64, device="cuda")
            own = (self.oa >= s0) & (self.oa < s1)
            oi = self.si[self.oa[own]]
            rhs[loc[oi], self.oa[own] - self.sptr[oi]] = -H[self.oblk[own]]
            L = torch.linalg.cholesky(A.permute(0, 1, 3, 2, 4).reshape(v.numel(), 3 * m, 3 * m))
            z = torch.cholesky_solve(rhs.reshape(v.numel(), 3 * m, 3), L).reshape(v.numel(), m, 3, 3)
            si = self.si[s0:s1]
            U[s0:s1] = z[loc[si], torch.arange(s0, s1, device="cuda") - self.sptr[si]]
        return U

    def rotations(self, x):
        off = self.brow != self.bcol
        r, c = self.brow[off], self.bcol[off]
        dx, dX = x[c] - x[r], self.X[c] - self.X[r]
        A = torch.zeros((self.n, 3, 3), dtype=torch.float64, device="cuda").index_add_(0, r, dx[:, :, None] * dX[:, None])
        C = torch.zeros_like(A).index_add_(0, r, dX[:, :, None] * dX[:, None])
        return self._polar(A @ torch.linalg.inv(C))[0]

    def sweep(self, x, U, colour, xt=None):
        upd = self.case["update"]
        if self.case["corotated"] and upd != "cd":
            U = self.rotations(x)[self.sj] @ U
        rounds = [None] if self.case["schedule"] == "jacobi" else range(int(colour.max()) + 1)
        for c in rounds:
            g, H = self.derivatives(x, xt)
            mine = self.free if c is None else self.free & (colour == c)
            zero = torch.zeros((self.n, 3, 3), dtype=torch.float64, device="cuda")
            Hii = H[self.diag]
            if upd == "cd":
                M, rhs = Hii, g
            else:
                on = mine[self.si[self.pa]]
                a, b, blk = self.pa[on], self.pb[on], self.pblk[on]
                Ht = zero.index_add(0, self.si[a], U[a].transpose(1, 2) @ H[blk] @ U[b])
                own = mine[self.si[self.oa]]
                a, blk = self.oa[own], self.oblk[own]
                A = zero.index_add(0, self.si[a], H[blk].transpose(1, 2) @ U[a])
                r = torch.zeros_like(g).index_add(0, self.si, torch.einsum("sab,sa->sb", U, g[self.sj]))
                if upd == "jgs2":
                    M, rhs = Hii + Ht, g + r
                else:
                    empty = self.sptr[1:] == self.sptr[:-1]
                    Ht = torch.where((mine & ~empty)[:, None, None], Ht, self.eye)
                    W = torch.linalg.solve(Ht, A.transpose(1, 2)).transpose(1, 2)
                    M, rhs = Hii - W @ A.transpose(1, 2), g - (W @ r[:, :, None])[:, :, 0]
            M = torch.where(mine[:, None, None], M, self.eye)
            x = x - torch.linalg.solve(M, rhs[:, :, None])[:, :, 0] * mine[:, None]
        return x

    def greedy(self):
        ptr, col = self.bptr.cpu().numpy(), self.bcol.cpu().numpy()
        out = np.full(self.n, -1)
        for v in range(self.n):
            used = {out[u] for u in col[ptr[v]:ptr[v + 1]] if u < v}
            out[v] = next(c for c in itertools.count() if c not in used)
        return torch.as_tensor(out).cuda()

    def solve(self, scenes):
        c = self.case
        x = torch.as_tensor(np.concatenate([s.x0 for s in scenes])).cuda()
        colour = torch.as_tensor(np.concatenate([s.lattice for s in scenes])).cuda() if c["colors"] == "lattice" else self.greedy()
        U = None
        if c["update"] != "cd":
            self.supports(c["k"])
            U = self.bases(self.X)
        xt, x_old = None, x
        if self.h:
            v = torch.as_tensor(scenes[0].v0).cuda()
            xt = x + self.h * v + self.h ** 2 * torch.as_tensor(scenes[0].gravity).cuda()
        g0 = self.derivatives(x, xt)[0].norm()
        for it in range(c["sweeps"]):
            if c.get("restart_every") and it and it % c["restart_every"] == 0:
                U = self.bases(x)
            y = self.sweep(x, U, colour, xt)
            if c.get("line_search"):
                e, a = self.energy(x, xt), 1.0
                while a > 0 and self.energy(x + a * (y - x), xt) > e:
                    a = a / 2 if a > 2.0 ** -29 else 0.0
                y = x + a * (y - x)
            x = y
        v = (x - x_old) / self.h if self.h else None
        return x, v, g0, self.derivatives(x, xt)[0]


def exact(case, seed):
    if case["kind"] == "train":
        return None
    if case["kind"] == "forward":
        X, _ = _net_inputs(case, seed)
        dims, params = _network(seed)
        p, y, at = torch.as_tensor(params).cuda().double(), X[:, :D_IN].double(), 0
        for l, (n_in, n_out) in enumerate(zip(dims[:-1], dims[1:])):
            W = p[at:at + n_in * n_out].reshape(n_out, n_in)
            b = p[at + n_in * n_out:at + n_in * n_out + n_out]
            at += n_in * n_out + n_out
            y = y @ W.T + b
            if l < len(dims) - 2:
                y = 0.5 * y * (1.0 + torch.erf(y * math.sqrt(0.5)))
        return y
    scenes = _scenes(case, seed)
    # dense patch solves in float64: a few seconds for these, far more for the largest bodies and rings
    patch = {1: 60, 2: 200, 3: 530}[case["k"]]
    if case["update"] != "cd" and sum(s.n for s in scenes[:1]) * patch ** 3 > 4e11:
        return None
    if case["kind"] == "concurrent":
        out = []
        for s in scenes:
            x, _, _, g = _Exact([s], case).solve([s])
            out.append({"x": x.T.contiguous(), "g_final": float(g.norm()), "iterations": None})
        return out
    ex = _Exact(scenes, case)
    x, v, g0, g = ex.solve(scenes)
    if case["kind"] == "sweep":
        return x.T.contiguous()
    if case["kind"] == "batch":
        off = np.cumsum([0] + [s.n for s in scenes])
        return {"x": x.T.contiguous(), "iterations": None, "status": None,
                "g_final": [float(g[a:b].norm()) for a, b in zip(off[:-1], off[1:])]}
    out = {"x": x.T.contiguous(), "g0": float(g0), "g_final": float(g.norm()), "iterations": None}
    if v is not None:
        out["v"] = v.T.contiguous()
    return out
