"""Performance cases of the thin plate / shell library: what its users have it do, through the public binding.

Every case is one call pattern of a user's program on the GPU:

* ``step``    one simulation: its state is set from device buffers, advanced ``steps`` time steps, and read
              back into device buffers (an interactive loop, a controller, a rollout from given states);
* ``batch``   many simulations of different sizes advanced together from packed, page-locked host buffers and
              back (``shell_batch_step_states``): the batched workload and the serving mix;
* ``eval``    elastic forces and energies of a given state (design evaluation, line searches, monitoring);
* ``static``  the quasi-static equilibrium of a loaded strip (Newton-Raphson with the displacement limit).

Each pass starts from the same given state, so every pass does the same work (a rollout from that state); the
solver's initial guess then comes from the steps of the pass before, as in any program that sets states. Sizes, materials and
time steps are those of the repository's benchmark workloads and tests (the 16 x 16 plate, the 128 x 128
cylinder panel, the 512 x 512-vertex jittered plate, the batch of 256 mixed instances, the serving mix, the
cantilever), with odd and ragged grids between them.

Results of the ``fp32_refine`` mode are handed on as single-precision vectors: that mode is chosen by programs
that go on in single precision (rendering, learning) and its states are accurate to a few 1e-7. FP64 results
are handed on as they are.

``exact`` restates the linearised backward-Euler step, the forces and the energies in plain torch (64 bits, forces by
automatic differentiation of the energy, direct or tightly converged linear solves).
"""
import concurrent.futures
import math

import numpy as np
import torch

import paper_2502_10872_gb300 as gb

MODELS = ("EP", "ES", "FP", "FS", "SP", "SS")


# ------------------------------------------------------------------------------------------------ the cases
def _step(name, mesh, nx, ny, model, precision, **kw):
    c = {"name": name, "kind": "step", "mesh": mesh, "nx": nx, "ny": ny, "model": model, "precision": precision,
         "E": 1e6, "t": 1e-3, "dt": 1e-2, "steps": 1, "chord": 0, "refine_rtol": 0.0}
    c.update(kw)
    return c


def _batch(name, instances, lo, hi, precision, **kw):
    c = {"name": name, "kind": "batch", "mesh": "mixed", "instances": instances, "lo": lo, "hi": hi,
         "precision": precision, "dt": 1e-2, "steps": 1, "ctas": 0, "share": 1.0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one interactive step of the 289-vertex plate, where latency is all there is
        _step("plate16", "plate", 16, 16, "EP", "fp32_refine"),
        # the same kind of call in the library's default precision, on a ragged shell panel
        _step("panel24_fp64", "cylinder", 24, 17, "SS", "fp64"),
        # a small time step (mass-dominated matrix: the automatic choice is the Jacobi preconditioner)
        _step("jacobi96", "cylinder", 96, 61, "ES", "fp32_refine", E=1e5, dt=1e-4, steps=8),
        # the ordinary single simulation: the 16,641-vertex cylinder panel
        _step("cyl128", "cylinder", 128, 128, "SS", "fp32_refine", dt=5e-3, steps=8),
        # the same panel in FP64
        _step("cyl128_fp64", "cylinder", 128, 128, "FS", "fp64", dt=5e-3, steps=4),
        # exact backward Euler by four chord iterations, ragged grid
        _step("chord64", "cylinder", 64, 49, "FS", "fp32_refine", dt=5e-3, steps=2, chord=4),
        # the largest single simulation: 262,144 vertices, jittered, refined to the workload's 1e-6
        _step("jitter512", "jitter", 511, 511, "SP", "fp32_refine", E=1e7, t=5e-4, dt=1.0 / 60.0, steps=4,
              refine_rtol=1e-6),
        # forces and energies of a mid-size shell
        {"name": "eval128", "kind": "eval", "mesh": "cylinder", "nx": 128, "ny": 128, "model": "SS",
         "precision": "fp64", "E": 1e6, "t": 1e-3, "dt": 1e-2},
        # the quasi-static cantilever: 51 nodes, some tens of Newton steps in one call
        {"name": "cantilever", "kind": "static", "mesh": "strip", "nx": 16, "ny": 2, "model": "FP",
         "precision": "fp64", "E": 1.2e6, "t": 0.1, "dt": 1.0, "load": 1.0, "eps_f": 1e-8},
        # the batched workload: 256 mixed instances, about 0.9 million vertices, its tuned launch shape
        _batch("batch256", 256, 8, 128, "fp32_refine", steps=8, ctas=5, share=2.0),
        # a small FP64 batch with the default launch shape
        _batch("batch24_fp64", 24, 8, 64, "fp64"),
        # requests of the serving mix as they sit in one batch, with the serving loop's launch shape
        _batch("serving12", 12, 32, 320, "fp32_refine", mesh="jitter", steps=8, ctas=5, share=0.125),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "batch", "eval"])
    model = rng.choice(MODELS)
    precision = rng.choice(["fp32_refine", "fp32_refine", "fp64"])
    if kind == "batch":
        n = _log_int(rng, 3, 192)
        hi = _log_int(rng, 24, 128 if precision == "fp32_refine" else 64)
        tuned = rng.random() < 0.5 and precision == "fp32_refine"
        return {k: v for k, v in _batch("", n, 8, hi, precision, mesh=rng.choice(["mixed", "mixed", "jitter"]),
                                        steps=rng.choice([1, 2, 4, 6]), ctas=5 if tuned else 0,
                                        share=2.0 if tuned else 1.0).items() if k != "name"}
    side = _log_int(rng, 9, 400 if precision == "fp32_refine" else 160)
    nx, ny = side, max(3, int(side * rng.uniform(0.5, 1.2)))
    mesh = rng.choice(["plate", "cylinder", "jitter"])
    if kind == "eval":
        return {"kind": "eval", "mesh": mesh, "nx": nx, "ny": ny, "model": model, "precision": "fp64",
                "E": 10 ** rng.uniform(5, 8), "t": 1e-3, "dt": 1e-2}
    c = _step("", mesh, nx, ny, model, precision, E=10 ** rng.uniform(5, 8), dt=rng.choice([2e-3, 5e-3, 1e-2]),
              steps=rng.choice([1, 2, 4, 6]), chord=rng.choice([0, 0, 0, 3]))
    return {k: v for k, v in c.items() if k != "name"}


# ------------------------------------------------------------------------------------------------ scenes
def _grid(nx, ny, lx, ly):
    """nx x ny cells on [0, lx] x [0, ly], each split along (i, j)-(i+1, j+1), counter-clockwise from +z."""
    gx, gy = np.meshgrid(np.linspace(0.0, lx, nx + 1), np.linspace(0.0, ly, ny + 1))
    i, j = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny)))
    a = j * (nx + 1) + i
    tris = np.stack([a, a + 1, a + nx + 2, a, a + nx + 2, a + nx + 1], axis=1).reshape(-1, 3)
    return np.stack([gx.ravel(), gy.ravel()], axis=1), tris.astype(np.int32)


def _scene(mesh, nx, ny, model, E, t, dt, rng, nu=0.3, radius=0.5, load=0.0, rho=1000.0):
    """A mesh with its material, constraints and a moving state: a smooth displacement from rest and a smooth
    velocity field drawn from rng, both zero at the constraints."""
    V = (nx + 1) * (ny + 1)
    width = radius * math.pi / 2 if mesh == "cylinder" else ny / nx
    if mesh == "strip":   # the cantilever strip: 10 x 1, two node columns held, end load
        xy, tris = _grid(nx, ny, 10.0, 1.0)
    else:
        xy, tris = _grid(nx, ny, 1.0, width)
    u, w = xy[:, 0] / xy[:, 0].max(), xy[:, 1] / xy[:, 1].max()
    if mesh == "jitter":
        d = rng.uniform(-0.2 / nx, 0.2 / nx, xy.shape)
        inner = (u > 0) & (u < 1) & (w > 0) & (w < 1)
        xy = np.where(inner[:, None], xy + d, xy)
    idx = np.arange(V).reshape(ny + 1, nx + 1)
    sides = [idx[:, 0]]
    weight = u
    normal = np.tile([0.0, 0.0, 1.0], (V, 1))
    rest = np.concatenate([xy, np.zeros((V, 1))], axis=1)
    start = rest
    if mesh == "cylinder":
        phi = (xy[:, 1] - 0.5 * width) / radius
        start = np.stack([xy[:, 0], radius * np.sin(phi), radius * np.cos(phi)], axis=1)
        normal = np.stack([np.zeros(V), np.sin(phi), np.cos(phi)], axis=1)
        rest = start if model[1] == "S" else rest
        sides = [idx[0], idx[-1]]
        weight = np.sin(np.pi * w)
    clamped = np.concatenate([np.stack([s[:-1], s[1:]], axis=1) for s in sides]).astype(np.int32)
    pinned = np.zeros(V, np.uint8)
    pinned[clamped.ravel()] = 1
    if mesh == "strip":
        pinned[idx[:, :2].ravel()] = 1
        clamped = clamped[:0]

    def field():
        return weight * sum(rng.normal() * np.sin((k + 0.5) * np.pi * u + rng.uniform(0, 6)) *
                            np.cos(k * np.pi * w + rng.uniform(0, 6)) / (k + 1) for k in range(3))
    moving = mesh != "strip"
    x0 = start + (1e-3 * field())[:, None] * normal * moving
    v0 = ((0.2 * field())[:, None] * normal + 0.02 * np.stack([field(), field(), field()], axis=1)) * moving
    lv, lf = np.zeros(0, np.int32), np.zeros((0, 3))
    if load:
        lv = idx[:, -1].astype(np.int32)
        share = np.full(ny + 1, 1.0 / (ny + 1))
        lf = np.stack([0 * share, 0 * share, load * share], axis=1)
    return {"tris": tris, "rest": np.ascontiguousarray(rest), "model": model, "E": E, "nu": nu, "t": t, "rho": rho, "dt": dt,
            "x0": np.ascontiguousarray(x0), "v0": np.ascontiguousarray(v0), "pinned": pinned, "clamped": clamped,
            "gravity": (0.0, 0.0, 0.0 if load else -9.81), "lv": lv, "lf": lf}


def _scene_of(case, seed):
    rng = np.random.default_rng([int(seed), 7])
    E = case["E"] * math.exp(rng.uniform(-0.1, 0.1))   # another seed: another material too
    load = case.get("load", 0.0) * math.exp(rng.uniform(-0.05, 0.05))
    strip = {"nu": 0.1, "rho": 1.0, "load": load} if case["mesh"] == "strip" else {}
    return _scene(case["mesh"], case["nx"], case["ny"], case["model"], E, case["t"], case["dt"], rng, **strip)


def _scenes_of(case, seed):
    """The instances of a batch: sizes and models are the case's own, states and materials the seed's."""
    size = np.random.default_rng([case["instances"], case["lo"], case["hi"]])
    rng = np.random.default_rng([int(seed), 11])
    out = []
    for k in range(case["instances"]):
        side = int(round(math.exp(size.uniform(math.log(case["lo"]), math.log(case["hi"])))))
        curved, model, radius = size.uniform() < 0.5, MODELS[int(size.integers(0, 6))], float(size.uniform(0.3, 2.0))
        E, nu = float(math.exp(rng.uniform(math.log(1e5), math.log(1e8)))), float(rng.uniform(0.2, 0.45))
        mesh = case["mesh"] if case["mesh"] != "mixed" else ("cylinder" if curved else "plate")
        out.append(_scene(mesh, side, side, model, E, 1e-3, case["dt"], rng, nu=nu, radius=radius))
    return out


def _create(sc, precision, refine_rtol=0.0):
    torch.cuda.set_device(0)   # the current device is per thread
    return gb.shell_create(sc["tris"], sc["rest"], sc["model"], sc["E"], sc["nu"], sc["t"], sc["rho"], init_xyz=sc["x0"],
                           init_vel=sc["v0"], pinned=sc["pinned"], clamped_edges=sc["clamped"],
                           gravity=sc["gravity"], load_vtx=sc["lv"], load_f=sc["lf"], dt=sc["dt"],
                           precision=precision, refine_rtol=refine_rtol)


# ------------------------------------------------------------------------------------------------ one pass
def prepare(case, seed):
    if case["kind"] == "batch":
        scenes = _scenes_of(case, seed)
        batch = gb.shell_batch_create(120 << 30)
        if case["ctas"]:
            gb.shell_batch_set_launch(batch, case["ctas"], case["share"])
        with concurrent.futures.ThreadPoolExecutor(8) as pool:   # set-up on the host's cores, as a server does
            for h in pool.map(lambda sc: _create(sc, case["precision"]), scenes):
                gb.shell_batch_admit(batch, h)
                del h
        rows = sum(len(sc["rest"]) for sc in scenes)
        s = {"case": case, "batch": batch}
        for k, src in (("x_in", "x0"), ("v_in", "v0"), ("x_out", None), ("v_out", None)):
            s[k] = torch.empty((rows, 3), dtype=torch.float64, pin_memory=True)
            if src:
                s[k].copy_(torch.from_numpy(np.concatenate([sc[src] for sc in scenes])))
        s["x32"], s["v32"] = torch.empty((rows, 3)), torch.empty((rows, 3))
        return s
    sc = _scene_of(case, seed)
    s = {"case": case, "h": _create(sc, case["precision"], case.get("refine_rtol", 0.0)), "sc": sc}
    if case.get("chord"):
        gb.shell_set_nonlinear(s["h"], case["chord"], 0.0)
    s["x_in"], s["v_in"] = torch.from_numpy(sc["x0"]).cuda(), torch.from_numpy(sc["v0"]).cuda()
    s["x_out"], s["v_out"] = torch.empty_like(s["x_in"]), torch.empty_like(s["v_in"])
    return s


def run(s):
    c = s["case"]
    if c["kind"] == "batch":
        gb.shell_batch_step_states(s["batch"], c["steps"], s["x_in"].numpy(), s["v_in"].numpy(), s["x_out"].numpy(),
                                   s["v_out"].numpy())
        if c["precision"] == "fp64":
            return {"x": s["x_out"], "v": s["v_out"]}
        return {"x": s["x32"].copy_(s["x_out"]), "v": s["v32"].copy_(s["v_out"])}
    gb.shell_set_state_device(s["h"], s["x_in"], s["v_in"])
    if c["kind"] == "eval":
        return {"forces": gb.shell_forces(s["h"]), "energy": gb.shell_energy(s["h"])}
    if c["kind"] == "static":
        gb.shell_solve_static(s["h"], c["eps_f"], 0.1)
        gb.shell_get_state_device(s["h"], s["x_out"])
        return {"x": s["x_out"]}
    gb.shell_step(s["h"], c["steps"])
    gb.shell_get_state_device(s["h"], s["x_out"], s["v_out"])
    if c["precision"] == "fp64":
        return {"x": s["x_out"], "v": s["v_out"]}
    return {"x": s["x_out"].float(), "v": s["v_out"].float()}


def _rows(case):
    """(vertices, model) of each instance."""
    if case["kind"] != "batch":
        return [((case["nx"] + 1) * (case["ny"] + 1), case["model"])]
    return [(len(sc["rest"]), sc["model"]) for sc in _scenes_of(case, 0)]


def work(case):
    """Per step: the state in and out, external forces and masses (FP64), every stencil operator once and the
    constant matrix once, with one product of it (a regular grid has 2 triangles and 3 edges per vertex, 13
    matrix entries per row of the edge hinge and 19 of the triangle-centred models)."""
    wide = 8 if case["precision"] == "fp64" else 4
    reps = {"step": case.get("steps", 1) * max(1, case.get("chord", 0)), "batch": case.get("steps", 1)}.get(case["kind"], 1)
    nbytes = flops = 0.0
    for V, m in _rows(case):
        if m[0] == "E":
            stencils, nnz, force = 2 * (12 + 24 + 4 * wide) + 3 * (17 + 6 * wide), 13, 2 * 200 + 3 * 150
        else:
            stencils, nnz, force = 2 * (25 + 24 + 31 * wide), 19, 2 * 500
        matrix = 0 if case["kind"] == "eval" else nnz * (wide + 2)
        nbytes += reps * V * (96 + 32 + stencils + matrix)
        flops += reps * V * (force + (0 if case["kind"] == "eval" else 6 * nnz + 60))
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------------ in 64 bits
FREE, CLAMPED = 1, 2


def _stencils(sc):
    """Vertex indices (virtual nodes -1) and boundary codes of the model's stencils: [S,4] / [S,6], [S,3]."""
    tris, V = sc["tris"].astype(np.int64), len(sc["rest"])
    p, q, r = (np.concatenate([tris[:, k], tris[:, (k + 1) % 3], tris[:, (k + 2) % 3]]) for k in range(3))
    key, twin = p * V + q, q * V + p
    order = np.argsort(key)
    at = np.minimum(np.searchsorted(key[order], twin), len(key) - 1)
    inner = key[order][at] == twin
    across = np.where(inner, r[order][at], -1)
    cl = np.concatenate([sc["clamped"], sc["clamped"][:, ::-1]]).astype(np.int64)
    code = np.where(inner, 0, np.where(np.isin(key, cl[:, 0] * V + cl[:, 1]), CLAMPED, FREE))
    if sc["model"][0] == "E":
        keep = (inner & (p < q)) | (code == CLAMPED)
        return np.stack([r, p, q, across], axis=1)[keep], code[keep]
    # triangle stencils, rotated so that the first free edge (12, 23, 31) becomes edge 12
    nb, cd = across.reshape(3, -1).T, code.reshape(3, -1).T
    rot = (np.argmax(cd == FREE, axis=1)[:, None] + np.arange(3)) % 3
    v, nb, cd = (np.take_along_axis(a, rot, 1) for a in (tris, nb, cd))
    turn = [1, 2, 0]   # neighbour i lies across the edge opposite vertex i
    return np.concatenate([v, nb[:, turn]], axis=1), cd[:, turn]


def _height(x, a, b):
    e = b - a
    s = ((x - a) * e).sum(-1) / (e * e).sum(-1)
    return (x - a - s[:, None] * e).norm(dim=-1), s


def _unit(a):
    return a / a.norm(dim=-1, keepdim=True)


def _tri_normal(a, b, c):
    return torch.linalg.cross(b - a, c - a)


class _Exact:
    """The constant system and the energy of one simulation."""

    def __init__(self, sc):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        f = lambda a: torch.as_tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.sc, self.X, self.dt = sc, f(sc["rest"]), sc["dt"]
        self.tris = torch.as_tensor(sc["tris"].astype(np.int64), device=dev)
        E, nu, t = sc["E"], sc["nu"], sc["t"]
        kb = E * t ** 3 / (12 * (1 - nu * nu))
        idx, code = _stencils(sc)
        self.idx, code = torch.as_tensor(idx, device=dev), torch.as_tensor(code, device=dev)
        self.edge = sc["model"][0] == "E"
        (self._edges if self.edge else self._triangles)(code, kb, nu)
        # membrane: constant-strain triangles, rest edges in their own plane
        a, b, c = (self.X[self.tris[:, k]] for k in range(3))
        n = _tri_normal(a, b, c)
        self.At = 0.5 * n.norm(dim=-1) * t
        ex = _unit(b - a)
        ey = torch.linalg.cross(_unit(n), ex)
        self.Di = torch.linalg.inv(torch.stack([torch.stack([(ex * (b - a)).sum(-1), (ex * (c - a)).sum(-1)], -1),
                                                torch.stack([(ey * (b - a)).sum(-1), (ey * (c - a)).sum(-1)], -1)], -2))
        self.mu, self.lam = E / (2 * (1 + nu)), E * nu / (1 - nu * nu)
        V = len(self.X)
        self.mass = torch.zeros(V, dtype=torch.float64, device=dev).index_add_(
            0, self.tris.reshape(-1), (self.At * sc["rho"] / 3).repeat_interleave(3))
        self.free = f(1.0 - sc["pinned"])[:, None]
        self.fext = self.mass[:, None] * f(sc["gravity"])
        if len(sc["lv"]):
            self.fext.index_add_(0, torch.as_tensor(sc["lv"].astype(np.int64), device=dev), f(sc["lf"]))

    def _gather(self, x):
        xs = x[self.idx.clamp(min=0)]
        return xs - xs[:, (1 if self.edge else 0), None]   # relative to the frame's origin

    def _edges(self, code, kb, nu):
        X = self.X[self.idx.clamp(min=0)]
        cl = code == CLAMPED
        virt = X[:, 1] + X[:, 2] - X[:, 0]
        x1, x2, x3, x4 = X[:, 0], X[:, 1], X[:, 2], torch.where(cl[:, None], virt, X[:, 3])
        (h1, s), (h4, q) = _height(x1, x2, x3), _height(x4, x2, x3)
        L = torch.stack([1 / h1, -((1 - s) / h1 + (1 - q) / h4), -(s / h1 + q / h4), 1 / h4], 1) * (2 / (h1 + h4))[:, None]
        L[:, 0] = torch.where(cl, L[:, 0] + L[:, 3], L[:, 0])
        L[:, 3] = torch.where(cl, torch.zeros_like(h1), L[:, 3])
        A1, A2 = (0.5 * _tri_normal(*v).norm(dim=-1) for v in ((x1, x2, x3), (x4, x3, x2)))
        self.L = L[:, None]
        self.W = (kb * torch.where(cl, A1, A1 + A2))[:, None, None]
        self._rest(cl, _unit(_tri_normal(x1, x2, x3)))

    def _triangles(self, code, kb, nu):
        X = self.X[self.idx.clamp(min=0)]
        hinge = ((1, 2), (2, 0), (0, 1))
        X = X.clone()
        for i, (a, b) in enumerate(hinge):
            X[:, 3 + i] = torch.where((code[:, i] > 0)[:, None], X[:, a] + X[:, b] - X[:, i], X[:, 3 + i])
        L = X.new_zeros((len(X), 3, 6))
        for i, (a, b) in enumerate(hinge):
            (h, s), (g, q) = _height(X[:, i], X[:, a], X[:, b]), _height(X[:, 3 + i], X[:, a], X[:, b])
            k = 2 / (h + g)
            L[:, i, i], L[:, i, 3 + i] = k / h, k / g
            L[:, i, a], L[:, i, b] = -k * ((1 - s) / h + (1 - q) / g), -k * (s / h + q / g)
        n = _tri_normal(X[:, 0], X[:, 1], X[:, 2])
        ex = _unit(X[:, 1] - X[:, 0])
        ey = torch.linalg.cross(_unit(n), ex)
        P = torch.stack([((X - X[:, :1]) * e[:, None]).sum(-1) for e in (ex, ey)], -1)
        D = kb * X.new_tensor([[1, nu, 0], [nu, 1, 0], [0, 0, 0.5 * (1 - nu)]])
        if self.sc["model"][0] == "F":
            R = X.new_zeros((len(X), 3, 3))
            for i, (a, b) in enumerate(hinge):
                m = _unit(P[:, b] - P[:, a])
                R[:, 0, i], R[:, 1, i], R[:, 2, i] = m[:, 1] ** 2, m[:, 0] ** 2, -2 * m[:, 0] * m[:, 1]
            R[:, 2] *= ~(code == FREE).any(1)[:, None]
            D = R.transpose(1, 2) @ D @ R
        else:
            C = torch.stack([0.5 * P[..., 0] ** 2, 0.5 * P[..., 1] ** 2, 0.5 * P[..., 0] * P[..., 1]], -1)
            L = torch.linalg.solve(L @ C, L)
        for i, (a, b) in enumerate(hinge):
            c = L[:, :, 3 + i].clone()
            cl, fr = (code[:, i] == CLAMPED)[:, None], (code[:, i] == FREE)[:, None]
            L[:, :, i] += c * cl - c * fr
            L[:, :, a] += c * fr
            L[:, :, b] += c * fr
            L[:, :, 3 + i] *= ~(cl | fr)
        self.L, self.W = L, 0.5 * n.norm(dim=-1)[:, None, None] * D
        self._rest((code == CLAMPED).any(1), _unit(n))

    def _rest(self, clamped, n0):
        """Rest curvatures and the fixed normals of the stencils at clamped edges."""
        self.cl, self.n0 = clamped[:, None], n0
        d = self._gather(self.X)
        n = n0
        if self.edge and self.sc["model"][1] == "S":
            n = torch.where(self.cl, n0, self._normal(d))
        k0 = torch.einsum("srk,skc,sc->sr", self.L, d, n)
        self.k0 = k0 if self.sc["model"][1] == "S" else torch.where(self.cl, k0, torch.zeros_like(k0))

    def _normal(self, d):
        if not self.edge:
            return _unit(_tri_normal(d[:, 0], d[:, 1], d[:, 2]))
        n1 = _unit(_tri_normal(d[:, 0], d[:, 1], d[:, 2]))
        n2 = _unit(_tri_normal(torch.where(self.cl, d[:, 1] + d[:, 2] - d[:, 0], d[:, 3]), d[:, 2], d[:, 1]))
        return _unit(n1 + n2)

    def energies(self, x):
        """(membrane, bending)."""
        a, b, c = (x[self.tris[:, k]] for k in range(3))
        F = torch.stack([b - a, c - a], -1) @ self.Di
        C = F.transpose(1, 2) @ F
        # the stretch S = sqrt(C) of a 2 x 2 matrix: (C + sqrt(det C) I) / tr S, tr S = sqrt(tr C + 2 sqrt(det C));
        # S - I = (C - I) (S + I)^-1 keeps its digits at small strains
        I2 = torch.eye(2, dtype=x.dtype, device=x.device)
        J = torch.sqrt(C[:, 0, 0] * C[:, 1, 1] - C[:, 0, 1] * C[:, 1, 0])
        ts = torch.sqrt(C[:, 0, 0] + C[:, 1, 1] + 2 * J)
        e = (C - I2) @ torch.linalg.inv((C + J[:, None, None] * I2) / ts[:, None, None] + I2)
        tr = e[:, 0, 0] + e[:, 1, 1]
        memb = (self.At * (self.mu * (e * e).sum((1, 2)) + 0.5 * self.lam * tr ** 2)).sum()
        d = self._gather(x)
        G = torch.einsum("srk,skc->src", self.L, d)
        if self.sc["model"][1] == "S":
            eps = torch.einsum("src,sc->sr", G, torch.where(self.cl, self.n0, self._normal(d))) - self.k0
            return memb, 0.5 * torch.einsum("sr,srq,sq->", eps, self.W, eps)
        eps = torch.where(self.cl, torch.einsum("src,sc->sr", G, self.n0) - self.k0, torch.zeros_like(self.k0))
        flat = torch.where(self.cl[..., None], torch.zeros_like(G), G)
        return memb, 0.5 * (torch.einsum("sr,srq,sq->", eps, self.W, eps) + torch.einsum("src,srq,sqc->", flat, self.W, flat))

    def forces(self, x):
        x = x.detach().clone().requires_grad_(True)
        memb, bend = self.energies(x)
        return -torch.autograd.grad(memb + bend, x)[0]

    def matrix(self):
        """M + dt^2 K with identity rows and columns at pinned vertices."""
        V = len(self.X)
        K = torch.einsum("sik,sil,slm->skm", self.L, self.W, self.L)
        G = torch.stack([-self.Di[:, 0] - self.Di[:, 1], self.Di[:, 0], self.Di[:, 1]], 1)
        Km = (2 * (self.mu + self.lam) * self.At)[:, None, None] * (G @ G.transpose(1, 2))
        rows, cols, vals = [], [], []
        for blk, ix in ((K, self.idx), (Km, self.tris)):
            k = ix.shape[1]
            i, j = ix[:, :, None].expand(-1, k, k), ix[:, None, :].expand(-1, k, k)
            keep = (i >= 0) & (j >= 0)
            rows, cols, vals = rows + [i[keep]], cols + [j[keep]], vals + [self.dt ** 2 * blk[keep]]
        d = torch.arange(V, device=self.X.device)
        free = self.free[:, 0]
        i, j = torch.cat(rows + [d]), torch.cat(cols + [d])
        val = torch.cat(vals + [self.mass]) * free[i] * free[j]
        i, j, val = torch.cat([i, d]), torch.cat([j, d]), torch.cat([val, 1 - free])
        return torch.sparse_coo_tensor(torch.stack([i, j]), val, (V, V)).coalesce()

    def solver(self):
        A = self.matrix()
        if len(self.X) <= 6000:
            chol = torch.linalg.cholesky(A.to_dense())
            return lambda b: torch.cholesky_solve(b, chol)
        i = A.indices()
        di = 1 / A.values()[i[0] == i[1]][:, None]
        A = A.to_sparse_csr()

        def cg(b):   # conjugate gradients, one recurrence for the three right-hand sides
            x, r = torch.zeros_like(b), b.clone()
            z = di * r
            p, g, stop = z.clone(), (r * z).sum(), 1e-28 * float((b * b).sum())
            for it in range(40000):
                w = A @ p
                a = g / (p * w).sum().clamp(min=1e-300)
                x += a * p
                r -= a * w
                z = di * r
                h = (r * z).sum()
                p = z + (h / g.clamp(min=1e-300)) * p
                g = h
                if it % 64 == 63 and float((r * r).sum()) <= stop:
                    break
            return x
        return cg


def _advance(sc, steps, chord):
    m = _Exact(sc)
    solve = m.solver()
    x, v = (torch.as_tensor(sc[k], device=m.X.device) for k in ("x0", "v0"))
    M = m.mass[:, None]
    for _ in range(steps):
        vk = torch.zeros_like(v)
        for _ in range(max(1, chord)):
            vk = vk - solve(m.free * (M * (vk - v) - m.dt * (m.forces(x + m.dt * vk) + m.fext)))
        x, v = x + m.dt * vk, vk
    return x, v


def exact(case, seed):
    if case["kind"] == "static":
        return None
    if case["kind"] == "batch":
        scenes = _scenes_of(case, seed)
        if sum(len(sc["rest"]) for sc in scenes) > 40000:
            return None
        both = [_advance(sc, case["steps"], 0) for sc in scenes]
        return {"x": torch.cat([b[0] for b in both]), "v": torch.cat([b[1] for b in both])}
    sc = _scene_of(case, seed)
    if case["kind"] == "eval":
        m = _Exact(sc)
        x, v = (torch.as_tensor(sc[k], device=m.X.device) for k in ("x0", "v0"))
        memb, bend = m.energies(x)
        kin, ext = 0.5 * (m.mass[:, None] * v * v).sum(), -(m.fext * (x - m.X)).sum()
        return {"forces": m.forces(x), "energy": torch.stack([memb, bend, kin, ext])}
    if len(sc["rest"]) * case["steps"] * max(1, case["chord"]) > 1100000:
        return None
    x, v = _advance(sc, case["steps"], case["chord"])
    return {"x": x, "v": v}
