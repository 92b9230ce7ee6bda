"""Performance cases: what programs built on this library ask of it.

Three entry points carry a user's work and are measured here, over the sizes,
precisions and modes they are used with:

  Scene.step           one backward-Euler time step of one scene, from host
                       targets to host positions
  ppn_step_batch       the same step for many scenes advanced together
  pcg_solve_static     the linear solve alone, on a caller's device-resident system

A step starts from a given displacement and velocity, which the program restores
before it (a rollout branched from a checkpoint, a line of a parameter sweep, one
candidate of a control search), so every pass does the same work.
"""

import numpy as np
import torch

import paper_2505_21013_gb300 as P
from ppn_inputs import cube_scene, kuhn_grid, press_scene, random_batch_scenes, twisting_beam_scene

MODES = {"ppn": P.MODE_PPN, "pn": P.MODE_PN, "newton": P.MODE_NEWTON, "pdn": P.MODE_PDN}


def listed():
    return [
        # an interactive toy body, the smallest parity scene: latency and launches decide
        {"name": "cube5_fp64", "kind": "cube", "n": 5, "precision": "fp64", "mode": "ppn", "tol": 1e-6},
        # a small body in a game-like loop, mixed precision
        {"name": "beam6_mixed", "kind": "beam", "nx": 6, "ny": 6, "nz": 21, "omega": 2.0, "E": 1e6,
         "precision": "mixed", "mode": "ppn", "tol": 1e-4},
        # the scene of the threshold sweep: violent, so that elements are projected
        {"name": "violent10_mixed", "kind": "beam", "nx": 10, "ny": 10, "nz": 40, "omega": 20.0, "E": 1e5,
         "precision": "mixed", "mode": "ppn", "tol": 1e-4},
        # the reference-accuracy path at an ordinary size
        {"name": "beam12_fp64", "kind": "beam", "nx": 12, "ny": 12, "nz": 45, "omega": 2.0, "E": 1e6,
         "precision": "fp64", "mode": "ppn", "tol": 1e-6},
        # the headline workload, and the projected-Newton baseline on it
        {"name": "beam20_mixed", "kind": "beam", "nx": 20, "ny": 20, "nz": 80, "omega": 2.0, "E": 1e6,
         "precision": "mixed", "mode": "ppn", "tol": 1e-4},
        {"name": "beam20_mixed_pn", "kind": "beam", "nx": 20, "ny": 20, "nz": 80, "omega": 2.0, "E": 1e6,
         "precision": "mixed", "mode": "pn", "tol": 1e-4},
        # the headline mesh turned violently: selection, projection and retries
        {"name": "violent20_mixed", "kind": "beam", "nx": 20, "ny": 20, "nz": 80, "omega": 20.0, "E": 1e5,
         "precision": "mixed", "mode": "ppn", "tol": 1e-4},
        # many independent scenes of mixed sizes per launch (data generation, serving)
        {"name": "batch64_mixed", "kind": "batch", "scenes": 64, "set": 0, "tmin": 1e3, "tmax": 5e4,
         "precision": "mixed", "mode": "ppn", "tol": 1e-4},
        # the largest scene: contact with moving obstacles, a matrix larger than L2
        {"name": "press4x40_mixed", "kind": "press", "boxes": 4, "n": 40, "precision": "mixed", "mode": "ppn",
         "tol": 1e-4},
        # the allocation-free solve: a few row tiles, and the headline mesh's size
        {"name": "solve_7x6x13", "kind": "solve", "nx": 7, "ny": 6, "nz": 13, "rel_tol": 1e-4},
        {"name": "solve_20x20x80", "kind": "solve", "nx": 20, "ny": 20, "nz": 80, "rel_tol": 1e-4},
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["beam", "beam", "beam", "cube", "batch", "press", "solve", "solve"])
    if kind == "solve":
        n = _log_int(rng, 60, 60000)
        nx = max(2, int(round((n / 4.0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.3))))
        ny = max(2, int(round((n / 4.0) ** (1.0 / 3.0) * rng.uniform(0.7, 1.3))))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": max(2, min(n, 65536) // (nx * ny)), "rel_tol": 1e-4}
    if kind == "batch":
        return {"kind": kind, "scenes": _log_int(rng, 3, 60), "set": rng.randrange(1, 1000), "tmin": 1e3, "tmax": float(_log_int(rng, 4000, 50000)),
                "precision": "mixed", "mode": rng.choice(["ppn", "ppn", "pn"]), "tol": 1e-4}
    if kind == "press":
        return {"kind": kind, "boxes": rng.choice([1, 2, 4]), "n": _log_int(rng, 6, 30), "precision": "mixed",
                "mode": "ppn", "tol": 1e-4}
    fp64 = rng.random() < 0.3
    common = {"precision": "fp64" if fp64 else "mixed", "mode": rng.choice(["ppn", "ppn", "ppn", "pn", "newton", "pdn"]),
              "tol": 1e-6 if fp64 else 1e-4}
    if kind == "cube":
        return {"kind": kind, "n": _log_int(rng, 4, 16 if fp64 else 36), **common}
    c = _log_int(rng, 3, 10 if fp64 else 21)
    omega, E = rng.choice([(2.0, 1e6), (2.0, 1e6), (5.0, 1e6), (20.0, 1e5)])
    return {"kind": kind, "nx": c, "ny": max(3, c + rng.choice([-1, 0, 0, 1])), "nz": 4 * c + rng.choice([-3, 0, 1, 2]),
            "omega": omega, "E": E, **common}


# ------------------------------------------------------------------ scenes

STEPS_BEFORE = 3  # the twist is this many time steps old when a pass starts


def _spec(case, seed):
    if case["kind"] == "cube":
        return cube_scene(case["n"], seed=seed)
    if case["kind"] == "press":
        return press_scene(n=case["n"], boxes=case["boxes"], seed=seed)
    return twisting_beam_scene(case["nx"], case["ny"], case["nz"], h=0.01, E=case["E"], nu=0.45, omega=case["omega"],
                               dt=1.0 / 30.0, seed=seed)


def _batch(case):
    return random_batch_scenes(case["scenes"], case["tmin"], case["tmax"], seed=case["set"])


def _start(spec, seed):
    """Displacement and velocity before the step."""
    X = spec.rest
    rng = np.random.default_rng(seed)
    if spec.meta["kind"] == "beam":  # twisted linearly along its axis by the turns done so far, still turning
        nx, ny, nz = spec.meta["dims"]
        h, omega = spec.meta["h"], spec.meta["omega"]
        s = (X[:, 2] / ((nz - 1) * h))
        c = np.array([0.5 * (nx - 1) * h, 0.5 * (ny - 1) * h])
        ang = omega * spec.dt * STEPS_BEFORE * s
        px, py = X[:, 0] - c[0], X[:, 1] - c[1]
        qx, qy = np.cos(ang) * px - np.sin(ang) * py, np.sin(ang) * px + np.cos(ang) * py
        u = np.stack([qx - px, qy - py, np.zeros_like(px)], axis=1)
        rate = omega * rng.uniform(0.95, 1.0) * s
        v = np.stack([-rate * qy, rate * qx, np.zeros_like(px)], axis=1)
        return u, v
    v = np.zeros_like(X)
    if spec.meta["kind"] == "cube":  # swaying: a shear growing with the height above the fixed face
        v[:, 0] = rng.uniform(0.2, 0.6) * X[:, 1]
        v[:, 2] = rng.uniform(-0.4, 0.4) * X[:, 1]
    else:  # the boxes settle from slightly different speeds
        v[:, 1] = -rng.uniform(0.0, 0.02)
    return np.zeros_like(X), v


class _Stepping:
    """A scene with the state it starts from, and what the step is given."""

    def __init__(self, spec, seed, precision):
        self.scene = P.Scene.from_spec(spec, precision=precision)
        self.u, self.v = _start(spec, seed)
        self.targets = spec.targets_at(STEPS_BEFORE)
        self.obstacles = spec.obstacles_at(0)
        if self.obstacles:
            self.scene.set_obstacles(spec.obstacles_at(-1))

    def load(self):
        self.scene.set_displacement(self.u, self.v)
        if len(self.targets):
            self.scene.set_targets(self.targets)
        if self.obstacles:
            self.scene.set_obstacles(self.obstacles)


# ------------------------------------------------------------------ linear systems

def _system(case, seed):
    """Springs and lumped masses on a tet grid's edges (SPD), and a load: row_ptr, col, 3x3 blocks, b."""
    h, dt = 0.01, 1.0 / 60.0
    X, tets = kuhn_grid(case["nx"], case["ny"], case["nz"], h, jitter=0.01, seed=seed)
    n = len(X)
    rng = np.random.default_rng([seed, 11])
    pairs = np.concatenate([tets[:, [a, b]] for a in range(4) for b in range(a + 1, 4)]).astype(np.int64)
    pairs.sort(axis=1)
    key = np.unique(pairs[:, 0] * n + pairs[:, 1])
    i, j = key // n, key % n
    d = X[j] - X[i]
    d /= np.linalg.norm(d, axis=1)[:, None]
    k = 1e5 * h * np.exp(rng.uniform(-1.0, 1.0, len(key)))
    K = k[:, None, None] * (d[:, :, None] * d[:, None, :] + 0.05 * np.eye(3))
    D = np.zeros((n, 3, 3))
    D[:] = 1000.0 * h**3 / dt**2 * np.eye(3)
    for c in range(9):
        D[:, c // 3, c % 3] += np.bincount(i, K[:, c // 3, c % 3], n) + np.bincount(j, K[:, c // 3, c % 3], n)
    row = np.concatenate([i, j, np.arange(n)])
    col = np.concatenate([j, i, np.arange(n)])
    order = np.argsort(row * n + col, kind="stable")
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=n))])
    b = 1000.0 * h**3 * (np.array([0.0, -9.81, 0.0]) + 5.0 * rng.standard_normal((n, 3)))
    return (row_ptr.astype(np.int32), col[order].astype(np.int32),
            np.concatenate([-K, -K, D])[order].astype(np.float32), b.astype(np.float32))


# ------------------------------------------------------------------ the contract

def prepare(case, seed):
    if case["kind"] == "solve":
        rp, col, val, b = _system(case, seed)
        n, nnzb = len(rp) - 1, len(col)
        comp = np.ascontiguousarray(val.reshape(nnzb, 9).T)  # component-major
        b4 = np.zeros((n, 4), np.float32)
        b4[:, :3] = b
        dev = torch.device("cuda", 0)
        return {"case": case, "n": n, "nnzb": nnzb, "row_ptr": torch.from_numpy(rp).to(dev),
                "col": torch.from_numpy(col).to(dev), "val": torch.from_numpy(comp).to(dev),
                "b": torch.from_numpy(b4).to(dev), "x": torch.zeros((n, 4), dtype=torch.float32, device=dev)}
    prec = P.PREC_FP64 if case["precision"] == "fp64" else P.PREC_MIXED
    if case["kind"] == "batch":
        specs = _batch(case)
    else:
        specs = [_spec(case, seed)]
    steps = [_Stepping(s, [seed, k], prec) for k, s in enumerate(specs)]
    return {"case": case, "steps": steps, "out": None if case["kind"] == "batch" else np.zeros_like(specs[0].rest)}


def run(state):
    case = state["case"]
    if case["kind"] == "solve":
        s = state
        info = P.ppn.pcg_solve_static(s["row_ptr"].data_ptr(), s["col"].data_ptr(), s["val"].data_ptr(), s["n"],
                                      s["nnzb"], s["b"].data_ptr(), s["x"].data_ptr(), rel_tol=case["rel_tol"])
        return {"x": s["x"][:, :3], "iters": info["iters"], "ind": info["ind"]}
    mode = MODES[case["mode"]]
    for s in state["steps"]:
        s.load()
    if case["kind"] == "batch":
        scenes = [s.scene for s in state["steps"]]
        P.ppn_step_batch(scenes, [mode] * len(scenes), case["tol"])
        return {"x": np.concatenate([s.get_state()[0] for s in scenes])}
    _, x, _ = state["steps"][0].scene.step(mode, case["tol"], out=state["out"])
    return {"x": x}


def _counts(case):
    """(vertices, tets, BSR blocks) of a case's scenes, from the grid sizes alone."""
    def grid(nx, ny, nz):
        cells = (nx - 1) * (ny - 1) * (nz - 1)
        # edges of the Kuhn split: along the axes, the face diagonals and the cell diagonal
        e = ((nx - 1) * ny * nz + nx * (ny - 1) * nz + nx * ny * (nz - 1) + (nx - 1) * (ny - 1) * nz
             + (nx - 1) * ny * (nz - 1) + nx * (ny - 1) * (nz - 1) + cells)
        return np.array([nx * ny * nz, 6 * cells, nx * ny * nz + 2 * e], dtype=np.float64)

    if case["kind"] == "cube":
        return grid(case["n"], case["n"], case["n"])
    if case["kind"] == "press":
        return case["boxes"] * grid(case["n"], case["n"], case["n"])
    if case["kind"] == "batch":
        return sum(grid(*s.meta["dims"]) for s in _batch(case))
    return grid(case["nx"], case["ny"], case["nz"])


def work(case):
    """One pass: a solve reads its matrix and load and writes its solution once; a time step does so for at
    least two Newton iterations, each with one evaluation of the elements and one linear solve, whose matrix
    it also has to form.  The iterations inside a solve are the method's and not counted."""
    nv, nt, nb = _counts(case)
    if case["kind"] == "solve":
        return {"bytes": nb * 40.0 + nv * 36.0, "flops": nb * 18.0}
    w = 8.0 if case["precision"] == "fp64" else 4.0
    per_newton = nt * (16.0 + 12 * w) + nb * (9 * w + 4.0) * 2 + nv * (24.0 * 4 + 12 * w)
    return {"bytes": 2 * per_newton + nv * 24.0 * 4, "flops": 2 * (nt * 2000.0 + nb * 18.0)}


# ------------------------------------------------------------------ 64-bit values

def _exact_solve(case, seed):
    """The solution in 64 bits: CG on the same (FP32-valued) system to 1e-13."""
    rp, col, val, b = _system(case, seed)
    n = len(rp) - 1
    dev = torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")
    row = np.repeat(np.arange(n), np.diff(rp))
    k = np.arange(3)
    r3 = np.broadcast_to((3 * row)[:, None, None] + k[None, :, None], val.shape).reshape(-1)
    c3 = np.broadcast_to((3 * col.astype(np.int64))[:, None, None] + k[None, None, :], val.shape).reshape(-1)
    A = torch.sparse_coo_tensor(torch.from_numpy(np.stack([r3, c3])), torch.from_numpy(val.astype(np.float64).reshape(-1)),
                                (3 * n, 3 * n)).coalesce().to_sparse_csr().to(dev)
    diag = torch.from_numpy(np.concatenate([val[rp[i] + np.searchsorted(col[rp[i]:rp[i + 1]], i)].diagonal()
                                            for i in range(n)]).astype(np.float64)).to(dev)
    f = torch.from_numpy(b.astype(np.float64).reshape(-1)).to(dev)
    x = torch.zeros_like(f)
    r = f.clone()
    z = r / diag
    p = z.clone()
    rz = torch.dot(r, z)
    for _ in range(20000):
        q = A @ p
        a = rz / torch.dot(p, q)
        x += a * p
        r -= a * q
        if float(r.norm()) <= 1e-13 * float(f.norm()):
            break
        z = r / diag
        rz, old = torch.dot(r, z), rz
        p = z + (rz / old) * p
    return {"x": x.reshape(n, 3).cpu(), "iters": None, "ind": None}


def _exact_step(case, seed):
    """The step's minimiser in 64 bits, by Newton's method with a dense Hessian (small bodies)."""
    spec = _spec(case, seed)
    u0, v0 = _start(spec, [seed, 0])
    X = torch.from_numpy(spec.rest)
    tets = torch.from_numpy(spec.tets.astype(np.int64))
    mu = spec.E / (2 * (1 + spec.nu))
    lam = spec.E * spec.nu / ((1 + spec.nu) * (1 - 2 * spec.nu)) + mu
    Dm = (X[tets[:, 1:]] - X[tets[:, :1]]).transpose(1, 2)
    vol = torch.linalg.det(Dm).abs() / 6.0
    Di = torch.linalg.inv(Dm)
    mass = torch.zeros(len(X), dtype=torch.float64).index_add_(0, tets.reshape(-1), (spec.rho * vol / 4.0).repeat_interleave(4))
    free = torch.ones(len(X), dtype=torch.bool)
    free[torch.from_numpy(spec.fixed.astype(np.int64))] = False
    dt = spec.dt
    hat = torch.from_numpy(u0 + dt * v0) + dt * dt * torch.tensor(spec.gravity, dtype=torch.float64)
    base = torch.from_numpy(u0.copy())
    base[torch.from_numpy(spec.fixed.astype(np.int64))] = torch.from_numpy(spec.targets_at(STEPS_BEFORE) - spec.rest[spec.fixed])

    def energy(y):
        u = base.clone()
        u[free] = y.reshape(-1, 3)
        H = (u[tets[:, 1:]] - u[tets[:, :1]]).transpose(1, 2) @ Di
        F = H + torch.eye(3, dtype=torch.float64)
        Jm1 = torch.linalg.det(F) - 1.0
        psi = 0.5 * mu * ((F * F).sum((1, 2)) - 3.0) - mu * Jm1 + 0.5 * lam * Jm1 * Jm1
        return (vol * psi).sum() + (0.5 / dt**2 * mass[free, None] * (u - hat)[free] ** 2).sum()

    y = base[free].reshape(-1).clone()
    for _ in range(12):
        g = torch.autograd.functional.jacobian(energy, y)
        Hs = torch.autograd.functional.hessian(energy, y, vectorize=True)
        dy = torch.linalg.solve(Hs, -g)
        t, e0 = 1.0, energy(y)
        while t > 1e-6 and not energy(y + t * dy) <= e0 + 1e-12 * e0.abs():
            t *= 0.5
        y = y + t * dy
        if float(dy.abs().max()) < 1e-14:
            break
    u = base.clone()
    u[free] = y.reshape(-1, 3)
    return {"x": (X + u).numpy()}


def exact(case, seed):
    if case["kind"] == "solve":
        return _exact_solve(case, seed)
    if case["kind"] == "cube" and case["n"] <= 6:
        return _exact_step(case, seed)
    return None  # a step of a larger scene: minutes in plain numpy
