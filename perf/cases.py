"""The workloads whose speed is measured: whole time steps through lfx.State (history in, step,
solution out, as a coupled or logged simulation drives it), a batch of meshes stepped as one system,
and the allocation-free preconditioner on device matrices.

A case is a dict of plain values.  Fields: flow (cavity, pipe, box, stenosis, moving, batch, precond),
n and nz (hexahedra across and along, each cut into six tetrahedra), order (BDF), precision, implicit,
stab and diffusion (indices of lfx_options), members (batch), riis, bf16 (storage of the mixed path's smoother).  Meshes are jittered, shuffled
Kuhn-split lattices: 5.6 to 6 tetrahedra and about 15 matrix blocks per node, as in the tetrahedral
meshes of the paper (Table tab:mesh).  The mesh belongs to the case; the flow fields, the time level
and the loads come from the seed."""
from __future__ import annotations

import ctypes
import functools
import json
import math

import numpy as np
import torch

from paper_2304_12032_gb300 import lfx as L

RHO, MU = 1.06, 0.035          # blood in CGS units, as in the repository's vessel workloads
C_R, RADIUS = 30.0, 1.2        # constant of tau_M; radius of the inlet profile (covers the duct's corners)
RTOL = 1e-11                   # as in the repository's comparisons with its oracle; the stenosis's rounding floor is 4e-12


def listed():
    step = dict(order=2, precision="mixed", implicit=False, stab=2, diffusion=0, members=1, riis=False, bf16=True)
    return [
        # the Beltrami cube of the convergence study: 3072 tetrahedra, FP64, latency and launches count
        dict(step, name="cavity_3k_fp64", flow="cavity", n=8, nz=8, order=1, precision="fp64"),
        # the smallest vessel meshes of a batch or a serving pool
        dict(step, name="pipe_19k", flow="pipe", n=11, nz=26),
        # a coarse vessel in the default (FP64) precision
        dict(step, name="pipe_100k_fp64", flow="pipe", n=15, nz=74, precision="fp64"),
        # SUPG-PSPG, BDF3, symmetric-gradient diffusion and a body force: the bifurcation workload's options
        dict(step, name="supg_60k_bdf3_fp64", flow="pipe", n=13, nz=59, order=3, precision="fp64", stab=1, diffusion=1),
        # a mesh of the serving pool's average size, ramped uniform inflow into a box
        dict(step, name="box_500k", flow="box", n=41, nz=50),
        # the headline: a Poiseuille cylinder of a million tetrahedra, BDF2, mixed precision
        dict(step, name="pipe_1m", flow="pipe", n=32, nz=166),
        # the same kind of mesh in FP64 throughout
        dict(step, name="pipe_600k_fp64", flow="pipe", n=27, nz=137, precision="fp64"),
        # stenosis with a resistive disk and a Womersley inlet: the largest single mesh in use
        dict(step, name="stenosis_4m", flow="stenosis", n=51, nz=257, riis=True),
        # the fully implicit formulation (Newton's method)
        dict(step, name="newton_150k", flow="pipe", n=17, nz=87, implicit=True),
        # a moving vessel wall (ALE): lifting, geometry and step
        dict(step, name="moving_80k", flow="moving", n=15, nz=59),
        # independent meshes of 10k to 90k tetrahedra stepped as one system
        dict(step, name="batch_16", flow="batch", n=15, nz=31, members=16),
        # the preconditioner alone on a caller's device matrix, near the largest size it takes
        dict(step, name="precond_60k_nodes", flow="precond", n=24, nz=95, precision="fp64"),
    ]


def draw(rng):
    flow = rng.choice(["cavity", "pipe", "pipe", "pipe", "box", "stenosis", "moving", "batch", "precond"])
    c = dict(flow=flow, order=rng.choice([1, 2, 2, 3]), precision=rng.choice(["fp64", "mixed", "mixed"]), implicit=False,
             stab=2, diffusion=0, members=1, riis=flow == "stenosis", bf16=rng.random() < 0.8)
    n = int(round(math.exp(rng.uniform(math.log(7), math.log(40)))))
    aspect = rng.uniform(1.0, 5.0)
    if flow == "cavity":
        c.update(precision="fp64", n=min(n, 17))
        aspect = 1.0
    elif flow == "pipe":
        c.update(n=n if c["precision"] == "mixed" else min(n, 27), stab=rng.choice([1, 2, 2]), diffusion=rng.choice([0, 0, 1]))
        if c["stab"] == 2 and rng.random() < 0.25:
            c.update(implicit=True, n=min(n, 18))
    elif flow == "moving":
        c.update(n=min(n, 18), order=rng.choice([1, 2]))
    elif flow == "batch":
        c.update(n=min(n, 15), members=rng.randint(2, 16))
        aspect = min(aspect, 2.5)
    elif flow == "precond":
        c.update(n=min(n, 24), precision="fp64")
        aspect = min(aspect, 4.0)
    else:
        c.update(n=n if c["precision"] == "mixed" else min(n, 27))
    c["nz"] = max(5, int(aspect * c.get("n", n)) + rng.randint(0, 3))
    return c


def _sizes(case):
    """(n, nz) of each mesh of the case: one, or members whose sizes fall from the largest."""
    m = case["members"]
    return [(max(5, int(case["n"] * (1.0 - 0.5 * k / m))), max(5, case["nz"] - (k * case["nz"]) // (2 * m))) for k in range(m)]


def work(case):
    T = sum(6 * n * n * nz for n, nz in _sizes(case))
    V = sum((n + 1) ** 2 * (nz + 1) for n, nz in _sizes(case))
    blocks = 15 * V
    if case["flow"] == "precond":   # matrix (FP64 blocks, columns, transposes) and two vectors
        return {"bytes": blocks * (128 + 8) + V * (8 + 64), "flops": blocks * 2 * (5 * 9 + 12 * 7)}
    # elements, coordinates, history in, solution out; the flops of the element matrices and of one
    # product with the matrix
    return {"bytes": 16 * T + 24 * V + 32 * V * (case["order"] + 1),
            "flops": 2948 * T + 32 * blocks}


# ---------------------------------------------------------------------------------- meshes
def _lattice(n, nz, flow, rng):
    """Nodes, tetrahedra, boundary faces and tags (wall 0, inlet 1, outlet 2; cavity: sides 1 to 6)."""
    ix, iy, iz = (a.ravel() for a in np.meshgrid(np.arange(n + 1), np.arange(n + 1), np.arange(nz + 1), indexing="ij"))
    X = np.stack([2.0 * ix / n - 1.0, 2.0 * iy / n - 1.0, 2.0 * iz / n], 1)
    inner = (ix > 0) & (ix < n) & (iy > 0) & (iy < n) & (iz > 0) & (iz < nz)
    X[inner] += (2.0 / n) * 0.12 * rng.uniform(-1, 1, (int(inner.sum()), 3))
    if flow == "cavity":
        X = 0.5 * (X + np.array([1.0, 1.0, 0.0]))
    elif flow != "box":             # a duct of rounded cross-section, narrowed to half its width for the stenosis
        x, y = X[:, 0].copy(), X[:, 1].copy()
        X[:, 0], X[:, 1] = x * np.sqrt(1 - 0.4 * y * y), y * np.sqrt(1 - 0.4 * x * x)
        if flow == "stenosis":
            s = np.clip((X[:, 2] - 0.3 * X[:, 2].max()) / 1.0, -1, 1)
            X[:, :2] *= (1 - 0.25 * (1 + np.cos(np.pi * s)))[:, None]
    at = lambda a, b, c: (a * (n + 1) + b) * (nz + 1) + c  # noqa: E731
    h = [a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), np.arange(nz), indexing="ij")]
    tets = []
    for order in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        p, v = [a.copy() for a in h], []
        v.append(at(*p))
        for axis in order:
            p[axis] = p[axis] + 1
            v.append(at(*p))
        tets.append(np.stack(v, 1))
    faces, tags = [], []
    for axis, side, tag in ((0, 0, 0), (0, n, 0), (1, 0, 0), (1, n, 0), (2, 0, 1), (2, nz, 2)):
        b, c = [k for k in range(3) if k != axis]
        m = (n, n, nz)
        g = [a.ravel() for a in np.meshgrid(np.arange(m[b]), np.arange(m[c]), indexing="ij")]

        def corner(db, dc):
            q = [None] * 3
            q[axis], q[b], q[c] = np.full_like(g[0], side), g[0] + db, g[1] + dc
            return at(*q)

        for tri in ((corner(0, 0), corner(1, 0), corner(1, 1)), (corner(0, 0), corner(0, 1), corner(1, 1))):
            faces.append(np.stack(tri, 1))
            tags.append(np.full(g[0].size, len(faces) // 2 + len(faces) % 2 if flow == "cavity" else tag))
    return X, np.concatenate(tets), np.concatenate(faces), np.concatenate(tags)


@functools.lru_cache(maxsize=16)
def _mesh(key):
    """Host arrays of the case's mesh in a shuffled numbering, as a mesh generator leaves it."""
    case = json.loads(key)
    rng = np.random.default_rng(17)
    parts, off, shift = [], 0, 0.0
    for n, nz in _sizes(case):
        X, t, f, g = _lattice(n, nz, case["flow"], rng)
        X[:, 0] += shift
        parts.append((X, t + off, f + off, g))
        off, shift = off + len(X), shift + 3.0
    X, t, f, g = (np.concatenate([p[k] for p in parts]) for k in range(4))
    new = rng.permutation(len(X))
    nodes = np.empty_like(X)
    nodes[new] = X
    t = new[t][rng.permutation(len(t))]
    return dict(nodes=nodes, tets=np.ascontiguousarray(t, np.int32), faces=np.ascontiguousarray(new[f], np.int32),
                tags=np.ascontiguousarray(g, np.int32), n=case["n"], length=float(X[:, 2].max()))


def _area_vectors(m, tags, nodes=None):
    """Outward area vector of each face with a tag in tags, and their faces (for convex-sided ducts)."""
    X = m["nodes"] if nodes is None else nodes
    f = m["faces"][np.isin(m["tags"], tags)]
    a = 0.5 * np.cross(X[f[:, 1]] - X[f[:, 0]], X[f[:, 2]] - X[f[:, 0]])
    out = X[f].mean(1) - m["nodes"].mean(0)
    return f, a * np.sign((a * out).sum(1))[:, None]


# ---------------------------------------------------------------------------------- problems
_WAVES = ([94.2, -60.0, 22.0, 9.0], [0.0, 18.0, -7.0, 4.0])   # Womersley inlet: cosine and sine coefficients (period 1)


def _conditions(case, m):
    centre = dict(center=(0.0, 0.0, 0.0), normal=(0.0, 0.0, -1.0))
    if case["flow"] == "cavity":
        return [L.BC(tag=t, kind="nodal") for t in range(1, 7)]
    if case["flow"] == "moving":
        return [L.BC(tag=0, kind="nodal"), L.BC(tag=1, kind="nodal"), L.BC(tag=2, kind="neumann", time="constant", p=(3.0,))]
    inlet = L.BC(tag=1, kind="dirichlet", profile="parabolic", time="pulsatile", p=(15.0, 40.0, 0.8), radius=RADIUS, **centre)
    if case["flow"] in ("box", "batch"):
        inlet = L.BC(tag=1, kind="dirichlet", profile="uniform", time="ramp", p=(0.0, 15.0, 0.0, 0.5), **centre)
    if case["flow"] == "stenosis":
        inlet = L.BC(tag=1, kind="dirichlet", profile="womersley", time="fourier", p=(1.0,), a=_WAVES[0], b=_WAVES[1],
                     radius=RADIUS, **centre)
    return [L.BC(tag=0, kind="noslip"), inlet, L.BC(tag=2, kind="neumann", time="constant", p=(3.0,))]


def _physics(case):
    if case["flow"] == "cavity":
        return dict(rho=1.0, mu=1.0, dt=1e-3, f=(0.0, 0.0, 0.0), disk=None)
    f = (0.1, -0.2, 0.3) if case["stab"] == 1 else (0.0, 0.0, 0.0)
    return dict(rho=RHO, mu=MU, dt=5e-4 if case["flow"] == "stenosis" else 1e-3, f=f,
                disk=dict(resistance=1e4, eps=4.0 / case["n"], radius=0.5) if case["riis"] else None)


@functools.lru_cache(maxsize=16)
def _problem(key):
    case, m = json.loads(key), _mesh(key)
    ph = _physics(case)
    mesh = L.Mesh(m["nodes"], m["tets"], m["faces"], m["tags"])
    opt = L.default_options(precision=case["precision"], stab=case["stab"], diffusion=case["diffusion"], f=ph["f"],
                            implicit=int(case["implicit"]), gmres_rtol=RTOL * (0.1 if case["flow"] == "cavity" else 1.0), smoother_bf16=int(case["bf16"]),
                            pin_pressure_node=0 if case["flow"] == "cavity" else -1)
    d = ph["disk"]
    riis = [L.RIIS(d["resistance"], d["eps"], (0.0, 0.0, 0.7 * m["length"]), (0.0, 0.0, 1.0), d["radius"])] if d else []
    return L.Problem(mesh, ph["rho"], ph["mu"], ph["dt"], case["order"], _conditions(case, m), riis, opt)


def _fields(case, m, seed):
    """History levels u, p, the time, and what the step takes besides (nodal values, displacements)."""
    rng = np.random.default_rng(seed)
    X, order, dt, V = m["nodes"], case["order"], _physics(case)["dt"], len(m["nodes"])
    more = {}
    if case["flow"] == "cavity":
        t0 = rng.uniform(0.0, 0.2)
        u = np.stack([_beltrami(X, t0 - k * dt)[0] for k in range(order)])
        p = np.stack([_beltrami(X, t0 - k * dt)[1] for k in range(order)])
        ue, pe = _beltrami(X, t0 + dt)
        f, a = _area_vectors(m, range(1, 7))
        w = np.zeros((V, 3))
        for k in range(3):
            np.add.at(w, f[:, k], a / 3.0)
        ue -= w * ((w * ue).sum() / (w * w).sum())      # no net flux through the sides
        return u, p, t0, dict(nodal={t: ue for t in range(1, 7)}, pin=float(pe[0]))
    x, y, z = X[:, 0], X[:, 1], X[:, 2]
    if case["flow"] == "batch":
        x = x - 3.0 * np.round(x / 3.0)
    t0 = rng.uniform(0.1, 0.6)
    u, p = np.zeros((order, V, 3)), np.zeros((order, V))
    base = 20.0 * np.clip(1.0 - 0.45 * (x * x + y * y), 0.05, None)
    waves = [(rng.normal(0, 1.0, 3), rng.uniform(0.5, 3.0, 3), rng.uniform(0, 2 * np.pi), rng.uniform(1, 6)) for _ in range(6)]
    noise = rng.standard_normal((V, 4))
    for k in range(order):
        t = t0 - k * dt
        u[k, :, 2] = base * (1.0 + 0.1 * math.sin(7.8 * t))
        p[k] = 2.8 * (m["length"] - z) * (1.0 + 0.1 * math.cos(7.8 * t))
        for amp, wave, phase, freq in waves:
            s = np.sin(X @ wave + phase + freq * t)
            u[k] += s[:, None] * amp
            p[k] += 0.5 * amp[0] * s
        u[k] += 0.05 * noise[:, :3]
        p[k] += 0.02 * noise[:, 3]
    if case["flow"] == "moving":
        wall = np.unique(m["faces"][m["tags"] == 0])
        pulse = lambda t: 0.04 * math.sin(5.0 * t) * np.concatenate([X[:, :2] * np.sin(np.pi * z / m["length"])[:, None], 0 * X[:, :1]], 1)  # noqa: E731
        hist = [pulse(t0 - k * dt) for k in range(order)]
        d1 = pulse(t0 + dt)
        inflow = np.zeros((V, 3))
        inflow[:, 2] = base
        more = dict(d_hist=np.stack(hist), wall=wall.astype(np.int32), d_wall=np.ascontiguousarray(d1[wall]),
                    nodal={0: (d1 - hist[0]) / dt, 1: inflow})
    return u, p, t0, more


def _beltrami(X, t, a=math.pi / 4, d=math.pi / 2):
    """The Ethier-Steinman solution with rho = mu = 1."""
    x, y, z = X.T
    e = math.exp(-d * d * t)
    s, c = np.sin, np.cos
    u = -a * e * np.stack([np.exp(a * x) * s(a * y + d * z) + np.exp(a * z) * c(a * x + d * y),
                           np.exp(a * y) * s(a * z + d * x) + np.exp(a * x) * c(a * y + d * z),
                           np.exp(a * z) * s(a * x + d * y) + np.exp(a * y) * c(a * z + d * x)], 1)
    p = -0.5 * a * a * e * e * (
        np.exp(2 * a * x) + np.exp(2 * a * y) + np.exp(2 * a * z)
        + 2 * s(a * x + d * y) * c(a * z + d * x) * np.exp(a * (y + z))
        + 2 * s(a * y + d * z) * c(a * x + d * y) * np.exp(a * (z + x))
        + 2 * s(a * z + d * x) * c(a * y + d * z) * np.exp(a * (x + y)))
    return u, p


def _pinned(a):
    t = torch.empty(a.shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())
    out = t.numpy()
    out[...] = a
    return out


# ---------------------------------------------------------------------------------- a pass
def prepare(case, seed):
    key = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    m = _mesh(key)
    if case["flow"] == "precond":
        return _precond_inputs(m, seed)
    problem = _problem(key)
    u, p, t0, more = _fields(case, m, seed)
    s = dict(kind="step", u=_pinned(u), p=_pinned(p), t0=t0, more=more, out=(_pinned(u[0]), _pinned(p[0])))
    s["state"] = L.State(problem, s["u"], s["p"], t0)
    run(s)      # the simulation's first step builds the multigrid hierarchy that the later ones keep
    return s


def run(s):
    if s["kind"] == "precond":
        lib, a = L.library(), s["args"]
        status = lib.lfx_asimple_apply_noalloc(*a, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if status != L.LFX_OK:
            raise RuntimeError(lib.lfx_last_error().decode())
        return {"z": s["z"]}
    state, more = s["state"], s["more"]
    state.set(s["u"], s["p"], s["t0"])
    if "d_hist" in more:
        state.set_displacement(more["d_hist"])
        state.set_boundary_displacement(more["wall"], more["d_wall"])
    for tag, values in more.get("nodal", {}).items():
        state.set_dirichlet_nodal(tag, values)
    if "pin" in more:
        state.set_pressure_pin(more["pin"])
    state.step()
    u, p = state.get(*s["out"])
    return {"u": u, "p": p}


def _precond_inputs(m, seed):
    """A diagonally dominant velocity block, gradient and divergence blocks and a Laplacian-like pressure
    block on the mesh's node graph, with a residual: what aSIMPLE meets in a time step."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    V = len(m["nodes"])
    t = torch.from_numpy(m["tets"]).to(dev).long()
    key = torch.unique((t[:, :, None] * V + t[:, None, :]).reshape(-1))
    row, col = key // V, key % V
    nb = row.numel()
    row_ptr = torch.zeros(V + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=V), 0)
    diag = torch.searchsorted(key, torch.arange(V, device=dev) * (V + 1))
    trans = torch.searchsorted(key, col * V + row)
    upper = torch.minimum(torch.arange(nb, device=dev), trans)     # one edge, one value for both directions
    on = row == col
    rnd = lambda *s: torch.randn(*s, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    B = torch.zeros(nb, 4, 4, dtype=torch.float64, device=dev)
    eye = torch.eye(3, dtype=torch.float64, device=dev)
    B[:, :3, :3] = (0.04 + 0.01 * rnd(nb)[upper])[:, None, None] * eye + 0.003 * rnd(nb, 3, 3)
    B[on, :3, :3] += eye * (1.0 + 0.05 * rnd(V))[:, None, None]
    grad = 0.1 * rnd(nb, 3)
    B[:, :3, 3] = grad
    B[:, 3, :3] = -grad[trans]
    link = 0.02 * (1.0 + 0.2 * rnd(nb)[upper]).abs()
    B[:, 3, 3] = torch.where(on, torch.zeros_like(link), -link)
    B[diag, 3, 3] = 0.002 - torch.zeros(V, dtype=torch.float64, device=dev).index_add_(0, row, B[:, 3, 3])
    i32 = [a.to(torch.int32).contiguous() for a in (row_ptr, col, diag, trans)]
    r, z = rnd(V, 4), torch.empty(V, 4, dtype=torch.float64, device=dev)
    args = (V, *(ctypes.c_void_p(a.data_ptr()) for a in (*i32, B, r, z)), None)
    return dict(kind="precond", z=z, keep=(i32, B, r), row=row, col=col, args=args)


# ---------------------------------------------------------------------------------- in 64 bits
def exact(case, seed):
    """The same results from the equations of the paper in plain torch: element matrices, Dirichlet rows,
    a Krylov solve to rounding error; the preconditioner from its definition.  None above 700k tetrahedra
    (160k with Newton's method), where that takes too long."""
    key = json.dumps({k: v for k, v in case.items() if k != "name"}, sort_keys=True)
    T = sum(6 * n * n * nz for n, nz in _sizes(case))
    if T > (160_000 if case["implicit"] else 700_000):
        return None
    m = _mesh(key)
    if case["flow"] == "precond":
        return {"z": _exact_precond(_precond_inputs(m, seed))}
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    u, p, t0, more = _fields(case, m, seed)
    X, order, ph = m["nodes"], case["order"], _physics(case)
    beta = [(1.0,), (2.0, -0.5), (3.0, -1.5, 1.0 / 3.0)][order - 1]
    gamma = [(1.0,), (2.0, -1.0), (3.0, -3.0, 1.0)][order - 1]
    alpha = (1.0, 1.5, 11.0 / 6.0)[order - 1]
    ub, ue, pe = (sum(c * a for c, a in zip(cs, b)) for cs, b in ((beta, u), (gamma, u), (gamma, p)))
    ua = None
    D = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
    tets = D(m["tets"]).long()
    if "d_hist" in more:
        d1 = _lifting(D(X), tets, D(more["wall"]).long(), D(more["d_wall"])).cpu().numpy()
        ua = (alpha * d1 - sum(c * d for c, d in zip(beta, more["d_hist"]))) / ph["dt"]
        X = X + d1
    fixed, values = _dirichlet(case, m, t0 + ph["dt"], more)
    load = np.zeros((len(X), 4))
    if case["flow"] != "cavity":
        f, a = _area_vectors(m, [2], X)
        for k in range(3):
            np.add.at(load[:, :3], f[:, k], -3.0 * a / 3.0)
    sdf = None
    if ph["disk"]:
        rad, h = np.hypot(X[:, 0], X[:, 1]), X[:, 2] - 0.7 * m["length"]
        sdf = np.where(rad > ph["disk"]["radius"], np.hypot(rad - ph["disk"]["radius"], h), np.abs(h)) * np.where(h >= 0, 1, -1)
    ctx = dict(case=case, ph=ph, alpha=alpha, X=D(X), tets=tets, ub=D(ub), ua=None if ua is None else D(ua), load=D(load),
               fixed=D(fixed), values=D(values), sdf=None if sdf is None else D(sdf))
    ue, pe = D(ue), D(pe)
    sol = _solve_step(ctx, ue, pe, torch.cat([ue, pe[:, None]], 1))
    if case["implicit"]:        # the fixed point of the step linearised at its own solution
        for _ in range(60):
            new = _solve_step(ctx, sol[:, :3].contiguous(), sol[:, 3].contiguous(), sol)
            done = (new - sol).norm() <= 1e-13 * new.norm()
            sol = new
            if done:
                break
    sol = sol.cpu().numpy()
    return {"u": sol[:, :3].copy(), "p": sol[:, 3].copy()}


def _dirichlet(case, m, t, more):
    """Mask [V][4] of the prescribed unknowns and their values at time t."""
    X, V = m["nodes"], len(m["nodes"])
    fixed, val = np.zeros((V, 4), bool), np.zeros((V, 4))
    on = lambda tag: np.unique(m["faces"][m["tags"] == tag])  # noqa: E731
    if case["flow"] == "cavity":
        for tag, v in more["nodal"].items():
            fixed[on(tag), :3], val[on(tag), :3] = True, v[on(tag)]
        fixed[0, 3], val[0, 3] = True, more["pin"]
        return fixed, val
    if case["flow"] == "moving":    # the first condition given wins where tags meet
        for tag in (1, 0):
            fixed[on(tag), :3], val[on(tag), :3] = True, more["nodal"][tag][on(tag)]
        return fixed, val
    inlet = on(1)
    r2 = X[inlet, 0] ** 2 + X[inlet, 1] ** 2
    if case["flow"] in ("box", "batch"):
        w = 0.5 * 15.0 * (1 - math.cos(math.pi * t / 0.5)) if t < 0.5 else 15.0
        w = np.full(inlet.size, w)
    elif case["flow"] == "stenosis":
        w = _womersley(np.sqrt(r2), t)
    else:
        g = 15.0 + 25.0 * 0.5 * (1 - math.cos(2 * math.pi * t / 0.8))
        w = g * 2.0 * (RADIUS ** 2 - r2) / (math.pi * RADIUS ** 4)
    fixed[inlet, :3], val[inlet, 2] = True, w
    fixed[on(0), :3], val[on(0), :3] = True, 0.0
    return fixed, val


def _womersley(r, t):
    def bessel(order, z):
        term = np.ones_like(z) if order == 0 else z / 2
        total = term.copy()
        for k in range(1, 80):
            term = term * (-(z * z) / 4) / (k * (k + order))
            total = total + term
        return total

    a, b = _WAVES
    w = a[0] * 2.0 * (RADIUS ** 2 - r * r) / (math.pi * RADIUS ** 4)
    for h in range(1, len(a)):
        z = np.asarray(complex(0, 1) ** 1.5 * RADIUS * math.sqrt(h * 2 * math.pi * RHO / MU), complex)
        shape = 1 - bessel(0, z * (r / RADIUS)) / bessel(0, z)
        flux = math.pi * RADIUS ** 2 * (1 - 2 * bessel(1, z) / (z * bessel(0, z)))
        w = w + ((a[h] - 1j * b[h]) * np.exp(2j * math.pi * h * t) * shape / flux).real
    return w


def _geometry(X):
    """Gradients of the four basis functions [t][4][3], J^-1 and volumes of the elements X [t][4][3]."""
    J = (X[:, 1:] - X[:, :1]).transpose(1, 2)
    Ji = torch.linalg.inv(J)
    return torch.cat([-Ji.sum(1, keepdim=True), Ji], 1), Ji, torch.linalg.det(J).abs() / 6.0


def _element_matrices(c, conn, ue, pe):
    """Matrices [t][4][4][4][4] (test node, component, trial node, component) and right-hand sides [t][4][4]."""
    ph, stab = c["ph"], c["case"]["stab"]
    rho, mu, dt = ph["rho"], ph["mu"], ph["dt"]
    # the reference coordinates (hence J, G, g) follow the orientation that the library fixes
    X = c["X"][conn]
    flip = torch.linalg.det(X[:, 1:] - X[:, :1]) < 0
    conn = torch.where(flip[:, None], conn[:, [0, 1, 3, 2]], conn)
    ga, Ji, vol = _geometry(c["X"][conn])
    G, g = torch.einsum("tmk,tml->tkl", Ji, Ji), Ji.sum(1)
    A = ga.new_zeros(len(conn), 4, 4, 4, 4)
    b = ga.new_zeros(len(conn), 4, 4)
    gab = torch.einsum("tai,tbi->tab", ga, ga)
    uen, ubn, pen = ue[conn], c["ub"][conn], pe[conn]
    f = torch.tensor(ph["f"], dtype=torch.float64, device=ga.device)
    grad_u, grad_p = torch.einsum("tai,taj->tij", uen, ga), torch.einsum("ta,tai->ti", pen, ga)
    for q in range(4):
        lam = ga.new_full((4,), (5 - math.sqrt(5)) / 20)
        lam[q] = (5 + 3 * math.sqrt(5)) / 20
        at = lambda v: torch.einsum("a,ta...->t...", lam, v)  # noqa: E731
        u_q, ub_q, w = at(uen), at(ubn), vol / 4
        us = u_q if c["ua"] is None else u_q - at(c["ua"][conn])
        sR = torch.zeros_like(vol)
        if c["sdf"] is not None:
            d, eps = at(c["sdf"][conn]), ph["disk"]["eps"]
            sR = torch.where(d.abs() <= eps, ph["disk"]["resistance"] / eps * (1 + torch.cos(math.pi * d / eps)) / (2 * eps), sR)
        tau = (c["case"]["order"] ** 2 * rho ** 2 / dt ** 2 + rho ** 2 * torch.einsum("ti,tij,tj->t", us, G, us)
               + C_R * mu ** 2 * (G * G).sum((1, 2)) + sR * sR).rsqrt()
        tau_c = 1.0 / (tau * (g * g).sum(1))
        m = rho * ub_q / dt + f
        res = rho * ((c["alpha"] * u_q - ub_q) / dt + torch.einsum("tij,tj->ti", grad_u, us)) + grad_p + sR[:, None] * u_q - f
        ugr = torch.einsum("ti,tai->ta", us, ga)
        mga = torch.einsum("ti,tai->ta", m, ga)
        ca = rho * c["alpha"] / dt + sR
        cb = ca[:, None] * lam + rho * ugr
        on = 1.0 if stab >= 1 else 0.0
        v = (rho * tau[:, None] * (us - tau[:, None] * res)) if stab >= 2 else torch.zeros_like(us)
        K = (ca[:, None, None] * lam[:, None] * lam + rho * lam[:, None] * ugr[:, None, :] + mu * gab
             + on * rho * tau[:, None, None] * ugr[:, :, None] * cb[:, None, :])
        Q = on * tau_c[:, None, None, None, None] * torch.einsum("tai,tbj->taibj", ga, ga)
        Q = Q + torch.einsum("ti,taj,tb->taibj", v, ga, cb)
        if c["case"]["diffusion"]:
            Q = Q + mu * torch.einsum("taj,tbi->taibj", ga, ga)
        wq = w[:, None, None, None]
        A[:, :, :3, :, :3] += wq[..., None] * Q
        for i in range(3):
            A[:, :, i, :, i] += w[:, None, None] * K
        A[:, :, :3, :, 3] += wq * (-torch.einsum("b,tai->taib", lam, ga) + torch.einsum("ti,tab->taib", v, gab)
                                   + on * rho * torch.einsum("t,ta,tbi->taib", tau, ugr, ga))
        A[:, :, 3, :, :3] += wq * (torch.einsum("a,tbj->tabj", lam, ga) + on * torch.einsum("t,tb,taj->tabj", tau, cb, ga))
        A[:, :, 3, :, 3] += on * (w * tau)[:, None, None] * gab
        b[:, :, :3] += w[:, None, None] * (lam[:, None] * m[:, None, :] + on * rho * (tau[:, None] * ugr)[:, :, None] * m[:, None, :]
                                           + mga[:, :, None] * v[:, None, :])
        b[:, :, 3] += on * (w * tau)[:, None] * mga
    return conn, A, b


def _csr(rows, cols, vals, n):
    order = torch.argsort(rows * n + cols)
    crow = torch.zeros(n + 1, dtype=torch.int64, device=rows.device)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=n), 0)
    return torch.sparse_csr_tensor(crow, cols[order], vals[order], (n, n))


def _solve_step(c, ue, pe, x0):
    V, tets = len(c["X"]), c["tets"]
    key = torch.unique((tets[:, :, None] * V + tets[:, None, :]).reshape(-1))
    blocks = torch.zeros(key.numel(), 16, dtype=torch.float64, device=key.device)
    rhs = c["load"].clone()
    for k in range(0, len(tets), 200_000):
        conn, A, b = _element_matrices(c, tets[k:k + 200_000], ue, pe)
        slot = torch.searchsorted(key, (conn[:, :, None] * V + conn[:, None, :]).reshape(-1))
        blocks.index_add_(0, slot, A.permute(0, 1, 3, 2, 4).reshape(-1, 16))
        rhs.index_add_(0, conn.reshape(-1), b.reshape(-1, 4))
    i = torch.arange(4, device=key.device)
    rows = ((key // V)[:, None, None] * 4 + i[:, None]).expand(-1, 4, 4).reshape(-1)
    cols = ((key % V)[:, None, None] * 4 + i).expand(-1, 4, 4).reshape(-1)
    vals, n = blocks.reshape(-1), 4 * V
    fixed, rhs = c["fixed"].reshape(-1), rhs.reshape(-1)
    diag = torch.zeros(n, dtype=torch.float64, device=key.device)
    diag[rows[rows == cols]] = vals[rows == cols].abs()
    vals = torch.where(fixed[rows], torch.where(rows == cols, diag[rows], torch.zeros_like(vals)), vals)
    rhs = torch.where(fixed, diag * c["values"].reshape(-1), rhs)
    x = torch.where(fixed, c["values"].reshape(-1), x0.reshape(-1))
    return _krylov(rows, cols, vals, n, rhs, x).reshape(V, 4)


def _bicgstab(apply, d, b, steps):
    """A few Jacobi-preconditioned BiCGStab steps from zero."""
    x, r = torch.zeros_like(b), b.clone()
    rt, p, rho = r.clone(), r.clone(), (r * r).sum()
    for _ in range(steps):
        q = d * p
        v = apply(q)
        alpha = rho / (rt * v).sum()
        s = r - alpha * v
        y = d * s
        t = apply(y)
        om = (t * s).sum() / (t * t).sum()
        x = x + alpha * q + om * y
        r = s - om * t
        new = (rt * r).sum()
        p = r + (new / rho) * (alpha / om) * (p - om * v)
        rho = new
    return torch.where(torch.isfinite(x).all(), x, d * b)


def _krylov(rows, cols, vals, n, b, x):
    """Flexible GMRES with a block factorisation (velocity, pressure Schur complement), to rounding error."""
    A = _csr(rows, cols, vals, n)
    p = torch.arange(n, device=b.device) % 4 == 3
    part = lambda sel: _csr(rows[sel], cols[sel], vals[sel], n)  # noqa: E731
    F, Gm, Dm, C = part(~p[rows] & ~p[cols]), part(~p[rows] & p[cols]), part(p[rows] & ~p[cols]), part(p[rows] & p[cols])
    at = rows == cols
    diag = torch.ones_like(b)
    diag[rows[at]] = vals[at]
    dF = torch.where(p, torch.zeros_like(b), 1.0 / diag)
    DF = torch.sparse.mm(Dm, torch.sparse_csr_tensor(Gm.crow_indices(), Gm.col_indices(),
                                                     Gm.values() * dF[torch.repeat_interleave(torch.arange(n, device=b.device), Gm.crow_indices().diff())], (n, n)))
    S = lambda v: C @ v - DF @ v  # noqa: E731
    R = torch.repeat_interleave(torch.arange(n, device=b.device), DF.crow_indices().diff())
    dS = torch.where(p, diag, torch.ones_like(b))
    own = R == DF.col_indices()
    dS[R[own]] -= DF.values()[own]
    dS = torch.where(p, 1.0 / dS, torch.zeros_like(b))

    def precond(r):
        ru = torch.where(p, torch.zeros_like(r), r)
        zu = _bicgstab(lambda v: F @ v, dF, ru, 6)
        zp = _bicgstab(S, dS, torch.where(p, r - Dm @ zu, torch.zeros_like(r)), 60)
        return zu - dF * (Gm @ zp) + zp

    bn, best, last = b.norm(), x, math.inf
    for _ in range(12):
        r = b - A @ x
        beta = r.norm()
        rel = (beta / bn).item()
        if rel < last:
            best = x
        if rel < 2e-15 or rel > 0.5 * last:
            break
        last = rel
        Q, Z, H = [r / beta], [], torch.zeros(41, 40, dtype=torch.float64)
        for j in range(40):
            Z.append(precond(Q[j]))
            w = A @ Z[j]
            for _twice in range(2):
                h = torch.stack([(q * w).sum() for q in Q])
                w = w - torch.stack(Q, 1) @ h
                H[:j + 1, j] += h.cpu()
            H[j + 1, j] = w.norm().item()
            Q.append(w / w.norm())
            e = torch.zeros(j + 2, 1, dtype=torch.float64)
            e[0] = beta.item()
            y = torch.linalg.lstsq(H[:j + 2, :j + 1], e).solution
            if (H[:j + 2, :j + 1] @ y - e).norm().item() < max(1e-9 * beta.item(), 1e-16 * bn.item()):
                break
        x = x + torch.stack(Z, 1) @ y[:, 0].to(b.device)
    return best


def _lifting(X, tets, fixed, values):
    """The harmonic extension of the displacements given at the fixed nodes (conjugate gradients)."""
    ga, _, vol = _geometry(X[tets])
    K = torch.einsum("t,tai,tbi->tab", vol, ga, ga)
    V = len(X)
    rows, cols = tets[:, :, None].expand(-1, 4, 4).reshape(-1), tets[:, None, :].expand(-1, 4, 4).reshape(-1)
    M = torch.sparse_coo_tensor(torch.stack([rows, cols]), K.reshape(-1), (V, V)).coalesce().to_sparse_csr()
    free = torch.ones(V, 1, dtype=torch.float64, device=X.device)
    free[fixed] = 0
    d = torch.zeros_like(X)
    d[fixed] = values
    inv = torch.zeros(V, dtype=torch.float64, device=X.device).index_add_(0, tets.reshape(-1), torch.diagonal(K, dim1=1, dim2=2).reshape(-1))
    inv = free / inv[:, None]
    r = -free * (M @ d)
    z = inv * r
    p, rz, r0 = z, (r * z).sum(0), r.norm()
    for _ in range(4000):
        q = free * (M @ p)
        a = rz / (p * q).sum(0).clamp_min(1e-300)
        d, r = d + a * p, r - a * q
        if r.norm() <= 1e-15 * r0:
            break
        z = inv * r
        new = (r * z).sum(0)
        p, rz = z + (new / rz.clamp_min(1e-300)) * p, new
    return d


def _exact_precond(s):
    """aSIMPLE with six Chebyshev steps on the velocity block (lmax / lmin = 60) and on the Schur
    complement (30), both from Gershgorin bounds: the entry point's defaults."""
    (_, B, r), row, col = s["keep"], s["row"], s["col"]
    V = len(r)

    def mul(blk, v):        # sum over a row's blocks of blk [nb][i][j] v[col][j]
        return torch.zeros(V, blk.shape[1], dtype=torch.float64, device=r.device).index_add_(
            0, row, (blk * v[col][:, None, :]).sum(2))

    F, Gm, Dm, C = B[:, :3, :3], B[:, :3, 3:], B[:, 3:, :3], B[:, 3:, 3:]
    on = row == col
    dF = torch.zeros(V, 3, dtype=torch.float64, device=r.device)
    dF[row[on]] = 1.0 / torch.diagonal(F[on], dim1=1, dim2=2)
    S = lambda v: mul(C, v) - mul(Dm, dF * mul(Gm, v))  # noqa: E731
    dS = torch.zeros(V, 1, dtype=torch.float64, device=r.device)
    dS[row[on]] = C[on][:, 0]
    pos = torch.searchsorted(row * V + col, col * V + row)      # block (j, i) of block (i, j)
    dS -= mul(Dm * Gm[pos].transpose(1, 2), dF)
    dS = 1.0 / dS
    one = torch.ones(V, 1, dtype=torch.float64, device=r.device)
    lam_f = (dF.abs() * mul(F.abs(), one.expand(-1, 3))).max().item()
    lam_s = (dS.abs() * (mul(C.abs(), one) + mul(Dm.abs(), dF.abs() * mul(Gm.abs(), one)))).max().item()

    def chebyshev(apply, d, b, lmax, ratio):
        theta, delta = 0.5 * (lmax + lmax / ratio), 0.5 * (lmax - lmax / ratio)
        rho = delta / theta
        res = d * b
        step = res / theta
        x = step
        for _ in range(5):
            res = res - d * apply(step)
            new = 1.0 / (2.0 * theta / delta - rho)
            step = new * rho * step + 2.0 * new / delta * res
            x, rho = x + step, new
        return x

    zu = chebyshev(lambda v: mul(F, v), dF, r[:, :3], lam_f, 60.0)
    zp = chebyshev(S, dS, r[:, 3:] - mul(Dm, zu), lam_s, 30.0)
    return torch.cat([zu - dF * mul(Gm, zp), zp], 1)
