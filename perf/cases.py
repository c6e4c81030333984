"""Performance cases of the red-blood-cell solver: the work a program has it do, through
the public Python binding (paper_1903_06479_gb300.npfem).

A simulation keeps one handle per mesh topology, device arrays of positions, velocities
and forces, and calls `step` (or replays a captured graph of steps) in a time loop; a
coupled one computes the forces from the fluid's stress lattice before every step, and a
dense suspension detects collisions first.  The fluid side calls the multi-direct forcing;
the warm-start network is fitted by loss/gradient and Adam calls.  The cases are those
calls over the sizes of this repository's configurations, tests and benchmark: one cell to
16384, meshes of 66 to 2562 vertices, each precision of the solver.

A pass of the stepping cases is a stretch of `steps` time steps from a stored state (a
program that restarts from a checkpoint, or that looks ahead, copies the state and steps
the copy).  Inputs are drawn on the GPU from the seed: discocytes with random
orientations and positions in a 100 um box of a plasma shear flow, moving with the flow.

`exact` follows the same definitions in FP64 with plain torch: rest-state tables, the
energies' gradient, a quasi-Newton iteration run to rounding level, the dissipation step,
the immersed-boundary sums, the network's gradient.
"""
import functools
import math

import numpy as np
import torch

from paper_1903_06479_gb300 import learn
from paper_1903_06479_gb300 import npfem
from paper_1903_06479_gb300 import workloads

DT = 0.1  # us
BOX = 100.0  # um
LATTICE_N = 121  # nodes per side of the fluid lattice: the box and ten nodes around it
LATTICE_DX = 1.0
W_COL = 2000.0  # pN/um
CUTOFF = 0.6  # um


def listed():
    return [
        # one cell in FP64 at a tight tolerance: parameter studies and references; latency
        dict(name="one_cell_fp64", kind="steps", groups="258x1", precision="fp64", tol=1e-8, steps=4, graph=False),
        # one cell with the library's defaults (FP32): the smallest time loop, launches count
        dict(name="one_cell", kind="steps", groups="642x1", precision="fp32", tol=1e-6, steps=8, graph=False),
        # a few dozen cells of the paper's finest resolution with the defaults: fewer cells than SMs
        dict(name="few_fine_cells", kind="steps", groups="1026x37", precision="fp32", tol=1e-6, steps=4, graph=False),
        # a suspension of the paper's middle resolution with the defaults (FP32), odd count
        dict(name="suspension_fp32", kind="steps", groups="258x3001", precision="fp32", tol=1e-6, steps=4, graph=False),
        # the benchmark's population through the plain FP32 path
        dict(name="population_fp32", kind="steps", groups="642x1024", precision="fp32", tol=1e-6, steps=4, graph=False),
        # the benchmark's population, tensor-core contraction, a captured stretch of the time loop
        dict(name="population_bf16", kind="steps", groups="642x1024", precision="bf16", tol=1e-6, steps=10, graph=True),
        # the same coupled to the fluid: forces from the stress lattice and thermal noise before every step
        dict(name="coupled_bf16", kind="coupled", groups="642x1024", precision="bf16", tol=1e-6, steps=4, graph=False),
        # the largest population of the repository's configurations
        dict(name="large_bf16", kind="steps", groups="642x16384", precision="bf16", tol=1e-6, steps=2, graph=False),
        # mixed resolutions in one call (40 % / 40 % / 20 %)
        dict(name="mixed_bf16", kind="steps", groups="258x1638+642x1638+2562x820", precision="bf16", tol=1e-6, steps=2,
             graph=False),
        # a dense suspension: collisions detected before every step (TF32 contraction, refined)
        dict(name="dense_tf32", kind="dense", groups="642x500", precision="tf32", tol=1e-6, steps=2, graph=False),
        # the fluid side: multi-direct forcing of the benchmark's population on the lattice
        dict(name="forcing", kind="forcing", groups="642x1024", cycles=3),
        # fitting the warm-start network: one minibatch's loss, gradient and Adam update
        dict(name="network_fit", kind="fit", batch=8192),
    ]


# Vertex counts a program meets: subdivided octahedra and icosahedra and, between them, the
# geodesic grids of other frequencies (10 f^2 + 2, 4 f^2 + 2, 5 f^2 + 2 on the icosahedron,
# octahedron and pentagonal bipyramid, the last with odd counts).
DRAW_VERTS = (66, 127, 162, 198, 258, 362, 407, 607, 642, 786, 1002, 1026, 1442, 2562)
# vertex-steps of a pass, by precision (a large mesh's contraction grows with n^2)
DRAW_WORK = dict(fp64=4.0e3, fp32=2.0e6, tf32=2.0e6, bf16=8.0e6)


def draw(rng):
    kind = rng.choices(("steps", "coupled", "dense", "forcing", "fit"), (9, 2, 1, 1, 1))[0]
    log_int = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if kind == "fit":
        return dict(kind=kind, batch=log_int(500, 60000))
    n = rng.choice(DRAW_VERTS)
    if kind == "forcing":
        return dict(kind=kind, groups="%dx%d" % (n, max(1, log_int(2000, 1.2e6) // n)), cycles=rng.randint(1, 5))
    if kind == "dense":
        prec = rng.choice(("fp32", "tf32", "bf16"))
        return dict(kind=kind, groups="%dx%d" % (n, max(2, log_int(1e4, 4e5) // n)), precision=prec, tol=1e-6, steps=2,
                    graph=False)
    prec = rng.choices(("fp64", "fp32", "tf32", "bf16"), (1, 3, 1, 3))[0] if kind == "steps" else "bf16"
    if prec == "fp64":
        n = min(n, 362)
    steps = rng.randint(2, 4)
    most = DRAW_WORK[prec] / (1.0 + n / 642.0)
    first = max(1, log_int(n, most) // (n * steps))
    groups = "%dx%d" % (n, first)
    if prec != "fp64" and rng.random() < 0.25:
        other = rng.choice([k for k in DRAW_VERTS if k != n])
        groups += "+%dx%d" % (other, max(1, log_int(other, DRAW_WORK[prec] / (2.0 + other / 321.0)) // (other * steps)))
    return dict(kind=kind, groups=groups, precision=prec, tol=1e-8 if prec == "fp64" else 1e-6, steps=steps,
                graph=kind == "steps" and rng.random() < 0.3)


# ---------------------------------------------------------------------------------------
# meshes
# ---------------------------------------------------------------------------------------
def _bases():
    octa = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    g = (1.0 + 5.0 ** 0.5) / 2.0
    ico = [(0, s, t * g) for s in (1, -1) for t in (1, -1)]
    ico = ico + [(b, c, a) for a, b, c in ico] + [(c, a, b) for a, b, c in ico]
    penta = [(math.cos(2 * math.pi * k / 5), math.sin(2 * math.pi * k / 5), 0.0) for k in range(5)] + [(0, 0, 1), (0, 0, -1)]
    return {4: octa, 5: penta, 10: ico}


def _hull_faces(v):
    """Triangles of a deltahedron's convex hull (a plane through three corners with the rest behind it)."""
    out = []
    for i in range(len(v)):
        for j in range(i + 1, len(v)):
            for k in range(j + 1, len(v)):
                nrm = np.cross(v[j] - v[i], v[k] - v[i])
                d = (v - v[i]) @ nrm
                if np.linalg.norm(nrm) > 1e-9 and (np.all(d < 1e-9) or np.all(d > -1e-9)):
                    out.append((i, j, k) if np.all(d < 1e-9) else (i, k, j))
    return out


def _geodesic(corners, f):
    """Class I geodesic grid of frequency f on a deltahedron: unit vectors and outward faces."""
    v = np.asarray(corners, dtype=np.float64)
    v = v / np.linalg.norm(v, axis=1, keepdims=True)
    index, points, tris = {}, [], []

    def at(face, a, b, c):
        key = tuple(sorted((face[q], w) for q, w in enumerate((a, b, c)) if w))
        if key not in index:
            p = (a * v[face[0]] + b * v[face[1]] + c * v[face[2]]) / f
            index[key] = len(points)
            points.append(p / np.linalg.norm(p))
        return index[key]

    for face in _hull_faces(v):
        for a in range(f):
            for b in range(f - a):
                c = f - 1 - a - b
                tris.append((at(face, a + 1, b, c), at(face, a, b + 1, c), at(face, a, b, c + 1)))
                if c:
                    tris.append((at(face, a + 1, b + 1, c - 1), at(face, a, b + 1, c), at(face, a + 1, b, c)))
    p, t = np.asarray(points), np.asarray(tris, dtype=np.int32)
    out = np.einsum("ij,ij->i", np.cross(p[t[:, 1]] - p[t[:, 0]], p[t[:, 2]] - p[t[:, 0]]), p[t].sum(1)) > 0
    t[~out] = t[~out][:, [0, 2, 1]]
    return p, t


@functools.lru_cache(maxsize=None)
def _mesh(n):
    """Rest positions [n, 3] and triangles of the discocyte with n vertices."""
    try:
        return workloads.discocyte(n)
    except ValueError:
        pass
    for m, corners in _bases().items():
        f = math.isqrt((n - 2) // m)
        if m * f * f + 2 == n:
            s, t = _geodesic(corners, f)
            break
    else:
        raise ValueError("no geodesic grid with %d vertices" % n)
    d = workloads.DISCOCYTE_D
    r2 = (0.25 * d * d) * (s[:, :2] ** 2).sum(1)
    q = np.clip(1.0 - 4.0 * r2 / d ** 2, 0.0, None)
    z = np.sign(s[:, 2]) * d * np.sqrt(q) * (workloads.ES_A0 + workloads.ES_A1 * r2 / d ** 2 + workloads.ES_A2 * r2 ** 2 / d ** 4)
    return np.column_stack([0.5 * d * s[:, :2], z]), t


def _groups(case):
    return [tuple(int(k) for k in g.split("x")) for g in case["groups"].split("+")]


@functools.lru_cache(maxsize=None)
def _fans(n):
    """[n, most] triangles around every vertex, padded with the number of triangles."""
    t = _mesh(n)[1]
    around = [[] for _ in range(n)]
    for k, tri in enumerate(t):
        for i in tri:
            around[i].append(k)
    most = max(map(len, around))
    return np.asarray([a + [len(t)] * (most - len(a)) for a in around])


def _area_normals(x, n):
    """Vertex shares A_k n_k of the area-weighted normals; x: [cells, n, 3]."""
    t = torch.as_tensor(_mesh(n)[1].astype(np.int64), device=x.device)
    a = torch.cross(x[:, t[:, 1]] - x[:, t[:, 0]], x[:, t[:, 2]] - x[:, t[:, 0]], dim=2) / 6.0
    a = torch.cat([a, torch.zeros_like(a[:, :1])], 1)
    fan = torch.as_tensor(_fans(n), device=x.device)
    return sum(a[:, fan[:, q]] for q in range(fan.shape[1]))


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _population(n, cells, gen, dense=False):
    """Positions, velocities and forces [cells, n, 3] (FP64) of cells moving with a shear
    flow u_x = gamma y: the centre's velocity and half the vorticity as a rotation; the
    force is the traction of the plasma's shear stress and thermal noise."""
    kw = dict(generator=gen, device="cuda", dtype=torch.float64)
    rest = torch.as_tensor(_mesh(n)[0], device="cuda")
    if dense:
        # stacks of aligned cells with small tilts, rims just touching
        side = math.ceil(cells ** (1 / 3))
        k = torch.arange(cells, device="cuda")
        grid = torch.stack([k % side, (k // side) % side, k // (side * side)], 1).double()
        centre = 8.0 + grid * torch.tensor([7.9, 7.9, 2.65], device="cuda") + 0.1 * torch.randn(cells, 3, **kw)
        tilt = 0.03
        q = torch.cat([torch.ones(cells, 1, device="cuda", dtype=torch.float64), tilt * torch.randn(cells, 3, **kw)], 1)
    else:
        centre = BOX * torch.rand(cells, 3, **kw)
        q = torch.randn(cells, 4, **kw)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                       2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                       2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    off = torch.einsum("cij,nj->cni", rot, rest)
    gamma = 1e-6 * (10.0 + 990.0 * torch.rand(cells, 1, 1, **kw))  # 1/us
    pos = off + centre[:, None]
    vel = torch.zeros_like(pos)
    vel[..., 0] = gamma[..., 0] * (centre[:, None, 1] + 0.5 * off[..., 1])
    vel[..., 1] = -0.5 * gamma[..., 0] * off[..., 0]
    an = _area_normals(pos, n)
    frc = 0.5 * torch.randn(cells, n, 3, **kw)
    frc[..., 0] += workloads.PLASMA_ETA * gamma[..., 0] * an[..., 1]
    frc[..., 1] += workloads.PLASMA_ETA * gamma[..., 0] * an[..., 0]
    return pos, vel, frc


def _soa(parts, dtype):
    """[cells, n, 3] arrays of every group as one flat component-major array."""
    return torch.cat([p.transpose(1, 2).reshape(-1) for p in parts]).to(dtype).contiguous()


def _lattice():
    lo = -0.5 * ((LATTICE_N - 1) * LATTICE_DX - BOX)
    return npfem.lattice((lo, lo, lo), LATTICE_DX, (LATTICE_N,) * 3)


def _field(gen, width, kind):
    """A lattice field [z, y, x, width]: the plasma's shear stress (rate rising across the
    box) or velocity, with small smooth fluctuations."""
    g = torch.arange(LATTICE_N, device="cuda", dtype=torch.float64) / (LATTICE_N - 1)
    z, y, x = torch.meshgrid(g, g, g, indexing="ij")
    rate = 1e-6 * (10.0 + 990.0 * z)
    out = torch.zeros(LATTICE_N, LATTICE_N, LATTICE_N, width, device="cuda", dtype=torch.float64)
    used = 6 if kind == "stress" else 3
    size = workloads.PLASMA_ETA * 1e-4 if kind == "stress" else 2e-3
    for c in range(used):
        a = torch.randn(3, 4, generator=gen, device="cuda", dtype=torch.float64)
        for k in range(3):
            out[..., c] += size * a[k, 0] * torch.sin((k + 1) * math.pi * (a[k, 1] * x + a[k, 2] * y + a[k, 3] * z))
    if kind == "stress":
        out[..., 3] += workloads.PLASMA_ETA * rate
    else:
        out[..., 0] += rate * BOX * y
    return out.float().contiguous()


def _fit_inputs(case, seed):
    gen = _generator(seed)
    kw = dict(generator=gen, device="cuda")
    samples = 8 * case["batch"]
    scale = torch.tensor([4e-2, 4e-2, 3e-2, 2e-2, 2e-2, 2e-2, 5e-5, 5e-5, 5e-5], device="cuda")
    feat = torch.randn(samples, 9, **kw) * scale
    target = 2e-4 * (torch.tanh(feat[:, :3] / scale[:3] - feat[:, 3:6] / scale[3:6]) + 0.3 * torch.randn(samples, 3, **kw))
    params = torch.as_tensor(learn.set_normalisation(learn.init_params(seed % 2 ** 31), feat, target), device="cuda")
    idx = torch.randint(0, samples, (case["batch"],), dtype=torch.int32, **kw)
    return params, feat, target, idx


def _inputs(case, seed):
    """The arrays of a case on the GPU, from the seed alone."""
    gen = _generator(seed)
    dtype = torch.float64 if case.get("precision") == "fp64" else torch.float32
    pops = [_population(n, cells, gen, case["kind"] == "dense") for n, cells in _groups(case)]
    s = {k: _soa([p[q] for p in pops], dtype) for q, k in enumerate(("x0", "v0", "f"))}
    if case["kind"] == "coupled":
        s["sigma"] = _field(gen, 8, "stress")
        s["noise"] = 0.5 * torch.randn(case["steps"], s["x0"].numel(), generator=gen, device="cuda")
    if case["kind"] == "forcing":
        s["u_lattice"] = _field(gen, 4, "velocity")
    return s


def prepare(case, seed):
    if case["kind"] == "fit":
        params, feat, target, idx = _fit_inputs(case, seed)
        return dict(case=case, params=params, feat=feat, target=target, idx=idx, m=torch.zeros_like(params),
                    v=torch.zeros_like(params), grad=torch.zeros_like(params), loss=torch.zeros(1, device="cuda"), step=0)
    s = _inputs(case, seed)
    s["case"], s["cells"] = case, [c for _, c in _groups(case)]
    opts = npfem.default_opts(precision=case.get("precision", "fp32"), tol=case.get("tol", 1e-6),
                              refine=int(case.get("precision") == "tf32"))
    s["handles"] = [npfem.Handle(*_mesh(n), npfem.material(), opts, dt=DT) for n, _ in _groups(case)]
    s["lattice"] = _lattice()
    s["x"], s["v"] = s["x0"].clone(), s["v0"].clone()
    if case["kind"] == "dense":
        verts = sum(n * c for n, c in _groups(case))
        s["planes"] = torch.zeros(verts, 4, device="cuda")
        s["found"] = torch.zeros(2, dtype=torch.int32, device="cuda")
        s["handles"][0].set_collisions(s["planes"], W_COL)
    if case["kind"] == "forcing":
        s["f_lattice"] = torch.zeros(LATTICE_N, LATTICE_N, LATTICE_N, 4, device="cuda")
    if case.get("graph"):
        s["loop"] = npfem.StepGraph(s["handles"], s["cells"], s["x"], s["v"], s["f"], DT, steps=case["steps"])
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "fit":
        s["step"] += 1
        npfem.mlp_loss_grad(s["params"], s["feat"], s["target"], s["idx"], case["batch"], s["grad"], s["loss"])
        npfem.mlp_adam(s["params"], s["m"], s["v"], s["grad"], s["step"], lr=1e-3)
        return [s["loss"], s["grad"], s["params"], s["m"], s["v"]]
    if case["kind"] == "forcing":
        npfem.ibm_forcing(s["handles"], s["cells"], s["x"], s["v"], s["lattice"], s["u_lattice"], DT, case["cycles"],
                          s["f"], s["f_lattice"])
        return [s["f"], s["f_lattice"]]
    handles, cells, x, v, f = s["handles"], s["cells"], s["x"], s["v"], s["f"]
    x.copy_(s["x0"])
    v.copy_(s["v0"])
    if case["graph"]:
        s["loop"].launch()
        return [x, v]
    for k in range(case["steps"]):
        if case["kind"] == "coupled":
            npfem.ibm_forces(handles, cells, x, s["lattice"], s["sigma"], f)
            f += s["noise"][k]
        elif case["kind"] == "dense":
            npfem.collision_detect(handles, cells, x, CUTOFF, s["planes"], s["found"])
        npfem.step(handles, cells, x, v, f, DT)
    if case["kind"] == "coupled":
        return [x, v, f]
    return [x, v, s["planes"], s["found"]] if case["kind"] == "dense" else [x, v]


def work(case):
    """Bytes: the state in and out of every step (5 vectors), the fields and the network's
    arrays once.  Flops: an evaluation is about 700 per vertex (two triangles and a bending
    ring each) and a direction about 200; a step of these populations takes about 4 of
    each.  The application of the prefactored inverse is counted as the two sparse
    triangular solves it stands for, about 60 entries per vertex each."""
    if case["kind"] == "fit":
        b = case["batch"]
        return dict(bytes=52 * b + 9 * 4 * 5016, flops=6 * b * (9 * 64 + 64 * 64 + 64 * 3))
    verts = sum(n * c for n, c in _groups(case))
    nodes = LATTICE_N ** 3
    if case["kind"] == "forcing":
        k = case["cycles"]
        return dict(bytes=36 * verts + 32 * nodes, flops=verts * (2 * k + 2) * 64 * 8)
    size = 8 if case["precision"] == "fp64" else 4
    per = 15 * size * verts
    flops = verts * (4 * (700 + 200 + 12 * 60) + 700)
    if case["kind"] == "coupled":
        return dict(bytes=case["steps"] * (per + 9 * size * verts) + 24 * nodes,
                    flops=case["steps"] * (flops + verts * 64 * 15))
    if case["kind"] == "dense":
        per += 28 * verts
    return dict(bytes=case["steps"] * per, flops=case["steps"] * flops)


# ---------------------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------------------
class _Membrane:
    """Rest-state tables and the objective's gradient of one topology in FP64."""

    def __init__(self, n):
        m = workloads.DEFAULT_MATERIAL
        X, t = _mesh(n)
        X, t = np.asarray(X, dtype=np.float64), np.asarray(t, dtype=np.int64)
        self.n, self.m = n, m
        e1, e2 = X[t[:, 1]] - X[t[:, 0]], X[t[:, 2]] - X[t[:, 0]]
        cr = np.cross(e1, e2)
        two = np.linalg.norm(cr, axis=1)
        l1 = np.linalg.norm(e1, axis=1)
        a, b, c = l1, (e1 * e2).sum(1) / l1, two / l1
        dm = np.stack([1 / a, -b / (a * c), 1 / c], 1)  # upper-triangular D_m^-1
        area = 0.5 * two
        v0 = (X[t[:, 0]] * cr).sum() / 6.0
        bary, vor, lap = np.zeros(n), np.zeros(n), np.zeros((n, n))
        P = X[t]
        cot = np.empty((len(t), 3))
        for q in range(3):
            u, w = P[:, (q + 1) % 3] - P[:, q], P[:, (q + 2) % 3] - P[:, q]
            cot[:, q] = (u * w).sum(1) / np.linalg.norm(np.cross(u, w), axis=1)
            np.add.at(lap, (t[:, (q + 1) % 3], t[:, (q + 2) % 3]), cot[:, q])
            np.add.at(lap, (t[:, (q + 2) % 3], t[:, (q + 1) % 3]), cot[:, q])
            np.add.at(bary, t[:, q], area / 3.0)
        obtuse = (cot < 0).any(1)
        for q in range(3):
            q1, q2 = (q + 1) % 3, (q + 2) % 3
            fine = 0.125 * (((P[:, q1] - P[:, q]) ** 2).sum(1) * cot[:, q2] + ((P[:, q2] - P[:, q]) ** 2).sum(1) * cot[:, q1])
            np.add.at(vor, t[:, q], np.where(obtuse, np.where(cot[:, q] < 0, 0.5, 0.25) * area, fine))
        adj = np.zeros((n, n), dtype=bool)
        for q in range(3):
            adj[t[:, q], t[:, (q + 1) % 3]] = adj[t[:, (q + 1) % 3], t[:, q]] = True
        lap /= 2.0 * vor[:, None]
        lap[np.arange(n), np.arange(n)] = -lap.sum(1)  # delta = lap x
        mass = m["density"] * v0 * bary / area.sum()
        # the constant quasi-Newton matrix M/h^2 + sum w G^T G
        gj, gk = np.stack([dm[:, 0], dm[:, 1]], 1), np.stack([0 * dm[:, 0], dm[:, 2]], 1)
        G = np.stack([-(gj + gk), gj, gk], 1)  # [nt, corner, column]
        H = np.diag(mass / DT ** 2 + m["k_vol"]) + lap.T @ ((m["k_bend"] * vor)[:, None] * lap)
        loc = np.einsum("t,tpc,tqc->tpq", (m["C"] + m["k_mat_hess"]) * area, G, G)
        np.add.at(H, (np.repeat(t, 3, 1).ravel(), np.tile(t, (1, 3)).ravel()), loc.ravel())
        most = int(adj.sum(1).max())
        ring = np.argsort(~adj, axis=1, kind="stable")[:, :most]
        on = np.take_along_axis(adj, ring, 1)
        dev = lambda v: torch.as_tensor(v, device="cuda")
        rc = np.where(on, np.take_along_axis(lap, ring, 1), 0.0)
        rt = np.where(on, np.take_along_axis(lap.T, ring, 1), 0.0)
        self.t, self.dm, self.area, self.v0 = dev(t), dev(dm), dev(area), v0
        self.ring, self.rc, self.rt, self.diag = dev(ring), dev(rc), dev(rt), dev(np.diag(lap).copy())
        self.vor, self.mass = dev(vor), dev(mass)
        self.dg = dev(np.linalg.norm(lap @ X, axis=1))
        self.inv = torch.linalg.inv(dev(H))
        e = np.triu(adj)
        i, j = np.nonzero(e)
        self.lbar = np.linalg.norm(X[i] - X[j], axis=1).mean()

    def laplacian(self, f, weights):
        return self.diag[:, None] * f + sum(weights[:, q, None] * f[:, self.ring[:, q]] for q in range(self.ring.shape[1]))

    def gradient(self, x, uy, u, planes):
        """Gradient of the objective at x + u (x relative to each cell's vertex 0), uy = y - x."""
        m, t, dm, p = self.m, self.t, self.dm, x + u
        pi = p[:, t[:, 0]]
        e1, e2 = p[:, t[:, 1]] - pi, p[:, t[:, 2]] - pi
        d0, d1, d3 = dm[:, 0, None], dm[:, 1, None], dm[:, 2, None]
        f0, f1 = e1 * d0, e1 * d1 + e2 * d3
        aa, bb, cc = (f0 * f0).sum(-1), (f0 * f1).sum(-1), (f1 * f1).sum(-1)
        mean, dif = 0.5 * ((aa - 1) + (cc - 1)), 0.5 * (aa - cc)
        rad = torch.sqrt(dif * dif + bb * bb)
        s1, s2 = torch.sqrt(1 + mean + rad), torch.sqrt(1 + mean - rad)
        a1, a2 = (mean + rad) / (s1 + 1), (mean - rad) / (s2 + 1)
        r = 0.5 * (a1 - a2)  # nearest area-preserving stretches (1 + r, 1 / (1 + r))
        for _ in range(8):
            q = 1 + r
            r = r - ((r - a1) * q ** 3 + r * (1 + a2) + a2) / (q ** 3 + 3 * (r - a1) * q * q + 1 + a2)
        k1 = self.area * (m["C"] * (a1 - r) + 0.5 * m["B"] * s1 * a1 * (2 + a1) + m["D"] * a1 ** 3) / s1
        k2 = self.area * (m["C"] * (a2 + r / (1 + r)) + 0.5 * m["B"] * s2 * a2 * (2 + a2) + m["D"] * a2 ** 3) / s2
        pos = dif >= 0
        vx, vy = torch.where(pos, dif + rad, bb), torch.where(pos, bb, rad - dif)
        vx = torch.where(rad == 0, torch.ones_like(vx), vx)
        s = 1 / torch.sqrt(vx * vx + vy * vy)
        vx, vy = vx * s, vy * s
        k00, k11, k01 = k1 * vx * vx + k2 * vy * vy, k1 * vy * vy + k2 * vx * vx, (k1 - k2) * vx * vy
        g0 = f0 * k00[..., None] + f1 * k01[..., None]
        g1 = f0 * k01[..., None] + f1 * k11[..., None]
        cj, ck = g0 * d0 + g1 * d1, g1 * d3
        cr = torch.cross(e1, e2, dim=2)
        g, gc = torch.zeros_like(p), torch.zeros_like(p)
        for q, part in enumerate((-(cj + ck), cj, ck)):
            g.index_add_(1, t[:, q], part)
            gc.index_add_(1, t[:, q], cr / 6.0)
        df = self.laplacian(p, self.rc)
        nf = df.norm(dim=2, keepdim=True)
        w = (m["k_bend"] * self.vor)[:, None] * df * (1 - self.dg[:, None] / nf)
        g += self.laplacian(w, self.rt)
        vol = (pi * cr).sum((1, 2)) / 6.0
        g += (m["k_vol"] * (vol - self.v0) / (gc * gc).sum((1, 2)))[:, None, None] * gc
        g += (self.mass / DT ** 2)[:, None] * (u - uy)
        if planes is not None:
            d = planes[..., 3] - (planes[..., :3] * p).sum(-1)
            g -= W_COL * torch.clamp(d, min=0.0)[..., None] * planes[..., :3]
        return g

    def minimise(self, x, uy, planes, most=80, tol=1e-12):
        """Unit-step L-BFGS from y with the constant matrix, every cell to rounding level."""
        dot = lambda a, b: (a * b).sum((1, 2), keepdim=True)
        u, pairs = uy.clone(), []
        g = self.gradient(x, uy, u, planes)
        for _ in range(most):
            res = (((DT ** 2 / self.mass[:, None] * g) ** 2).sum((1, 2)) / self.n).sqrt().max() / self.lbar
            if not float(res) > tol:
                break
            q, al = g.clone(), []
            for s, y, sy in reversed(pairs):
                a = dot(s, q) / sy
                al.append(a)
                q -= a * y
            q = torch.einsum("ij,cjk->cik", self.inv, q)
            for (s, y, sy), a in zip(pairs, reversed(al)):
                q += (a - dot(y, q) / sy) * s
            u2 = u - q
            g2 = self.gradient(x, uy, u2, planes)
            s, y = u2 - u, g2 - g
            sy = dot(s, y)
            pairs = (pairs + [(s, y, torch.where(sy > 0, sy, torch.full_like(sy, math.inf)))])[-8:]
            u, g = u2, g2
        return u

    def step(self, x, v, f, planes=None):
        """One time step of [cells, n, 3] arrays: the converged positions, damped velocities."""
        uy = DT * v + DT ** 2 * f / self.mass[:, None]
        u = torch.empty_like(uy)
        some = max(1, int(4e6) // len(self.t))
        for a in range(0, len(x), some):
            c = slice(a, a + some)
            u[c] = self.minimise(x[c] - x[c, :1], uy[c], None if planes is None else planes[c])
        xr = x - x[:, :1] + u
        v = u / DT
        mass, tot = self.mass[:, None], self.mass.sum()
        xc, vc = (mass * xr).sum(1, keepdim=True) / tot, (mass * v).sum(1, keepdim=True) / tot
        r = xr - xc
        spin = (mass * torch.cross(r, v - vc, dim=2)).sum(1)
        inertia = (mass[..., None] * ((r * r).sum(-1)[..., None, None] * torch.eye(3, device="cuda", dtype=torch.float64) -
                                      r[..., :, None] * r[..., None, :])).sum(1)
        omega = torch.linalg.solve(inertia, spin)
        rigid = vc + torch.cross(omega[:, None].expand_as(r), r, dim=2)
        return x + u, v + self.m["kappa"] * (rigid - v)


def _split(case, flat, width=3):
    out, at = [], 0
    for n, c in _groups(case):
        out.append(flat[at:at + width * n * c].double().view(c, width, n).transpose(1, 2).contiguous())
        at += width * n * c
    return out


def _weight(r):
    """The four-point kernel."""
    a = r.abs()
    near = 3 - 2 * a + torch.sqrt(torch.clamp(1 + 4 * a - 4 * a * a, min=0.0))
    far = 5 - 2 * a - torch.sqrt(torch.clamp(-7 + 12 * a - 4 * a * a, min=0.0))
    return torch.where(a <= 1, near, torch.where(a <= 2, far, torch.zeros_like(a))) / 8


class _Stencil:
    """The 64 lattice nodes around points [m, 3] and their weights, one after the other."""

    def __init__(self, p):
        r = (p + 0.5 * ((LATTICE_N - 1) * LATTICE_DX - BOX)) / LATTICE_DX
        self.base = torch.floor(r).long() - 1
        self.w = [_weight(r - (self.base + q)) for q in range(4)]

    def nodes(self):
        for c in range(4):
            for b in range(4):
                for a in range(4):
                    k = self.base + torch.tensor([a, b, c], device="cuda")
                    w = self.w[a][:, 0] * self.w[b][:, 1] * self.w[c][:, 2]
                    w = w * ((k >= 0) & (k < LATTICE_N)).all(1)
                    k = k.clamp(0, LATTICE_N - 1)
                    yield (k[:, 2] * LATTICE_N + k[:, 1]) * LATTICE_N + k[:, 0], w[:, None]

    def gather(self, field):
        return sum(w * field[k] for k, w in self.nodes())

    def spread(self, values):
        out = torch.zeros(LATTICE_N ** 3, values.shape[1], device="cuda", dtype=torch.float64)
        for k, w in self.nodes():
            out.index_add_(0, k, w * values)
        return out


def _vertex_areas(x, n):
    t = torch.as_tensor(_mesh(n)[1].astype(np.int64), device="cuda")
    a = torch.cross(x[:, t[:, 1]] - x[:, t[:, 0]], x[:, t[:, 2]] - x[:, t[:, 0]], dim=2).norm(dim=2) / 6.0
    a = torch.cat([a, torch.zeros_like(a[:, :1])], 1)
    fan = torch.as_tensor(_fans(n), device="cuda")
    return sum(a[:, fan[:, q]] for q in range(fan.shape[1]))


def _exact_forces(case, xs, sigma):
    out = []
    for x, (n, c) in zip(xs, _groups(case)):
        nrm = _area_normals(x, n)
        nrm = nrm / nrm.norm(dim=2, keepdim=True) * _vertex_areas(x, n)[..., None]
        s = _Stencil(x.view(-1, 3)).gather(sigma.view(-1, 8).double()).view(c, n, 8)
        full = torch.stack([s[..., 0], s[..., 3], s[..., 4], s[..., 3], s[..., 1], s[..., 5], s[..., 4], s[..., 5], s[..., 2]],
                           -1).view(c, n, 3, 3)
        out.append((full @ nrm[..., None])[..., 0])
    return out


def _exact_planes(case, xs):
    """The tangent plane at the nearest vertex of another cell, per vertex, by brute force."""
    cell, pos, nrm, org, at = [], [], [], [], 0
    for x, (n, c) in zip(xs, _groups(case)):
        a = _area_normals(x, n)
        pos.append(x.view(-1, 3))
        nrm.append((a / a.norm(dim=2, keepdim=True)).view(-1, 3))
        org.append(x[:, :1].expand_as(x).reshape(-1, 3))
        cell.append(torch.arange(at, at + c, device="cuda").repeat_interleave(n))
        at += c
    cell, pos, nrm, org = (torch.cat(v) for v in (cell, pos, nrm, org))
    planes = torch.zeros(len(pos), 4, device="cuda", dtype=torch.float64)
    some = max(1, int(4e8) // len(pos))
    for a in range(0, len(pos), some):
        s = slice(a, a + some)
        d2 = sum((pos[s, None, k] - pos[None, :, k]) ** 2 for k in range(3))
        d2.masked_fill_(cell[s, None] == cell[None, :], math.inf)
        best, j = d2.min(1)
        hit = best <= CUTOFF ** 2
        off = (nrm[j] * (pos[j] - org[s])).sum(1, keepdim=True)
        planes[s] = torch.where(hit[:, None], torch.cat([nrm[j], off], 1), torch.zeros_like(planes[s]))
    return planes


def _exact_fit(case, seed):
    params, feat, target, idx = _fit_inputs(case, seed)
    p = params.double()
    sizes, at, part = [(64, 9), (64,), (64, 64), (64,), (3, 64), (3,), (9,), (9,), (3,)], 0, []
    for shape in sizes:
        k = math.prod(shape)
        part.append(p[at:at + k].view(shape))
        at += k
    low = lambda v: v.to(torch.bfloat16).double()
    w1, b1, w2, b2, w3, b3, mu, sd, so = part
    w1, w2, w3 = low(w1), low(w2), low(w3)
    z = low((feat[idx.long()].double() - mu) / sd)
    h1 = torch.tanh(z @ w1.T + b1)
    h1r = low(h1)
    h2 = torch.tanh(h1r @ w2.T + b2)
    r = h2 @ w3.T + b3 - target[idx.long()].double() / so
    n = case["batch"]
    do = 2 * r / n
    d2 = (do @ w3) * (1 - h2 * h2)
    d1 = (d2 @ w2) * (1 - h1 * h1)
    grads = [d1.T @ z, d1.sum(0), d2.T @ h1r, d2.sum(0), do.T @ h2, do.sum(0)]
    g = torch.cat([q.reshape(-1) for q in grads] + [torch.zeros(21, device="cuda", dtype=torch.float64)])
    m, v = 0.1 * g, 1e-3 * g * g
    new = p - 1e-3 * (m / 0.1) / (torch.sqrt(v / 1e-3) + 1e-8)
    return [(r * r).sum().reshape(1) / n, g, new, m, v]


def exact(case, seed):
    if case["kind"] == "fit":
        return _exact_fit(case, seed)
    s = _inputs(case, seed)
    groups = _groups(case)
    xs, vs, fs = (_split(case, s[k]) for k in ("x0", "v0", "f"))
    if case["kind"] == "forcing":
        stencils = [_Stencil(x.view(-1, 3)) for x in xs]
        area = [_vertex_areas(x, n).view(-1, 1) for x, (n, _) in zip(xs, groups)]
        u = s["u_lattice"].view(-1, 4)[:, :3].double()
        spread = lambda fv: sum(t.spread(f * a) for t, f, a in zip(stencils, fv, area)) / LATTICE_DX ** 2
        fv = [(v.view(-1, 3) - t.gather(u)) / DT for t, v in zip(stencils, vs)]
        for _ in range(case["cycles"]):
            ul = u + DT * spread(fv)
            fv = [f + (v.view(-1, 3) - t.gather(ul)) / DT for t, f, v in zip(stencils, fv, vs)]
        body = spread(fv).view(LATTICE_N, LATTICE_N, LATTICE_N, 3)
        body = torch.cat([body, torch.zeros_like(body[..., :1])], -1)
        return [_soa([f.view(c, n, 3) for f, (n, c) in zip(fv, groups)], torch.float64), body]
    # the dense FP64 work of a step grows with the vertices of a mesh
    if case["steps"] * sum(n * c * (1 + n / 300) for n, c in groups) > 4e7 or max(n for n, _ in groups) > 2562:
        return None
    solids = [_Membrane(n) for n, _ in groups]
    planes = None
    for k in range(case["steps"]):
        if case["kind"] == "coupled":
            fs = _exact_forces(case, xs, s["sigma"])
            fs = [f + e for f, e in zip(fs, _split(case, s["noise"][k]))]
        per = [None] * len(groups)
        if case["kind"] == "dense":
            planes = _exact_planes(case, xs)
            at = np.cumsum([0] + [n * c for n, c in groups])
            per = [planes[at[g]:at[g + 1]].view(c, n, 4) for g, (n, c) in enumerate(groups)]
        new = [m.step(x, v, f, q) for m, x, v, f, q in zip(solids, xs, vs, fs, per)]
        xs, vs = [a for a, _ in new], [b for _, b in new]
    out = [_soa(xs, torch.float64), _soa(vs, torch.float64)]
    if case["kind"] == "coupled":
        out.append(_soa(fs, torch.float64))
    return out + [planes, None] if case["kind"] == "dense" else out
