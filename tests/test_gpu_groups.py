"""What the groups of one call share: the collision planes of the first handle, whichever
kernel solves a group, and the carried pairs of handles that differ in their L-BFGS window."""
import numpy as np
import pytest

from helpers import DT, fp32_store_allowance, gpu_step_device, max_rel_disp, oracle_steps, population32
from paper_1903_06479_gb300 import workloads as W

pytestmark = pytest.mark.gpu
WCOL = 2000.0


@pytest.fixture(scope="module")
def N():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_06479_gb300 import npfem
    npfem.lib()
    return npfem


def octahedral_discocyte(f):
    """The discocyte on an octahedron's faces cut into f x f triangles: 4 f^2 + 2 vertices."""
    index, points, tris = {}, [], []

    def at(i, j, s):
        key = (i * s[0], j * s[1], (f - i - j) * s[2])
        if key not in index:
            index[key] = len(points)
            points.append(key)
        return index[key]

    for s in np.array(np.meshgrid([1, -1], [1, -1], [1, -1])).reshape(3, -1).T:
        for i in range(f):
            for j in range(f - i):
                tris.append((at(i, j, s), at(i + 1, j, s), at(i, j + 1, s)))
                if i + j < f - 1:
                    tris.append((at(i + 1, j, s), at(i + 1, j + 1, s), at(i, j + 1, s)))
    p, t = np.asarray(points, dtype=np.float64), np.asarray(tris, dtype=np.int32)
    p /= np.linalg.norm(p, axis=1, keepdims=True)
    flip = (np.cross(p[t[:, 1]] - p[t[:, 0]], p[t[:, 2]] - p[t[:, 0]]) * p[t].sum(1)).sum(1) < 0
    t[flip] = t[flip][:, [0, 2, 1]]
    d = W.DISCOCYTE_D
    xy = 0.5 * d * p[:, :2]
    r2 = (xy ** 2).sum(1) / d ** 2
    z = d * np.sqrt(np.clip(1.0 - 4.0 * r2, 0.0, None)) * (W.ES_A0 + W.ES_A1 * r2 + W.ES_A2 * r2 ** 2)
    return np.column_stack([xy, np.sign(p[:, 2]) * z]), t


def _call(N, sizes, cells, precision, seed=900, **opts):
    """Handles and the concatenated state of a call's groups."""
    import torch
    hs, pops = [], []
    for k, (n, c) in enumerate(zip(sizes, cells)):
        rest, tris = W.discocyte(n)
        kw = {q: v[k] if isinstance(v, (list, tuple)) else v for q, v in opts.items()}
        hs.append(N.Handle(rest, tris, N.material(), N.default_opts(precision=precision, tol=1e-6, **kw), dt=DT))
        pops.append(population32(n, max(c, 1), seed=seed + n, forces="shear", noise_pN=0.5, box=40.0))
    cat = lambda k: torch.tensor(np.concatenate([W.to_soa(p[k])[:c].ravel() for p, c in zip(pops, cells)]),
                                 dtype=torch.float32, device="cuda")
    return hs, pops, [cat(k) for k in "xvf"]


# the pressed group: SIMT beside clusters; SIMT and clusters behind a first group without cells; a
# second cluster group
@pytest.mark.parametrize("precision,sizes,cells", [("bf16", (642, 2562), (3, 4)), ("fp32", (258, 642), (0, 4)),
                                                   ("bf16", (258, 642), (0, 4)), ("bf16", (642, 258), (3, 5)),
                                                   ("fp64", (258, 642), (0, 4))])
def test_planes_of_the_first_handle_press_every_group(N, precision, sizes, cells):
    """Planes installed on the first handle press the last group's last cell after three steps
    without them (so that BF16 cells pass through the first-iterate pass): its mean velocity
    gains about w d h / m, the other cells' none."""
    import torch
    hs, pops, (x, v, f) = _call(N, sizes, cells, precision)
    if precision == "fp64":
        x, v, f = x.double(), v.double(), f.double()
    f.zero_()
    for _ in range(3):
        N.step(hs, cells, x, v, f, DT)
    n, verts = sizes[-1], sum(a * b for a, b in zip(sizes, cells))
    mean = lambda: v.view(-1)[-3 * n * cells[-1]:].view(cells[-1], 3, n)[:, 0].mean(1).double().cpu().numpy()
    before = mean()
    planes = torch.zeros((verts, 4), device="cuda")
    xl = x[-3 * n:].view(3, n)[0]
    planes[-n:, 0] = 1.0
    planes[-n:, 3] = (xl - xl[0] + 0.01).float()
    hs[0].set_collisions(planes, WCOL)
    N.step(hs, cells, x, v, f, DT)
    torch.cuda.synchronize()
    gain = mean() - before
    push = WCOL * 0.01 * DT / (94e3 / n)
    assert gain[-1] > 0.5 * push and np.abs(gain[:-1]).max() < 0.2 * push


@pytest.mark.parametrize("precision,sizes,windows", [("bf16", (162, 258), (2, 8)), ("bf16", (258, 1026), (1, 8)),
                                                     ("fp32", (162, 258), (8, 2)), ("fp64", (66, 162), (2, 8))])
def test_groups_with_different_windows(N, precision, sizes, windows):
    """Each group of a call, stepped with carried pairs, agrees with the group stepped alone (every
    cell converges to 1e-6 in both)."""
    import torch
    cells = (5, 6)
    hs, pops, (x, v, f) = _call(N, sizes, cells, precision, lbfgs_m=windows)
    td = torch.float64 if precision == "fp64" else torch.float32
    x, v, f = x.to(td), v.to(td), f.to(td)
    x0, v0 = x.clone(), v.clone()
    st = torch.zeros((sum(cells), 32), dtype=torch.uint8, device="cuda")
    for _ in range(4):
        N.step(hs, cells, x, v, f, DT, stats=st)
    torch.cuda.synchronize()
    st = st.cpu().numpy().view(N.CELL_STATS_DTYPE).reshape(-1)
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()
    at = 0
    for h, n, c in zip(hs, sizes, cells):
        part = slice(at, at + 3 * n * c)
        xa, va = x0[part].clone(), v0[part].clone()
        rest, tris = W.discocyte(n)
        alone = N.Handle(rest, tris, N.material(), h.opts, dt=DT)
        for _ in range(4):
            N.step([alone], [c], xa, va, f[part], DT)
        torch.cuda.synchronize()
        lb = alone.rest_info()[1]["lbar"]
        X = lambda t: W.from_soa(t.double().cpu().numpy().reshape(c, 3, n))
        assert max_rel_disp(X(x[part]), X(xa), lb) <= 4e-5
        at += 3 * n * c


@pytest.mark.parametrize("windows", [(5, 2), (2, 5)])
def test_cluster_groups_of_different_shared_memory(N, windows):
    """Two groups of one cluster kernel whose launches need different amounts of shared memory, step
    after step."""
    import torch
    cells = (4, 5)
    hs, pops, (x, v, f) = _call(N, (642, 642), cells, "bf16", lbfgs_m=windows)
    st = torch.zeros((sum(cells), 32), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        N.step(hs, cells, x, v, f, DT, stats=st)
    torch.cuda.synchronize()
    assert all(h.tuning()["tensor_core"] for h in hs)
    st = st.cpu().numpy().view(N.CELL_STATS_DTYPE).reshape(-1)
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()


# alone and beside finer or damped meshes; few cells (one launch for all) and more than one per SM
@pytest.mark.parametrize("sizes,cells,damped", [((642, 1026), (20, 10), None), ((258, 1026), (20, 3), None),
                                                ((642, 1026), (160, 160), None), ((642, 258), (20, 10), 1),
                                                ((162, 1026), (5, 3), 0), ((1026, 642), (9, 30), None)])
def test_first_group_does_not_depend_on_its_companions(N, sizes, cells, damped):
    """What a cell's mesh applies (dense inverse or sparse factor) is a matter of the mesh: the first
    group's cells come out bit for bit as in a call of their own where both calls run them in
    blocks of one size, and to the rounding of the reductions otherwise."""
    import torch
    mats = [N.material(beta_D=0.3) if damped == k else N.material() for k in range(2)]
    hs, pops, (x, v, f) = _call(N, sizes, cells, "fp32")
    make = lambda k: N.Handle(*W.discocyte(sizes[k]), mats[k], N.default_opts(precision="fp32", tol=1e-6), dt=DT)
    x0, v0, f0 = (t[:3 * sizes[0] * cells[0]].clone() for t in (x, v, f))
    hs = [make(0), make(1)]
    alone = make(0)
    st = torch.zeros((sum(cells), 32), dtype=torch.uint8, device="cuda")
    for _ in range(3):
        N.step(hs, cells, x, v, f, DT, stats=st)
        N.step([alone], cells[:1], x0, v0, f0, DT)
    torch.cuda.synchronize()
    st = st.cpu().numpy().view(N.CELL_STATS_DTYPE).reshape(-1)
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()
    xa, va = x[:x0.numel()], v[:x0.numel()]
    if sum(cells) <= 152:
        assert torch.equal(xa, x0) and torch.equal(va, v0)
    else:
        lb = alone.rest_info()[1]["lbar"]
        X = lambda t: W.from_soa(t.double().cpu().numpy().reshape(cells[0], 3, sizes[0]))
        assert max_rel_disp(X(xa), X(x0), lb) <= 3e-5


@pytest.mark.parametrize("n,cells", [(642, 3), (1026, 9), (258, 320)])
def test_tf32_handles_are_fp32_handles(N, n, cells):
    """TF32 handles run the FP32 path: the same bits (but in launches of at most eight cells of 701 to
    1100 vertices, where FP32 handles keep the dense inverse)."""
    import torch
    out = []
    for precision in ("fp32", "tf32"):
        hs, _, (x, v, f) = _call(N, (n,), (cells,), precision, refine=int(precision == "tf32"))
        for _ in range(2):
            N.step(hs, (cells,), x, v, f, DT)
        N.step_static(hs, (cells,), x, v, f, DT)
        torch.cuda.synchronize()
        out.append((x, v))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])


# 786 vertices: the finest cluster kernel; with damping its first guess solves with M~'s factor
@pytest.mark.parametrize("precision,refine,cells", [("bf16", 0, 1), ("bf16", 1, 9), ("bf16", 0, 160), ("fp32", 0, 3)])
def test_damped_cells_between_the_dense_and_the_cluster_limit(N, precision, refine, cells):
    """Damped cells (beta_D > 0) of 786 vertices against the FP64 oracle after two steps."""
    import torch
    from oracle import oracle as O
    rest, tris = octahedral_discocyte(14)
    assert len(rest) == 786
    m = O.Model(rest, tris, W.material_vector(beta_D=0.01), DT)
    rng = np.random.default_rng(960)
    x = (rest[None] + 20.0 * rng.random((cells, 1, 3))).astype(np.float32).astype(np.float64)
    v = (0.01 * rng.standard_normal(x.shape)).astype(np.float32).astype(np.float64)
    f = (0.5 * rng.standard_normal(x.shape)).astype(np.float32).astype(np.float64)
    h = N.Handle(rest, tris, N.material(beta_D=0.01), N.default_opts(precision=precision, tol=1e-6, refine=refine), dt=DT)
    assert h.tuning()["tensor_core"] == (precision == "bf16")
    xg, vg, st = gpu_step_device(h, x, v, f, steps=2)
    h.check_device()
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()
    pick = sorted({0, cells - 1})
    xo, vo, _ = oracle_steps(m, x[pick], v[pick], f[pick], steps=2, tol=1e-10, max_iter=200)
    assert max_rel_disp(xg[pick], xo, m.lbar) <= 2e-5 + fp32_store_allowance(x, m.lbar)


@pytest.mark.parametrize("n", [258, 642])
def test_idle_sms_are_filled(N, n):
    """Clusters of three or six blocks leave SMs of a 152-SM GPU idle; with fill_idle_sms a step of
    more cells than cluster blocks launches the SIMT kernel on them, small meshes included."""
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("needs 152 SMs")
    launches = []
    for fill in (0, 1):
        hs, _, (x, v, f) = _call(N, (n,), (300,), "bf16", warm_history=0, fill_idle_sms=fill)
        N.step(hs, (300,), x, v, f, DT)
        before = N.launch_count()
        N.step(hs, (300,), x, v, f, DT)
        launches.append(N.launch_count() - before)
    torch.cuda.synchronize()
    assert launches[1] == launches[0] + 1


def test_tf32_limit(N):
    """npfem_step refuses cells of a TF32 mesh above 4096 vertices, also in a group behind others;
    npfem_step_static and empty groups are not refused."""
    import torch
    (small, big), _, (x, v, f) = _call(N, (66, 4098), (2, 1), "tf32")
    x0 = x.clone()
    for hs, cells, at in (((small, big), (2, 1), 0), ((big,), (1,), 3 * 66 * 2)):
        with pytest.raises(N.NpfemError) as e:
            N.step(hs, cells, x[at:], v[at:], f[at:], DT)
        assert e.value.code == -1
    torch.cuda.synchronize()
    assert torch.equal(x, x0)
    N.step((small, big), (2, 0), x, v, f, DT)
    N.step_static((big,), (1,), x[396:], v[396:], f[396:], DT)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(x).all()) and not torch.equal(x[:396], x0[:396]) and not torch.equal(x[396:], x0[396:])


@pytest.mark.parametrize("precision,n,cells,want", [("fp32", 258, 400, 128), ("fp32", 642, 200, 256),
                                                    ("fp32", 642, 3, 512), ("fp64", 66, 200, 128)])
def test_tuning_reports_the_block_size(N, precision, n, cells, want):
    import torch
    (h,), _, (x, v, f) = _call(N, (n,), (cells,), precision)
    if precision == "fp64":
        x, v, f = x.double(), v.double(), f.double()
    assert h.tuning()["simt_threads"] == 512
    N.step([h], [cells], x, v, f, DT)
    assert h.tuning()["simt_threads"] == want
    shape = N.autotune([h], [cells], x, v, f, DT, trial_steps=1)[0]
    assert shape["simt_threads"] == want and set(shape["trial_ms"]) == {"simt512"}


@pytest.mark.parametrize("sizes,cells", [((66,), (1,)), ((66,), (700,)), ((162,), (320,)), ((162,), (9,)), ((66, 162), (140, 20)),
                                         ((66, 258), (3, 2))])
def test_static_step_of_small_fp64_meshes(N, sizes, cells):
    """npfem_step_static in 128-thread blocks (66 vertices; 162 with more than a cell per SM) and in
    512: a fixed number of iterations differs from npfem_step by rounding only."""
    import torch
    hs, _, (x, v, f) = _call(N, sizes, cells, "fp64", warm_history=0, max_iter=4, armijo_noise=0.0)
    for h in hs:
        h.close()
    hs = [N.Handle(*W.discocyte(n), N.material(), N.default_opts(precision="fp64", tol=0.0, max_iter=4, warm_history=0,
                                                               armijo_noise=0.0), dt=DT) for n in sizes]
    x, v, f = x.double(), v.double(), f.double()
    xs, vs = x.clone(), v.clone()
    for _ in range(2):
        N.step(hs, cells, x, v, f, DT)
        N.step_static(hs, cells, xs, vs, f, DT)
    torch.cuda.synchronize()
    lb = min(h.rest_info()[1]["lbar"] for h in hs)
    assert float((x - xs).abs().max()) <= 1e-10 * lb and float((v - vs).abs().max()) * DT <= 1e-10 * lb


def test_stretched_equilibria_of_the_dense_inverse_and_the_factor(N):
    """A 1026-vertex cell stretched to 200 pN: an FP32 handle alone (dense inverse) and a TF32 handle
    (the same FP32 path with the sparse factor) reach the same equilibrium, by the tolerance of the
    equilibria against the oracle (2e-3 of the diameters)."""
    from paper_1903_06479_gb300 import validation as V
    forces = (100.0, 200.0)
    r = {p: V.stretching(sizes=(1026,), forces_pN=forces, precision=p)[1026] for p in ("fp32", "tf32")}
    for p in r:
        assert max(r[p]["move"]) < 1e-4, (p, r[p]["move"])  # settled
    for k in ("DA", "DT"):
        a, b = np.array(r["fp32"][k]), np.array(r["tf32"][k])
        assert (np.abs(a - b) <= 2e-3 * a).all(), (k, a, b)
