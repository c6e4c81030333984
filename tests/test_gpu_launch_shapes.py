"""The launch shapes of a step by mesh size and number of cells: clusters of blocks per
cell for few cells, one 512-thread block per SM, two of 256 and four of 128 threads for
small meshes, each with the sparse solve at sizes around its tree's leaves.  The vector
paths of the spreading and of the network's gradient at their edges.

Tolerances: FP64 runs a fixed number of iterations, so it differs from the FP64 oracle by
rounding order only (1e-10 mean edge lengths, as the other fixed-iteration tests); FP32
converges to 1e-6 (one step within 1e-5 mean edge lengths and the rounding of storing x).
"""
import numpy as np
import pytest

from helpers import DT, fp32_store_allowance, gpu_step_device, max_rel_disp, oracle_model, oracle_steps, population32
from oracle import oracle as O
from paper_1903_06479_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def N():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1903_06479_gb300 import npfem
    npfem.lib()
    return npfem


# 18: one leaf holds the mesh; 42: two leaves; 38 SMs' worth of cells and more per size
@pytest.mark.parametrize("n,cells", [(18, 1), (18, 320), (42, 3), (66, 20), (66, 160), (162, 1), (162, 70), (258, 1)])
def test_fp64_fixed_iterations(N, n, cells):
    m, rest, tris = oracle_model(n)
    h = N.Handle(rest, tris, N.material(), N.default_opts(precision="fp64", tol=0.0, max_iter=5, armijo_noise=0.0,
                                                          warm_history=0), dt=DT)
    p = population32(n, cells, seed=300 + n, forces="shear", noise_pN=0.5, box=20.0)
    pick = sorted({0, cells // 2, cells - 1})
    xo, vo, _ = oracle_steps(m, p["x"][pick], p["v"][pick], p["f"][pick], tol=0.0, max_iter=5)
    xg, vg, _ = gpu_step_device(h, p["x"], p["v"], p["f"], dtype="float64")
    assert max_rel_disp(xg[pick], xo, m.lbar) <= 1e-10
    assert max_rel_disp(DT * vg[pick], DT * vo, m.lbar) <= 1e-10


@pytest.mark.parametrize("n,cells", [(18, 2), (66, 1), (66, 400), (162, 19), (258, 38), (258, 320), (642, 1), (642, 76),
                                     (642, 160), (1026, 2), (1026, 37), (1026, 160)])
def test_fp32_converged_step(N, n, cells):
    m, rest, tris = oracle_model(n)
    h = N.Handle(rest, tris, N.material(), N.default_opts(precision="fp32", tol=1e-6), dt=DT)
    p = population32(n, cells, seed=400 + n, forces="shear", noise_pN=0.5, box=20.0)
    pick = sorted({0, cells - 1})
    xo, _, _ = oracle_steps(m, p["x"][pick], p["v"][pick], p["f"][pick], steps=2, tol=1e-10, max_iter=200)
    xg, _, st = gpu_step_device(h, p["x"], p["v"], p["f"], steps=2)  # the second with carried pairs
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()
    assert max_rel_disp(xg[pick], xo, m.lbar) <= 2e-5 + fp32_store_allowance(p["x"], m.lbar)


def test_few_cells_of_several_meshes(N):
    """A cluster per cell over three meshes in one call, statistics included."""
    sizes, cells = (66, 258, 642), (3, 2, 4)
    import torch
    hs, pops, ms = [], [], []
    for n, c in zip(sizes, cells):
        m, rest, tris = oracle_model(n)
        hs.append(N.Handle(rest, tris, N.material(), N.default_opts(precision="fp64", tol=1e-9), dt=DT))
        pops.append(population32(n, c, seed=500 + n, forces="shear", noise_pN=0.5, box=20.0))
        ms.append(m)
    cat = lambda k: torch.tensor(np.concatenate([W.to_soa(p[k]).ravel() for p in pops]), device="cuda")
    x, v, f = cat("x"), cat("v"), cat("f")
    st = torch.zeros((sum(cells), 32), dtype=torch.uint8, device="cuda")
    N.step(hs, cells, x, v, f, DT, stats=st)
    torch.cuda.synchronize()
    st = st.cpu().numpy().view(N.CELL_STATS_DTYPE).reshape(-1)
    assert (st["status"] == 0).all()
    at = ct = 0
    for m, p, n, c in zip(ms, pops, sizes, cells):
        xo, _, so = oracle_steps(m, p["x"], p["v"], p["f"], tol=1e-9, max_iter=50)
        xg = W.from_soa(x[at:at + 3 * n * c].cpu().numpy().reshape(c, 3, n))
        assert max_rel_disp(xg, xo, m.lbar) <= 1e-8
        assert [int(k) for k in st["iterations"][ct:ct + c]] == [s.iterations for s in so]
        at += 3 * n * c
        ct += c


@pytest.mark.parametrize("samples,offset", [(1, 0), (63, 0), (64, 1), (65, 0), (20001, 0)])
def test_network_gradient_edges(N, samples, offset):
    """Partial and full tiles, several tiles per block, a gradient buffer that is not 16-byte
    aligned; the tolerance of the gradient's parity test."""
    import torch
    rng = np.random.default_rng(600 + samples)
    from paper_1903_06479_gb300 import learn
    P = learn.init_params(3)
    P[-12:-3] = 1.0 + 0.1 * rng.random(9)
    feat = rng.normal(0, 1, (samples, 9)).astype(np.float32)
    tgt = rng.normal(0, 1, (samples, 3)).astype(np.float32)
    dev = lambda a: torch.tensor(a, device="cuda")
    buf = torch.full((N.mlp_nparam() + 4,), 7.0, device="cuda")
    grad = buf[offset:offset + N.mlp_nparam()]
    loss = torch.full((1,), 7.0, device="cuda")
    N.mlp_loss_grad(dev(P), dev(feat), dev(tgt), None, samples, grad, loss)
    lo, go = O.mlp_loss_grad(P.astype(np.float64), feat.astype(np.float64), tgt.astype(np.float64), True)
    assert abs(float(loss.item()) - lo) <= 1e-5 * lo
    assert np.abs(grad.cpu().numpy() - go).max() <= 1e-4 * np.abs(go).max()
    assert (buf[offset + N.mlp_nparam():] == 7.0).all()


@pytest.mark.parametrize("offset", [0, 1])
def test_spread_alignment(N, offset):
    """The spread force with 16-byte reductions and, for a lattice that is not 16-byte
    aligned, scalar ones: the same sums in another order (1e-5 of the largest value)."""
    import torch
    rest, tris = W.discocyte(162)
    h = N.Handle(rest, tris, N.material(), N.default_opts(), dt=DT)
    p = population32(162, 5, seed=700, forces="noise", box=10.0)
    x = torch.tensor(W.to_soa(p["x"]), dtype=torch.float32, device="cuda")
    v = torch.randn_like(x)
    side = 45
    lat = N.lattice((-6.0, -6.0, -6.0), 0.5, (side,) * 3)
    u = torch.randn(side ** 3 * 4, device="cuda")
    ref = None
    for off in (0, offset):
        buf = torch.zeros(side ** 3 * 4 + 4, device="cuda")
        fl, fv = buf[off:off + side ** 3 * 4], torch.zeros_like(x)
        N.ibm_forcing([h], [5], x, v, lat, u, DT, 0, fv, fl)
        torch.cuda.synchronize()
        got = fl.double().cpu().numpy()
        ref = got if ref is None else ref
        assert np.abs(ref).max() > 0 and np.abs(got - ref).max() <= 1e-5 * np.abs(ref).max()
        assert (buf[off + side ** 3 * 4:] == 0).all()


@pytest.mark.parametrize("dx", [1.0, 0.3])
def test_forcing_cell_by_cell(N, dx):
    """130 cells in one call (a block per cell, the box of lattice nodes in shared memory; at
    dx 0.3 the boxes do not fit and the blocks fall back) against two calls of 65 (vertex by
    vertex): interpolation, slip and spread agree to the order of the sums (1e-5 of the
    largest value).  Some cells lie partly outside the lattice."""
    import torch
    rest, tris = W.discocyte(258)
    h = N.Handle(rest, tris, N.material(), N.default_opts(), dt=DT)
    cells, half = 130, 65
    p = population32(258, cells, seed=701, forces="noise", box=20.0)
    x = torch.tensor(W.to_soa(p["x"]), dtype=torch.float32, device="cuda")
    v = torch.randn_like(x)
    side = int(20.0 / dx)
    lat = N.lattice((0.0, 0.0, 0.0), dx, (side, side + 1, side + 2))
    nodes = side * (side + 1) * (side + 2)
    u = torch.randn(nodes * 4, device="cuda")
    close = lambda a, b: float((a.double() - b.double()).abs().max()) <= 1e-5 * float(b.double().abs().max())
    whole, parts = torch.zeros_like(x), torch.zeros_like(x)
    N.ibm_interpolate([h], [cells], x, lat, u, whole)
    for a in (0, half):
        N.ibm_interpolate([h], [half], x[a:a + half], lat, u, parts[a:a + half])
    assert float(parts.abs().max()) > 0 and close(whole, parts)
    fl, fv = torch.zeros(nodes * 4, device="cuda"), torch.zeros_like(x)
    N.ibm_forcing([h], [cells], x, v, lat, u, DT, 0, fv, fl)
    sums = torch.zeros_like(fl)
    for a in (0, half):
        one, fp = torch.zeros_like(fl), torch.zeros_like(x[a:a + half])
        N.ibm_forcing([h], [half], x[a:a + half], v[a:a + half], lat, u, DT, 0, fp, one)
        assert close(fv[a:a + half], fp)
        sums += one
    torch.cuda.synchronize()
    assert float(sums.abs().max()) > 0 and close(fl, sums)
    # a cycle of the iteration reads the spread force back
    N.ibm_forcing([h], [cells], x, v, lat, u, DT, 1, fv, fl)
    torch.cuda.synchronize()
    assert bool(torch.isfinite(fv).all()) and bool(torch.isfinite(fl).all())


def test_groups_of_several_block_sizes_share_options_and_planes(N):
    """A call whose groups run in separate launches (by block size): every group takes the
    options and the collision planes of the call's first handle, as in one launch."""
    import torch
    sizes, cells = (258, 1026), (310, 160)
    hs, pops = [], []
    for k, (n, c) in enumerate(zip(sizes, cells)):
        rest, tris = W.discocyte(n)
        # the second handle's own tolerance would stop it at the first iterate
        hs.append(N.Handle(rest, tris, N.material(), N.default_opts(precision="fp32", tol=1e-6 if k == 0 else 1e3,
                                                                    lbfgs_m=5 if k == 0 else 2), dt=DT))
        pops.append(population32(n, c, seed=800 + n, forces="shear", noise_pN=0.5, box=40.0))
    cat = lambda k: torch.tensor(np.concatenate([W.to_soa(p[k]).ravel() for p in pops]), dtype=torch.float32, device="cuda")
    x, v, f = cat("x"), cat("v"), cat("f")
    verts = sum(n * c for n, c in zip(sizes, cells))
    planes = torch.zeros((verts, 4), device="cuda")
    first = sizes[0] * cells[0]
    # the second group's last cell: every vertex 0.01 um behind a plane normal to x
    xl = W.to_soa(pops[1]["x"])[-1]
    planes[verts - sizes[1]:, 0] = 1.0
    planes[verts - sizes[1]:, 3] = torch.tensor(xl[0] - xl[0, 0] + 0.01, dtype=torch.float32, device="cuda")
    hs[0].set_collisions(planes, 2000.0)
    st = torch.zeros((sum(cells), 32), dtype=torch.uint8, device="cuda")
    for _ in range(2):
        N.step(hs, cells, x, v, f, DT, stats=st)
    torch.cuda.synchronize()
    st = st.cpu().numpy().view(N.CELL_STATS_DTYPE).reshape(-1)
    assert (st["status"] == 0).all() and (st["residual"] <= 1e-6).all()
    vx = v[3 * first:].view(cells[1], 3, sizes[1])[:, 0].mean(1).cpu().numpy()
    # the push is w_col d h / m per step on every vertex, far above the noise's mean velocity
    push = 2000.0 * 0.01 * DT / (94e3 / sizes[1])
    assert vx[-1] > 0.5 * push and np.abs(vx[:-1]).max() < 0.2 * push
